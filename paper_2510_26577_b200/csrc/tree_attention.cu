// cast_tree_attention: tree-masked verification attention.
//
// CUDA-core path (fp32 inputs, and bf16 caches the tensor-core path does not take: pages other than 8, 16, 32 and 64
// positions, pointers not aligned for it): a flash-style kernel. One CTA owns (sequence, kv-head, block of 32 query rows, KV split); a
// query row is a (tree token, head of the GQA group) pair, so a K/V tile fetched once serves
// all tree tokens and all heads of the group. Tiles of 64 positions are converted to fp32 in
// shared memory; S = QK^T and O += PV are register-tiled FFMA loops; the softmax is online.
// Prefix positions need no mask; a tree position L+j is visible to row (t, g) iff bit j of
// anc_mask[t] is set. KV splits write (max, sum, unnormalised O) partials; the CTA of a row block
// that finishes last (an atomic ticket, nothing spins) merges them, or a second kernel when they are many.
// Bound by instruction issue, shared-memory reads of the products first: both go by 16-byte vectors, the first product by
// packed multiply-adds (60 tokens, 4 sequences of 2048, 32/8 heads of 64: 233 us, 276 without the packing; 128 dims 450 and
// 511). A 64-row tile of 8 x 4 per thread is as fast from 200 rows per kv-head on and up to twice as slow below.
#include <math.h>

#include "cast_internal.h"

using namespace cast;

namespace cast {
// implemented in tree_attention_tc.cu; returns false when the shape is not taken there
bool tree_attention_tc_launch(cast_ctx* c, const void* q, const void* k, const void* v, int B, int Hq, int Hkv, int D,
                              int page_size, const int32_t* page_table, int seq_capacity, int num_pages,
                              const int32_t* kv_len, const uint32_t* anc, const int32_t* n_tree, const int32_t* first_row,
                              float scale, void* out, cudaStream_t stream, cast_status* status);
bool tree_attention_tc_takes(const cast_ctx* c, int B, int Hq, int Hkv, int D, int page_size, int seq_capacity);
size_t tree_attention_tc_workspace(const cast_ctx* c, int B, int Hq, int Hkv, int D, int page_size, int seq_capacity);
cast_status tree_attention_tc_reserve(cast_ctx* c, size_t bytes);
}

namespace {

constexpr int kRB = 32;   // query rows per CTA
constexpr int kPT = 64;   // positions per tile
constexpr int kThreads = 256;
constexpr int kMaxSplit = 64;
constexpr int kMergeHere = 16;  // up to this many splits the last CTA merges (a second launch costs 4 us)
// A ticket per row block of a split launch, of which there are at most kOwn / 2 per SM: room for 4096 SMs.
constexpr size_t kCcTicketBytes = (size_t)32768 * sizeof(int32_t);

struct AttnParams {
  const void* q;
  const void* k;
  const void* v;
  void* out;
  int B, Ncap, Nmax, Hq, Hkv, G, page_size, seq_capacity, num_pages, words, nsplit, nrowblk;  // Nmax: most tokens of a tree
  const int32_t* page_table;
  const int32_t* kv_len;
  const int32_t* n_tree;
  const int32_t* first_row;  // [B] or null: output rows start at this tree token
  const uint32_t* anc;
  float scale;
  int32_t* ticket;  // [B][Hkv][nrowblk] splits finished
  float* part_o;    // [B][Hkv][nrowblk][nsplit][kRB][D]
  float* part_ml;   // [B][Hkv][nrowblk][nsplit][kRB][2]
  DevState* st;
};

template <typename T> __device__ __forceinline__ void load_chunk(const T* p, float* out);
template <> __device__ __forceinline__ void load_chunk<float>(const float* p, float* out) {
  const float4 a = *reinterpret_cast<const float4*>(p);
  out[0] = a.x; out[1] = a.y; out[2] = a.z; out[3] = a.w;
}
template <> __device__ __forceinline__ void load_chunk<__nv_bfloat16>(const __nv_bfloat16* p, float* out) {
  const uint4 a = *reinterpret_cast<const uint4*>(p);
  const uint32_t w[4] = {a.x, a.y, a.z, a.w};
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    out[2 * i] = __uint_as_float(w[i] << 16);
    out[2 * i + 1] = __uint_as_float(w[i] & 0xffff0000u);
  }
}
__device__ __forceinline__ void store4(float* p, const float (&x)[4], float f) {
  *reinterpret_cast<float4*>(p) = make_float4(x[0] * f, x[1] * f, x[2] * f, x[3] * f);
}
__device__ __forceinline__ void store4(__nv_bfloat16* p, const float (&x)[4], float f) {
  const __nv_bfloat162 a = __floats2bfloat162_rn(x[0] * f, x[1] * f), b = __floats2bfloat162_rn(x[2] * f, x[3] * f);
  *reinterpret_cast<uint2*>(p) = make_uint2(*reinterpret_cast<const uint32_t*>(&a), *reinterpret_cast<const uint32_t*>(&b));
}

// Packed fp32 pairs: one instruction, two multiply-adds with IEEE results each.
typedef unsigned long long f32x2;
__device__ __forceinline__ f32x2 fma2(f32x2 a, f32x2 b, f32x2 c) {
  f32x2 r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
  return r;
}
__device__ __forceinline__ float sum2(f32x2 v) {
  float a, b;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(v));
  return a + b;
}

// Merge of a row block's splits: this warp's rows r0, r0 + step, ... (ROWS of them). The splits' weights H per lane, then the
// columns, four per lane (at D = 64 each half of the warp takes every other split). The rows advance together and their first
// loads go out ahead of the weights: row after row, each with two round trips to L2, four rows were 6 us of a launch of 14.
template <typename T, int D, int ROWS, int H>
__device__ __forceinline__ void merge_splits(const AttnParams& p, int b, int kvh, int rb, int F, int row0, int r0, int step,
                                             int rows_here) {
  static_assert(kMaxSplit <= 64 && kMergeHere <= 32, "H splits per lane");
  constexpr int C4 = D / 4, kHalves = 32 / C4, UN = ROWS > 1 ? 2 : 8;
  const int lane = threadIdx.x & 31, c = lane % C4 * 4, half = lane / C4;
  const size_t part0 = (((size_t)b * p.Hkv + kvh) * p.nrowblk + rb) * p.nsplit * kRB;
  const float2* ml = reinterpret_cast<const float2*>(p.part_ml) + part0;
  float2 x[ROWS][H];
  float4 v[ROWS][UN];
  auto load = [&](int s0) {
#pragma unroll
    for (int u = 0; u < ROWS; ++u)
#pragma unroll
      for (int k = 0; k < UN; ++k) {
        const int s = s0 + k * kHalves + half, r = r0 + u * step;
        v[u][k] = s < p.nsplit && r < rows_here
                      ? __ldcg(reinterpret_cast<const float4*>(p.part_o + (part0 + (size_t)s * kRB + r) * D + c))
                      : make_float4(0.f, 0.f, 0.f, 0.f);
      }
  };
#pragma unroll
  for (int u = 0; u < ROWS; ++u)
#pragma unroll
    for (int h = 0; h < H; ++h)
      x[u][h] = lane + 32 * h < p.nsplit && r0 + u * step < rows_here ? __ldcg(ml + (size_t)(lane + 32 * h) * kRB + r0 + u * step)
                                                                      : make_float2(-INFINITY, 0.f);
  load(0);
  float w[ROWS][H], l[ROWS], acc[ROWS][4];
#pragma unroll
  for (int u = 0; u < ROWS; ++u) {
    float M = x[u][0].x;
    if (H == 2) M = fmaxf(M, x[u][H - 1].x);
    l[u] = 0.f;
#pragma unroll
    for (int of = 16; of > 0; of >>= 1) M = fmaxf(M, __shfl_xor_sync(0xffffffffu, M, of));
#pragma unroll
    for (int h = 0; h < H; ++h) {
      w[u][h] = x[u][h].x > -INFINITY ? expf(x[u][h].x - M) : 0.f;
      l[u] += x[u][h].y * w[u][h];
    }
#pragma unroll
    for (int of = 16; of > 0; of >>= 1) l[u] += __shfl_xor_sync(0xffffffffu, l[u], of);
#pragma unroll
    for (int e = 0; e < 4; ++e) acc[u][e] = 0.f;
  }
#pragma unroll 1
  for (int s0 = 0;;) {
#pragma unroll
    for (int k = 0; k < UN; ++k) {
      const int s = s0 + k * kHalves + half;
#pragma unroll
      for (int u = 0; u < ROWS; ++u) {
        // (a split that saw nothing weighs 0, and its sums are 0)
        const float ws = __shfl_sync(0xffffffffu, H == 1 || s0 + k * kHalves < 32 ? w[u][0] : w[u][H - 1], s & 31);
        acc[u][0] += v[u][k].x * ws;
        acc[u][1] += v[u][k].y * ws;
        acc[u][2] += v[u][k].z * ws;
        acc[u][3] += v[u][k].w * ws;
      }
    }
    s0 += UN * kHalves;
    if (s0 >= p.nsplit) break;
    load(s0);
  }
#pragma unroll
  for (int u = 0; u < ROWS; ++u) {
    if (kHalves == 2) {
#pragma unroll
      for (int e = 0; e < 4; ++e) acc[u][e] += __shfl_xor_sync(0xffffffffu, acc[u][e], 16);
    }
    const int r = r0 + u * step, row = row0 + r, t = F + row / p.G;
    T* out = reinterpret_cast<T*>(p.out) + (((size_t)b * p.Ncap + t) * p.Hq + kvh * p.G + row % p.G) * D;
    if (half == 0 && r < rows_here) store4(out + c, acc[u], l[u] > 0.f ? 1.f / l[u] : 0.f);
  }
}

template <typename T, int D>
__global__ void __launch_bounds__(kThreads) tree_attn_cc_kernel(const AttnParams p) {
  constexpr int KS = D + 4;          // padded row stride of Qs / Ks (floats)
  constexpr int SS = kPT + 4;        // row stride of Ss: rows 16-byte aligned
  constexpr int CH = 16 / sizeof(T); // elements per 16-byte chunk
  constexpr int CPR = D / CH;        // chunks per cache row
  constexpr int DC = D / 32;         // output columns per lane
  extern __shared__ __align__(16) float smem[];
  float* Qs = smem;                       // [kRB][KS]
  float* Ks = Qs + kRB * KS;              // [kPT][KS]
  float* Vs = Ks + kPT * KS;              // [kPT][D]
  float* Ss = Vs + kPT * D;               // [kRB][SS]
  __shared__ float row_m[kRB], row_l[kRB], row_alpha[kRB];
  __shared__ uint32_t anc_s[kRB][CAST_MAX_TREE / 32];
  __shared__ long long slot_s[2][kPT];
  __shared__ int s_last;
  asm volatile("griddepcontrol.wait;" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");

  const int split = blockIdx.x % p.nsplit, rb = blockIdx.x / p.nsplit;
  const int kvh = blockIdx.y, b = blockIdx.z;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  int N = p.n_tree[b];
  if (N > p.Nmax) {  // row blocks are launched for Nmax tokens: the rows past it stay untouched, and the caller is told
    if (blockIdx.x == 0 && kvh == 0 && tid == 0) report(p.st, CAST_ERR_BAD_TREE, b);
    N = p.Nmax;
  }
  N = N < 0 ? 0 : N;
  int L = p.kv_len[b];
  if (L < 0) L = 0;
  const int G = p.G;
  int F = p.first_row != nullptr ? p.first_row[b] : 0;  // tokens before F are context only
  F = F < 0 ? 0 : (F > N ? N : F);
  const int rows_total = (N - F) * G;
  const int row0 = rb * kRB;
  if (row0 >= rows_total) return;
  const int max_pos = p.page_size == 0 ? p.seq_capacity : p.seq_capacity * p.page_size;
  int total = L + N;
  if (total > max_pos) {
    if (tid == 0) report(p.st, CAST_ERR_BAD_PAGE, b);
    total = max_pos;
  }
  const int ntiles = (total + kPT - 1) / kPT;
  const int t0 = (int)((long long)split * ntiles / p.nsplit), t1 = (int)((long long)(split + 1) * ntiles / p.nsplit);

  auto find_slots = [&](int tile) {  // cache slots of a tile's positions, a tile ahead of their use
    if (tid >= kPT) return;
    const int pos = tile * kPT + tid;
    long long slot = -1;
    if (tile < t1 && pos < total) {
      if (p.page_size == 0) {
        slot = (long long)b * p.seq_capacity + pos;
      } else {
        const int page = p.page_table[(size_t)b * p.seq_capacity + pos / p.page_size];
        if (page < 0 || page >= p.num_pages) report(p.st, CAST_ERR_BAD_PAGE, b);
        else slot = (long long)page * p.page_size + pos % p.page_size;
      }
    }
    slot_s[tile & 1][tid] = slot;
  };
  find_slots(t0);
  // query rows (pre-scaled), their ancestor masks, running softmax state
  const T* q = reinterpret_cast<const T*>(p.q);
  for (int i = tid; i < kRB * CPR; i += kThreads) {
    const int r = i / CPR, ch = i % CPR, row = row0 + r;
    float f[CH];
    if (row < rows_total) {
      const int t = F + row / G, g = row % G;
      load_chunk<T>(q + (((size_t)b * p.Ncap + t) * p.Hq + kvh * G + g) * D + ch * CH, f);
    } else {
#pragma unroll
      for (int e = 0; e < CH; ++e) f[e] = 0.f;
    }
#pragma unroll
    for (int e = 0; e < CH; ++e) Qs[r * KS + ch * CH + e] = f[e] * p.scale;
  }
  if (tid < kRB) {
    row_m[tid] = -INFINITY;
    row_l[tid] = 0.f;
    const int row = row0 + tid;
    for (int w = 0; w < CAST_MAX_TREE / 32; ++w)
      anc_s[tid][w] = (row < rows_total && w < p.words) ? p.anc[((size_t)b * p.Ncap + F + row / G) * p.words + w] : 0u;
  }
  float o[4][DC];
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int e = 0; e < DC; ++e) o[i][e] = 0.f;

  const T* kc = reinterpret_cast<const T*>(p.k);
  const T* vc = reinterpret_cast<const T*>(p.v);
  const int ty = tid / 16, tx = tid % 16;

  for (int tile = t0; tile < t1; ++tile) {
    const int pbase = tile * kPT;
    __syncthreads();  // previous tile fully consumed; the slots (and Qs, anc_s on the first pass) visible
#pragma unroll 4
    for (int i = tid; i < kPT * CPR; i += kThreads) {
      const int pl = i / CPR, ch = i % CPR;
      const long long slot = slot_s[tile & 1][pl];
      float fk[CH], fv[CH];
      if (slot >= 0) {
        const size_t off = ((size_t)slot * p.Hkv + kvh) * D + ch * CH;
        load_chunk<T>(kc + off, fk);
        load_chunk<T>(vc + off, fv);
      } else {
#pragma unroll
        for (int e = 0; e < CH; ++e) fk[e] = fv[e] = 0.f;
      }
#pragma unroll
      for (int e = 0; e < CH; e += 4) {
        *reinterpret_cast<float4*>(Ks + pl * KS + ch * CH + e) = make_float4(fk[e], fk[e + 1], fk[e + 2], fk[e + 3]);
        *reinterpret_cast<float4*>(Vs + pl * D + ch * CH + e) = make_float4(fv[e], fv[e + 1], fv[e + 2], fv[e + 3]);
      }
    }
    __syncthreads();
    find_slots(tile + 1);
    // S = Q K^T: thread (ty, tx) owns rows 2ty, 2ty+1 and positions tx, tx+16, tx+32, tx+48
    {
      // (the inner index in pairs: a packed instruction does two multiply-adds, and the operands lie in pairs anyway)
      f32x2 acc[2][4];
#pragma unroll
      for (int i = 0; i < 2; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i][j] = 0ull;
#pragma unroll 8
      for (int d = 0; d < D; d += 4) {
        const ulonglong2 q0 = *reinterpret_cast<const ulonglong2*>(Qs + (2 * ty) * KS + d);
        const ulonglong2 q1 = *reinterpret_cast<const ulonglong2*>(Qs + (2 * ty + 1) * KS + d);
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          const ulonglong2 kk = *reinterpret_cast<const ulonglong2*>(Ks + (tx + 16 * j) * KS + d);
          acc[0][j] = fma2(q0.y, kk.y, fma2(q0.x, kk.x, acc[0][j]));
          acc[1][j] = fma2(q1.y, kk.y, fma2(q1.x, kk.x, acc[1][j]));
        }
      }
#pragma unroll
      for (int i = 0; i < 2; ++i) {
        const int r = 2 * ty + i;
        const bool row_ok = row0 + r < rows_total;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          const int pl = tx + 16 * j, pos = pbase + pl;
          bool vis = row_ok && pos < total;
          if (vis && pos >= L) {
            const int jt = pos - L;
            vis = (anc_s[r][jt >> 5] >> (jt & 31)) & 1u;
          }
          Ss[r * SS + pl] = vis ? sum2(acc[i][j]) : -INFINITY;
        }
      }
    }
    __syncthreads();
    // online softmax and O += P V: warp w owns rows 4w .. 4w+3
#pragma unroll
    for (int rr = 0; rr < 4; ++rr) {
      const int r = 4 * warp + rr;
      const float s0 = Ss[r * SS + lane], s1 = Ss[r * SS + lane + 32];
      float mx = fmaxf(s0, s1);
#pragma unroll
      for (int of = 16; of > 0; of >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, of));
      const float m_old = row_m[r];
      const float m_new = fmaxf(m_old, mx);
      float p0 = 0.f, p1 = 0.f, alpha = 1.f;
      if (m_new > -INFINITY) {
        p0 = expf(s0 - m_new);
        p1 = expf(s1 - m_new);
        alpha = expf(m_old - m_new);
      }
      float sum = p0 + p1;
#pragma unroll
      for (int of = 16; of > 0; of >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, of);
      __syncwarp();
      Ss[r * SS + lane] = p0;
      Ss[r * SS + lane + 32] = p1;
      if (lane == 0) {
        row_m[r] = m_new;
        row_l[r] = row_l[r] * alpha + sum;
        row_alpha[r] = alpha;
      }
    }
    __syncwarp();
#pragma unroll
    for (int rr = 0; rr < 4; ++rr) {
      const float a = row_alpha[4 * warp + rr];
#pragma unroll
      for (int e = 0; e < DC; ++e) o[rr][e] *= a;
    }
#pragma unroll 4
    for (int pl = 0; pl < kPT; pl += 4) {
      float4 pv[4];
#pragma unroll
      for (int rr = 0; rr < 4; ++rr) pv[rr] = *reinterpret_cast<const float4*>(Ss + (4 * warp + rr) * SS + pl);
#pragma unroll
      for (int x = 0; x < 4; ++x) {
        float vv[DC];
        if constexpr (DC == 4) {
          const float4 t4 = *reinterpret_cast<const float4*>(Vs + (pl + x) * D + lane * 4);
          vv[0] = t4.x; vv[1] = t4.y; vv[2] = t4.z; vv[3] = t4.w;
        } else {
          const float2 t2 = *reinterpret_cast<const float2*>(Vs + (pl + x) * D + lane * 2);
          vv[0] = t2.x; vv[1] = t2.y;
        }
#pragma unroll
        for (int rr = 0; rr < 4; ++rr) {
          const float w = x == 0 ? pv[rr].x : x == 1 ? pv[rr].y : x == 2 ? pv[rr].z : pv[rr].w;
#pragma unroll
          for (int e = 0; e < DC; ++e) o[rr][e] += w * vv[e];
        }
      }
    }
  }
  __syncthreads();
  // rows to shared memory (the keys' place), then in contiguous pieces: the output, or this split's partial
  float* Os = Ks;
#pragma unroll
  for (int rr = 0; rr < 4; ++rr)
#pragma unroll
    for (int e = 0; e < DC; ++e) Os[(4 * warp + rr) * KS + lane * DC + e] = o[rr][e];
  __syncthreads();
  const int rows_here = rows_total - row0 < kRB ? rows_total - row0 : kRB;
  constexpr int C4 = D / 4;
  T* out = reinterpret_cast<T*>(p.out);
  auto out_row = [&](int r) {
    const int row = row0 + r, t = F + row / G;
    return out + (((size_t)b * p.Ncap + t) * p.Hq + kvh * G + row % G) * D;
  };
  if (p.nsplit == 1) {
    for (int i = tid; i < rows_here * C4; i += kThreads) {
      const int r = i / C4, c = i % C4 * 4;
      const float4 v = *reinterpret_cast<const float4*>(Os + r * KS + c);
      const float x[4] = {v.x, v.y, v.z, v.w};
      store4(out_row(r) + c, x, row_l[r] > 0.f ? 1.f / row_l[r] : 0.f);
    }
    return;
  }
  const size_t item = ((size_t)b * p.Hkv + kvh) * p.nrowblk + rb, part0 = item * p.nsplit * kRB;
  float2* ml = reinterpret_cast<float2*>(p.part_ml) + part0;
  for (int i = tid; i < rows_here * C4; i += kThreads) {
    const int r = i / C4, c = i % C4 * 4;
    __stcg(reinterpret_cast<float4*>(p.part_o + (part0 + (size_t)split * kRB + r) * D + c), *reinterpret_cast<const float4*>(Os + r * KS + c));
  }
  if (tid < rows_here) __stcg(ml + (size_t)split * kRB + tid, make_float2(row_m[tid], row_l[tid]));
  if (p.nsplit > kMergeHere) return;  // attn_merge_kernel
  __syncthreads();
  if (tid == 0) {
    // releases this CTA's partial (the barrier made it this thread's to release), acquires those that came earlier
    int t;
    asm volatile("atom.acq_rel.gpu.global.add.s32 %0, [%1], 1;" : "=r"(t) : "l"(p.ticket + item) : "memory");
    s_last = t == p.nsplit - 1;
    if (t == p.nsplit - 1) p.ticket[item] = 0;  // ready for the next launch
  }
  __syncthreads();
  if (!s_last) return;
  merge_splits<T, D, kRB / (kThreads / 32), 1>(p, b, kvh, rb, F, row0, warp, kThreads / 32, rows_here);
}

// The same as a kernel of its own, a warp per row: for launches of many splits, whose partials (a quarter of a megabyte and
// more per row block) one CTA would take several us to read.
template <typename T, int D>
__global__ void __launch_bounds__(kThreads) attn_merge_kernel(const AttnParams p) {
  asm volatile("griddepcontrol.wait;" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  constexpr int kPer = kRB / (kThreads / 32);  // CTAs per row block
  const int rb = blockIdx.x / kPer, kvh = blockIdx.y, b = blockIdx.z;
  int N = p.n_tree[b];
  N = N < 0 ? 0 : (N > p.Nmax ? p.Nmax : N);
  int F = p.first_row != nullptr ? p.first_row[b] : 0;
  F = F < 0 ? 0 : (F > N ? N : F);
  const int row0 = rb * kRB, rows_here = min((N - F) * p.G - row0, kRB);
  const int r = (blockIdx.x % kPer) * (kThreads / 32) + (threadIdx.x >> 5);
  merge_splits<T, D, 1, 2>(p, b, kvh, rb, F, row0, r, kRB, rows_here);
}

// Row blocks and KV splits of a launch, and the bytes of workspace it needs.
struct CcPlan {
  int nsplit, nrowblk;
  size_t bytes;
};
// per_sm: CTAs per SM at most, which bounds the workspace: kOwn (40 MB) for the shapes this path is for, kFallback (5 MB) for
// those that come here only when a pointer is not aligned for the tensor path, whose callers reserve both workspaces.
constexpr int kOwn = 16, kFallback = 2;
CcPlan cc_plan(const cast_ctx* c, int per_sm, int B, int Hq, int Hkv, int D, int page_size, int seq_capacity) {
  CcPlan pl;
  pl.nrowblk = (c->cfg.total_token * (Hq / Hkv) + kRB - 1) / kRB;
  const int base = B * Hkv * pl.nrowblk;
  const int max_pos = page_size == 0 ? seq_capacity : seq_capacity * page_size;
  const int max_tiles = (max_pos + kPT - 1) / kPT;
  // The count for which a machine evenly loaded with all tiles, half a tile added per CTA for its prologue and partial, and
  // one CTA left running alone at its end (1.3 times as slow a tile) take least; past kMergeHere splits a second launch, as
  // long as a tile. Sequences differ in length, so more and shorter CTAs than the machine holds at once are no loss:
  // 8 sequences of 300-2000, 128 rows, 3 splits (one round of resident CTAs) 98 us, 8 splits 62.
  int nsplit = 1;
  float best = 0.f;
  for (int n = 1; n <= kMaxSplit && n <= max_tiles && (n == 1 || (long long)base * n <= (long long)per_sm * c->num_sms); ++n) {
    const float cost = (float)base * ((float)max_tiles + 0.5f * (float)n) / (float)c->num_sms +
                       1.3f * ((float)((max_tiles + n - 1) / n) + 0.5f) + (n > kMergeHere ? 1.f : 0.f);
    if (n == 1 || cost < best) {
      best = cost;
      nsplit = n;
    }
  }
  pl.nsplit = nsplit;
  pl.bytes = nsplit == 1 ? 0 : kCcTicketBytes + (size_t)base * nsplit * kRB * (D + 2) * sizeof(float);
  return pl;
}

template <typename T, int D>
cast_status launch_cc(cast_ctx* c, AttnParams& p, int per_sm, cudaStream_t s) {
  const CcPlan pl = cc_plan(c, per_sm, p.B, p.Hq, p.Hkv, D, p.page_size, p.seq_capacity);
  // compute calls never allocate: the workspace comes from cast_reserve_attention
  if (pl.bytes > c->attn_ws_bytes) return CAST_ERR_CAPACITY;
  p.nsplit = pl.nsplit;
  p.nrowblk = pl.nrowblk;
  if (pl.nsplit > 1) {
    p.ticket = reinterpret_cast<int32_t*>(c->attn_ws);
    p.part_o = reinterpret_cast<float*>(reinterpret_cast<char*>(c->attn_ws) + kCcTicketBytes);
    p.part_ml = p.part_o + (size_t)p.B * p.Hkv * pl.nrowblk * pl.nsplit * kRB * D;
  }
  const size_t smem = (size_t)(kRB * (D + 4) + kPT * (D + 4) + kPT * D + kRB * (kPT + 4)) * sizeof(float);
  auto kern = tree_attn_cc_kernel<T, D>;
  CAST_CUDA_OK(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(pl.nsplit * pl.nrowblk, p.Hkv, p.B);
  cfg.blockDim = dim3(kThreads, 1, 1);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;  // launched while its predecessor drains; waits for it
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  cudaError_t e = cudaLaunchKernelEx(&cfg, kern, p);
  if (e == cudaSuccess && pl.nsplit > kMergeHere) {
    cfg.gridDim = dim3(pl.nrowblk * (kRB / (kThreads / 32)), p.Hkv, p.B);
    cfg.dynamicSmemBytes = 0;
    e = cudaLaunchKernelEx(&cfg, attn_merge_kernel<T, D>, p);
  }
  if (e != cudaSuccess) {
    cudaGetLastError();
    return CAST_ERR_CUDA;
  }
  return CAST_OK;
}

}  // namespace

extern "C" cast_status cast_set_attention_early_reads(cast_ctx* c, int promise) {
  if (!c) return CAST_ERR_INVALID_ARG;
  c->attn_early = promise ? 1 : 0;
  c->wl_valid = 0;
  return CAST_OK;
}

extern "C" cast_status cast_reserve_attention(cast_ctx* c, cast_dtype dtype, int B, int Hq, int Hkv, int D, int page_size,
                                              int seq_capacity) {
  if (!c || B < 1 || Hq < 1 || Hkv < 1 || page_size < 0 || seq_capacity < 1) return CAST_ERR_INVALID_ARG;
  if (dtype != CAST_F32 && dtype != CAST_BF16) return CAST_ERR_DTYPE;
  if (B > c->cfg.max_batch) return CAST_ERR_CAPACITY;
  if (Hq % Hkv != 0 || (D != 64 && D != 128)) return CAST_ERR_SHAPE;
  // a bf16 call takes the tensor-core path when shape and pointer alignment allow and the CUDA-core path
  // otherwise: both workspaces are sized, so the choice at call time never needs memory
  bool own = true;
  if (dtype == CAST_BF16) {
    own = !tree_attention_tc_takes(c, B, Hq, Hkv, D, page_size, seq_capacity);
    const cast_status st = tree_attention_tc_reserve(c, tree_attention_tc_workspace(c, B, Hq, Hkv, D, page_size, seq_capacity));
    if (st != CAST_OK) return st;
  }
  const size_t need = cc_plan(c, own ? kOwn : kFallback, B, Hq, Hkv, D, page_size, seq_capacity).bytes;
  if (need > c->attn_ws_bytes) {
    CAST_CUDA_OK(cudaDeviceSynchronize());
    if (c->attn_ws) cudaFree(c->attn_ws);
    c->attn_ws = nullptr;
    c->attn_ws_bytes = 0;
    CAST_CUDA_OK(cudaMalloc(&c->attn_ws, need));
    // tickets start at zero; every merge leaves its ticket at zero again
    CAST_CUDA_OK(cudaMemset(c->attn_ws, 0, kCcTicketBytes));
    c->attn_ws_bytes = need;
  }
  return CAST_OK;
}

extern "C" cast_status cast_tree_attention_rows(cast_ctx* c, const void* q, const void* k_cache, const void* v_cache,
                                                cast_dtype dtype, int B, int Hq, int Hkv, int D, int page_size,
                                                const int32_t* page_table, int seq_capacity, int num_pages,
                                                const int32_t* kv_len, const uint32_t* anc_mask, const int32_t* n_tree,
                                                const int32_t* first_row, float scale, void* out, void* stream) {
  if (!c || !q || !k_cache || !v_cache || !kv_len || !anc_mask || !n_tree || !out || B < 1 || Hq < 1 || Hkv < 1 ||
      page_size < 0 || seq_capacity < 1 || (page_size > 0 && (!page_table || num_pages < 1)))
    return CAST_ERR_INVALID_ARG;
  if (dtype != CAST_F32 && dtype != CAST_BF16) return CAST_ERR_DTYPE;
  if (B > c->cfg.max_batch) return CAST_ERR_CAPACITY;
  if (Hq % Hkv != 0 || (D != 64 && D != 128)) return CAST_ERR_SHAPE;
  if (((uintptr_t)q | (uintptr_t)k_cache | (uintptr_t)v_cache | (uintptr_t)out) & 15) return CAST_ERR_SHAPE;
  if (scale == 0.f) scale = 1.0f / sqrtf((float)D);
  cudaStream_t s = (cudaStream_t)stream;
  const int fresh = c->tree_inputs_fresh;
  if (fresh) c->wl_valid = 0;  // also where this call takes no list itself: a later one must not find the old one
  c->tree_inputs_fresh = 0;  // whatever is launched below waits for its predecessor before it releases its own dependents
  if (dtype == CAST_BF16) {
    cast_status st = CAST_OK;
    c->tree_inputs_fresh = fresh;
    const bool taken = tree_attention_tc_launch(c, q, k_cache, v_cache, B, Hq, Hkv, D, page_size, page_table, seq_capacity,
                                                num_pages, kv_len, anc_mask, n_tree, first_row, scale, out, s, &st);
    c->tree_inputs_fresh = 0;
    if (taken) return st;
  }
  AttnParams p;
  p.q = q; p.k = k_cache; p.v = v_cache; p.out = out;
  p.B = B; p.Ncap = c->cfg.max_tree; p.Nmax = c->cfg.total_token; p.Hq = Hq; p.Hkv = Hkv; p.G = Hq / Hkv;
  p.page_size = page_size; p.seq_capacity = seq_capacity; p.num_pages = num_pages; p.words = c->words;
  p.page_table = page_table; p.kv_len = kv_len; p.n_tree = n_tree; p.first_row = first_row; p.anc = anc_mask;
  p.scale = scale; p.ticket = nullptr; p.part_o = nullptr; p.part_ml = nullptr; p.st = c->state;
  if (dtype == CAST_F32) return D == 64 ? launch_cc<float, 64>(c, p, kOwn, s) : launch_cc<float, 128>(c, p, kOwn, s);
  const int per_sm = tree_attention_tc_takes(c, B, Hq, Hkv, D, page_size, seq_capacity) ? kFallback : kOwn;
  return D == 64 ? launch_cc<__nv_bfloat16, 64>(c, p, per_sm, s) : launch_cc<__nv_bfloat16, 128>(c, p, per_sm, s);
}

extern "C" cast_status cast_tree_attention(cast_ctx* c, const void* q, const void* k_cache, const void* v_cache,
                                           cast_dtype dtype, int B, int Hq, int Hkv, int D, int page_size,
                                           const int32_t* page_table, int seq_capacity, int num_pages,
                                           const int32_t* kv_len, const uint32_t* anc_mask, const int32_t* n_tree,
                                           float scale, void* out, void* stream) {
  return cast_tree_attention_rows(c, q, k_cache, v_cache, dtype, B, Hq, Hkv, D, page_size, page_table, seq_capacity,
                                  num_pages, kv_len, anc_mask, n_tree, nullptr, scale, out, stream);
}
