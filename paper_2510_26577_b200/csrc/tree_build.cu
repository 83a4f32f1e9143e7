// Draft-tree construction: cast_step_begin, cast_tree_expand, cast_select_nodes.
//
// cast_tree_expand is ONE kernel per draft layer, launched as thread-block clusters (the chunks of
// one logits row form a cluster) with programmatic dependent launch between the layers:
//   1. vocabulary sweep - one CTA per chunk: streaming 16-byte loads, two buffers of them in flight, online max / sum-exp
//      in base 2, and a list of candidates per warp, filtered against a threshold the CTA's warps share (the K-th largest
//      of the maxima of sixteen parts: a lower bound on the CTA's K-th largest, so the result is exact and only a
//      logit or two per warp survives the filter);
//   2. the chunk's candidates, maxima and sums go straight into the shared memory of the cluster's
//      first CTA, which merges the row after the cluster barrier (log-sum-exp in fp64, the candidates ranked by
//      counting) and appends the K children to the node pool;
//   3. the last row-merging CTA of the layer (an atomic ticket; nothing spins) ranks each
//      sequence's candidates, forms the utility u (Eq. 1) and the cost c (Eq. 2), runs Algorithm 1
//      (breadth pruning), the depth-pruning test and the FIFO update, and publishes the retained
//      nodes and the layer's sorted list.
// cast_select_nodes ranks the pool by merging the per-layer sorted lists (binary searches), forms
// the batch-mean utility, runs Algorithm 1 with the target-cost ratio and linearises the tree.
#include <math.h>

#include "cast_internal.h"

using namespace cast;

namespace {

// ------------------------------------------------------------------ expand
struct ExpandParams {
  const void* logits;
  int V, K, W, H, P, layer, nchunks, chunk_elems;
  int prefetch;  // the layer's logits are small enough to be worth asking for ahead of the dependency wait
  double* pool_score;
  int32_t* pool_token;
  int32_t* pool_parent;
  int32_t* pool_depth;
  uint8_t* pool_kept;
  int32_t* retained;
  int32_t* lsort;
  double* lscore;
  DevState* st;
  int32_t* layer_ticket;
  int32_t* seq_ticket;
  double* tail_vs;
  int32_t* tail_sorted;
  int32_t* tail_tok;
  double* fifo_vals;
  int32_t* fifo_cnt;
  int R;
  DevTable tab;
  double C1, C2;
  int enable_bp, enable_dp, ctx_base_mode;
  int32_t* next_tokens;
  int32_t* next_parent_row;
  int32_t* next_count;
  // the step's root tokens and prefix lengths (read by layer 1, which also resets the per-step state)
  const int32_t* root_token;
  const int32_t* kv_len;
};

__device__ __forceinline__ float ex2f(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
// log2(e) split into a float just below it and a positive residual: x * log2(e) to better than one ulp
// of the product, and -inf logits stay -inf through both FMAs (no inf - inf)
// Packed fp32 pairs: one instruction, two lanes of the FMA pipe, the same IEEE results per element.
__device__ __forceinline__ unsigned long long pack2(float a, float b) {
  unsigned long long r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
  return r;
}
__device__ __forceinline__ void unpack2(unsigned long long v, float& a, float& b) {
  asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(v));
}
__device__ __forceinline__ unsigned long long fma2(unsigned long long a, unsigned long long b, unsigned long long c) {
  unsigned long long r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
  return r;
}
__device__ __forceinline__ unsigned long long add2(unsigned long long a, unsigned long long b) {
  unsigned long long r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
constexpr float kLog2eHi = 1.4426950216293335f;
constexpr float kLog2eLo = 1.925963033500011e-08f;  // log2(e) - kLog2eHi

// exp(s) for s <= 0 to about 1.2e-7 relative: the product with log2(e) and the integer part in fp64, the
// fractional power by the fp32 unit, exact scaling. (A node value needs no more: the decision margins that
// the parity contract asks for are 2e-6 relative.)
__device__ __forceinline__ double fast_exp_neg(double s) {
  const double t = s * 1.4426950408889634074;
  if (!(t > -1000.0)) return 0.0;
  const double n = floor(t);
  return ldexp((double)ex2f((float)(t - n)), (int)n);
}
// log2(S), S > 0, to about 1e-7 absolute: exact exponent split, fp32 logarithm of the mantissa
__device__ __forceinline__ double fast_log2(double S) {
  int e;
  const double m = frexp(S, &e);
  return (double)e + (double)log2f((float)m);
}

// ---- thread-block cluster primitives (a logits row is swept by one cluster)
__device__ __forceinline__ uint32_t smem_addr(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ uint32_t map_to_rank(uint32_t saddr, uint32_t rank) {
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(saddr), "r"(rank));
  return r;
}
__device__ __forceinline__ void st_cluster_u64(uint32_t addr, unsigned long long v) {
  asm volatile("st.shared::cluster.u64 [%0], %1;" ::"r"(addr), "l"(v) : "memory");
}
__device__ __forceinline__ void st_cluster_f32(uint32_t addr, float v) {
  asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(addr), "f"(v) : "memory");
}
__device__ __forceinline__ void st_cluster_u32(uint32_t addr, uint32_t v) {
  asm volatile("st.shared::cluster.u32 [%0], %1;" ::"r"(addr), "r"(v) : "memory");
}
__device__ __forceinline__ void st_cluster_f64(uint32_t addr, double v) {
  asm volatile("st.shared::cluster.f64 [%0], %1;" ::"r"(addr), "d"(v) : "memory");
}
__device__ __forceinline__ void cluster_arrive_release() { asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait_acquire() { asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory"); }

// Programmatic dependent launch (both are no-ops for a grid launched without the attribute).
__device__ __forceinline__ void grid_dependency_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void grid_launch_dependents() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

// State fields the layer tail needs; every CTA reads them at its start (same cache lines as the row
// count it needs anyway), so the tail itself starts without a round trip to memory.
struct TailState {
  int ctx_sum, n0, kept_total;
  double u_last;
};

// The ticket of the "last CTA" pattern: the caller has passed a CTA barrier after its global
// writes; one thread takes the ticket with release-acquire semantics (cumulative over the CTA's writes).
__device__ __forceinline__ bool take_ticket(int32_t* counter, int expected, int* flag_s) {
  if (threadIdx.x == 0) {
    // one acquire-release atomic at device scope: releases this CTA's writes (the barrier before the
    // call made them this thread's to release), acquires those of the CTAs that came earlier
    int t;
    asm volatile("atom.acq_rel.gpu.global.add.s32 %0, [%1], 1;" : "=r"(t) : "l"(counter) : "memory");
    const int last = (t == expected - 1);
    if (last) *counter = 0;
    *flag_s = last;
  }
  __syncthreads();
  return *flag_s != 0;
}

// Layer tail (Eq. 1, Eq. 2, Algorithm 1, depth pruning) in two parts. tail_rank orders the candidates of
// some sequences and is what costs time with many sequences; tail_decide is the batch-wide rest. With up to
// four sequences (eight, of few candidates) the last CTA of the layer runs both from shared memory; with more, the last CTA
// of every sequence ranks that sequence (so the sequences are ranked in parallel) and leaves the first n sorted
// nodes in global memory, and the last of those CTAs decides.

constexpr int kTailScratch = 28672;  // bytes of shared memory the tail works in
// Up to this many sequences, or candidates, the one-CTA tail is faster than a second ticket (V = 32000, 8 sequences: 92 -> 89 us).
constexpr int kTailSingleMaxB = 8, kTailAlwaysSingleB = 4, kTailSingleCands = 512;

// Candidates Algorithm 1 looks at: the first n of the sorted list.
__device__ __forceinline__ int tail_width(const ExpandParams& p, int n_prev) {
  const int Ni = n_prev * p.K;
  int n = Ni < p.W ? Ni : p.W;
  if ((p.enable_bp || p.enable_dp) && p.tab.Ntab < n) n = p.tab.Ntab;
  return n;
}

// Ranking by counting. A warp's lanes hold 32 of the items; the items they are compared with are read one at a
// time, the same in all lanes; the warps share out the comparisons and their counts meet in shared memory. (With a lane
// per share of one item's comparisons the shared-memory reads made 126 keys take 1.7 us.) A comparison of 64-bit keys is a
// subtraction whose borrow is counted.
__device__ __forceinline__ void count_less64(int& neg, uint32_t alo, uint32_t ahi, uint32_t blo, uint32_t bhi) {
  asm("{\n\t.reg .u32 t;\n\tsub.cc.u32 t, %1, %3;\n\tsubc.cc.u32 t, %2, %4;\n\tsubc.u32 %0, %0, 0;\n\t}"
      : "+r"(neg)
      : "r"(alo), "r"(ahi), "r"(blo), "r"(bhi));
}

// log2 of the warps per group when `nw` warps share `groups` groups (an integer division is a chain of some 130 cycles)
__device__ __forceinline__ int share_log(int groups, int nw) {
  int l = 0;
  while (groups << (l + 1) <= nw) ++l;
  return l;
}

// A candidate as one 128-bit number, smaller = earlier in the order (value desc, token asc, creation order): the value's
// bits mapped so that larger values come first, the token, the place. (Equal siblings are everywhere with half-precision
// logits: comparisons that look at the token on equality only took 4 us for 144 candidates, these 1.2.)
__device__ __forceinline__ uint4 make_cand(double score, int token, int place) {
  uint64_t b = (uint64_t)__double_as_longlong(score + 0.0);  // (-0 as +0)
  b = (b >> 63) ? b : ~(b | 0x8000000000000000ull);
  return make_uint4((uint32_t)place, (uint32_t)token, (uint32_t)b, (uint32_t)(b >> 32));
}
__device__ __forceinline__ double cand_score(const uint4& c) {
  const uint64_t b = ((uint64_t)c.w << 32) | c.z;
  return __longlong_as_double((long long)((b >> 63) ? b : ~b & 0x7fffffffffffffffull));
}
__device__ __forceinline__ void count_less(int& neg, const uint4& a, const uint4& b) {  // neg -= a < b
  asm("{\n\t.reg .u32 t;\n\t"
      "sub.cc.u32 t, %1, %5;\n\tsubc.cc.u32 t, %2, %6;\n\tsubc.cc.u32 t, %3, %7;\n\tsubc.cc.u32 t, %4, %8;\n\t"
      "subc.u32 %0, %0, 0;\n\t}"
      : "+r"(neg)
      : "r"(a.x), "r"(a.y), "r"(a.z), "r"(a.w), "r"(b.x), "r"(b.y), "r"(b.z), "r"(b.w));
}

// rank_s[i] -= the number of candidates of i's sequence that come before it; nb sequences of Ni candidates, one after the
// other. Groups of 32 candidates of one sequence, one per lane; the warps left over split a group's comparisons. Bound by
// the ALU: more candidates per lane only add padding.
__device__ __forceinline__ void rank_candidates(const uint4* cand, int* rank_s, int nb, int Ni) {
  const int lane = threadIdx.x & 31, nw = blockDim.x >> 5;
  const int gps = (Ni + 31) >> 5, groups = nb * gps;
  int shares = 1;
  while ((shares + 1) * groups <= nw) ++shares;
  const int len = div_small(Ni + shares - 1, shares, __fdividef(1.f, (float)shares));
#pragma unroll 1
  for (int w = threadIdx.x >> 5; w < groups * shares; w += nw) {
    const int wg = div_small(w, shares, __fdividef(1.f, (float)shares));
    const int j0 = (w - wg * shares) * len, j1 = min(j0 + len, Ni);
    int bl = 0, g = wg;
    for (; g >= gps; g -= gps) ++bl;
    const uint4* list = cand + bl * Ni;
    const int ci = g * 32 + lane;
    const uint4 mine = list[ci < Ni ? ci : 0];
    int neg = 0;
#pragma unroll 8
    for (int j = j0; j < j1; ++j) count_less(neg, list[j], mine);
    if (ci < Ni) atomicAdd(&rank_s[bl * Ni + ci], neg);
  }
}

// Ranks the layer's candidates of the sequences [b_begin, b_begin + b_count): writes every sequence's sorted
// list for the rerank (lsort, lscore) and, for rank < n, pool index, token and value to sorted_o, stok_o,
// vs_o at [b * CAST_MAX_WIDTH + rank] (shared or global memory).
__device__ __forceinline__ void tail_rank(const ExpandParams& p, int b_begin, int b_count, int n, int n_prev, int base,
                                          unsigned char* scratch, int* sorted_o, int* stok_o, double* vs_o) {
  const int tid = threadIdx.x, nt = blockDim.x;
  const int P = p.P;
  const int Ni = n_prev * p.K;
  uint4* cand = reinterpret_cast<uint4*>(scratch);            // 1024 candidates
  int* rank_s = reinterpret_cast<int*>(scratch + 16384);      // 1024 ranks, negated
  const float inv_Ni = __fdividef(1.f, (float)Ni);
  const int group = div_small(1024, Ni, inv_Ni);              // sequences ranked per pass
#pragma unroll 1
  for (int b0 = 0; b0 < b_count; b0 += group) {
    const int nb = (b_count - b0) < group ? (b_count - b0) : group;
    const int tot = nb * Ni;
    for (int i = tid; i < tot; i += nt) {
      const int bl = div_small(i, Ni, inv_Ni), ci = i - bl * Ni;
      const size_t o = (size_t)(b_begin + b0 + bl) * P + base + ci;
      cand[i] = make_cand(__ldcg(p.pool_score + o), __ldcg(p.pool_token + o), ci);
      rank_s[i] = 0;
    }
    __syncthreads();
    // Rank under the order (value desc, token asc, creation order): the number of the sequence's candidates that come first.
    rank_candidates(cand, rank_s, nb, Ni);
    __syncthreads();
#pragma unroll 1
    for (int i = tid; i < tot; i += nt) {
      const int bl = div_small(i, Ni, inv_Ni), ci = i - bl * Ni, rank = -rank_s[i];
      const uint4 mine = cand[i];
      {
        const int bg = b_begin + b0 + bl;
        const size_t o = (size_t)bg * P + base + rank;
        p.lsort[o] = base + ci;  // the layer's sorted list, for the rerank
        const double s = cand_score(mine);
        p.lscore[o] = s;
        if (rank < n) {
          sorted_o[bg * CAST_MAX_WIDTH + rank] = base + ci;
          stok_o[bg * CAST_MAX_WIDTH + rank] = (int)mine.y;
          vs_o[bg * CAST_MAX_WIDTH + rank] = fast_exp_neg(s);
        }
      }
    }
    __syncthreads();
  }
}

// What the deciding warp needs from memory, requested as soon as the CTA knows that it ranks (the first warp; per lane).
struct DecideIn {
  double c;              // Eq. 2's cost of rank lane + 1
  double prev[2], cur[2];  // entries lane and lane + 32 of the buffers A_{i-1} (to be pushed to) and A_i (to be averaged)
  int prev_n, cur_n;
  int n0;                // layer 1: the longest of two sequences' prefixes
};
__device__ __forceinline__ DecideIn decide_load(const ExpandParams& p, const TailState& ts, int B, int n) {
  DecideIn d;
  const int lane = threadIdx.x & 31;
  d.c = 0.0;
  d.prev[0] = d.prev[1] = d.cur[0] = d.cur[1] = 0.0;
  d.prev_n = d.cur_n = 0;
  d.n0 = ts.n0;
  if (threadIdx.x >= 32) return d;
  static_assert(CAST_MAX_BATCH <= 64 && kMaxFifo <= 64, "two entries per lane");
  if (p.layer == 1) d.n0 = max(lane < B ? p.kv_len[lane] : 0, lane + 32 < B ? p.kv_len[lane + 32] : 0);
  if ((p.enable_bp || p.enable_dp) && lane < n && !(p.layer == 1 && p.ctx_base_mode)) {
    const int g = select_grid(ts.ctx_sum + (p.ctx_base_mode ? ts.n0 : 0), p.tab.L, p.tab.M);
    d.c = p.tab.fD[(size_t)(g - 1) * p.tab.Ntab + lane] / p.tab.fT[(size_t)(g - 1) * p.tab.Ntab];
  }
  if (p.enable_dp) {
    if (p.layer >= 2) {
      const double* A = p.fifo_vals + (size_t)(p.layer - 2) * p.R;
      if (lane < p.R) d.prev[0] = A[lane];
      if (lane + 32 < p.R) d.prev[1] = A[lane + 32];
      d.prev_n = p.fifo_cnt[p.layer - 2];
    }
    if (p.layer < p.H) {
      const double* A = p.fifo_vals + (size_t)(p.layer - 1) * p.R;
      if (lane < p.R) d.cur[0] = A[lane];
      if (lane + 32 < p.R) d.cur[1] = A[lane + 32];
      d.cur_n = p.fifo_cnt[p.layer - 1];
    }
  }
  return d;
}

// a / B; for a power of two by an exact product (a division in fp64 is a chain of some 200 cycles)
__device__ __forceinline__ double mean_of(double a, int B) {
  if ((B & (B - 1)) == 0) return a * __longlong_as_double((long long)(1023 - (31 - __clz(B))) << 52);
  return a / (double)B;
}

// The batch-wide part: Eq. 1 over the sequences' first n sorted values, Eq. 2, Algorithm 1, the depth test,
// the state for the next layer and the layer's outputs. GLOBAL: the inputs were written to global memory by
// other CTAs (read past L1). One warp decides (n <= CAST_MAX_WIDTH <= 32: a rank per lane, no barriers); the next layer's
// CTAs wait for this, so it is a chain of shuffles and arithmetic only.
template <bool GLOBAL>
__device__ __forceinline__ void tail_decide(const ExpandParams& p, const TailState& ts, const DecideIn& d, int B, int n, int n_prev,
                                            int base, const int* sorted_i, const int* stok_i, const double* vs_i) {
  __shared__ double vbar[CAST_MAX_WIDTH];
  __shared__ int s_ni;
  constexpr unsigned kAll = 0xffffffffu;
  const int tid = threadIdx.x, nt = blockDim.x, lane = tid & 31;
  DevState* st = p.st;
  const int K = p.K, W = p.W, P = p.P;
  const int Ni = n_prev * K;
  if (p.layer == 1) {
    // The first layer of a step also starts the step (cast_step_begin launches nothing): the padded context
    // length n_0 = max_b kv_len[b] and every sequence's root node (value 1, depth 0) at pool index 0.
    for (int b = tid - 32; b >= 0 && b < B; b += nt - 32) {
      const size_t o = (size_t)b * P;
      p.pool_score[o] = 0.0;
      p.pool_token[o] = p.root_token[b];
      p.pool_parent[o] = -1;
      p.pool_depth[o] = 0;
      p.pool_kept[o] = 1;
      p.lsort[o] = 0;
      p.lscore[o] = 0.0;
    }
  }
  const float inv_W = __fdividef(1.f, (float)W), inv_K = __fdividef(1.f, (float)K);
  // the nodes that may be retained, requested together with their values
  constexpr int kOut = CAST_MAX_BATCH * CAST_MAX_WIDTH / kSweepThreads;
  int idx_k[kOut], tok_k[kOut];
  if (GLOBAL) {
#pragma unroll
    for (int k = 0; k < kOut; ++k) {
      const int i = tid + k * nt, b = div_small(i, W, inv_W), s = i - b * W;
      idx_k[k] = tok_k[k] = 0;
      if (i < B * W && s < n) {
        idx_k[k] = __ldcg(sorted_i + b * CAST_MAX_WIDTH + s);
        tok_k[k] = __ldcg(stok_i + b * CAST_MAX_WIDTH + s);
      }
    }
  }
  // Eq. 1: batch mean of the rank-wise values
  if (GLOBAL) {
    // many sequences: a warp per rank sums over the sequences, two per lane, then a fixed shuffle tree
    static_assert(CAST_MAX_BATCH <= 64, "two sequences per lane");
    for (int j = tid >> 5; j < n; j += nt >> 5) {
      double a = (lane < B ? __ldcg(vs_i + lane * CAST_MAX_WIDTH + j) : 0.0) +
                 (lane + 32 < B ? __ldcg(vs_i + (lane + 32) * CAST_MAX_WIDTH + j) : 0.0);
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) a += __shfl_xor_sync(kAll, a, o);
      if (lane == 0) vbar[j] = mean_of(a, B);
    }
    __syncthreads();
  }
  if (tid < 32) {
    int n0 = d.n0;
    if (p.layer == 1) n0 = __reduce_max_sync(kAll, n0);
    double c = d.c;
    if ((p.enable_bp || p.enable_dp) && p.layer == 1 && p.ctx_base_mode && lane < n) {
      const int g = select_grid(ts.ctx_sum + n0, p.tab.L, p.tab.M);
      c = p.tab.fD[(size_t)(g - 1) * p.tab.Ntab + lane] / p.tab.fT[(size_t)(g - 1) * p.tab.Ntab];
    }
    double u = 0.0;
    if (lane < n) {
      if (GLOBAL) {
        u = vbar[lane];
      } else {
#pragma unroll 1
        for (int b = 0; b < B; ++b) u += vs_i[b * CAST_MAX_WIDTH + lane];
        u = mean_of(u, B);
      }
    }
#pragma unroll
    for (int o = 1; o < CAST_MAX_WIDTH; o <<= 1) {  // prefix sums
      const double t = __shfl_up_sync(kAll, u, o);
      if (lane >= o) u += t;
    }
    // Algorithm 1: mark[j] survives iff no earlier i has (u_j - u_i) < C1 (c_j - c_i); n_i = the largest marked index
    bool ok = lane < n;
    if (p.enable_bp) {
#pragma unroll 4
      for (int i = 0; i < n - 1; ++i) {
        const double ui = __shfl_sync(kAll, u, i), ci = __shfl_sync(kAll, c, i);
        if (i < lane && (u - ui) < p.C1 * (c - ci)) ok = false;
      }
    }
    const unsigned marks = __ballot_sync(kAll, ok);
    const int n_i = marks != 0u ? 32 - __clz(marks) : 1;
    if (lane == 0) s_ni = n_i;
    const double u_n = __shfl_sync(kAll, u, n_i - 1), c_n = __shfl_sync(kAll, c, n_i - 1);
    bool go = true;
    if (p.enable_dp) {
      if (p.layer >= 2) {  // gain ratio of the previous layer goes into its buffer, FIFO
        const double phi = u_n / ts.u_last;
        double* A = p.fifo_vals + (size_t)(p.layer - 2) * p.R;
        if (d.prev_n < p.R) {
          if (lane == 0) {
            A[d.prev_n] = phi;
            p.fifo_cnt[p.layer - 2] = d.prev_n + 1;
          }
        } else {
          if (lane >= 1 && lane < p.R) A[lane - 1] = d.prev[0];
          if (lane + 32 < p.R) A[lane + 31] = d.prev[1];
          if (lane == 0) A[p.R - 1] = phi;
        }
      }
      if (p.layer < p.H) {  // generate layer i+1 only if Avg(A_i) * u / c >= C2
        double a = 0.0;
        for (int k = 0; k < d.cur_n; ++k) a += __shfl_sync(kAll, k < 32 ? d.cur[0] : d.cur[1], k & 31);
        const double alpha = a / (double)d.cur_n;
        go = (alpha * u_n / c_n) >= p.C2;
      }
    }
    const int next = (p.layer < p.H && go) ? n_i : 0;
    if (p.layer == 1) {  // per-step state (rows[]: a later layer that is never reached must read 0)
      for (int i = lane + 2; i <= CAST_MAX_DEPTH; i += 32) {
        st->n_hist[i] = 0;
        st->layer_base[i] = 0;
        st->layer_n[i] = 0;
      }
      for (int i = lane; i < CAST_MAX_DEPTH + 2; i += 32)
        if (i != 2) st->rows[i] = (i == 1) ? 1 : 0;
      if (lane == 0) {
        st->B = B;
        st->n0 = n0;
        st->n_tree = 0;
        st->n_hist[0] = 1;
        st->layer_base[0] = 0;
        st->layer_n[0] = 1;
      }
    }
    if (lane == 0) {
      st->rows[p.layer + 1] = next;
      st->n_hist[p.layer] = n_i;
      st->layer_base[p.layer] = base;
      st->layer_n[p.layer] = Ni;
      st->ctx_sum = ts.ctx_sum + n_i;
      st->kept_total = ts.kept_total + n_i;
      st->u_last = u_n;
      st->pool_size = base + Ni;
      st->layers_done = p.layer;
      *p.next_count = next;
    }
  }
  __syncthreads();
  const int n_i = s_ni;
#pragma unroll
  for (int k = 0; k < kOut; ++k) {
    const int i = tid + k * nt;
    if (i >= B * W) break;
    const int b = div_small(i, W, inv_W), s = i - b * W;
    int tok = -1, prow = -1;
    if (s < n_i) {
      const int idx = GLOBAL ? idx_k[k] : sorted_i[b * CAST_MAX_WIDTH + s];
      tok = GLOBAL ? tok_k[k] : stok_i[b * CAST_MAX_WIDTH + s];
      prow = div_small(idx - base, K, inv_K);
      p.retained[b * W + s] = idx;
      p.pool_kept[(size_t)b * P + idx] = 1;
    }
    p.next_tokens[i] = tok;
    p.next_parent_row[i] = prow;
  }
}

// ---- vocabulary sweep of one chunk -------------------------------------------------------------------------------
// A chunk's logits are read in buffers of 64 bytes per thread, two of them in flight: while one is worked on the next is on
// its way. Per logit the work is a maximum, the exponential and its sum (about five instructions); candidates for the
// top K are found by one comparison of the buffer's maximum with a threshold, below which almost all buffers lie.
//
// Candidates: every warp has a list in shared memory, to which a lane appends what reaches the threshold. The threshold
// is a lower bound on the CTA's K-th largest logit, shared by its warps: the K-th largest of the sixteen warps' maxima over
// the first two buffers (K of the chunk's logits are at least that large), raised once more in long chunks. A dozen
// logits per 16 K pass it, so a list is not put in order until it overflows (a rising row, ties): then the warp ranks
// it, keeps its K best and raises its own threshold to the K-th; if a single buffer overflows it (constant rows) the K
// best come from K rounds of a warp-wide maximum. What reaches the threshold is never dropped except for K better
// ones, and every threshold is at most the K-th largest: the chunk's top K is always among the lists.
constexpr int kBufVecs = 4;     // 16-byte vectors per thread and buffer
constexpr int kGroups = kSweepThreads / 32;  // parts of a CTA whose maxima give the threshold: its warps
constexpr int kListCap = 64;    // keys per warp list
constexpr int kPushCap = 32;    // keys a warp hands on at most
static_assert(kGroups == 16, "a group's number takes the last four bits of its maximum");
static_assert(CAST_MAX_TOP_K <= kGroups, "the K-th largest of the groups' maxima needs K <= groups");
static_assert(CAST_MAX_TOP_K <= kPushCap, "a warp hands on its K best");

// OUT: the overflow handling is a function of its own. Inlined twice it is half of the sweep's code, and in the short launches,
// which run everything once, the warps wait for instructions (1-2 us per tree); in the 64-register launches the call costs
// more registers than there are (batch 64 307 -> 329 us).
template <typename T, bool OUT>
struct Sweep {
  static constexpr int VEC = Vec<T>::N;
  static constexpr int kSlots = kBufVecs * VEC;                      // logits of a thread per buffer
  static constexpr int kBufElems = kSweepThreads * kSlots;                      // of the CTA
  uint4 raw[kBufVecs];

  // First element (of the aligned view) of this thread's vector v in the buffer that starts at `base`.
  static __device__ __forceinline__ int elem(int base, int v) { return base + (v * kSweepThreads + (int)threadIdx.x) * VEC; }

  // A whole buffer; `at`: this thread's first vector of it. (One address per buffer, the rest are immediate offsets.)
  __device__ __forceinline__ void load(const uint4* at) {
#pragma unroll
    for (int v = 0; v < kBufVecs; ++v) raw[v] = __ldcs(at + v * kSweepThreads);
  }
  // A buffer that is not all there. xa: the row from the 16-byte boundary at or below its start; elements [lo, end) of it
  // exist.
  __device__ __forceinline__ void load_part(const T* xa, int base, int lo, int end) {
#pragma unroll
    for (int v = 0; v < kBufVecs; ++v) {
      const int idx = elem(base, v);
      if (idx >= lo && idx + VEC <= end) {
        raw[v] = __ldcs(reinterpret_cast<const uint4*>(xa + idx));
      } else {
        raw[v] = make_uint4(Vec<T>::kMinusInf, Vec<T>::kMinusInf, Vec<T>::kMinusInf, Vec<T>::kMinusInf);
        if (idx < end) {
#pragma unroll
          for (int e = 0; e < VEC; ++e)
            if (idx + e >= lo && idx + e < end) Vec<T>::put(raw[v], e, to_float(xa[idx + e]));
        }
      }
    }
  }
  static __device__ __forceinline__ int slot_elem(int base, int i) {
    return base + ((i / VEC) * kSweepThreads + (int)threadIdx.x) * VEC + (i % VEC);
  }
  // the logit of slot i (not a constant)
  __device__ __forceinline__ float slot(int i) const {
    const int w = i * kBufVecs * 4 / kSlots;  // its word of the sixteen
    const uint4 q = (w & 8) ? ((w & 4) ? raw[3] : raw[2]) : ((w & 4) ? raw[1] : raw[0]);
    const uint32_t u = (w & 2) ? ((w & 1) ? q.w : q.z) : ((w & 1) ? q.y : q.x);
    if (VEC == 4) return __uint_as_float(u);
    return __uint_as_float((i & 1) ? (u & 0xffff0000u) : (u << 16));
  }
  __device__ __forceinline__ float max() const {
    float m = Vec<T>::max(raw[0]);
#pragma unroll
    for (int v = 1; v < kBufVecs; ++v) m = fmaxf(m, Vec<T>::max(raw[v]));
    return m;
  }
  // Running maximum M2 (log2 units) and sum of 2^(x log2e - M2) of this thread; m: the buffer's maximum. NaN and +inf
  // logits poison the sum.
  __device__ __forceinline__ void sum(float m, float& M2, float& s_run) const {
    const float t2 = m * kLog2eHi;
    if (t2 > M2) {
      s_run *= ex2f(M2 - t2);
      M2 = t2;
    }
    if (!(M2 > -INFINITY)) {  // nothing finite so far: -inf adds nothing, NaN has to be noticed
      float t = 0.f;
#pragma unroll
      for (int v = 0; v < kBufVecs; ++v) {
        float x[VEC];
        Vec<T>::unpack(raw[v], x);
#pragma unroll
        for (int i = 0; i < VEC; ++i) t += x[i];
      }
      if (t != t) s_run = t;
      return;
    }
    // x * log2(e) - M2 with log2(e) in two parts (the product is exact to fp32's last bit and beyond), two logits per
    // instruction
    const unsigned long long hi2 = pack2(kLog2eHi, kLog2eHi), lo2 = pack2(kLog2eLo, kLog2eLo), nm2 = pack2(-M2, -M2);
    unsigned long long acc2 = pack2(0.f, 0.f);
#pragma unroll
    for (int v = 0; v < kBufVecs; ++v) {
      float x[VEC];
      Vec<T>::unpack(raw[v], x);
#pragma unroll
      for (int i = 0; i < VEC; i += 2) {
        const unsigned long long x2 = pack2(x[i], x[i + 1]);
        float e0, e1;
        unpack2(fma2(x2, hi2, fma2(x2, lo2, nm2)), e0, e1);
        acc2 = add2(acc2, pack2(ex2f(e0), ex2f(e1)));
      }
    }
    float a0, a1;
    unpack2(acc2, a0, a1);
    s_run += a0 + a1;
  }
  // Appends what reaches `thr` to the warp's list (all 32 lanes call; `thr` is finite, so padding does not pass).
  // shift: elements of the aligned view before token 0.
  __device__ __forceinline__ void extract(float m, float& thr, int base, int shift, int K, unsigned long long* list, int* count) const {
    if (!__any_sync(0xffffffffu, m >= thr)) return;
    const int lane = threadIdx.x & 31;
    const int have0 = *count;
    __syncwarp();
    // a lane's passing slots as a bit mask, then a loop over its set bits (one round as a rule; unrolled over the slots
    // the code of the empty ones was most of the sweep's): the slot's logit by selects
    uint32_t mask = 0u;
#pragma unroll
    for (int v = 0; v < kBufVecs; ++v) {
      float x[VEC];
      Vec<T>::unpack(raw[v], x);
#pragma unroll
      for (int e = 0; e < VEC; ++e) mask |= x[e] >= thr ? 1u << (v * VEC + e) : 0u;
    }
#pragma unroll 1
    while (mask != 0u) {
      const int i = __ffs(mask) - 1;
      mask &= mask - 1u;
      const int pos = atomicAdd(count, 1);
      if (pos < kListCap) list[pos] = make_key(slot(i), slot_elem(base, i) - shift);
    }
    __syncwarp();
    const int n = *count;
    if (n > kListCap - 16) {
      uint4 copy[kBufVecs];
#pragma unroll
      for (int v = 0; v < kBufVecs; ++v) copy[v] = raw[v];
      thr = OUT ? overflow_call(copy, thr, base, shift, K, list, count, have0, n) : overflow(copy, thr, base, shift, K, list, count, have0, n);
    }
  }
  static __device__ __noinline__ float overflow_call(const uint4 (&buf)[kBufVecs], float thr, int base, int shift, int K,
                                                     unsigned long long* list, int* count, int have0, int n) {
    return overflow(buf, thr, base, shift, K, list, count, have0, n);
  }
  // The list has run over, or will soon: its K best stay, in order; returns the threshold (the K-th, once there are K).
  static __device__ __forceinline__ float overflow(const uint4 (&buf)[kBufVecs], float thr, int base, int shift, int K,
                                                unsigned long long* list, int* count, int have0, int n) {
    const int lane = threadIdx.x & 31;
    unsigned long long mine = 0ull;
    int kept = 0;
    if (n > kListCap) {
      // K rounds of "largest key below the last one taken" over the old list and this buffer; lane r keeps the r-th
      unsigned long long bound = ~0ull;
#pragma unroll 1
      for (int round = 0; round < K; ++round) {
        unsigned long long best = 0ull;
#pragma unroll
        for (int v = 0; v < kBufVecs; ++v) {
          float x[VEC];
          Vec<T>::unpack(buf[v], x);
          const int id = elem(base, v) - shift;
#pragma unroll
          for (int e = 0; e < VEC; ++e)
            if (x[e] >= thr) {
              const unsigned long long k2 = make_key(x[e], id + e);
              if (k2 < bound && k2 > best) best = k2;
            }
        }
#pragma unroll 1
        for (int i = lane; i < have0; i += 32)
          if (list[i] < bound && list[i] > best) best = list[i];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
          const unsigned long long other = __shfl_xor_sync(0xffffffffu, best, o);
          best = other > best ? other : best;
        }
        if (best == 0ull) break;
        if (lane == round) mine = best;
        bound = best;
        ++kept;
      }
    } else {
      kept = keep_best(list, n, K, mine);
    }
    __syncwarp();
    if (lane < kept) list[lane] = mine;
    if (lane == 0) *count = kept;
    if (kept == K) thr = fmaxf(thr, key_value(__shfl_sync(0xffffffffu, mine, K - 1)));
    __syncwarp();
    return thr;
  }
  // The min(n, K) largest of the list's n <= 64 keys, in order, one per lane.
  static __device__ __forceinline__ int keep_best(unsigned long long* list, int n, int K, unsigned long long& mine) {
    const int lane = threadIdx.x & 31;
    const unsigned long long k0 = lane < n ? list[lane] : 0ull, k1 = lane + 32 < n ? list[lane + 32] : 0ull;
    int r0 = 0, r1 = 0;
#pragma unroll 1
    for (int j = 0; j < n; ++j) {
      const unsigned long long kj = list[j];
      r0 += (kj > k0);
      r1 += (kj > k1);
    }
    __syncwarp();
    if (lane < n && r0 < K) list[r0] = k0;
    if (lane + 32 < n && r1 < K) list[r1] = k1;
    __syncwarp();
    const int kept = n < K ? n : K;
    mine = lane < kept ? list[lane] : 0ull;
    return kept;
  }
};

__device__ __forceinline__ float warp_max(float x) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) x = fmaxf(x, __shfl_xor_sync(0xffffffffu, x, o));
  return x;
}
// A thread's share in the groups' maxima, which go to shared memory as integers: the value's ordered bits, the last four
// replaced by the group's number, so that they are distinct and one comparison orders two of them.
__device__ __forceinline__ void group_max(float x, uint32_t* v) {
  x = warp_max(x);
  if ((threadIdx.x & 31) == 0) v[threadIdx.x >> 5] = (ordered_bits(x) & ~15u) | (threadIdx.x >> 5);
}
// The K-th largest of the groups' maxima, rounded down in its last bits: still a lower bound on the K-th largest of the
// logits. At least -FLT_MAX. (Every warp for itself.)
__device__ __forceinline__ float kth_of_groups(const uint32_t* v, int K) {
  const uint32_t mine = v[threadIdx.x & (kGroups - 1)];
  int r = 0;
#pragma unroll
  for (int j = 0; j < kGroups; j += 4) {
    const uint4 o = *reinterpret_cast<const uint4*>(v + j);
    r += (o.x > mine) + (o.y > mine) + (o.z > mine) + (o.w > mine);
  }
  const unsigned who = __ballot_sync(0xffffffffu, r == K - 1);
  return fmaxf(from_ordered_bits(__shfl_sync(0xffffffffu, mine, __ffs(who) - 1) & ~15u), -3.402823466e38f);
}

// MINB = 2 compiles the same code for two CTAs per SM (half the registers): for launches with more CTAs than
// SMs, where a second resident CTA hides the first one's latencies; MINB = 1 is for the short launches.
template <typename T, int MINB>
__global__ void __launch_bounds__(kSweepThreads, MINB) expand_kernel(const ExpandParams p) {
  // filled in the first CTA of the row's cluster by all CTAs of the cluster: chunk c's candidate keys, and per warp of
  // chunk c its maximum (log2 units) and sum of 2^(. - maximum); later the tail's arrays
  constexpr int kWarps = kSweepThreads / 32, kChunkCap = kWarps * kPushCap;
  __shared__ __align__(16) unsigned char scratch[kSweepMaxChunks * kChunkCap * 8 > kTailScratch ? kSweepMaxChunks * kChunkCap * 8 : kTailScratch];
  __shared__ float row_max[kSweepMaxChunks * kWarps];
  __shared__ double row_sum[kSweepMaxChunks * kWarps];
  __shared__ int row_n[kSweepMaxChunks];
  __shared__ float row_bound[kSweepMaxChunks];  // the chunks' thresholds: lower bounds on the row's K-th largest logit
  constexpr int kListMax = kWarps * kListCap;
  __shared__ int rank_s[kListMax], list_n;
  __shared__ __align__(16) unsigned long long wlist[kWarps * kListCap];
  __shared__ unsigned long long topk[CAST_MAX_TOP_K];
  __shared__ int wcount[kWarps];
  __shared__ __align__(16) uint32_t gmax[2][kGroups];
  __shared__ int sorted[kTailSingleMaxB * CAST_MAX_WIDTH];  // small batches: pool indices of the first sorted candidates
  __shared__ int s_flag, push_n;
  __shared__ double s_lse, s_parent_score;
  __shared__ TailState s_ts;
  __shared__ int s_base, s_n_prev, s_parent;
  unsigned long long* row_keys = reinterpret_cast<unsigned long long*>(scratch);

  const int chunk = blockIdx.x, r = blockIdx.y, b = blockIdx.z, B = gridDim.z;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  DevState* st = p.st;
  const int K = p.K;
  const int row = b * p.W + r;
  using S = Sweep<T, MINB == 1>;
  constexpr int E = S::kBufElems;
  // the row from the 16-byte boundary at or below its start: its tokens are elements [shift, V + shift) of that view
  const T* x = reinterpret_cast<const T*>(p.logits) + (size_t)row * p.V;
  const int shift = (int)((reinterpret_cast<uintptr_t>(x) & 15) / sizeof(T));
  const T* xa = x - shift;
  const int begin = chunk * p.chunk_elems;
  const int end = min(begin + p.chunk_elems, p.V + shift);
  if (p.nchunks > 1) cluster_arrive_release();  // (waited for before the first store to another CTA: all of them run by then)
  if (tid < kWarps) wcount[tid] = 0;
  if (tid == 0) push_n = list_n = 0;
  // Programmatic dependent launch: this grid may have become resident while the previous kernel of the
  // stream was still finishing. Nothing that kernel may have written is read above this line - not the
  // logits either: in a serving loop the previous kernel is the draft model's, and it writes them. What a
  // CTA may do is ask the L2 cache for its chunk: a prefetch returns no value, and a line that the previous
  // kernel writes afterwards is written in that same cache, so the loads below see it. When the previous kernel
  // is not the one that writes the logits (layers queued back to back) the first loads then cost a round trip
  // to L2 instead of one to HBM; rows that turn out not to exist are fetched for nothing, hence only for small
  // layers.
  if (p.prefetch) {
    const char* cb = reinterpret_cast<const char*>(chunk == 0 ? x : xa + begin);
    const int bytes = (int)(reinterpret_cast<const char*>(xa + end) - cb);
#pragma unroll 1
    for (int off = tid * 128; off < bytes; off += kSweepThreads * 128)
      asm volatile("prefetch.global.L2 [%0];" ::"l"(cb + off));
  }
  grid_dependency_wait();
  grid_launch_dependents();  // the next grid may now take the SMs this one leaves idle
  // the first logits are requested before the state is read (every row r < W exists in memory): one memory round trip
  S q0, q1;
  const uint4* at_mine = reinterpret_cast<const uint4*>(xa + begin) + tid;  // this thread's place in buffer `at`
  constexpr int kStep = kBufVecs * kSweepThreads;                                       // vectors per buffer
  if (begin >= shift && begin + 2 * E <= end) {
    q0.load(at_mine);
    q1.load(at_mine + kStep);
  } else {
    q0.load_part(xa, begin, shift, end);
    q1.load_part(xa, begin + E, shift, end);
  }
  // what the layer tail needs of the state is read now, together with the row count: one round trip; it waits in shared
  // memory, out of the sweep's registers. (Layer 1 starts the step: one row per sequence, the root at pool index 0 with
  // value 1.)
  {
    int n_prev = 1;
    if (p.layer > 1) n_prev = st->rows[p.layer];
    if (tid == 0) {
      s_ts.ctx_sum = 0;
      s_ts.n0 = 0;  // layer 1: the deciding CTA works it out from kv_len
      s_ts.kept_total = 1;
      s_ts.u_last = 1.0;
      s_base = 1;
      if (p.layer > 1) {
        s_ts.ctx_sum = st->ctx_sum;
        s_ts.n0 = st->n0;
        s_ts.kept_total = st->kept_total;
        s_ts.u_last = st->u_last;
        s_base = st->pool_size;
      }
      s_n_prev = n_prev;
    }
    if (n_prev == 0) {
      if (chunk == 0 && r == 0 && b == 0 && tid == 0) *p.next_count = 0;
      return;
    }
    if (r >= n_prev) return;
    // the parent of this row's children and its log-value
    if (tid == 32 && chunk == 0) {
      const int parent = p.layer > 1 ? p.retained[b * p.W + r] : 0;
      s_parent = parent;
      s_parent_score = p.layer > 1 ? p.pool_score[(size_t)b * p.P + parent] : 0.0;
    }
  }

  // ---- sweep
  unsigned long long* list = wlist + warp * kListCap;
  float m_run = -INFINITY, M2 = -INFINITY, s_run = 0.f, thr = 0.f;
  auto work = [&](S& q, float m, int at, const uint4* mine) {
    q.extract(m, thr, at, shift, K, list, &wcount[warp]);
    if (at + 3 * E <= end) q.load(mine + 2 * kStep);
    else if (at + 2 * E < end) q.load_part(xa, at + 2 * E, shift, end);
  };
  auto threshold = [&](float m, uint32_t* g) {
    group_max(m, g);
    __syncthreads();
    return kth_of_groups(g, K);
  };
#pragma unroll 1
  for (int at = begin; at < end; at += 2 * E, at_mine += 2 * kStep) {  // (two copies of the work: a buffer that is moved is waited for)
    const float m0 = q0.max();
    m_run = fmaxf(m_run, m0);
    q0.sum(m0, M2, s_run);
    // the threshold from the first two buffers, and once more when four of seven buffers or more are done
    if (at == begin) thr = threshold(fmaxf(m0, q1.max()), gmax[0]);
    else if (at == begin + 4 * E && end - at > 2 * E) thr = fmaxf(thr, threshold(m_run, gmax[1]));
    work(q0, m0, at, at_mine);
    if (at + E >= end) break;
    const float m1 = q1.max();
    m_run = fmaxf(m_run, m1);
    q1.sum(m1, M2, s_run);
    work(q1, m1, at + E, at_mine + kStep);
  }

  // ---- chunk result: what is left of the warps' lists above the threshold, and every warp's maximum and sum, straight
  // into the shared memory of the cluster's first CTA, which merges the row
  {
    const float Mw = warp_max(M2);
    double sd = (M2 > -INFINITY) ? (double)s_run * (double)ex2f(M2 - Mw) : (double)s_run;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) sd += __shfl_xor_sync(0xffffffffu, sd, o);
    const int n = wcount[warp];
    unsigned long long k0 = lane < n ? list[lane] : 0ull, k1 = lane + 32 < n ? list[lane + 32] : 0ull;
    if (k0 != 0ull && key_value(k0) < thr) k0 = 0ull;  // (appended before the threshold was raised)
    if (k1 != 0ull && key_value(k1) < thr) k1 = 0ull;
    unsigned m0 = __ballot_sync(0xffffffffu, k0 != 0ull), m1 = __ballot_sync(0xffffffffu, k1 != 0ull);
    if (__popc(m0) + __popc(m1) > kPushCap) {  // (warp-uniform) its K best
      __syncwarp();
      S::keep_best(list, n, K, k0);
      k1 = 0ull;
      m0 = __ballot_sync(0xffffffffu, k0 != 0ull);
      m1 = 0u;
    }
    const int total = __popc(m0) + __popc(m1);
    int pos = 0;
    if (lane == 0 && total > 0) pos = atomicAdd(&push_n, total);
    pos = chunk * kChunkCap + __shfl_sync(0xffffffffu, pos, 0);
    const unsigned below = (1u << lane) - 1u;
    const int p0 = pos + __popc(m0 & below), p1 = pos + __popc(m0) + __popc(m1 & below);
    if (p.nchunks == 1) {
      if (k0 != 0ull) row_keys[p0] = k0;
      if (k1 != 0ull) row_keys[p1] = k1;
      if (lane == 0) {
        row_max[warp] = Mw;
        row_sum[warp] = sd;
      }
      __syncthreads();
      if (tid == 0) {
        row_n[0] = push_n;
        row_bound[0] = thr;
      }
      __syncthreads();
    } else {
      cluster_wait_acquire();
      if (k0 != 0ull) st_cluster_u64(map_to_rank(smem_addr(&row_keys[p0]), 0u), k0);
      if (k1 != 0ull) st_cluster_u64(map_to_rank(smem_addr(&row_keys[p1]), 0u), k1);
      if (lane == 0) {
        st_cluster_f32(map_to_rank(smem_addr(&row_max[chunk * kWarps + warp]), 0u), Mw);
        st_cluster_f64(map_to_rank(smem_addr(&row_sum[chunk * kWarps + warp]), 0u), sd);
      }
      __syncthreads();
      if (tid == 0) {
        st_cluster_u32(map_to_rank(smem_addr(&row_n[chunk]), 0u), (uint32_t)push_n);
        st_cluster_f32(map_to_rank(smem_addr(&row_bound[chunk]), 0u), thr);
      }
      cluster_arrive_release();
      if (chunk != 0) return;  // the results are on their way; the first CTA waits for them
      cluster_wait_acquire();
    }
  }

  // ---- row merge by the first CTA of the row's cluster: the candidates (a dozen or two per chunk) that reach the largest
  // of the chunks' thresholds go side by side, then the last warp forms the log-sum-exp while the others rank them
  const float row_thr = [&] {
    float t = row_bound[0];
#pragma unroll
    for (int c = 1; c < kSweepMaxChunks; ++c) t = c < p.nchunks ? fmaxf(t, row_bound[c]) : t;
    return t;
  }();
  if (tid < K) topk[tid] = 0ull;
  {
    constexpr int kLanes = kSweepThreads / kSweepMaxChunks;  // threads per chunk: whole warps
    static_assert(kLanes % 32 == 0, "a warp looks at one chunk");
    const int c = tid / kLanes, nc = c < p.nchunks ? row_n[c] : 0;
#pragma unroll 1
    for (int i0 = (tid % kLanes) - lane; i0 < nc; i0 += kLanes) {
      const int i = i0 + lane;
      const unsigned long long key = i < nc ? row_keys[c * kChunkCap + i] : 0ull;
      const bool keep = key != 0ull && key_value(key) >= row_thr;
      const unsigned m = __ballot_sync(0xffffffffu, keep);
      int pos = 0;
      if (lane == 0 && m != 0u) pos = atomicAdd(&list_n, __popc(m));
      pos = __shfl_sync(0xffffffffu, pos, 0) + __popc(m & ((1u << lane) - 1u));
      if (keep && pos < kListMax) {
        wlist[pos] = key;
        rank_s[pos] = 0;
      }
    }
  }
  __syncthreads();
  const int total = list_n;
  const bool packed = total <= kListMax;  // (else: ties without number, ranked where they are)
  if (warp == kWarps - 1) {
    constexpr int kPer = kSweepMaxChunks * kWarps / 32;
    float Mv[kPer], Mr = -INFINITY;
    double Sv[kPer], term = 0.0;
#pragma unroll
    for (int i = 0; i < kPer; ++i) {
      const int at = lane + 32 * i;
      const bool in = at < p.nchunks * kWarps;
      Mv[i] = in ? row_max[at] : -INFINITY;
      Sv[i] = in ? row_sum[at] : 0.0;
      Mr = fmaxf(Mr, Mv[i]);
    }
    Mr = warp_max(Mr);
    // weights by the fp32 unit, sums in fp64 (a warp without a finite maximum adds 0, or the NaN it met)
#pragma unroll
    for (int i = 0; i < kPer; ++i) term += Mv[i] > -INFINITY ? Sv[i] * (double)ex2f(Mv[i] - Mr) : Sv[i];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) term += __shfl_xor_sync(0xffffffffu, term, o);
    const double lse = ((double)Mr + fast_log2(term)) * 0.69314718055994530942;
    if (lane == 0) {
      if (!(term > 0.0 && isfinite(lse))) report(st, CAST_ERR_NONFINITE, row);
      s_lse = lse;
    }
  } else if (packed) {
    const int groups = (total + 31) >> 5, nw = kWarps - 1;
    const int sl = share_log(groups, nw), shares = 1 << sl, len = (total + shares - 1) >> sl;
#pragma unroll 1
    for (int w = warp; w < groups << sl; w += nw) {
      const int j0 = (w & (shares - 1)) * len, j1 = min(j0 + len, total), i = (w >> sl) * 32 + lane;
      const unsigned long long key = wlist[i < total ? i : 0];
      int neg = 0;
#pragma unroll 8
      for (int j = j0; j < j1; ++j) {
        const uint2 o = *reinterpret_cast<const uint2*>(wlist + j);
        count_less64(neg, (uint32_t)key, (uint32_t)(key >> 32), o.x, o.y);
      }
      if (i < total) atomicAdd(&rank_s[i], neg);
    }
  } else {
#pragma unroll 1
    for (int c1 = 0; c1 < p.nchunks; ++c1)
#pragma unroll 1
      for (int i = tid; i < row_n[c1]; i += kSweepThreads - 32) {
        const unsigned long long key = row_keys[c1 * kChunkCap + i];
        int cnt = 0;
#pragma unroll 1
        for (int c = 0; c < p.nchunks; ++c)
#pragma unroll 4
          for (int j = 0; j < row_n[c]; ++j) cnt += row_keys[c * kChunkCap + j] > key;
        if (cnt < K) topk[cnt] = key;
      }
  }
  __syncthreads();
  if (packed) {
    for (int i = tid; i < total; i += kSweepThreads)
      if (-rank_s[i] < K) topk[-rank_s[i]] = wlist[i];
    __syncthreads();
  }
  const int base = s_base;
  if (tid < K) {  // the K children join the pool
    const unsigned long long key = topk[tid];
    const float val = key_value(key);
    int tok = key_token(key);
    if (key == 0ull || !(val > -INFINITY) || tok < 0 || tok >= p.V) {  // fewer than K finite logits
      report(st, CAST_ERR_NONFINITE, row);
      tok = 0;
    }
    const size_t o = (size_t)b * p.P;
    const int idx = base + r * K + tid;
    p.pool_score[o + idx] = s_parent_score + ((double)val - s_lse);
    p.pool_token[o + idx] = tok;
    p.pool_parent[o + idx] = s_parent;
    p.pool_depth[o + idx] = p.layer;
    p.pool_kept[o + idx] = 0;
  }

  // ---- layer tail
  __syncthreads();
  const int n_prev = s_n_prev, n_tail = tail_width(p, n_prev);
  const TailState ts = s_ts;
  if (B <= kTailAlwaysSingleB || (B <= kTailSingleMaxB && B * n_prev * K <= kTailSingleCands)) {  // the last CTA of the layer ranks and decides, everything in shared memory
    if (!take_ticket(p.layer_ticket, B * n_prev, &s_flag)) return;
    double* vs = reinterpret_cast<double*>(scratch + 20480);  // [B][CAST_MAX_WIDTH] sorted values
    int* stok = reinterpret_cast<int*>(scratch + 24576);      // [B][CAST_MAX_WIDTH] tokens of the sorted nodes
    const DecideIn d = decide_load(p, ts, B, n_tail);
    tail_rank(p, 0, B, n_tail, n_prev, base, scratch, sorted, stok, vs);
    tail_decide<false>(p, ts, d, B, n_tail, n_prev, base, sorted, stok, vs);
  } else {  // the last CTA of every sequence ranks that sequence; the last of those decides for the batch
    if (!take_ticket(p.seq_ticket + b, n_prev, &s_flag)) return;
    tail_rank(p, b, 1, n_tail, n_prev, base, scratch, p.tail_sorted, p.tail_tok, p.tail_vs);
    // (tail_rank ends with a CTA barrier: the ticket below releases what all threads wrote)
    const DecideIn d = decide_load(p, ts, B, n_tail);
    if (!take_ticket(p.layer_ticket, B, &s_flag)) return;
    tail_decide<true>(p, ts, d, B, n_tail, n_prev, base, p.tail_sorted, p.tail_tok, p.tail_vs);
  }
}

// ------------------------------------------------------------------ rerank + linearise
struct SelectParams {
  const double* pool_score;
  const int32_t* pool_token;
  const int32_t* pool_parent;
  const int32_t* pool_depth;
  const int32_t* lsort;
  const double* lscore;
  DevState* st;
  int P, Ncap, words, m, pool_mode, enable_dr, per_row;
  int list_cap;  // entries of the lists in shared memory: (H + 1) m, rounded up
  double C3;
  DevTable tab;
  double* sel_score;
  double* sel_value;
  int32_t* sel_idx;
  int32_t* tokens;
  int32_t* parent;
  int32_t* depth;
  uint32_t* anc;
  int32_t* pool_idx;
  double* scores;
  int32_t* n_tree;
};

// Phase 1: rank sequence b's pool under (value desc, depth asc, token asc, creation order) and
// publish the best min(pool, m) nodes with their values. The pool is the root plus one sorted list
// per layer (written by the layer tails in exactly that order restricted to the layer), so the rank
// of the k-th node of a list is k plus, for every other list, the number of its nodes that come
// first: a binary search each. Lists are cut to their first m nodes (later ones cannot rank < m), and a node below
// the m-th of any list is passed over. The searches of a node are shared by as many threads as the CTA has to spare.
__device__ __forceinline__ void select_rank_phase(const SelectParams& p, int b, unsigned char* smem) {
  __shared__ int lbase[CAST_MAX_DEPTH + 1], llen[CAST_MAX_DEPTH + 1], loff[CAST_MAX_DEPTH + 2];
  const int tid = threadIdx.x, nt = blockDim.x;
  const size_t o = (size_t)b * p.P;
  const int nl = p.st->layers_done + 1;  // lists: depth 0 (the root) .. layers_done
  if (tid < 32) {  // one memory round trip for all lists
    static_assert(CAST_MAX_DEPTH + 1 <= 32, "a list per lane");
    int len = 0, at = 0;
    if (tid < nl) {
      len = p.pool_mode == 0 ? p.st->layer_n[tid] : p.st->n_hist[tid];
      at = p.st->layer_base[tid];
    }
    len = len > p.m ? p.m : len;
    int incl = len;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
      const int t = __shfl_up_sync(0xffffffffu, incl, d);
      if (tid >= d) incl += t;
    }
    if (tid < nl) {
      llen[tid] = len;
      lbase[tid] = at;
      loff[tid + 1] = incl;
    }
    if (tid == 0) loff[0] = 0;
  }
  const int peff = p.pool_mode == 0 ? p.st->pool_size : p.st->kept_total;  // (needed further down)
  __syncthreads();
  const int total = loff[nl];
  double* ls = reinterpret_cast<double*>(smem);                  // the lists' values, list l at loff[l]
  int* rank_s = reinterpret_cast<int*>(ls + p.list_cap);         // ranks
  unsigned char* lst = reinterpret_cast<unsigned char*>(rank_s + p.list_cap);  // which list
#pragma unroll 1
  for (int i = tid; i < total; i += nt) {
    int l = 0;
    while (i >= loff[l + 1]) ++l;
    ls[i] = p.lscore[o + lbase[l] + (i - loff[l])];
    rank_s[i] = i - loff[l];
    lst[i] = (unsigned char)l;
  }
  __syncthreads();
  const int n_out = min(min(peff, p.m), p.Ncap);
  double bound = -INFINITY;
#pragma unroll 4
  for (int l = 0; l < nl; ++l)
    if (llen[l] >= p.m) bound = fmax(bound, ls[loff[l] + p.m - 1]);
  int parts = 1;  // threads per node, a multiple of four lists each at a time
  while ((parts + 1) * total <= nt && parts < nl) ++parts;
  int half0 = 1;  // first stride of the searches: positions up to 2 half0 - 1 >= the longest list are reachable
  while (2 * half0 - 1 < p.m && half0 < CAST_MAX_TREE) half0 <<= 1;
  int part = 0, i = tid;
  while (i >= total && part < parts) {
    i -= total;
    ++part;
  }
#pragma unroll 1
  for (; part < parts && i < total; i += nt) {  // (more nodes than threads: parts is 1)
    const int l = lst[i];
    const double s = ls[i];
    if (s < bound) {
      if (part == 0) rank_s[i] = 0x40000000;
      continue;
    }
    int before = 0;
    // nodes of another list l2 that come first: value > s, or value == s when their depth is smaller.
    // Lower-bound searches, four lists in lockstep and branch-free so that their loads overlap.
#pragma unroll 1
    for (int l0 = part; l0 < nl; l0 += 4 * parts) {
      int pos[4] = {0, 0, 0, 0}, len4[4], off4[4];
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const int l2 = l0 + q * parts;
        const bool valid = l2 < nl && l2 != l;
        len4[q] = valid ? llen[l2] : 0;
        off4[q] = valid ? loff[l2] : 0;
      }
#pragma unroll 1
      for (int half = half0; half >= 1; half >>= 1) {
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          const int idx = pos[q] + half - 1;
          const bool inb = idx < len4[q];
          const double a = ls[off4[q] + (inb ? idx : 0)];
          const bool first = inb && ((l0 + q * parts < l) ? (a >= s) : (a > s));
          pos[q] += first ? half : 0;
        }
      }
      before += pos[0] + pos[1] + pos[2] + pos[3];
    }
    if (before != 0) atomicAdd(&rank_s[i], before);
  }
  __syncthreads();
#pragma unroll 1
  for (int j = tid; j < total; j += nt) {
    const int rank = rank_s[j];
    if (rank < n_out) {
      const int l = lst[j];
      const double s = ls[j];
      p.sel_score[(size_t)b * p.Ncap + rank] = s;
      p.sel_value[(size_t)b * p.Ncap + rank] = fast_exp_neg(s);
      p.sel_idx[(size_t)b * p.Ncap + rank] = p.lsort[o + lbase[l] + (j - loff[l])];
    }
  }
}

// Phase 2: batch-mean utility, target-cost ratio, Algorithm 1 -> N; then sequence b's tree. Four threads per rank in the
// phases that loop over the ranks (512 threads): with one, those loops were most of this phase.
constexpr int kSelThreads = 512, kSelShares = kSelThreads / CAST_MAX_TREE;
static_assert(kSelShares == 4, "four lanes of a warp share a rank");
__device__ __forceinline__ void select_finalize_phase(const SelectParams& p, int b, int B) {
  __shared__ double u[CAST_MAX_TREE], c[CAST_MAX_TREE];
  __shared__ int kept[CAST_MAX_TREE], lin_parent[CAST_MAX_TREE];
  __shared__ short lin_of[1 + CAST_MAX_TOP_K + (CAST_MAX_DEPTH - 1) * CAST_MAX_WIDTH * CAST_MAX_TOP_K];
  __shared__ int s_N;
  const int tid = threadIdx.x, lane = tid & 31;
  const int rk = tid >> 2, sub = tid & 3;  // this thread's rank (or node) and share
  const size_t o = (size_t)b * p.P;
  const int pool = p.st->pool_size;
  const int peff = p.pool_mode == 0 ? pool : p.st->kept_total;
  int n = min(min(peff, p.m), p.Ncap);
  if (p.enable_dr && p.tab.Ntab < n) n = p.tab.Ntab;
  if (tid == 0) s_N = 1;
  if (p.enable_dr) {
    const int g0 = select_grid(p.st->n0, p.tab.L, p.tab.M);
    const double* f = p.tab.fT + (size_t)(g0 - 1) * p.tab.Ntab;
    if (tid < n) c[tid] = f[tid] / f[0];
  }
  // u_k = sum_{s<=k} v(s), v(s) = batch mean of the rank-s values (Eq. 1), or this sequence's own
  // rank-s value when every sequence sizes its tree by itself. The means first (u doubles as their buffer), then the
  // prefix sums in one warp. (Without the dynamic rerank nothing of this is used.)
  if (p.enable_dr) {
    double a = 0.0;
    if (rk < n) {
      if (p.per_row) {
        a = sub == 0 ? p.sel_value[(size_t)b * p.Ncap + rk] : 0.0;
      } else {
#pragma unroll 16
        for (int bb = sub; bb < B; bb += kSelShares) a += p.sel_value[(size_t)bb * p.Ncap + rk];
      }
    }
    a += __shfl_xor_sync(0xffffffffu, a, 1);
    a += __shfl_xor_sync(0xffffffffu, a, 2);
    if (sub == 0 && rk < n) u[rk] = p.per_row ? a : a / (double)B;
    __syncthreads();
    if (tid < 32) {
      double v[4], run = 0.0;
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        const int s = lane * 4 + e;
        run += s < n ? u[s] : 0.0;
        v[e] = run;
      }
      double incl = run;  // inclusive scan of the lane totals
#pragma unroll
      for (int d = 1; d < 32; d <<= 1) {
        const double t = __shfl_up_sync(0xffffffffu, incl, d);
        if (lane >= d) incl += t;
      }
      const double excl = incl - run;
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        const int s = lane * 4 + e;
        if (s < n) u[s] = excl + v[e];
      }
    }
    __syncthreads();
    bool ok = rk < n;
    const double uj = ok ? u[rk] : 0.0, cj = ok ? c[rk] : 0.0;
#pragma unroll 4
    for (int i = sub; i < rk && i < n; i += kSelShares)
      if ((uj - u[i]) < p.C3 * (cj - c[i])) ok = false;
    const unsigned good = __ballot_sync(0xffffffffu, ok);
    if (sub == 0 && ((good >> (lane & ~3)) & 15u) == 15u) atomicMax(&s_N, rk + 1);
    __syncthreads();
  }
  const int N = p.enable_dr ? s_N : n;
  // linearise: kept nodes in creation order (ascending pool index)
  if (tid < N) kept[tid] = p.sel_idx[(size_t)b * p.Ncap + tid];
  __syncthreads();
  const int pi = rk < N ? kept[rk] : 0;
  int tok = 0, par = -1, dep = 0;
  double score = 0.0;
  if (rk < N && sub == 0) {  // requested now, used once the order is known
    tok = p.pool_token[o + pi];
    par = p.pool_parent[o + pi];
    dep = p.pool_depth[o + pi];
    score = p.pool_score[o + pi];
  }
  int t = 0;
#pragma unroll 4
  for (int j = sub; j < N; j += kSelShares) t += kept[j] < pi;
  t += __shfl_xor_sync(0xffffffffu, t, 1);
  t += __shfl_xor_sync(0xffffffffu, t, 2);
  if (rk < N && sub == 0) lin_of[pi] = (short)t;
  __syncthreads();
  if (rk < N && sub == 0) {
    const int lp = par >= 0 ? (int)lin_of[par] : -1;
    lin_parent[t] = lp;
    const size_t q = (size_t)b * p.Ncap + t;
    p.tokens[q] = tok;
    p.parent[q] = lp;
    p.depth[q] = dep;
    p.pool_idx[q] = pi;
    if (p.scores) p.scores[q] = score;
  }
  __syncthreads();
  if (tid < p.Ncap) {
    uint32_t w[CAST_MAX_TREE / 32] = {0u, 0u, 0u, 0u};
    const size_t q = (size_t)b * p.Ncap + tid;
    if (tid < N) {
      int a = tid, guard = 0;
      while (a >= 0 && a < N && guard++ <= CAST_MAX_DEPTH + 1) {  // walk to the root, one bit per ancestor
        const uint32_t bit = 1u << (a & 31);
#pragma unroll
        for (int k = 0; k < CAST_MAX_TREE / 32; ++k) w[k] |= (a >> 5) == k ? bit : 0u;
        a = lin_parent[a];
      }
    } else {
      p.tokens[q] = -1;
      p.parent[q] = -1;
      p.depth[q] = -1;
      p.pool_idx[q] = -1;
      if (p.scores) p.scores[q] = 0.0;
    }
#pragma unroll
    for (int k = 0; k < CAST_MAX_TREE / 32; ++k)
      if (k < p.words) p.anc[q * p.words + k] = w[k];
  }
  if (tid == 0) {
    p.n_tree[b] = N;
    if (b == 0) p.st->n_tree = N;
  }
}

__global__ void __launch_bounds__(kSelThreads) select_rank_kernel(const SelectParams p) {
  extern __shared__ __align__(16) unsigned char smem[];
  grid_dependency_wait();
  grid_launch_dependents();
  select_rank_phase(p, blockIdx.x, smem);
}
__global__ void __launch_bounds__(kSelThreads) select_finalize_kernel(const SelectParams p) {
  grid_dependency_wait();
  select_finalize_phase(p, blockIdx.x, gridDim.x);
}
__global__ void __launch_bounds__(kSelThreads) select_fused_kernel(const SelectParams p) {  // batch 1: one launch
  extern __shared__ __align__(16) unsigned char smem[];
  grid_dependency_wait();
  select_rank_phase(p, 0, smem);
  __syncthreads();
  select_finalize_phase(p, 0, 1);
}

}  // namespace

// ------------------------------------------------------------------ C-ABI
extern "C" cast_status cast_step_begin(cast_ctx* c, int B, const int32_t* root_token, const int32_t* kv_len,
                                       void* stream) {
  if (!c || !root_token || !kv_len || B < 1) return CAST_ERR_INVALID_ARG;
  if (B > c->cfg.max_batch) return CAST_ERR_CAPACITY;
  const bool need = c->cfg.enable_bp || c->cfg.enable_dp || c->cfg.enable_dr;
  auto it = c->tables->find(B);
  if (it != c->tables->end()) {
    c->cur_table = it->second.dev;
  } else {
    if (need) return CAST_ERR_COST_TABLE;
    c->cur_table = DevTable{1, 1, 1 << 30, nullptr, nullptr};
  }
  c->cur_B = B;
  c->next_layer = 1;
  // Nothing is launched here: the first cast_tree_expand of the step reads root_token and kv_len and resets
  // the per-step state in its own kernel (one launch and one dependent round trip fewer per step).
  c->step_root = root_token;
  c->step_kv_len = kv_len;
  c->tree_inputs_fresh = 1;  // a new step: the engine may have moved the lengths (an attention call decodes afresh)
  (void)stream;
  return CAST_OK;
}

extern "C" cast_status cast_tree_expand(cast_ctx* c, int layer, const void* draft_logits, cast_dtype dtype,
                                        int32_t* next_tokens, int32_t* next_parent_row, int32_t* next_count,
                                        void* stream) {
  if (!c || !draft_logits || !next_tokens || !next_parent_row || !next_count) return CAST_ERR_INVALID_ARG;
  if (dtype != CAST_F32 && dtype != CAST_BF16) return CAST_ERR_DTYPE;
  if (c->cur_B < 1 || layer < 1 || layer > c->cfg.max_depth || layer != c->next_layer) return CAST_ERR_INVALID_ARG;
  c->next_layer = layer + 1;
  const int B = c->cur_B, V = c->cfg.vocab;
  const int rows_per_seq = layer == 1 ? 1 : c->W;
  // A logits row is swept by one cluster of 1 to 8 CTAs. A CTA pays for its fixed phases (prologue, chunk result, cluster
  // barrier and row merge when there is more than one chunk: about 2.5 us, 2 without) and about 2 us per buffer of 64 bytes a
  // thread, whether the buffer is full or not; CTAs beyond one per SM queue up (figures fitted to the measured layer times of
  // the benchmark shapes). The chunk count with the smallest estimate wins: few rows get many short chunks (latency), many
  // rows get few chunks of several full buffers (throughput).
  const int rows = B * rows_per_seq;
  // (a row's aligned view starts up to one vector before the row; V % 8 == 0 keeps every row as aligned as the first)
  const int room = V + (V % 8 != 0 || ((uintptr_t)draft_logits & 15) != 0 ? 7 : 0);
  const int buf_elems = kSweepThreads * 64 / (dtype == CAST_F32 ? 4 : 2);
  int nchunks = 1, chunk_elems = (room + 7) / 8 * 8;
  {
    double best = 1e30;
    for (int n = 1; n <= kSweepMaxChunks; ++n) {
      int ce = ((room + n - 1) / n + 7) / 8 * 8;
      if (n > 1 && ce < 2048) break;  // below this a chunk is all overhead
      const int ne = (room + ce - 1) / ce;
      const int bufs = (ce + buf_elems - 1) / buf_elems;
      const double per_cta = (ne == 1 ? 2.0 : 2.5) + 2.0 * bufs;
      // (a launch a little larger than the machine costs a good part of a second round: the few CTAs left over
      // run while the other SMs idle)
      const double queue = (double)rows * ne / c->num_sms;
      const double cost = per_cta * (queue <= 1.0 ? 1.0 : (queue < 1.5 ? 1.5 : queue));
      if (cost < best - 1e-9) {
        best = cost;
        nchunks = ne;
        chunk_elems = ce;
      }
    }
  }

  ExpandParams p;
  p.logits = draft_logits;
  p.V = V; p.K = c->cfg.top_k; p.W = c->W; p.H = c->cfg.max_depth; p.P = c->P; p.layer = layer;
  p.nchunks = nchunks; p.chunk_elems = chunk_elems;
  // every row that can exist is asked for, whether the previous layer kept it or not: worth it while the
  // whole layer is a small part of the L2 cache
  p.prefetch = (double)rows * V * (dtype == CAST_F32 ? 4 : 2) <= 24e6;
  p.pool_score = c->pool_score; p.pool_token = c->pool_token; p.pool_parent = c->pool_parent;
  p.pool_depth = c->pool_depth; p.pool_kept = c->pool_kept; p.retained = c->retained;
  p.lsort = c->lsort; p.lscore = c->lscore;
  p.st = c->state;
  p.layer_ticket = c->layer_ticket;
  p.seq_ticket = c->seq_ticket; p.tail_vs = c->tail_vs; p.tail_sorted = c->tail_sorted; p.tail_tok = c->tail_tok;
  p.fifo_vals = c->fifo_vals; p.fifo_cnt = c->fifo_cnt; p.R = c->cfg.fifo_len;
  p.tab = c->cur_table;
  p.C1 = c->cfg.C1; p.C2 = c->cfg.C2;
  p.enable_bp = c->cfg.enable_bp; p.enable_dp = c->cfg.enable_dp; p.ctx_base_mode = c->cfg.ctx_base_mode;
  p.next_tokens = next_tokens; p.next_parent_row = next_parent_row; p.next_count = next_count;
  p.root_token = c->step_root; p.kv_len = c->step_kv_len;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(nchunks, rows_per_seq, B);
  const bool queued = (long long)rows * nchunks > c->num_sms;
  cfg.blockDim = dim3(kSweepThreads, 1, 1);
  cfg.dynamicSmemBytes = 0;
  cfg.stream = (cudaStream_t)stream;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = (unsigned)nchunks;  // the chunks of one row
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  // may start before the previous kernel of the stream has drained (the kernel waits where it must)
  attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 2;
  cudaError_t e;
  if (dtype == CAST_F32)
    e = queued ? cudaLaunchKernelEx(&cfg, expand_kernel<float, 2>, p) : cudaLaunchKernelEx(&cfg, expand_kernel<float, 1>, p);
  else
    e = queued ? cudaLaunchKernelEx(&cfg, expand_kernel<__nv_bfloat16, 2>, p)
               : cudaLaunchKernelEx(&cfg, expand_kernel<__nv_bfloat16, 1>, p);
  if (e != cudaSuccess) {
    cudaGetLastError();
    return CAST_ERR_CUDA;
  }
  return CAST_OK;
}

extern "C" cast_status cast_select_nodes(cast_ctx* c, int32_t* tokens, int32_t* parent, int32_t* depth,
                                         uint32_t* anc_mask, int32_t* pool_idx, double* scores, int32_t* n_tree,
                                         void* stream) {
  if (!c || !tokens || !parent || !depth || !anc_mask || !pool_idx || !n_tree) return CAST_ERR_INVALID_ARG;
  if (c->cur_B < 1 || c->next_layer < 2) return CAST_ERR_INVALID_ARG;  // a step with at least one layer
  c->tree_inputs_fresh = 1;  // n_tree and the masks: the next attention call reads them after its dependency wait
  SelectParams p;
  p.pool_score = c->pool_score; p.pool_token = c->pool_token; p.pool_parent = c->pool_parent;
  p.pool_depth = c->pool_depth; p.lsort = c->lsort; p.lscore = c->lscore; p.st = c->state;
  p.P = c->P;
  p.Ncap = c->cfg.max_tree; p.words = c->words; p.m = c->cfg.total_token;
  p.pool_mode = c->cfg.pool_mode; p.enable_dr = c->cfg.enable_dr; p.C3 = c->cfg.C3;
  p.per_row = c->cfg.enable_dr && c->cfg.rerank_per_row;
  p.tab = c->cur_table;
  p.sel_score = c->sel_score; p.sel_value = c->sel_value; p.sel_idx = c->sel_idx;
  p.tokens = tokens; p.parent = parent; p.depth = depth; p.anc = anc_mask; p.pool_idx = pool_idx;
  p.scores = scores; p.n_tree = n_tree;
  // (H + 1) lists of at most m nodes: value, rank, list
  p.list_cap = ((c->cfg.max_depth + 1) * c->cfg.total_token + 15) / 16 * 16;
  const size_t smem = (size_t)p.list_cap * (sizeof(double) + sizeof(int32_t) + 1);
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(c->cur_B, 1, 1);
  cfg.blockDim = dim3(kSelThreads, 1, 1);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = (cudaStream_t)stream;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;  // see cast_tree_expand
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  cudaError_t e;
  if (c->cur_B == 1) {
    e = cudaLaunchKernelEx(&cfg, select_fused_kernel, p);
  } else {
    e = cudaLaunchKernelEx(&cfg, select_rank_kernel, p);
    cfg.dynamicSmemBytes = 0;
    if (e == cudaSuccess) e = cudaLaunchKernelEx(&cfg, select_finalize_kernel, p);
  }
  if (e != cudaSuccess) {
    cudaGetLastError();
    return CAST_ERR_CUDA;
  }
  return CAST_OK;
}
