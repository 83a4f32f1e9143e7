// cast_accept (target argmax sweep + greedy walk) and cast_compact_kv.
#include <math.h>

#include "cast_internal.h"

using namespace cast;

namespace {

constexpr int kArgThreads = 256;
constexpr int kArgUnroll = 8;

// One CTA per (chunk, tree token, sequence): the largest (logit, lowest token id) of the chunk. (Consecutive CTAs
// sweep consecutive memory; with the token index slowest, so that the rows past the trees come last, the large
// batches lost a sixth of their bandwidth.)
// Bound by memory once a logit costs little: a thread takes the maximum of a whole 16-byte vector (packed maxima for
// bf16: about one instruction per logit), keeps the raw vector that holds its best, and only the CTA's winner looks for
// the element in it at the end. With a compare and two selects per unpacked logit the bf16 sweep ran at 2.6 TB/s.
// A row whose start is not 16-byte aligned (an odd vocabulary) is swept from the boundary below it: element v of the
// aligned view is token v - shift, and only the vectors at the row's two ends are assembled element by element.
// (Those apart from the rest, and whole rounds without tests: with the assembly inside the unrolled loop the fp32 sweep took
// 102 registers, two CTAs per SM instead of four, and 1.2 GB of logits 223 us instead of 170.)
template <typename T>
__global__ void __launch_bounds__(kArgThreads) argmax_sweep_kernel(const T* __restrict__ logits, int V, int Ncap,
                                                                   int chunk_elems, const int32_t* __restrict__ n_tree,
                                                                   unsigned long long* __restrict__ part) {
  __shared__ unsigned long long red[kArgThreads / 32];
  const int chunk = blockIdx.x, t = blockIdx.y, b = blockIdx.z;
  // the walk kernel that follows may become resident now (it waits for this grid before it reads the winners)
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  if (t >= n_tree[b]) return;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const size_t row = (size_t)b * Ncap + t;
  const T* x = logits + row * V;
  constexpr int VEC = Vec<T>::N;
  const int shift = (int)((reinterpret_cast<uintptr_t>(x) & 15) / sizeof(T));
  const T* xa = x - shift;  // 16-byte aligned; token id = element - shift
  const int begin = chunk * chunk_elems;
  const int end = min(begin + chunk_elems, V + shift);
  const uint32_t none = Vec<T>::kMinusInf;
  float best = -INFINITY;
  int bvec = -1;  // first element of the best vector
  uint4 braw = make_uint4(none, none, none, none);
  for (int base = begin; base < end; base += kArgThreads * VEC * kArgUnroll) {
    uint4 raw[kArgUnroll];
    if (base >= shift && base + kArgThreads * VEC * kArgUnroll <= end) {  // a whole round: nothing to test per vector
#pragma unroll
      for (int v = 0; v < kArgUnroll; ++v) raw[v] = __ldcs(reinterpret_cast<const uint4*>(xa + base + (v * kArgThreads + tid) * VEC));
    } else {
#pragma unroll
      for (int v = 0; v < kArgUnroll; ++v) {
        const int idx = base + (v * kArgThreads + tid) * VEC;
        raw[v] = make_uint4(none, none, none, none);
        if (idx >= shift && idx + VEC <= end) raw[v] = __ldcs(reinterpret_cast<const uint4*>(xa + idx));
      }
#pragma unroll 1
      for (int v = 0; v < kArgUnroll; ++v) {  // at most one vector at each end of the row
        const int idx = base + (v * kArgThreads + tid) * VEC;
        if (idx >= end || (idx >= shift && idx + VEC <= end)) continue;
        uint4 a = make_uint4(none, none, none, none);
#pragma unroll
        for (int e = 0; e < VEC; ++e)
          if (idx + e >= shift && idx + e < end) Vec<T>::put(a, e, to_float(xa[idx + e]));
        const float m = Vec<T>::max(a);
        if (m > best || (m == best && idx < bvec)) {
          best = m;
          bvec = idx;
          braw = a;
        }
      }
    }
#pragma unroll
    for (int v = 0; v < kArgUnroll; ++v) {
      const float m = Vec<T>::max(raw[v]);
      const int idx = base + (v * kArgThreads + tid) * VEC;
      if (m > best || (m == best && idx < bvec)) {  // (bvec is past idx where an end's vector came first)
        best = m;
        bvec = idx;
        braw = raw[v];
      }
    }
  }
  const unsigned long long mine = bvec >= 0 ? make_key(best, bvec) : 0ull;
  unsigned long long key = mine;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const unsigned long long other = __shfl_xor_sync(0xffffffffu, key, o);
    key = other > key ? other : key;
  }
  if (lane == 0) red[warp] = key;
  __syncthreads();
#pragma unroll
  for (int w = 0; w < kArgThreads / 32; ++w) key = red[w] > key ? red[w] : key;
  // vectors are distinct, so the winner is one thread (nobody, in a chunk without a finite logit)
  if (key == 0ull ? tid == 0 : key == mine) {
    int id = bvec - shift;
#pragma unroll
    for (int e = VEC - 1; e >= 0; --e)
      if (Vec<T>::get(braw, e) == best) id = bvec - shift + e;
    part[row * kAcceptMaxChunks + chunk] = key == 0ull ? 0ull : make_key(best, id);
  }
}

// One CTA per sequence: merge the chunk winners into g[t], then walk from the root.
__global__ void __launch_bounds__(CAST_MAX_TREE) accept_walk_kernel(
    const unsigned long long* __restrict__ part, int nchunks, int Ncap, int Nmax, int H, const int32_t* __restrict__ tokens,
    const int32_t* __restrict__ parent, const int32_t* __restrict__ n_tree, int32_t* __restrict__ accept_len,
    int32_t* __restrict__ accept_path, int32_t* __restrict__ bonus, DevState* st) {
  __shared__ int g[CAST_MAX_TREE], tok[CAST_MAX_TREE], par[CAST_MAX_TREE];
  const int b = blockIdx.x, t = threadIdx.x, lane = t & 31;
  int N = n_tree[b];
  if (N > Nmax) N = 0;  // rows past Nmax were not swept: refused like an empty tree
  if (N < 1) {
    if (t == 0) {
      report(st, CAST_ERR_BAD_TREE, b);
      accept_len[b] = 0;
      bonus[b] = 0;
      for (int j = 0; j <= H; ++j) accept_path[b * (H + 1) + j] = -1;
    }
    asm volatile("griddepcontrol.wait;" ::: "memory");  // (the launch must not be over before the sweep is)
    return;
  }
  // the tree arrays were written before the sweep was launched; the sweep's winners are read after the wait
  // (programmatic dependent launch: this grid may be resident while the sweep still runs; a no-op otherwise)
  int tok_mine = 0, par_mine = -1;
  if (t < N) {
    tok_mine = tokens[(size_t)b * Ncap + t];
    par_mine = parent[(size_t)b * Ncap + t];
  }
  asm volatile("griddepcontrol.wait;" ::: "memory");
  if (t < N) {
    unsigned long long key = 0ull;
    for (int c = 0; c < nchunks; ++c) {
      const unsigned long long k = part[((size_t)b * Ncap + t) * kAcceptMaxChunks + c];
      key = k > key ? k : key;
    }
    g[t] = key ? key_token(key) : 0;
    tok[t] = tok_mine;
    par[t] = par_mine;
    if ((t == 0 && par[t] != -1) || (t > 0 && (par[t] < 0 || par[t] >= t))) report(st, CAST_ERR_BAD_TREE, b * Ncap + t);
  }
  __syncthreads();
  if (t >= 32) return;
  int cur = 0, len = 0;
  if (lane == 0) accept_path[b * (H + 1)] = 0;
  while (true) {
    const int want = g[cur];
    int found = 0x7fffffff;
    for (int c = lane; c < N; c += 32)
      if (par[c] == cur && tok[c] == want) {
        found = c;
        break;
      }
    found = __reduce_min_sync(0xffffffffu, found);
    if (found == 0x7fffffff) break;
    if (len == H || found <= cur) {  // deeper than the path buffer, or not a forward edge
      if (lane == 0) report(st, CAST_ERR_BAD_TREE, b * Ncap + found);
      break;
    }
    cur = found;
    ++len;
    if (lane == 0) accept_path[b * (H + 1) + len] = cur;
  }
  if (lane == 0) {
    for (int j = len + 1; j <= H; ++j) accept_path[b * (H + 1) + j] = -1;
    accept_len[b] = len;
    bonus[b] = g[cur];
  }
}

// ------------------------------------------------------------------ compaction
constexpr int kCompactThreads = 256;
constexpr int kMaxPath = CAST_MAX_DEPTH + 1;

struct CompactParams {
  char* k;
  char* v;
  size_t layer_stride;
  int row_bytes, page_size, seq_capacity, num_pages, H1;  // row_bytes: one position, all kv-heads
  const int32_t* page_table;
  const int32_t* accept_path;
  const int32_t* accept_len;
  int32_t* kv_len;
  int32_t* ticket;
  DevState* st;
};

// Slot of position `pos` of sequence b, or -1 for a page id out of range.
__device__ __forceinline__ long long cache_slot(const CompactParams& p, int b, int pos) {
  if (p.page_size == 0) return (long long)b * p.seq_capacity + pos;
  const int page = p.page_table[(size_t)b * p.seq_capacity + pos / p.page_size];
  return page < 0 || page >= p.num_pages ? -1 : (long long)page * p.page_size + pos % p.page_size;
}

// One CTA per (layer, sequence, up to 256 16-byte columns of the position rows of K and V). A position's heads are
// contiguous in memory, so a row is copied whole: with a CTA per kv-head, 4096 CTAs of a few hundred bytes each, the
// launch of 32 layers at batch 16 took 28 us; this one is bound by three dependent round trips (lengths and path, page
// ids, the rows). The destinations and sources of the sequence are worked out once per CTA, one path entry per
// lane; a row that is already in place (path 0, 1, 2, ...: the usual case of the root) is not touched.
// Column by column the copy is safe in any order of the stores: a path entry is no smaller than its place, so a
// destination slot is never the source of a later entry, and all loads come before the stores.
__global__ void __launch_bounds__(kCompactThreads) compact_kernel(const CompactParams p) {
  __shared__ long long src_s[kMaxPath], dst_s[kMaxPath];
  __shared__ int n_moves;
  const int layer = blockIdx.y, b = blockIdx.z, tid = threadIdx.x;
  asm volatile("griddepcontrol.wait;" ::: "memory");
  const int L = p.kv_len[b];
  bool bad = false;
  int a = 0;
  if (tid < 32) {
    a = p.accept_len[b];
    const int src = tid < p.H1 ? p.accept_path[b * p.H1 + tid] : 0;
    a = a < 0 ? 0 : (a > p.H1 - 1 ? p.H1 - 1 : a);
    const int max_pos = p.page_size == 0 ? p.seq_capacity : p.seq_capacity * p.page_size;
    long long from = 0, to = 0;
    if (tid <= a) {
      // a path element is a tree index no smaller than its place on the path (parents precede children), so
      // the destination L + j never lies past the source; anything else is a malformed path
      bad = L < 0 || src < tid || L + src >= max_pos;
      if (!bad) {
        from = cache_slot(p, b, L + src);
        to = cache_slot(p, b, L + tid);
        bad = from < 0 || to < 0;
      }
    }
    const unsigned moves = __ballot_sync(0xffffffffu, tid <= a && from != to);
    if (tid <= a && from != to) {
      const int at = __popc(moves & ((1u << tid) - 1u));
      src_s[at] = from;
      dst_s[at] = to;
    }
    if (tid == 0) n_moves = __popc(moves);
  }
  const int any_bad = __syncthreads_or(bad ? 1 : 0);
  if (tid == 0) {
    if (any_bad) report(p.st, CAST_ERR_BAD_PAGE, b);
    // every CTA of the sequence has read kv_len[b] once all have taken the ticket: the last one publishes the new length
    // (the rows themselves are the next kernel's business, which starts after this grid)
    const int t = atomicAdd(&p.ticket[b], 1);
    if (t == (int)(gridDim.x * gridDim.y) - 1) {
      p.ticket[b] = 0;
      if (!any_bad) p.kv_len[b] = L + a + 1;
    }
  }
  const int cols = p.row_bytes / 16;
  const int i = blockIdx.x * kCompactThreads + tid, n = n_moves;
  if (any_bad || i >= 2 * cols) return;
  char* base = (i < cols ? p.k : p.v) + (size_t)layer * p.layer_stride + (size_t)(i < cols ? i : i - cols) * 16;
  uint4 buf[kMaxPath];
#pragma unroll
  for (int j = 0; j < kMaxPath; ++j)
    if (j < n) buf[j] = *reinterpret_cast<const uint4*>(base + src_s[j] * p.row_bytes);
#pragma unroll
  for (int j = 0; j < kMaxPath; ++j)
    if (j < n) *reinterpret_cast<uint4*>(base + dst_s[j] * p.row_bytes) = buf[j];
}

// Elements per chunk when a row of V logits is swept in (about) nchunks chunks, which is updated. A row's aligned view
// starts up to one vector before the row (V % 8 == 0 keeps every row as aligned as the first).
int sweep_chunk(const void* logits, int V, int& nchunks) {
  const int room = V + (V % 8 != 0 || ((uintptr_t)logits & 15) != 0 ? 7 : 0);
  const int elems = ((room + nchunks - 1) / nchunks + 7) / 8 * 8;
  nchunks = (room + elems - 1) / elems;
  return elems;
}

}  // namespace

extern "C" cast_status cast_accept(cast_ctx* c, const void* target_logits, cast_dtype dtype, int B,
                                   const int32_t* tokens, const int32_t* parent, const int32_t* depth,
                                   const uint32_t* anc_mask, const int32_t* n_tree, int32_t* accept_len,
                                   int32_t* accept_path, int32_t* bonus_token, void* stream) {
  (void)depth;
  (void)anc_mask;
  if (!c || !target_logits || !tokens || !parent || !n_tree || !accept_len || !accept_path || !bonus_token || B < 1)
    return CAST_ERR_INVALID_ARG;
  if (dtype != CAST_F32 && dtype != CAST_BF16) return CAST_ERR_DTYPE;
  if (B > c->cfg.max_batch) return CAST_ERR_CAPACITY;
  const int V = c->cfg.vocab, Ncap = c->cfg.max_tree;
  // Chunks per logits row: enough CTAs to keep four per SM streaming when every sequence verifies its full
  // budget (the context's total_token; the row slots beyond a tree exit at once), and never chunks of more
  // than 32 K logits, so that a batch whose trees came out far below the budget still has several live CTAs
  // per SM; at least 4096 logits per chunk.
  const int budget = c->cfg.total_token < Ncap ? c->cfg.total_token : Ncap;
  int nchunks = (4 * c->num_sms + B * budget - 1) / (B * budget);
  if (nchunks < (V + 32767) / 32768) nchunks = (V + 32767) / 32768;
  if (nchunks > kAcceptMaxChunks) nchunks = kAcceptMaxChunks;
  if (nchunks > V / 4096) nchunks = V / 4096;
  if (nchunks < 1) nchunks = 1;
  // A CTA sweeps its chunk in rounds of kArgThreads * kArgUnroll vectors, each a full memory latency whether
  // the round is full or not: among the counts within two of the one above, the one whose last round is
  // fullest (V = 128 256 fp32 at batch 1: 8 chunks of 1.96 rounds instead of 10 of 1.57, 10.3 -> 9.4 us).
  {
    const int round_elems = kArgThreads * kArgUnroll * (dtype == CAST_F32 ? 4 : 8);
    const int lo = (V + 32767) / 32768 > nchunks - 2 ? (V + 32767) / 32768 : nchunks - 2;
    int hi = nchunks + 2 < kAcceptMaxChunks ? nchunks + 2 : kAcceptMaxChunks;
    if (hi > V / 4096) hi = V / 4096;
    const int n0 = nchunks;
    long long best = -1;
    for (int n = lo < 1 ? 1 : lo; n <= hi; ++n) {
      const int ce = ((V + n - 1) / n + 7) / 8 * 8;
      const long long padded = (long long)((ce + round_elems - 1) / round_elems) * round_elems * n;  // logits' worth of rounds
      const int dist = n > n0 ? n - n0 : n0 - n, dist_best = nchunks > n0 ? nchunks - n0 : n0 - nchunks;
      if (best < 0 || padded < best || (padded == best && dist <= dist_best)) {  // ties: nearest to n0, the larger of two
        best = padded;
        nchunks = n;
      }
    }
  }
  const int chunk_elems = sweep_chunk(target_logits, V, nchunks);
  cudaStream_t s = (cudaStream_t)stream;
  const dim3 grid(nchunks, budget, B);  // rows a tree of this context can have; a larger n_tree is BAD_TREE
  if (dtype == CAST_F32)
    argmax_sweep_kernel<float><<<grid, kArgThreads, 0, s>>>((const float*)target_logits, V, Ncap, chunk_elems, n_tree,
                                                            c->acc_part);
  else
    argmax_sweep_kernel<__nv_bfloat16><<<grid, kArgThreads, 0, s>>>((const __nv_bfloat16*)target_logits, V, Ncap,
                                                                    chunk_elems, n_tree, c->acc_part);
  {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(B, 1, 1);
    cfg.blockDim = dim3(CAST_MAX_TREE, 1, 1);
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;  // resident while the sweep drains
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    const unsigned long long* part = c->acc_part;
    const int H = c->cfg.max_depth;
    DevState* st = c->state;
    if (cudaLaunchKernelEx(&cfg, accept_walk_kernel, part, nchunks, Ncap, budget, H, tokens, parent, n_tree, accept_len,
                           accept_path, bonus_token, st) != cudaSuccess) {
      cudaGetLastError();
      return CAST_ERR_CUDA;
    }
  }
  return launch_status();
}

// ---- cast_accept_static: the acceptance step for callers that must not allocate ----------------
// Scratch for the chunk winners of the target argmax sweep. It lives in the library image: every GPU
// that loads the library holds these 512 KB until the process exits.
constexpr int kStaticAcceptRows = 2048;  // B * Ncap at most
static __device__ __align__(256) unsigned long long g_accept_static_scratch[kStaticAcceptRows * kAcceptMaxChunks];
// The walk kernel records a malformed tree in a state block. Without a context there is none, so the
// record goes to this one, which nobody reads (first record sticks; it never needs clearing).
static __device__ __align__(256) cast::DevState g_accept_static_sink;

namespace {
// Device address of the scratch array, looked up once per device. In host code the array's name is
// only a stand-in for the symbol; the address a kernel can use comes from cudaGetSymbolAddress.
cast_status static_scratch_address(unsigned long long** out, DevState** sink) {
  constexpr int kMaxDevices = 64;
  static unsigned long long* addr[kMaxDevices] = {nullptr};
  static DevState* sink_addr[kMaxDevices] = {nullptr};
  int dev = -1;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) return CAST_ERR_CUDA;
  if (addr[dev] == nullptr || sink_addr[dev] == nullptr) {
    void* p = nullptr;
    void* q = nullptr;
    if (cudaGetSymbolAddress(&p, g_accept_static_scratch) != cudaSuccess || p == nullptr) return CAST_ERR_CUDA;
    if (cudaGetSymbolAddress(&q, g_accept_static_sink) != cudaSuccess || q == nullptr) return CAST_ERR_CUDA;
    addr[dev] = static_cast<unsigned long long*>(p);
    sink_addr[dev] = static_cast<DevState*>(q);
  }
  *out = addr[dev];
  *sink = sink_addr[dev];
  return CAST_OK;
}
}  // namespace

extern "C" cast_status cast_accept_static(const void* target_logits, cast_dtype dtype, int B, int n_cap, int vocab,
                                          int max_depth, const int32_t* tokens, const int32_t* parent,
                                          const int32_t* n_tree, int32_t* accept_len, int32_t* accept_path,
                                          int32_t* bonus_token, void* stream) {
  if (!target_logits || !tokens || !parent || !n_tree || !accept_len || !accept_path || !bonus_token || B < 1 ||
      n_cap < 1 || vocab < 1 || max_depth < 1)
    return CAST_ERR_INVALID_ARG;
  if (dtype != CAST_F32 && dtype != CAST_BF16) return CAST_ERR_DTYPE;
  if (n_cap > CAST_MAX_TREE || max_depth > CAST_MAX_DEPTH || (long long)B * n_cap > kStaticAcceptRows)
    return CAST_ERR_CAPACITY;
  unsigned long long* scratch = nullptr;
  DevState* sink = nullptr;
  const cast_status st = static_scratch_address(&scratch, &sink);
  if (st != CAST_OK) return st;
  int num_sms = 0, dev = 0;
  CAST_CUDA_OK(cudaGetDevice(&dev));
  CAST_CUDA_OK(cudaDeviceGetAttribute(&num_sms, cudaDevAttrMultiProcessorCount, dev));
  int nchunks = (4 * num_sms + B * n_cap - 1) / (B * n_cap);
  if (nchunks > kAcceptMaxChunks) nchunks = kAcceptMaxChunks;
  if (nchunks > vocab / 4096) nchunks = vocab / 4096;
  if (nchunks < 1) nchunks = 1;
  const int chunk_elems = sweep_chunk(target_logits, vocab, nchunks);
  cudaStream_t s = (cudaStream_t)stream;
  const dim3 grid(nchunks, n_cap, B);
  // every chunk winner that the walk reads is written by this call's sweep first: nothing to clear
  if (dtype == CAST_F32)
    argmax_sweep_kernel<float><<<grid, kArgThreads, 0, s>>>((const float*)target_logits, vocab, n_cap, chunk_elems,
                                                            n_tree, scratch);
  else
    argmax_sweep_kernel<__nv_bfloat16><<<grid, kArgThreads, 0, s>>>((const __nv_bfloat16*)target_logits, vocab, n_cap,
                                                                    chunk_elems, n_tree, scratch);
  accept_walk_kernel<<<B, CAST_MAX_TREE, 0, s>>>(scratch, nchunks, n_cap, n_cap, max_depth, tokens, parent, n_tree, accept_len,
                                                 accept_path, bonus_token, sink);
  return launch_status();
}

extern "C" cast_status cast_compact_kv(cast_ctx* c, void* k_cache, void* v_cache, cast_dtype dtype, int B,
                                       int n_layers, size_t layer_stride_bytes, int Hkv, int D, int page_size,
                                       const int32_t* page_table, int seq_capacity, int num_pages,
                                       const int32_t* accept_path, const int32_t* accept_len, int32_t* kv_len,
                                       void* stream) {
  if (!c || !k_cache || !v_cache || !accept_path || !accept_len || !kv_len || B < 1 || n_layers < 1 || Hkv < 1 ||
      D < 1 || page_size < 0 || seq_capacity < 1 || (page_size > 0 && (!page_table || num_pages < 1)))
    return CAST_ERR_INVALID_ARG;
  if (dtype != CAST_F32 && dtype != CAST_BF16) return CAST_ERR_DTYPE;
  if (B > c->cfg.max_batch) return CAST_ERR_CAPACITY;
  const int row_bytes = D * (dtype == CAST_F32 ? 4 : 2);
  if (row_bytes % 16 != 0) return CAST_ERR_SHAPE;
  if (((uintptr_t)k_cache | (uintptr_t)v_cache | layer_stride_bytes) & 15) return CAST_ERR_SHAPE;
  const int H1 = c->cfg.max_depth + 1;
  c->tree_inputs_fresh = 1;  // kv_len and cache rows: an attention call that follows reads them after its dependency wait
  CompactParams p;
  p.k = (char*)k_cache; p.v = (char*)v_cache; p.layer_stride = layer_stride_bytes;
  p.row_bytes = Hkv * row_bytes; p.page_size = page_size; p.seq_capacity = seq_capacity;
  p.num_pages = num_pages; p.H1 = H1;
  p.page_table = page_table; p.accept_path = accept_path; p.accept_len = accept_len; p.kv_len = kv_len;
  p.ticket = c->compact_ticket; p.st = c->state;
  const int cols = 2 * (p.row_bytes / 16);
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((cols + kCompactThreads - 1) / kCompactThreads, n_layers, B);
  cfg.blockDim = dim3(kCompactThreads, 1, 1);
  cfg.stream = (cudaStream_t)stream;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;  // launched while the walk finishes; waits for it
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  if (cudaLaunchKernelEx(&cfg, compact_kernel, p) != cudaSuccess) {
    cudaGetLastError();
    return CAST_ERR_CUDA;
  }
  return CAST_OK;
}
