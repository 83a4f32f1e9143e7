// cast_accept_stochastic: acceptance at temperature T > 0 (Sec. "Speculative Decoding": a draft token with
// draft probability q and target probability p is accepted iff u <= min(1, p/q); after a rejection the
// target distribution is replaced by the residual norm(max(0, P_T - P_D))), walked over the draft tree.
//
// One thread-block cluster per sequence walks the accepted path. At a node every warp of the cluster holds a
// contiguous segment of the vocabulary: it reads the segment's target and draft logits once, keeps exp(logit / T) of
// both in fp64 (target: registers, draft: shared memory), and the warps hand their partial sums to every CTA of the
// cluster through distributed shared memory. The j-th residual has the closed form
//     P_j(x) = max(0, P_T(x) - a_j P_D(x)) / F_j,   a_0 = 0, F_0 = 1, a_{j+1} = a_j + F_j, F_j = F(a_j),
//     F(a) = sum_x max(0, P_T(x) - a P_D(x)),
// (by induction: max(0, max(0, s - a q)/F - q) = max(0, s - (a + F) q)/F), so a rejection costs one sweep
// over the cached segments plus one cluster-wide sum, and the test of a child x is
//     u * P_D(x) * F_j <= max(0, P_T(x) - a_j P_D(x)).
// All arithmetic is fp64: the bonus token is an inverse-CDF sample over up to 150k tokens, where fp32
// rounding would move the result in about one draw of a hundred.
// Every warp of a cluster computes the same decisions from the same numbers (sums are taken in one fixed order),
// so the control flow, and with it the sequence of cluster barriers, is uniform across the cluster.
//
// What bounds it: fp64 issue in the exponentials (64 lanes per SM: 2 V / cluster-size of them per node and CTA at about
// a dozen fp64 instructions each; with the rest of an exponential 3.1 us a node at V = 128256 and 16 CTAs, 6.4 with 8) and
// the chain of cluster-wide sums (about 1.2 us each). Hence: no pass for the maximum (fp64 has the exponent range to sum
// exp(logit / T) as it is; the row is evaluated again against its maximum only if the sum leaves 1e-280 .. 1e280), one
// exchange per node and per rejection and none for the bonus token, whose segment sums are those of the last exchange.
// Measured alone (T = 0.8, trees of 24, fp32, means over three or four sets of trees; before the exponentials went side by
// side -> now): V = 128256 1 sequence 32.3 -> 28.3 us, 8 67.3 -> 58.2, 16 84.6 -> 74.9; V = 32000 16 sequences 37.7 -> 35.2;
// all but 50 tokens of a row ruled out, V = 128256, 16 sequences 86.6 -> 87.3.
#include <math.h>

#include "cast_internal.h"

using namespace cast;

namespace {

constexpr int kStoThreads = 512;
constexpr int kStoWarps = kStoThreads / 32;
constexpr int kStoMaxCluster = 16;
constexpr int kStoInFlight = 8;  // logits of a row that a lane has in flight and exponentials that it works on side by side
// Vocabulary entries per CTA up to which the plan caches segments (196 608 tokens in clusters of 16): the rule that
// cast_accept_stochastic_plan has always answered by, set when a slice of both rows filled shared memory. The kernels hold
// up to 38 x 512 entries now, so the times do not cross here: V = 262144, one sequence, 76 us recomputing and 41 cached.
constexpr int kStoMaxSlice = 12288;

struct StoParams {
  const void* target_logits;
  const void* draft_logits;
  int V, Ncap, max_depth, ne, cs;  // ne: elements per lane; a CTA's slice is ne * kStoThreads
  double inv_T, T;
  double c_hi, c_lo;  // 32 / (T ln2) in two parts
  const int32_t* tokens;
  const int32_t* parent;
  const int32_t* n_tree;
  const double* u_accept;
  const double* u_bonus;
  int32_t* accept_len;
  int32_t* accept_path;
  int32_t* bonus_token;
  DevState* st;
};

__device__ __forceinline__ uint32_t sto_smem_addr(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ void sto_st_remote_f64x2(const double* local, uint32_t rank, double v0, double v1) {
  uint32_t ra;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(ra) : "r"(sto_smem_addr(local)), "r"(rank));
  asm volatile("st.shared::cluster.v2.f64 [%0], {%1, %2};" ::"r"(ra), "d"(v0), "d"(v1) : "memory");
}
__device__ __forceinline__ void sto_cluster_sync() {
  asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
  asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}

// exp(x) for x <= 700 in fp64 to about 3e-16 relative: x = n ln2 + r with n = round(x log2 e) (ln2 split in
// two so that n ln2_hi is exact: the split of fdlibm's e_exp.c), the degree-12 Taylor polynomial of e^r on |r| <= ln2 / 2 (remainder below
// 2e-16), scaling by 2^n through the exponent field. Arguments below -708 (results near the subnormal
// range) give 0; NaN gives NaN. For the values computed one at a time.
__device__ __forceinline__ double sto_exp_any(double x) {
  const double xin = x;
  x = fmax(x, -708.0);
  const double kMagic = 6755399441055744.0;  // 1.5 * 2^52: adding it rounds to an integer in the low word
  const double tn = fma(x, 1.4426950408889634074, kMagic);
  const int n = __double2loint(tn);
  const double nd = tn - kMagic;
  double r = fma(nd, -6.93147180369123816490e-01, x);
  r = fma(nd, -1.90821492927058770002e-10, r);
  double y = 2.08767569878680989792e-09;  // 1/12!
  y = fma(y, r, 2.50521083854417187751e-08);
  y = fma(y, r, 2.75573192239858906526e-07);
  y = fma(y, r, 2.75573192239858906526e-06);
  y = fma(y, r, 2.48015873015873015873e-05);
  y = fma(y, r, 1.98412698412698412698e-04);
  y = fma(y, r, 1.38888888888888888889e-03);
  y = fma(y, r, 8.33333333333333333333e-03);
  y = fma(y, r, 4.16666666666666666667e-02);
  y = fma(y, r, 1.66666666666666666667e-01);
  y = fma(y, r, 0.5);
  y = fma(y, r, 1.0);
  y = fma(y, r, 1.0);
  const double res = __hiloint2double(__double2hiint(y) + n * 1048576, __double2loint(y));
  return xin >= -708.0 ? res : (xin != xin ? xin : 0.0);
}

// A row's reference and the logits between which exp(logit / T - ref) keeps to the exponent range (fp32: they only have
// to be right within a few units of the exponent).
struct StoRef {
  double ref;
  float lo, hi;
  __device__ __forceinline__ StoRef(double r, double T) : ref(r) {
    lo = (float)fmax((r - 690.0) * T, -3e38);
    hi = (float)fmin((r + 690.0) * T, 3e38);
  }
};

// exp(logit / T - ref) to the same accuracy: x = (32 n + j) ln2/32 + r, |r| <= ln2/64, e^x = 2^n * tab[j] * (degree-6
// Taylor polynomial of e^r, remainder below 4e-18), tab[j] = 2^(j/32) held by lane j and fetched by shuffle (a table in
// shared memory is a gather with four-way bank conflicts; 32 lanes must call). Twelve fp64 instructions; the range tests
// are fp32: below r.lo the result is 0, above r.hi, or for NaN, infinity, which sends the caller to another reference.
__device__ __forceinline__ double sto_exp_row(float logit, const StoRef& row, double inv_T, double tab) {
  const float lc = fminf(fmaxf(logit, row.lo), row.hi);
  const double x = fma((double)lc, inv_T, -row.ref);
  const double kMagic = 6755399441055744.0;
  const double tn = fma(x, 32.0 * 1.4426950408889634074, kMagic);
  const int k = __double2loint(tn);  // round(x * 32 / ln2)
  const double kd = tn - kMagic;
  double r = fma(kd, -6.93147180369123816490e-01 / 32.0, x);
  r = fma(kd, -1.90821492927058770002e-10 / 32.0, r);
  double y = 1.38888888888888888889e-03;
  y = fma(y, r, 8.33333333333333333333e-03);
  y = fma(y, r, 4.16666666666666666667e-02);
  y = fma(y, r, 1.66666666666666666667e-01);
  y = fma(y, r, 0.5);
  y = fma(y, r, 1.0);
  y *= r;
  const double t = __hiloint2double(__shfl_sync(0xffffffffu, __double2hiint(tab), k & 31),
                                    __shfl_sync(0xffffffffu, __double2loint(tab), k & 31));
  y = fma(t, y, t);
  const int hi = __double2hiint(y) + (max(k, -32600) >> 5) * 1048576;  // (a reference of 1e9 leaves lo a coarse bound)
  const bool zero = logit < row.lo, big = !(logit <= row.hi);
  return __hiloint2double(big ? 0x7ff00000 : (zero ? 0 : hi), big || zero ? 0 : __double2loint(y));
}

// The same for a group of logits, a reference of 0 and logits within the limits on either side (the caller has looked), as
// almost all are. Step by step for M of them side by side: each is a chain of a dozen dependent fp64 instructions, and taken
// one after the other they left the pipe half idle (cycles of a warp per exponential, V = 128256: 56 before, 48 now, of which
// the fp64 instructions take 29 and the two shuffles and the conversion, which other pipes run, 8 each). No range tests, and
// the argument is reduced from the logit itself, t = logit * 32 / (T ln2) = k + f, |f| <= 1/2, by a factor in two parts: f's two
// roundings are 2^-54 each, 2e-18 in the result, where x = logit / T carried its own, up to 690 * 2^-53. What is left is the
// table entry's 2^-52 and the last step's 2^-53. The polynomial of e^r is taken in f.
// (The conversion by integer instructions: 80.9 -> 83.5 us for 16 sequences of V = 128256; M = 2 or 4: 86.1, 82.9.)
template <int M>
__device__ __forceinline__ void sto_exp_plain(const float (&logit)[M], double c_hi, double c_lo, double tab, double (&e)[M]) {
  constexpr double kL = 6.93147180559945309417e-01 / 32.0;
  const double kMagic = 6755399441055744.0;
  const double c[6] = {kL * kL * kL * kL * kL * kL / 720.0, kL * kL * kL * kL * kL / 120.0, kL * kL * kL * kL / 24.0,
                       kL * kL * kL / 6.0, kL * kL / 2.0, kL};
  double f[M], y[M];
  int k[M];
#pragma unroll
  for (int i = 0; i < M; ++i) f[i] = (double)logit[i];
#pragma unroll
  for (int i = 0; i < M; ++i) y[i] = fma(f[i], c_hi, kMagic);
#pragma unroll
  for (int i = 0; i < M; ++i) {
    k[i] = __double2loint(y[i]);
    y[i] -= kMagic;
  }
#pragma unroll
  for (int i = 0; i < M; ++i) y[i] = fma(f[i], c_hi, -y[i]);
#pragma unroll
  for (int i = 0; i < M; ++i) f[i] = fma(f[i], c_lo, y[i]);
#pragma unroll
  for (int i = 0; i < M; ++i) y[i] = c[0];
#pragma unroll
  for (int d = 1; d < 6; ++d)
#pragma unroll
    for (int i = 0; i < M; ++i) y[i] = fma(y[i], f[i], c[d]);
#pragma unroll
  for (int i = 0; i < M; ++i) y[i] *= f[i];
#pragma unroll
  for (int i = 0; i < M; ++i) {
    const double t = __hiloint2double(__shfl_sync(0xffffffffu, __double2hiint(tab), k[i] & 31),
                                      __shfl_sync(0xffffffffu, __double2loint(tab), k[i] & 31));
    const double v = fma(t, y[i], t);
    e[i] = __hiloint2double(__double2hiint(v) + (k[i] & ~31) * 32768, __double2loint(v));
  }
}

struct StoShared {
  double xch[2][kStoMaxCluster * kStoWarps][2];  // the cluster's warps' records, in vocabulary order, double-buffered
  int32_t par[CAST_MAX_TREE];
  int32_t tok[CAST_MAX_TREE];
  uint8_t kids[kStoWarps][CAST_MAX_TREE];  // every warp's own list of the current node's children
};

__device__ __forceinline__ double sto_warp_sum(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// Every warp hands its two values to every CTA of the cluster; after the barrier sh.xch[parity] holds all records.
// `meanwhile` runs while the others' records are on their way.
template <typename F>
__device__ __forceinline__ void sto_exchange(StoShared& sh, int parity, int rank, int cs, double v0, double v1, F meanwhile) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  double* slot = sh.xch[parity][rank * kStoWarps + warp];
  if (cs == 1) {
    if (lane == 0) {
      slot[0] = v0;
      slot[1] = v1;
    }
    meanwhile();
    __syncthreads();
    return;
  }
  if (lane < cs) sto_st_remote_f64x2(slot, (uint32_t)lane, v0, v1);
  asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
  meanwhile();
  asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ void sto_exchange(StoShared& sh, int parity, int rank, int cs, double v0, double v1) {
  sto_exchange(sh, parity, rank, cs, v0, v1, [] {});
}

// The records' sums, in the same order in every warp.
__device__ __forceinline__ void sto_fold(const StoShared& sh, int parity, int cs, double& s0, double& s1) {
  const int lane = threadIdx.x & 31;
  s0 = s1 = 0.0;
  for (int i = lane; i < cs * kStoWarps; i += 32) {
    s0 += sh.xch[parity][i][0];
    s1 += sh.xch[parity][i][1];
  }
  s0 = sto_warp_sum(s0);
  s1 = sto_warp_sum(s1);
}

// Target values a lane keeps in registers; the rest of a long segment joins the draft values in shared memory (with 32 or
// 38 in registers the sweep spilled and a node of 152064 tokens took as long as with the recomputing kernel).
__host__ __device__ constexpr int sto_in_registers(int NE) { return NE < 24 ? NE : 24; }
// Doubles per lane in shared memory.
__host__ __device__ constexpr int sto_in_shared(int NE) { return 2 * NE - sto_in_registers(NE); }

// NE > 0: up to NE elements per lane are cached; NE == 0: every sweep recomputes them from the logits.
template <typename T, int NE>
__global__ void __launch_bounds__(kStoThreads, 1) accept_stochastic_kernel(const StoParams p) {
  extern __shared__ __align__(16) unsigned char sto_dyn[];
  __shared__ StoShared sh;
  constexpr bool CACHED = NE > 0;
  constexpr int kP = CACHED ? sto_in_registers(NE) : 1;
  // The children's exponentials are formed while the sums are exchanged, but not where a segment's values leave no registers
  // for them (us, formed after / during: one sequence of V = 128256 42.3 / 40.3, 64 of 32000 105.6 / 104.2, with 32 entries a
  // lane, 16 of 128256, 80.5 / 82.2), nor where a node is short (up to four entries a lane, fp32, this launch alone, means over
  // four sets of trees: 16 sequences of V = 4099 30.8 / 32.0, of 1000 31.4 / 32.1, of 16001 30.2 / 30.8, of 32000 35.1 / 35.2,
  // eight of 4099 in bf16 23.0 / 23.5; one of 1000 22.7 / 22.3).
  constexpr bool kOverlap = NE > 4 && NE <= 24;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int cs = p.cs, rank = blockIdx.x, b = blockIdx.y;
  const int ne = CACHED ? NE : p.ne;
  const int begin = rank * p.ne * kStoThreads + warp * p.ne * 32 + lane;  // lane's j-th element: begin + 32 j
  const int mine = min(p.ne, max(0, (p.V - begin + 31) / 32));            // how many of them exist
  double ep[kP];                                                          // exp(target logit / T), j < kP
  // exp(draft logit / T) at eq[32 j], then the target's from kP on
  double* eq = reinterpret_cast<double*>(sto_dyn) + (size_t)warp * sto_in_shared(NE) * 32 + lane;
  int N = p.n_tree[b];
  if (N < 1 || N > p.Ncap) {
    if (rank == 0 && tid == 0) report(p.st, CAST_ERR_BAD_TREE, b);
    N = N < 1 ? 1 : p.Ncap;
  }
  const double tab = exp2((double)lane * (1.0 / 32.0));
  if (tid < CAST_MAX_TREE) {
    sh.par[tid] = tid < N ? p.parent[(size_t)b * p.Ncap + tid] : -2;
    sh.tok[tid] = tid < N ? p.tokens[(size_t)b * p.Ncap + tid] : 0;
  }
  const double u_bonus = p.u_bonus[b];
  // the peers' shared memory may be written once all CTAs of the cluster run
  if (cs > 1) sto_cluster_sync(); else __syncthreads();

  int parity = 0;
  int cur = 0, plen = 1;           // current node, nodes on the path so far
  double a = 0.0;                  // the distribution that stands at `cur`: max(0, P_T - a P_D) / F(a)
  double cp = 1.0, cq = 0.0;       // P_T(x) = e_p(x) cp, P_D(x) = e_q(x) cq
  StoRef ref_p(0.0, p.T), ref_q(0.0, p.T);  // e(x) = exp(logit / T - ref)
  int held = 0;                    // buffer with the segment sums of the distribution that stands
  double held_scale = 1.0;
  const T* lp = nullptr;
  const T* lq = nullptr;
  bool has_q = false;
  uint8_t* kids = sh.kids[warp];
  if (rank == 0 && tid == 0) p.accept_path[(size_t)b * (p.max_depth + 1)] = 0;

  auto logit = [&](const T* row, int j) -> float { return j < mine ? to_float(row[begin + 32 * j]) : -INFINITY; };
  auto value = [&](float x, const StoRef& row) -> double { return sto_exp_row(x, row, p.inv_T, tab); };
  auto pt = [&](int j) -> double {  // (cached: j is a constant wherever this is called)
    if (!CACHED) return value(logit(lp, j), ref_p);
    return j < kP ? ep[j < kP ? j : 0] : eq[32 * (NE + j - kP)];
  };
  auto qt = [&](int j) -> double { return CACHED ? eq[32 * j] : value(logit(lq, j), ref_q); };
  // the node's rows evaluated: this lane's sums
  auto evaluate = [&](double& sp, double& sq, bool zero_refs) {
    sp = sq = 0.0;
    if constexpr (CACHED) {
      constexpr int U = NE < kStoInFlight ? NE : kStoInFlight;  // the next group is loaded while this one is evaluated
      float xp[U], xq[U];
#pragma unroll
      for (int j = 0; j < U; ++j) {
        xp[j] = logit(lp, j);
        xq[j] = has_q ? logit(lq, j) : 0.f;
      }
#pragma unroll
      for (int j0 = 0; j0 < NE; j0 += U) {
        float np[U], nq[U];
#pragma unroll
        for (int j = 0; j < U; ++j) {
          np[j] = j0 + U + j < NE ? logit(lp, j0 + U + j) : 0.f;
          nq[j] = j0 + U + j < NE && has_q ? logit(lq, j0 + U + j) : 0.f;
        }
        bool plain_p = zero_refs, plain_q = zero_refs;
#pragma unroll
        for (int j = 0; j < U; ++j) {
          plain_p = plain_p && fabsf(xp[j]) <= ref_p.hi;
          plain_q = plain_q && fabsf(xq[j]) <= ref_p.hi;
        }
#pragma unroll
        for (int side = 0; side < 2; ++side) {  // target, draft
          if (side == 1 && !has_q) break;
          double e[U];
          bool plain = false;
          // (segments of four entries a lane are mostly padding, which is not within the limits: one sequence of V = 4099
          // 28.4 us with the look, 27.5 without)
          if constexpr (NE > 4) {
            plain = __all_sync(0xffffffffu, side == 0 ? plain_p : plain_q);
            if (plain) sto_exp_plain(side == 0 ? xp : xq, p.c_hi, p.c_lo, tab, e);
          }
          if (!plain) {
#pragma unroll
            for (int j = 0; j < U; ++j)
              e[j] = value(side == 0 ? xp[j] : xq[j], side == 0 ? ref_p : ref_q);
          }
#pragma unroll
          for (int j = 0; j < U; ++j) {
            if (j0 + j >= NE) break;
            if (side == 1) eq[32 * (j0 + j)] = e[j];
            else if (j0 + j < kP) ep[j0 + j < kP ? j0 + j : 0] = e[j];
            else eq[32 * (NE + j0 + j - kP)] = e[j];
          }
          // the group's sum in pairs (one after the other they are a chain)
#pragma unroll
          for (int j = 0; j < U; ++j)
            if (j0 + j >= NE) e[j] = 0.0;
#pragma unroll
          for (int o = 1; o < U; o *= 2)
#pragma unroll
            for (int j = 0; j + o < U; j += 2 * o) e[j] += e[j + o];
          if (side == 1) sq += e[0];
          else sp += e[0];
        }
#pragma unroll
        for (int j = 0; j < U; ++j) {
          xp[j] = np[j];
          xq[j] = nq[j];
        }
      }
    } else {
#pragma unroll 4
      for (int j = 0; j < ne; ++j) {
        sp += value(logit(lp, j), ref_p);
        if (has_q) sq += value(logit(lq, j), ref_q);
      }
    }
  };
  // P_T - a P_D at this lane's j-th token, aq = a cq. Each row is scaled by its own sum: both products are of order one. (One
  // multiply-add less per entry with the quotient a Sp / Sq of the sums: that leaves fp64 where the rows lie far apart, T = 0.05
  // and tops of 32 and -4.) The residual sums and the search for the bonus token both call this: a residual may be nothing but
  // the last bits of two equal rows, and a segment whose sum is positive must hold a token of positive mass.
  auto left = [&](int j, double aq) -> double { return __fma_rn(pt(j), cp, -__dmul_rn(qt(j), aq)); };
  // this lane's share of sum_x max(0, P_T - a2 P_D)
  auto residual = [&](double a2) -> double {
    const double aq = a2 * cq;
    double s = 0.0;
    auto add = [&](int j) {
      const double v = left(j, aq);
      s += v > 0.0 ? v : 0.0;
    };
#pragma unroll
    for (int j = 0; j < (CACHED ? NE : 1); ++j)
      if (CACHED) add(j);
    if (!CACHED) {
#pragma unroll 4
      for (int j = 0; j < ne; ++j) add(j);
    }
    return s;
  };

  for (;;) {
    // ---- children of `cur` in tree order (every warp for itself)
    int k = 0;
    for (int base = 0; base < N; base += 32) {
      const int c = base + lane;
      const bool is = c < N && c > cur && sh.par[c] == cur;
      const unsigned m = __ballot_sync(0xffffffffu, is);
      if (is) kids[k + __popc(m & ((1u << lane) - 1u))] = (uint8_t)c;
      k += __popc(m);
    }
    __syncwarp();
    if (k > 0 && plen > p.max_depth) {  // a path longer than the output has room for
      if (rank == 0 && tid == 0) report(p.st, CAST_ERR_BAD_TREE, b);
      k = 0;
    }
    has_q = k > 0;
    lp = reinterpret_cast<const T*>(p.target_logits) + ((size_t)b * p.Ncap + cur) * p.V;
    lq = reinterpret_cast<const T*>(p.draft_logits) + ((size_t)b * p.Ncap + cur) * p.V;
    // the children's tests need two logits and a uniform number each, lane j for child j: asked for now, used after
    // the sweep (a node with more than 32 children asks again)
    float raw_p = 0.f, raw_q = 0.f;
    double u = 0.0;
    bool token_ok = false;
    auto ask = [&](int j0) {
      const int j = j0 + lane;
      token_ok = false;
      if (j < k) {
        const int c = kids[j], x = sh.tok[c];
        token_ok = x >= 0 && x < p.V;
        if (token_ok) {
          raw_p = to_float(lp[x]);
          raw_q = to_float(lq[x]);
        }
        u = p.u_accept[(size_t)b * p.Ncap + c];
      }
    };
    ask(0);
    if (k > 0) {
      // the eldest child is the likeliest next node: its segments are asked into L2 while this node is worked on
      const size_t row = ((size_t)b * p.Ncap + kids[0]) * p.V + (begin - lane);
      const char* np = reinterpret_cast<const char*>(reinterpret_cast<const T*>(p.target_logits) + row);
      const char* nq = reinterpret_cast<const char*>(reinterpret_cast<const T*>(p.draft_logits) + row);
      const int bytes = min(p.ne * 32, p.V - (begin - lane)) * (int)sizeof(T);
      for (int off = lane * 128; off < bytes; off += 32 * 128) {
        asm volatile("prefetch.global.L2 [%0];" ::"l"(np + off));
        asm volatile("prefetch.global.L2 [%0];" ::"l"(nq + off));
      }
    }

    // ---- softmax sums of the node's rows
    double Sp, Sq = 1.0;
    ref_p = ref_q = StoRef(0.0, p.T);
    double child_p = 0.0, child_q = 0.0;  // exp(logit / T) of lane j's child
    auto child_exps = [&] {
      child_p = sto_exp_any(fma((double)raw_p, p.inv_T, -ref_p.ref));
      child_q = sto_exp_any(fma((double)raw_q, p.inv_T, -ref_q.ref));
    };
    for (int attempt = 0;; ++attempt) {
      double sp, sq;
      evaluate(sp, sq, attempt == 0);
      if constexpr (kOverlap) sto_exchange(sh, parity, rank, cs, sto_warp_sum(sp), sto_warp_sum(sq), child_exps);
      else sto_exchange(sh, parity, rank, cs, sto_warp_sum(sp), sto_warp_sum(sq));
      sto_fold(sh, parity, cs, Sp, Sq);
      held = parity;
      parity ^= 1;
      if (attempt == 1 || (Sp > 1e-280 && Sp < 1e280 && (!has_q || (Sq > 1e-280 && Sq < 1e280)))) break;
      // logits / T far from zero (or not finite): once more, against the rows' maxima
      double mp = -INFINITY, mq = -INFINITY;
      for (int j = 0; j < mine; ++j) {
        mp = fmax(mp, (double)logit(lp, j) * p.inv_T);
        if (has_q) mq = fmax(mq, (double)logit(lq, j) * p.inv_T);
      }
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
        mp = fmax(mp, __shfl_xor_sync(0xffffffffu, mp, o));
        mq = fmax(mq, __shfl_xor_sync(0xffffffffu, mq, o));
      }
      sto_exchange(sh, parity, rank, cs, mp, mq);
      for (int i = 0; i < cs * kStoWarps; ++i) {
        mp = fmax(mp, sh.xch[parity][i][0]);
        mq = fmax(mq, sh.xch[parity][i][1]);
      }
      parity ^= 1;
      if (isfinite(mp)) ref_p = StoRef(mp, p.T);
      if (isfinite(mq)) ref_q = StoRef(mq, p.T);
    }
    if (!(Sp > 0.0) || !isfinite(Sp) || (has_q && (!(Sq > 0.0) || !isfinite(Sq)))) {
      if (rank == 0 && tid == 0) report(p.st, CAST_ERR_NONFINITE, b * p.Ncap + cur);
      Sp = 1.0;  // keep the arithmetic finite; the result of this sequence is void
      Sq = 1.0;
      k = 0;
      has_q = false;
    }
    cp = 1.0 / Sp;
    cq = has_q ? 1.0 / Sq : 0.0;
    held_scale = cp;

    // ---- the children, one after the other, each against the residual its elder siblings left
    a = 0.0;
    double F = 1.0;
    int next = -1;
    for (int j0 = 0; j0 < k && next < 0; j0 += 32) {
      if (j0 > 0) ask(j0);
      if (j0 > 0 || !kOverlap) child_exps();
      const double px_l = child_p * cp, qx_l = child_q * cq;
      const unsigned valid = __ballot_sync(0xffffffffu, token_ok);
      bool empty = false;
      for (int j = j0; j < min(k, j0 + 32); ++j) {
        if (!((valid >> (j - j0)) & 1u)) {
          if (rank == 0 && tid == 0) report(p.st, CAST_ERR_BAD_TREE, b);
          continue;  // not a token: never accepted
        }
        const double px = __shfl_sync(0xffffffffu, px_l, j - j0), qx = __shfl_sync(0xffffffffu, qx_l, j - j0);
        const double uj = __shfl_sync(0xffffffffu, u, j - j0);
        if (uj * qx * F <= fmax(0.0, px - a * qx)) {
          next = kids[j];
          break;
        }
        // rejected: the residual of the residual
        const double a2 = a + F;
        sto_exchange(sh, parity, rank, cs, sto_warp_sum(residual(a2)), 0.0);
        double F2, none;
        sto_fold(sh, parity, cs, F2, none);
        if (!(F2 > 0.0)) {  // an empty residual: the distribution before it stands (and so do its segment sums)
          empty = true;
          break;
        }
        held = parity;
        held_scale = 1.0;
        parity ^= 1;
        a = a2;
        F = F2;
      }
      if (empty) break;
    }
    if (next < 0) break;
    cur = next;
    if (rank == 0 && tid == 0) p.accept_path[(size_t)b * (p.max_depth + 1) + plen] = cur;
    ++plen;
  }

  // ---- bonus token: inversion of the cumulative sum, in token order, of max(0, P_T - a P_D) at `cur`: first among the
  // cluster's warps, whose segment sums are at hand, then inside the segment. Where rounding leaves the goal unreached,
  // the last place that has mass is taken.
  if (rank == 0 && tid == 0) {
    p.accept_len[b] = plen - 1;
    for (int j = plen; j <= p.max_depth; ++j) p.accept_path[(size_t)b * (p.max_depth + 1) + j] = -1;
  }
  int owner = -1, last = -1;
  double before = 0.0, goal;
  {
    constexpr int kPer = kStoMaxCluster * kStoWarps / 32;  // consecutive segments per lane
    double s[kPer], run = 0.0;
#pragma unroll
    for (int i = 0; i < kPer; ++i) {
      const int at = lane * kPer + i;
      s[i] = at < cs * kStoWarps ? sh.xch[held][at][0] * held_scale : 0.0;
      run += s[i];
    }
    double incl = run;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const double t = __shfl_up_sync(0xffffffffu, incl, o);
      if (lane >= o) incl += t;
    }
    goal = u_bonus * __shfl_sync(0xffffffffu, incl, 31);
    double at = incl - run;
    int own_l = -1, last_l = -1;
    double before_l = 0.0, last_before_l = 0.0;
#pragma unroll
    for (int i = 0; i < kPer; ++i) {
      if (s[i] > 0.0) {
        last_l = lane * kPer + i;
        last_before_l = at;
        if (own_l < 0 && at + s[i] >= goal) {
          own_l = last_l;
          before_l = at;
        }
      }
      at += s[i];
    }
    const unsigned hit = __ballot_sync(0xffffffffu, own_l >= 0), mass = __ballot_sync(0xffffffffu, last_l >= 0);
    if (hit != 0u) {
      owner = __shfl_sync(0xffffffffu, own_l, __ffs(hit) - 1);
      before = __shfl_sync(0xffffffffu, before_l, __ffs(hit) - 1);
    } else if (mass != 0u) {
      owner = __shfl_sync(0xffffffffu, last_l, 31 - __clz(mass));
      before = __shfl_sync(0xffffffffu, last_before_l, 31 - __clz(mass));
    }
  }
  if (owner < 0) {  // nothing has mass (a void sequence): token 0
    if (rank == 0 && tid == 0) p.bonus_token[b] = 0;
  } else if (owner == rank * kStoWarps + warp) {
    // rows of 32 consecutive tokens, one per lane: the row in which the goal is reached, then the lane
    const double aq = has_q ? a * cq : 0.0;
    double run = before;
    double pick_v = 0.0, pick_at = 0.0;  // this lane's mass in the row that was picked, and the sum before that row
    int pick = -1;
    bool found = false;
    auto mass_of = [&](int j) -> double { return fmax(0.0, has_q ? left(j, aq) : pt(j) * cp); };
    auto visit = [&](int j, double v, double row) {
      if (!found && row > 0.0) {
        pick = j;
        pick_v = v;
        pick_at = run;
        found = run + row >= goal;
      }
      run += row;
    };
    constexpr int kRows = !CACHED ? 1 : NE < 8 ? NE : 8;  // rows summed side by side (a sum is a chain of five shuffles and additions)
#pragma unroll
    for (int j0 = 0; j0 < NE; j0 += kRows) {
      double v[kRows], row[kRows];
#pragma unroll
      for (int i = 0; i < kRows; ++i) row[i] = v[i] = j0 + i < NE ? mass_of(j0 + i) : 0.0;
#pragma unroll
      for (int o = 16; o > 0; o >>= 1)
#pragma unroll
        for (int i = 0; i < kRows; ++i) row[i] += __shfl_xor_sync(0xffffffffu, row[i], o);
#pragma unroll
      for (int i = 0; i < kRows; ++i)
        if (j0 + i < NE) visit(j0 + i, v[i], row[i]);
      if (found) break;  // (the same in all lanes)
    }
    if (!CACHED)
      for (int j = 0; j < ne; ++j) {
        const double v = mass_of(j);
        visit(j, v, sto_warp_sum(v));
      }
    double incl = pick_v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const double t = __shfl_up_sync(0xffffffffu, incl, o);
      if (lane >= o) incl += t;
    }
    const unsigned reach = __ballot_sync(0xffffffffu, pick_v > 0.0 && pick_at + incl >= goal);
    const unsigned mass = __ballot_sync(0xffffffffu, pick_v > 0.0);
    const int l = reach != 0u ? __ffs(reach) - 1 : (mass != 0u ? 31 - __clz(mass) : 0);
    if (lane == 0) p.bonus_token[b] = pick >= 0 ? begin + 32 * pick + l : 0;
  }
}

template <typename T, int NE>
cudaError_t sto_attributes(size_t dyn, int cs) {
  auto kern = accept_stochastic_kernel<T, NE>;
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)dyn);
  if (e == cudaSuccess && cs > 8) e = cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
  return e;
}
template <typename T, int NE>
void sto_config(cudaLaunchConfig_t& cfg, cudaLaunchAttribute* attr, int cs, int B, size_t dyn, cudaStream_t s) {
  cfg = {};
  cfg.gridDim = dim3(cs, B, 1);
  cfg.blockDim = dim3(kStoThreads, 1, 1);
  cfg.dynamicSmemBytes = dyn;
  cfg.stream = s;
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = cs;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
}
constexpr size_t sto_cache_bytes(int NE) { return (size_t)sto_in_shared(NE) * kStoThreads * sizeof(double); }

template <typename T, int NE>
cast_status sto_launch(const StoParams& p, int B, cudaStream_t s) {
  CAST_CUDA_OK((sto_attributes<T, NE>(sto_cache_bytes(NE), p.cs)));
  cudaLaunchConfig_t cfg;
  cudaLaunchAttribute attr[1];
  sto_config<T, NE>(cfg, attr, p.cs, B, sto_cache_bytes(NE), s);
  CAST_CUDA_OK(cudaLaunchKernelEx(&cfg, accept_stochastic_kernel<T, NE>, p));
  return CAST_OK;
}
// Clusters of cs CTAs that the device runs at once (0: it cannot run one).
template <typename T, int NE>
int sto_resident(int cs) {
  int n = 0;
  cudaLaunchConfig_t cfg;
  cudaLaunchAttribute attr[1];
  sto_config<T, NE>(cfg, attr, cs, 1, sto_cache_bytes(NE), nullptr);
  if (sto_attributes<T, NE>(sto_cache_bytes(NE), cs) == cudaSuccess &&
      cudaOccupancyMaxActiveClusters(&n, accept_stochastic_kernel<T, NE>, &cfg) == cudaSuccess)
    return n;
  (void)cudaGetLastError();
  return 0;
}

int elements_per_lane(int V, int cs) { return ((V + cs - 1) / cs + kStoThreads - 1) / kStoThreads; }

// The kernel for `ne` elements per lane: the smallest cached one that holds them, or the one that caches nothing. Slots
// past ne cost as much as live ones, hence the steps. 38 is what fits on chip: 76 doubles per lane, 24 of them in registers
// and 52 in shared memory (213 KB of 227). Clusters of 16 use the steps up to 24 (kStoMaxSlice), clusters of 8 all of them.
#define STO_PICK(T, ne, cached, call)      \
  (!(cached)    ? call<T, 0>               \
   : (ne) <= 4  ? call<T, 4>               \
   : (ne) <= 8  ? call<T, 8>               \
   : (ne) <= 16 ? call<T, 16>              \
   : (ne) <= 20 ? call<T, 20>              \
   : (ne) <= 24 ? call<T, 24>              \
   : (ne) <= 32 ? call<T, 32>              \
                : call<T, 38>)
constexpr int kStoMaxCached = 38;

// Largest cluster size (16, else 8) that runs with this context's vocabulary and a logits dtype, whether segments are
// cached at that size, and how many such clusters run at once; looked up once per context.
template <typename T>
void sto_plan(cast_ctx* c, int di) {
  if (c->sto_cs[di] != 0) return;
  const int V = c->cfg.vocab;
  int cs = 0, n = 0, cached = 0;
  for (cached = 1; cached >= 0 && n == 0; --cached)
    for (cs = 16; cs >= 8; cs >>= 1) {
      const int ne = elements_per_lane(V, cs);
      if (cached && (V > cs * kStoMaxSlice || ne > kStoMaxCached)) continue;
      n = STO_PICK(T, ne, cached, sto_resident)(cs);
      if (n > 0) break;
    }
  c->sto_cached[di] = n > 0 ? cached + 1 : 0;
  c->sto_resident[di] = n > 0 ? n : 1;
  c->sto_cs[di] = n > 0 ? cs : 1;
}

template <typename T>
cast_status sto_run(cast_ctx* c, StoParams& p, int B, int di, cudaStream_t s) {
  sto_plan<T>(c, di);  // first call with this dtype: a host-side query, no device work
  p.cs = c->sto_cs[di];
  const bool cached = c->sto_cached[di] != 0;
  // With more sequences than clusters of 16 run at once, clusters of 8: a node takes less than twice as long (the chain of
  // exchanges does not grow) and twice as many sequences run. Only where those hold the segments as well (155 648 tokens):
  // 16 sequences of V = 190000 take 82 us in clusters of 16 one after the other, 207 recomputing in clusters of 8.
  if (p.cs == 16 && B > c->sto_resident[di] && (!cached || elements_per_lane(p.V, 8) <= kStoMaxCached)) p.cs = 8;
  p.ne = elements_per_lane(p.V, p.cs);
  return STO_PICK(T, p.ne, cached, sto_launch)(p, B, s);
}

}  // namespace

extern "C" cast_status cast_accept_stochastic_plan(cast_ctx* c, cast_dtype dtype, int* cluster_size, int* cached) {
  if (!c || !cluster_size || !cached) return CAST_ERR_INVALID_ARG;
  if (dtype != CAST_F32 && dtype != CAST_BF16) return CAST_ERR_DTYPE;
  if (dtype == CAST_F32) sto_plan<float>(c, 0);
  else sto_plan<__nv_bfloat16>(c, 1);
  *cluster_size = c->sto_cs[dtype == CAST_F32 ? 0 : 1];
  *cached = c->sto_cached[dtype == CAST_F32 ? 0 : 1];
  return CAST_OK;
}

extern "C" cast_status cast_accept_stochastic(cast_ctx* c, const void* target_logits, const void* draft_logits,
                                              cast_dtype dtype, int B, double temperature, const int32_t* tokens,
                                              const int32_t* parent, const int32_t* n_tree, const double* u_accept,
                                              const double* u_bonus, int32_t* accept_len, int32_t* accept_path,
                                              int32_t* bonus_token, void* stream) {
  if (!c || !target_logits || !draft_logits || !tokens || !parent || !n_tree || !u_accept || !u_bonus || !accept_len ||
      !accept_path || !bonus_token || B < 1 || !(temperature > 0.0) || !isfinite(temperature))
    return CAST_ERR_INVALID_ARG;
  if (dtype != CAST_F32 && dtype != CAST_BF16) return CAST_ERR_DTYPE;
  if (B > c->cfg.max_batch) return CAST_ERR_CAPACITY;
  StoParams p;
  p.target_logits = target_logits;
  p.draft_logits = draft_logits;
  p.V = c->cfg.vocab;
  p.Ncap = c->cfg.max_tree;
  p.max_depth = c->cfg.max_depth;
  p.inv_T = 1.0 / temperature;
  p.T = temperature;
  {
    const long double c = 32.0L * 1.442695040888963407359924681001892137L / (long double)temperature;
    p.c_hi = (double)c;
    p.c_lo = (double)(c - (long double)p.c_hi);
    if (!isfinite(p.c_hi)) p.c_hi = p.c_lo = 0.0;  // (temperatures of 1e-307: zero is the one logit within the limits)
  }
  p.tokens = tokens;
  p.parent = parent;
  p.n_tree = n_tree;
  p.u_accept = u_accept;
  p.u_bonus = u_bonus;
  p.accept_len = accept_len;
  p.accept_path = accept_path;
  p.bonus_token = bonus_token;
  p.st = c->state;
  cudaStream_t s = (cudaStream_t)stream;
  return dtype == CAST_F32 ? sto_run<float>(c, p, B, 0, s) : sto_run<__nv_bfloat16>(c, p, B, 1, s);
}
