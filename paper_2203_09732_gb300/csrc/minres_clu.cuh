// Preconditioned MINRES of Algorithm 2 (Appendix A) inside one thread-block
// cluster, for chains of up to 16384 rows: the device side, shared by the
// single solve (minres_clu.cu) and the batched sweep (sweep.cu).
//
// What bounds a small solve is latency: two reductions per iteration over all
// rows, and the FP64 pipe, which takes 64 cycles per warp instruction and SM
// quarter whatever the number of active lanes (measured: dependent or not, 1
// lane or 32). So:
//   * the CTAs of a cluster exchange through distributed shared memory: every
//     warp sends its partial sum to every CTA (st.async, counted by an mbarrier
//     in the receiving CTA, about 450 cycles), no grid barrier and no trip
//     through L2 (about 2500 cycles a reduction in the grid forms);
//   * every CTA holds a full copy of q; the owner of a row sends the new entry
//     to all copies the same way, so the product's gathers are shared-memory
//     loads from per-row neighbour lists;
//   * a thread owns RPT rows for the whole solve and keeps their vectors in
//     registers: CLU_NW compute warps, one per SM quarter, saturate the FP64 pipe;
//   * three control warps per CTA take the scalars off the compute warps' path:
//     one adds the partials of alpha_k and forms the coefficient that needs it,
//     one adds those of beta_k^2 and has 1 / beta_k and its powers ready by then,
//     one runs the Givens rotation of Algorithm 2 an iteration behind; the compute
//     warps apply its d/x update two iterations behind, while they wait for
//     alpha. Where several scalars need the same operation, each takes a lane.
// All CTAs sum the same numbers in the same order, so they hold identical
// scalars and take the same branches.
#pragma once
#include "minres_smem.cuh"

namespace hs {

constexpr int CLU_NW = 4;                       // compute warps per CTA
constexpr int CLU_CW = 3;                       // control warps (warps 0, 1 and 2)
constexpr int CLU_NT = 32 * (CLU_NW + CLU_CW);
constexpr int CLU_SIZE_MAX = 16;                // CTAs per cluster
constexpr int CLU_RPT_MAX = 8;                  // rows per thread
static_assert(CLU_ROWS == CLU_SIZE_MAX * 32 * CLU_NW * CLU_RPT_MAX, "rows of the largest cluster");
// polls of an mbarrier before a wait gives up with HS_TIMEOUT (HS_BARRIER_LIMIT
// sets another number for single solves and sweeps)
constexpr unsigned CLU_WAIT_LIMIT = 1u << 22;

// Exchange words of one CTA (shared memory). What one warp hands to a later
// iteration of another has two places, used in turn.
struct CluShared {
  double slotA[CLU_SIZE_MAX * CLU_NW];          // partials of alpha_k
  double slotB[CLU_SIZE_MAX * CLU_NW];          // partials of beta_{k+1}^2
  unsigned long long barA, barB;                // remote data of the two phases
  unsigned long long barC;                      // alpha warp -> compute warps
  unsigned long long barF[2];                   // beta warp -> alpha warp
  unsigned long long barE[2];                   // alpha warp -> rotation warp
  unsigned long long barD[2];                   // rotation warp -> the others
  double c[3];                                  // coefficients of q_{k+1}, of type T
  double f[2][8];                               // F: sum = beta_k^2, beta_k, 1/beta_{k-1}, 1/beta_k,
                                                //    1/(2 beta_k^2), 1/(2 beta_k^3), beta_k/beta_{k-1}
  double alpha[2];                              // E: alpha_k
  struct { double co[4]; int apply, stop; } d[2];   // D: cq, cd1, cd2, tau (of type T)
  int fail;                                     // a wait of this CTA gave up
  int gave_up;                                  // a wait of any CTA did (clu_agree)
  unsigned phase[4];                            // compute warps' parities after a solve: b, c, d
  MinresState S;                                // the solve's state (rotation warp)
};

__device__ __forceinline__ uint32_t smem_u32(const void* p) {
  return (uint32_t)__cvta_generic_to_shared(p);
}
__device__ __forceinline__ uint32_t clu_map(uint32_t addr, uint32_t cta) {
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(cta));
  return r;
}
__device__ __forceinline__ void clu_sync() {
  asm volatile("barrier.cluster.arrive.release.aligned;\n"
               "barrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ uint32_t clu_rank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
__device__ __forceinline__ uint32_t clu_size() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_nctarank;" : "=r"(r));
  return r;
}
__device__ __forceinline__ void bar_init(unsigned long long* b, unsigned count) {
  asm volatile("mbarrier.init.shared.b64 [%0], %1;" ::"r"(smem_u32(b)), "r"(count) : "memory");
}
__device__ __forceinline__ void bar_arm(unsigned long long* b, unsigned bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared.b64 _, [%0], %1;" ::"r"(smem_u32(b)), "r"(bytes)
               : "memory");
}
__device__ __forceinline__ void bar_arrive(unsigned long long* b) {
  asm volatile("mbarrier.arrive.shared.b64 _, [%0];" ::"r"(smem_u32(b)) : "memory");
}
// Waits for the phase of the given parity (whole warps); false in every lane
// after limit polls. The vote that makes the answer the warp's is the loop's only
// branch: with a vote behind a loop per lane an iteration took 4 to 9 % longer.
__device__ __forceinline__ bool bar_wait(unsigned long long* b, unsigned parity, unsigned limit) {
  const uint32_t a = smem_u32(b);
  for (unsigned it = 0; it != limit; ++it) {
    uint32_t done;
    asm volatile("{\n.reg .pred p;\n"
                 "mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n"
                 "selp.u32 %0, 1, 0, p;\n}"
                 : "=r"(done) : "r"(a), "r"(parity) : "memory");
    if (__all_sync(0xffffffffu, done)) return true;
  }
  return false;
}
// One or two values into another CTA's shared memory, counted by its mbarrier.
__device__ __forceinline__ void clu_send(uint32_t dst, double v, uint32_t bar) {
  asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.b64 [%0], %1, [%2];" ::"r"(dst),
               "l"(__double_as_longlong(v)), "r"(bar) : "memory");
}
__device__ __forceinline__ void clu_send(uint32_t dst, float v, uint32_t bar) {
  asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.b32 [%0], %1, [%2];" ::"r"(dst),
               "r"(__float_as_uint(v)), "r"(bar) : "memory");
}
__device__ __forceinline__ void clu_send2(uint32_t dst, double v, double w, uint32_t bar) {
  asm volatile(
      "st.async.shared::cluster.mbarrier::complete_tx::bytes.v2.b64 [%0], {%1, %2}, [%3];" ::"r"(dst),
      "l"(__double_as_longlong(v)), "l"(__double_as_longlong(w)), "r"(bar) : "memory");
}
__device__ __forceinline__ void clu_send2(uint32_t dst, float v, float w, uint32_t bar) {
  asm volatile(
      "st.async.shared::cluster.mbarrier::complete_tx::bytes.v2.b32 [%0], {%1, %2}, [%3];" ::"r"(dst),
      "r"(__float_as_uint(v)), "r"(__float_as_uint(w)), "r"(bar) : "memory");
}

// Rows per CTA. With two or more rows a thread holds pairs of consecutive rows
// (one message per pair and copy: sending costs by the message), pair i of
// thread t at 2 (128 i + t): wider runs per thread would put the lanes of a
// gather on the same banks. Rows past n (in the last CTAs) are sent as zeros.
__host__ __device__ inline int clu_rows(int n, int cs, int rpt) {
  const int r = (n + cs - 1) / cs;
  return rpt == 1 ? r : (r + 1) & ~1;
}
// Dynamic shared memory of a CTA: the copy of q with one zero element behind
// it, then the neighbour lists (pairs of 16-bit row numbers, [pair][j][thread]).
template <typename T>
__host__ __device__ inline size_t clu_q_bytes(int n, int cs, int rpt) {
  return (((size_t)cs * clu_rows(n, cs, rpt) + 1) * sizeof(T) + 15) & ~size_t(15);
}
template <typename T>
__host__ __device__ inline size_t clu_bytes(int n, int L, int cs, int rpt) {
  return clu_q_bytes<T>(n, cs, rpt) + sizeof(uint32_t) * (size_t)(L / 2) * 32 * CLU_NW * rpt;
}

// Phase parities of a cluster's barriers, carried from solve to solve, and the
// polls of a wait. Every warp keeps its own; a compute warp without rows in a
// solve waits for nothing in it and takes compute warp 0's at its end, so solves
// of one kernel may follow each other in any order of sizes.
struct CluPhase {
  unsigned limit;
  unsigned a = 0, b = 0, c = 0, d[2] = {0, 0}, e[2] = {0, 0}, f[2] = {0, 0};
};

// Barriers of a CTA, once per kernel, before the first solve (all threads).
__device__ __forceinline__ void clu_setup(CluShared& sh) {
  if (threadIdx.x == 0) {
    bar_init(&sh.barA, 1);
    bar_init(&sh.barB, 1);
    bar_init(&sh.barC, 1);
    for (int i = 0; i < 2; ++i) {
      bar_init(&sh.barF[i], 1);
      bar_init(&sh.barE[i], 1);
      bar_init(&sh.barD[i], 1);
    }
    sh.fail = sh.gave_up = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncthreads();
  clu_sync();
}

// Whether a wait of any CTA of the cluster gave up, the same answer in all of
// them (all threads, after a CTA barrier behind the last write of sh.fail). If
// so, messages sent to a CTA that stopped waiting may still be under way: every
// CTA waits a while after all have stopped sending, so that none leaves before
// they have landed, and the barriers are out of step: no solve may follow.
__device__ __forceinline__ bool clu_agree(CluShared& sh) {
  if (sh.fail && threadIdx.x < clu_size())
    asm volatile("st.shared::cluster.s32 [%0], %1;" ::"r"(
                     clu_map(smem_u32(&sh.gave_up), threadIdx.x)), "r"(1) : "memory");
  __syncwarp();
  clu_sync();
  if (sh.gave_up == 0) return true;
  for (int i = 0; i < 100; ++i) __nanosleep(1000);
  clu_sync();
  return false;
}

// Sum of the np partials of all warps of the cluster, in every lane.
__device__ __forceinline__ double clu_total(const double* slot, int np) {
  const int lane = threadIdx.x & 31;
  double v = lane < np ? slot[lane] : 0.0;
  if (np > 32) v += lane + 32 < np ? slot[lane + 32] : 0.0;
  // a tree over the lanes that hold partials only: each level costs an FP64 add
  for (int o = np > 16 ? 16 : np > 8 ? 8 : np > 4 ? 4 : np > 2 ? 2 : np > 1 ? 1 : 0; o > 0; o >>= 1)
    v += __shfl_xor_sync(0xffffffffu, v, o);
  return __shfl_sync(0xffffffffu, v, 0);
}
static_assert(CLU_SIZE_MAX * CLU_NW <= 64, "clu_total adds two partials per lane");

// alpha_k = q_k . p_k / beta_k^2 in odd lanes, alpha_k / beta_k in even ones, from
// q_k . p_k (doubled) and the words of F. beta_1 carries the scale of the right-hand
// side, and 1 / (2 beta_1^3) leaves the range of doubles beyond 1e102 and below
// 1e-103: from 2^+-330 on the quotient takes two steps there. (The later beta_k are
// on the scale of M^-1 H, whose q . p overflows first.)
__device__ __forceinline__ double clu_alpha(const double* f, int k, double qp2) {
  const bool odd = threadIdx.x & 1;
  if (k == 1) {
    const double ib = f[3];
    if (((unsigned)__double2hiint(ib) >> 20) - (1023u - 330u) > 660u)
      return odd ? qp2 * f[4] : qp2 * f[4] * ib;
  }
  return qp2 * f[odd ? 4 : 5];
}

// The Givens rotation of step k (Algorithm 2) and its d/x coefficients: the
// quantities of givens_fast, with a reciprocal square root instead of a root
// and divisions, and one lane per scalar where the operation is the same
// (every lane computes; lanes past the first few repeat them). sumsq =
// beta_{k+1}^2, bn = beta_{k+1}, ib = 1 / beta_k.
__device__ __forceinline__ void clu_givens(MinresState& S, double sumsq, double bn, double ib) {
  constexpr unsigned full = 0xffffffffu;
  const int lane = threadIdx.x & 7;
  const double cp = S.c_prev, sp = S.s_prev;
  // lane 0: delta_k = c dh + s alpha; lane 1: hat gamma_k = c alpha - s dh
  const double u = lane & 1 ? S.alpha : S.delta_hat, w = lane & 1 ? -S.delta_hat : S.alpha;
  const double r = cp * u + sp * w;
  const double delta = __shfl_sync(full, r, 0), gh = __shfl_sync(full, r, 1);
  const double g2 = gh * gh + sumsq;                         // gamma_k^2
  if (!isfinite(bn) || !isfinite(g2)) {
    S.status = HS_NONFINITE; S.done = 2; S.pending = 0;
    return;
  }
  if (g2 == 0.0) {
    S.status = HS_BREAKDOWN; S.done = 2; S.pending = 0;
    return;
  }
  const double rg = rsqrt(g2);
  // times 1 / gamma_k: c_k, s_k, the three coefficients of d_k
  const double v = lane == 0 ? gh : lane == 1 ? bn : lane == 2 ? ib : lane == 3 ? -delta : -S.eps;
  const double t = v * rg;
  const double c = __shfl_sync(full, t, 0), sn = __shfl_sync(full, t, 1);
  S.cq = __shfl_sync(full, t, 2);
  S.cd1 = __shfl_sync(full, t, 3);
  S.cd2 = __shfl_sync(full, t, 4);
  // tau_k = c phi, phi_k = -s phi, epsilon_{k+1} = s_{k-1} beta, hat delta_{k+1} = c_{k-1} beta
  const double x = lane == 0 ? c : lane == 1 ? -sn : lane == 2 ? sp : cp;
  const double y = x * (lane < 2 ? S.phi : bn);
  S.tau = __shfl_sync(full, y, 0);
  S.phi = __shfl_sync(full, y, 1);
  S.eps = __shfl_sync(full, y, 2);
  S.delta_hat = __shfl_sync(full, y, 3);
  S.pending = 1;
  S.beta_prev = S.beta; S.beta = bn;
  S.c_prev = c; S.s_prev = sn;
  S.k = S.k + 1;
  if (fabs(S.phi) < S.tol_abs || bn == 0.0 || S.k > S.kmax) S.done = 1;
}

constexpr int PIPE_NV = 5;           // S1..S5 (S6 is carried)

// Smallest beta_{k+1}^2 / mag (mag: the sum of the expansion's terms in
// magnitude) that the expansion is trusted with: its relative error is about
// u mag / beta_{k+1}^2, at most 1e-8 (FP64) or 6e-5 (FP32) above the floor.
// Below it (in practice: a Krylov space that has run out, as for n <= 8 or a
// right-hand side inside an invariant subspace) the solve is handed back.
template <typename T>
constexpr double EXPANSION_FLOOR = sizeof(T) == 8 ? 1e-8 : 1e-3;

// The scalars of step k of the one-reduction form, by one warp: from the sums
// S1..S6, alpha_k, a = alpha_k / beta_k, c = beta_k / beta_{k-1} and the reciprocals
// ib = 1 / beta_k, ib2 = ib^2, ibp = 1 / beta_{k-1}: beta_{k+1}, the Givens rotation;
// ib and ibp move on a step. An FP64 instruction takes 64 cycles however many
// lanes want it, so each term of beta_{k+1}^2 has a lane: 31 of them instead of
// about 85 on one thread.
template <typename T>
__device__ __forceinline__ void pipe_scalars(MinresState& S, double S1, double S2, double S3,
                                             double S4, double S5, double S6, double alpha, double a,
                                             double c, double& ib, double ib2, double& ibp) {
  constexpr unsigned full = 0xffffffffu;
  const int lane = threadIdx.x & 31, tl = lane & 7;
  // S2 / beta_k^2 | c^2 | c / beta_k
  const double r = (tl == 0 ? S2 : c) * (tl == 0 ? ib2 : tl == 1 ? c : ib);
  const double t1 = __shfl_sync(full, r, 0), cc = __shfl_sync(full, r, 1);
  const double cb = __shfl_sync(full, r, 2);
  // the terms, lanes 0..5 and, in magnitude, 8..13: S2 / beta^2, a^2 S4, c^2 S6,
  // -2 a S1 / beta, -2 c S3 / beta, 2 a c S5
  const double u = tl == 0 ? t1 : tl == 2 ? cc : tl == 4 ? cb : tl < 6 ? a : 0.0;
  const double v = tl == 1 ? a : tl == 3 ? ib : tl == 5 ? c : 1.0;
  const double w = tl == 1 ? S4 : tl == 2 ? S6 : tl == 3 ? S1 : tl == 4 ? S3 : tl == 5 ? S5 : 1.0;
  const double f = tl < 3 ? 1.0 : tl < 5 ? -2.0 : 2.0;
  double term = (u * v) * (w * f);
  if (lane & 8) term = fabs(term);
#pragma unroll
  for (int o = 4; o > 0; o >>= 1) term += __shfl_xor_sync(full, term, o);
  // b2 carries a rounding error of about u mag, with mag the sum of the terms'
  // magnitudes and u the unit roundoff of the vectors
  const double b2 = __shfl_sync(full, term, 0), mag = __shfl_sync(full, term, 8);
  S.alpha = alpha;
  S.pending = 0;
  if (!isfinite(alpha) || !isfinite(b2)) {
    S.status = HS_NONFINITE; S.done = 2;
  } else if (!(b2 > EXPANSION_FLOOR<T> * mag)) {
    S.status = HS_BREAKDOWN; S.pad = PIPE_EXPANSION; S.done = 2;
  } else {
    const double ibn = rsqrt(b2);
    clu_givens(S, b2, b2 * ibn, ib);
    ibp = ib;
    ib = ibn;
  }
}

// The block of row i, among blocks lo .. hi: the last one that starts at or
// before it.
__device__ __forceinline__ int clu_block(const Geo& g, uint32_t i, int lo, int hi) {
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (__ldg(&g.blocks[mid].R) <= i) lo = mid;
    else hi = mid - 1;
  }
  return lo;
}

// Row i of H from the block tables (its block among lo .. hi): am = a_ii - sigma,
// naf = its antiparallel bonds, put(r) for the row r at the other end of each.
template <typename T, class F>
__device__ __forceinline__ void clu_row(const Geo& g, uint32_t i, int lo, int hi, double sigma, T& am,
                                        int& naf, F&& put) {
  lo = clu_block(g, i, lo, hi);
  const uint32_t* bw = reinterpret_cast<const uint32_t*>(g.blocks + lo);
  Hdr h;
  h.R = __ldg(bw);
  h.Rwrap = __ldg(bw + 1);
  h.bdelta = (int32_t)__ldg(bw + 2);
  const uint32_t meta = __ldg(bw + 3);
  h.w = meta & 0xFF;
  h.nh = (meta >> 8) & 0xFF;
  h.code = (meta >> 16) & 0xFF;
  h.off = g.cls_off[h.w];
  h.dhs = __hiloint2double((int)__ldg(bw + 5), (int)__ldg(bw + 4)) - sigma;
  h.dhs_f = (float)h.dhs;
  const LowEntry e = g.low[h.off + (int)(i - h.R)];
  const uint32_t xc = cut_mask(e.packed, h);
  for (int b = 0; b < le_cnt(e.packed); ++b)
    put(h.R + ((e.nbw[b >> 2] >> (8 * (b & 3))) & 0xFFu));
  for (int b = 0; b < h.nh; ++b) put((uint32_t)((int)i + (int)__ldg(bw + 6 + b)));
  if (xc & 1u) put((uint32_t)((int)i + h.bdelta));
  if (xc & 2u) put(h.Rwrap + e.wrap_r);
  am = diag_t<T>(e, h, xc);
  naf = naf_row(e.packed, h, xc);
}

// One solve by one cluster; every thread of every CTA calls it with the same
// job. Where trace is set, CTA 0 writes alpha_k to trace[2 (k - 1)] and beta_{k+1}
// to trace[2 (k - 1) + 1] (k = 1 .. kmax): the tridiagonal matrix of the Lanczos
// process that MINRES runs on. Rows are dealt to the CTAs in contiguous runs of rank order. Returns
// false in every CTA when a wait of any gave up (status HS_TIMEOUT). The final state
// is in sh.S of every CTA and, if job.st is set, in *job.st.
//
// Order of events (k = 1, 2, ...; the phases of a barrier follow each other
// because each is complete only when every warp of the cluster has sent, and a
// warp sends only after it has read what the phase before brought):
//   compute   wait B (q_k); p_k = (H - sigma) q_k; send alpha partials (A);
//             wait D (step k - 2): apply its d/x update, leave if it was the last;
//             wait C: q_{k+1}; send it and its norm's partials (B)
//   beta      wait B: beta_k and its reciprocal powers (F)
//   alpha     wait A, F, D (step k - 2): leave if it was the last; C: the
//             coefficients of q_{k+1}; E: alpha_k
//   rotation  wait F (beta_k) and E (alpha_{k-1}): the rotation of step k - 1; D: its
//             coefficients
template <typename T, int RPT>
__device__ bool clu_solve(const SmemJob& job, int pc, CluShared& sh, char* dyn, CluPhase& ph,
                          double* trace = nullptr) {
  const Geo& g = job.g;
  const int n = (int)g.n;
  const int cs = (int)clu_size(), me = (int)clu_rank();
  const int lane = threadIdx.x & 31;
  const int wid = (int)(threadIdx.x >> 5) - CLU_CW;   // compute warp, negative: control
  constexpr int SLOTS = 32 * CLU_NW * RPT;
  T* Q = reinterpret_cast<T*>(dyn);
  uint32_t* nbr = reinterpret_cast<uint32_t*>(dyn + clu_q_bytes<T>(n, cs, RPT));
  const int rpc = clu_rows(n, cs, RPT);
  const int r0 = me * rpc, zero = cs * rpc;           // first row, the zero element
  constexpr int V = RPT == 1 ? 1 : 2;                 // consecutive rows of a thread
  const int nwa = min(CLU_NW, (rpc / V + 31) / 32);   // compute warps with rows
  const int np = cs * nwa;
  const unsigned bytesA = 8u * np, bytesB = 8u * np + (unsigned)sizeof(T) * zero;
  const double sigma = job.sigma;
  if (threadIdx.x == 0) Q[zero] = T(0);
  clu_sync();                                    // every CTA has left the previous solve
  // A barrier's bytes are announced just before the wait of the warp that owns
  // it: data that came earlier has been counted (the count may be negative
  // meanwhile), and the phase cannot complete without this arrival.
  auto take = [&](unsigned long long* bar, unsigned bytes, unsigned& parity) {
    if (lane == 0) bar_arm(bar, bytes);
    __syncwarp();
    const bool got = bar_wait(bar, parity, ph.limit);
    parity ^= 1u;
    return got;
  };
  if (wid >= 0 && wid < nwa) {
    // ---- compute warps
    T q[RPT], qm[RPT], ql[RPT];                  // q_k, q_{k-1}, q_{k-2}
    T d1[RPT], d2[RPT], x[RPT], m[RPT], mi[RPT], dg[RPT];
    int np2[RPT];                                // neighbour pairs of the warp's longest row
    const int t0 = wid * 32 + lane;
    auto lrow = [&](int j) { return ((j / V) * 32 * CLU_NW + t0) * V + j % V; };   // in the CTA
    const uint32_t aBarA = smem_u32(&sh.barA), aBarB = smem_u32(&sh.barB);
    const uint32_t aSA = smem_u32(&sh.slotA[me * nwa + wid]);
    const uint32_t aSB = smem_u32(&sh.slotB[me * nwa + wid]);
    const uint32_t aQ = smem_u32(Q + r0 + t0 * V);
    auto slot_of = [&](int j) { return j * 32 * CLU_NW + t0; };
    auto owned = [&](int j) { return lrow(j) < rpc && r0 + lrow(j) < n; };
    T acc = T(0);
    double zm = 0.0;
#pragma unroll
    for (int j = 0; j < RPT; ++j) {
      const int slot = slot_of(j);
      q[j] = qm[j] = ql[j] = d1[j] = d2[j] = x[j] = m[j] = mi[j] = dg[j] = T(0);
      int cnt = 0;
      if (owned(j)) {
        const uint32_t i = (uint32_t)(r0 + lrow(j));
        uint16_t* out = reinterpret_cast<uint16_t*>(nbr);
        T am;
        int naf;
        clu_row<T>(g, i, 0, g.nblocks - 1, sigma, am, naf, [&](uint32_t r) {
          out[((cnt >> 1) * SLOTS + slot) * 2 + (cnt & 1)] = (uint16_t)r;
          ++cnt;
        });
        const T mm = pc == 0 ? precond_t<0, T>(am, naf)
                   : pc == 1 ? precond_t<1, T>(am, naf) : precond_t<2, T>(am, naf);
        const T b = reinterpret_cast<const T*>(job.b)[i];
        zm += mm == T(0) ? 1.0 : 0.0;
        const T im = mm == T(0) ? T(0) : T(1) / mm;
        q[j] = b * im;
        m[j] = mm;
        mi[j] = T(0.5) * im;                     // p is kept doubled, see below
        dg[j] = T(2) * am;
        acc += q[j] * b;
      }
      // a walk round the ring crosses an even number of antiparallel bonds
      np2[j] = __reduce_max_sync(0xffffffffu, cnt >> 1);
      for (int c = cnt >> 1; c < np2[j]; ++c)
        nbr[c * SLOTS + slot] = (uint32_t)zero | (uint32_t)zero << 16;
    }
    // q_{k+1} to every copy and the partial of its norm
    auto publish = [&](T part) {
      if (lrow(0) < rpc) {
#pragma unroll 4
        for (int c = 0; c < cs; ++c) {
          const int to = me + c < cs ? me + c : me + c - cs;
          const uint32_t rq = clu_map(aQ, to), rb = clu_map(aBarB, to);
#pragma unroll
          for (int j = 0; j < RPT; j += V)
            if (j == 0 || lrow(j) < rpc) {
              const uint32_t d = rq + (uint32_t)(j * 32 * CLU_NW * sizeof(T));
              if constexpr (V == 1) clu_send(d, q[j], rb);
              else clu_send2(d, q[j], q[j + 1], rb);
            }
        }
      }
      const double s = (double)warp_sum_all(part);
      if (lane < cs) clu_send(clu_map(aSB, lane), s, clu_map(aBarB, lane));
    };
    publish(acc);
    zm = warp_sum_all(zm);
    if (lane < cs) clu_send(clu_map(aSA, lane), zm, clu_map(aBarA, lane));
    // step 0 of D: the initial state
    bool ok = bar_wait(&sh.barD[0], ph.d[0], ph.limit);
    ph.d[0] ^= 1u;
    bool run = ok && sh.d[0].stop == 0;
    unsigned pb = ph.b;
    for (int k = 1; run; ++k) {
      if (!(ok = bar_wait(&sh.barB, pb, ph.limit))) break;   // q_k has arrived
      pb ^= 1u;
      // p_k, doubled: 2 (H - sigma) q = (2 a_ii - 2 sigma) q_i + sum over neighbours
      T p[RPT];
      acc = T(0);
#pragma unroll
      for (int j = 0; j < RPT; ++j) {
        const uint32_t* nl = nbr + slot_of(j);
        T s = T(0);
#pragma unroll 4
        for (int c = 0; c < np2[j]; ++c) {
          const uint32_t w = nl[c * SLOTS];
          s += Q[w & 0xFFFFu];
          s += Q[w >> 16];
        }
        p[j] = dg[j] * q[j] + s;
        acc += q[j] * p[j];
      }
      const double pa = (double)warp_sum_all(acc);
      if (lane < cs) clu_send(clu_map(aSA, lane), pa, clu_map(aBarA, lane));
      // d_{k-2} and x_{k-2} while alpha_k travels
      if (k > 2) {
        const int t = k & 1;
        if (!(ok = bar_wait(&sh.barD[t], ph.d[t], ph.limit))) break;
        ph.d[t] ^= 1u;
        if (sh.d[t].apply) {
          const T* co = reinterpret_cast<const T*>(sh.d[t].co);
          const T cq = co[0], e1 = co[1], e2 = co[2], tau = co[3];
#pragma unroll
          for (int j = 0; j < RPT; ++j) {
            const T d = cq * ql[j] + e1 * d1[j] + e2 * d2[j];
            d2[j] = d1[j];
            d1[j] = d;
            x[j] += tau * d;
          }
        }
        if (sh.d[t].stop) break;
      }
      if (!(ok = bar_wait(&sh.barC, ph.c, ph.limit))) break;
      ph.c ^= 1u;
      const T* co = reinterpret_cast<const T*>(sh.c);
      const T c1 = co[0], c2 = co[1], c3 = co[2];
      acc = T(0);
#pragma unroll
      for (int j = 0; j < RPT; ++j) {
        const T qn = p[j] * mi[j] * c1 - c2 * q[j] - c3 * qm[j];
        ql[j] = qm[j];
        qm[j] = q[j];
        q[j] = qn;
        acc += m[j] * qn * qn;
      }
      publish(acc);
    }
    if (!ok) sh.fail = 1;
    ph.b = pb;
    if (!run) ph.b ^= 1u;                        // nothing to do: B was not waited for
    T* xo = reinterpret_cast<T*>(job.x);         // may be null (trace runs)
#pragma unroll
    for (int j = 0; j < RPT; ++j)
      if (xo && owned(j)) xo[r0 + lrow(j)] = x[j];
    if (t0 == 0) {
      sh.phase[0] = ph.b; sh.phase[1] = ph.c;
      sh.phase[2] = ph.d[0]; sh.phase[3] = ph.d[1];
    }
  } else if (wid == -1) {
    // ---- beta warp
    double ib = 1.0;                             // 1 / beta_{k-1} (beta_0 = 1)
    bool ok = true;
    for (int k = 1;; ++k) {
      if (!(ok = take(&sh.barB, bytesB, ph.b))) break;
      const double sum = clu_total(sh.slotB, np);            // beta_k^2
      const double ibp = ib;
      ib = sum > 0.0 ? rsqrt(sum) : 0.0;
      // lane 0: beta_k, then beta_k / beta_{k-1}; lane 1: 1 / (2 beta_k^2), 1 / (2 beta_k^3)
      const double u = (lane & 1 ? 0.5 * ib : (sum >= 0.0 ? sum : NAN)) * ib;
      const double w = u * (lane & 1 ? ib : ibp);
      const int t = k & 1;
      if (lane < 2) {
        sh.f[t][lane ? 4 : 1] = u;
        sh.f[t][lane ? 5 : 6] = w;
        if (lane == 0) { sh.f[t][0] = sum; sh.f[t][2] = ibp; sh.f[t][3] = ib; }
      }
      if (trace && me == 0 && lane == 0 && k > 1 && k - 1 <= job.kmax) trace[2 * (k - 2) + 1] = u;
      __syncwarp();
      if (lane == 0) bar_arrive(&sh.barF[t]);
      // this iteration's B is the last one once step k - 2 (k = 1: the initial
      // state) says stop
      if (k == 1 || k > 2) {
        const int v = k == 1 ? 0 : t;
        if (!(ok = bar_wait(&sh.barD[v], ph.d[v], ph.limit))) break;
        ph.d[v] ^= 1u;
        if (sh.d[v].stop) break;
      }
    }
    if (!ok) sh.fail = 1;
  } else if (wid == -CLU_CW) {
    // ---- alpha warp (its first sum: the rows with M_ii = 0, handed on as alpha_0)
    bool ok = true;
    for (int k = 0;; ++k) {
      const int t = k & 1;
      if (!(ok = take(&sh.barA, bytesA, ph.a))) break;
      if (k > 0) {
        if (!(ok = bar_wait(&sh.barF[t], ph.f[t], ph.limit))) break;
        ph.f[t] ^= 1u;
      }
      if (k > 2) {
        if (!(ok = bar_wait(&sh.barD[t], ph.d[t], ph.limit))) break;
        ph.d[t] ^= 1u;
        if (sh.d[t].stop) break;
      }
      const double tot = clu_total(sh.slotA, np);
      if (k == 0) {
        if (lane == 0) { sh.alpha[0] = tot; bar_arrive(&sh.barE[0]); }
        if (!(ok = bar_wait(&sh.barD[0], ph.d[0], ph.limit))) break;
        ph.d[0] ^= 1u;
        if (sh.d[0].stop) {                      // beta_1 came, but no product follows
          ph.f[1] ^= 1u;
          break;
        }
        continue;
      }
      const double al = clu_alpha(sh.f[t], k, tot);
      if (lane == 0) {
        T* co = reinterpret_cast<T*>(sh.c);
        co[0] = (T)sh.f[t][3]; co[1] = (T)al; co[2] = (T)sh.f[t][6];
        bar_arrive(&sh.barC);
      }
      if (lane == 1) { sh.alpha[t] = al; bar_arrive(&sh.barE[t]); }
      if (trace && me == 0 && lane == 1 && k <= job.kmax) trace[2 * (k - 1)] = al;
    }
    if (!ok) sh.fail = 1;
  } else if (wid == 1 - CLU_CW) {
    // ---- rotation warp: step k - 1 in iteration k (k = 1: the initial state)
    MinresState S{};
    S.k = 1;
    bool ok = true;
    for (int k = 1;; ++k) {
      const int t = k & 1, u = t ^ 1;
      if (!(ok = bar_wait(&sh.barF[t], ph.f[t], ph.limit))) break;
      ph.f[t] ^= 1u;
      if (!(ok = bar_wait(&sh.barE[u], ph.e[u], ph.limit))) break;
      ph.e[u] ^= 1u;
      if (S.done != 0) break;                    // an iteration begun past the last step
      const double al = sh.alpha[u];
      if (k == 1) {
        init_state(S, sh.f[t][0], al, job.tol, job.kmax, sigma);
      } else {
        S.alpha = al;
        S.pending = 0;
        clu_givens(S, sh.f[t][0], sh.f[t][1], sh.f[t][2]);
      }
      if (lane == 0) {
        T* co = reinterpret_cast<T*>(sh.d[u].co);
        co[0] = (T)S.cq; co[1] = (T)S.cd1; co[2] = (T)S.cd2; co[3] = (T)S.tau;
        sh.d[u].apply = S.pending;
        sh.d[u].stop = S.done != 0;
        bar_arrive(&sh.barD[u]);
      }
      if (S.done != 0 && k == 1) break;
    }
    if (!ok) sh.fail = 1;
    S.pending = 0;
    S.done = 2;
    if (lane == 0) sh.S = S;
  }
  __syncthreads();
  if (wid >= nwa) {
    ph.b = sh.phase[0]; ph.c = sh.phase[1];
    ph.d[0] = sh.phase[2]; ph.d[1] = sh.phase[3];
  }
  const bool ok = clu_agree(sh);
  if (threadIdx.x == 0) {
    if (!ok) sh.S.status = HS_TIMEOUT;
    if (me == 0 && job.st) *job.st = sh.S;
  }
  __syncthreads();
  return ok;
}

// The rows per thread that a chain of n rows needs on cs CTAs; 0: too many.
__host__ __device__ inline int clu_rpt(int n, int cs) {
  const int need = ((n + cs - 1) / cs + 32 * CLU_NW - 1) / (32 * CLU_NW);
  return need <= 1 ? 1 : need <= 2 ? 2 : need <= 4 ? 4 : need <= CLU_RPT_MAX ? CLU_RPT_MAX : 0;
}

// clu_solve in FP64 with the rows per thread chosen at run time.
__device__ inline bool clu_solve64(int rpt, const SmemJob& job, int pc, CluShared& sh, char* dyn,
                                   CluPhase& ph, double* trace = nullptr) {
  switch (rpt) {
    case 1: return clu_solve<double, 1>(job, pc, sh, dyn, ph, trace);
    case 2: return clu_solve<double, 2>(job, pc, sh, dyn, ph, trace);
    case 4: return clu_solve<double, 4>(job, pc, sh, dyn, ph, trace);
    default: return clu_solve<double, CLU_RPT_MAX>(job, pc, sh, dyn, ph, trace);
  }
}

// Launch of a kernel on clusters of cs CTAs (grid: a multiple of cs); false
// when it is refused.
template <typename K, typename... A>
inline bool clu_launch(K kern, int grid, int cs, size_t smem, cudaStream_t s, A... args) {
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(grid);
  cfg.blockDim = dim3(CLU_NT);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = cs;
  at[0].val.clusterDim.y = 1;
  at[0].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  if (cs < 1 || cs > CLU_SIZE_MAX || !allow_smem(kern, smem) ||
      (cs > 8 && cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) !=
                     cudaSuccess) ||
      cudaLaunchKernelEx(&cfg, kern, args...) != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  count_launches(1);
  return true;
}

}  // namespace hs
