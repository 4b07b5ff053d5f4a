// Preconditioned MINRES of Algorithm 2 (Appendix A) on the whole GPU with one
// thread per row (up to three), for chains that a cluster cannot hold and that give
// a CTA at most 1248 rows (three for each of its 416 compute threads): L = 18 on 39
// SMs and more, L = 20 on 149 and more; a smaller share takes k_minres_smem. One cooperative launch, two reductions per iteration, the arithmetic
// of k_minres_smem.
//
// What bounded k_minres_smem (38 us per FP64 iteration at n = 184756, 19 of them
// the product): each warp gathered a 32-row chunk of q in four or five rounds of
// trips to L2, one after the other, and several chunks one after the other; the
// scalars ran on one thread between the reductions. Here
//   * each thread holds the vectors of its rows in registers and a list of its
//     rows' neighbours in shared memory, and issues the loads of a row's
//     neighbours sixteen at a time;
//   * three control warps per CTA run the reductions and the scalars as in the
//     cluster form (minres_clu.cuh): the Givens rotation of an iteration overlaps
//     the next one's product, its d/x update fills the wait for alpha;
//   * rows are dealt to threads by their number of neighbours, so that a warp's
//     rows have about the same (10.5 FP64 additions a row on average at L = 20,
//     16 to 18 for the longest of 32 rows in rank order);
//   * in a reduction only CTA 0 reads every CTA's partial sum (grid_total).
// Per iteration (us, row norm, 152 SMs, before -> here): L = 18 FP64 19.7 (one
// reduction) -> 11.4, FP32 17.9 -> 9.0; L = 20 FP64 37.7 -> 18.6, FP32 20.1 -> 10.0.
// At L = 20 the FP64 pipe takes about 10 us of it (26 instructions a row, 19
// cycles per warp and SM), the two exchanges about 3 us each.
#include <algorithm>
#include <cstdlib>

#include "minres_row.cuh"

namespace hs {

namespace {

constexpr int ROW_NW = 13;                      // compute warps (n = 184756: 1216 rows on 152
                                                // SMs, three per thread)
constexpr int ROW_NT = 32 * (ROW_NW + CLU_CW);  // and the control warps
constexpr int ROW_THREADS = 32 * ROW_NW;

struct RowShared {
  double partA[ROW_NW], partB[ROW_NW];          // the warps' partial sums
  unsigned long long barA, barB;                // compute warps -> control warps
  unsigned long long barQ;                      // q_k is complete
  unsigned long long barC, barF[2], barE[2], barD[2];   // as in CluShared
  double c[3], f[2][8], alpha[2];
  struct { double co[4]; int apply, stop; } d[2];
  int fail;
};

// Sum of the warps' partials, in every lane.
__device__ __forceinline__ double row_parts(const double* part, int nwa) {
  const int lane = threadIdx.x & 31;
  double v = lane < nwa ? part[lane] : 0.0;
#pragma unroll
  for (int o = 8; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return __shfl_sync(0xffffffffu, v, 0);
}

template <typename T, int RPT>
__global__ void __launch_bounds__(ROW_NT, 1) k_minres_row(RowArgs ra, int pc) {
  extern __shared__ __align__(16) char dyn[];
  __shared__ RowShared sh;
  const SmemJob& job = ra.job;
  const Geo& g = job.g;
  const int n = (int)g.n;
  const int G = gridDim.x, cta = blockIdx.x;
  const int lane = threadIdx.x & 31;
  const int wid = (int)(threadIdx.x >> 5) - CLU_CW;
  constexpr int SLOTS = ROW_THREADS * RPT;
  uint32_t* nbr = reinterpret_cast<uint32_t*>(dyn);   // [neighbour][slot]
  __shared__ uint16_t order[SLOTS];                   // rows by falling number of neighbours
  __shared__ uint8_t bonds[SLOTS];
  __shared__ int s_blk[2];                            // the CTA's blocks
  __shared__ int s_class[LMAX / 2];
  static_assert(ROW_NT / 32 >= LMAX / 2, "one warp per number of neighbours");
  const int rpc = (n + G - 1) / G;
  const int r0 = min(n, cta * rpc), rows = min(n, r0 + rpc) - r0;
  // compute warps with rows (RPT > 1: all, the last rows go to the last warps)
  const int nwa = rows > ROW_THREADS ? ROW_NW : (rows + 31) / 32;
  T* q_glob = reinterpret_cast<T*>(ra.q);
  GridWord* slotA = ra.slots;
  GridWord* slotB = ra.slots + GRID_WORDS * G;
  if (threadIdx.x == 0) {
    bar_init(&sh.barA, max(1, nwa));
    bar_init(&sh.barB, max(1, nwa));
    bar_init(&sh.barQ, 1);
    bar_init(&sh.barC, 1);
    for (int i = 0; i < 2; ++i) {
      bar_init(&sh.barF[i], 1);
      bar_init(&sh.barE[i], 1);
      bar_init(&sh.barD[i], 1);
    }
    sh.fail = 0;
  }
  row_deal<T>(g, r0, rows, order, bonds, s_blk, s_class);
  unsigned pd[2] = {0, 0};
  if (wid >= 0 && wid < nwa) {
    // ---- compute warps
    T q[RPT], qm[RPT], ql[RPT];                  // q_k, q_{k-1}, q_{k-2}
    T d1[RPT], d2[RPT], x[RPT], m[RPT], mi[RPT], dg[RPT];
    int cnt[RPT];
    const int t0 = wid * 32 + lane;
    // the j-th row: the longest third (or half) of the list forwards, the rest
    // backwards, so that the warps' sums are about the same
    auto place = [&](int j) { return j * ROW_THREADS + (j ? ROW_THREADS - 1 - t0 : t0); };
    auto owned = [&](int j) { return place(j) < rows; };
    int row[RPT];
#pragma unroll
    for (int j = 0; j < RPT; ++j) row[j] = owned(j) ? r0 + order[place(j)] : -1;
    auto send = [&](double* part, unsigned long long* bar, T v) {
      const double s = (double)warp_sum_all(v);
      __syncwarp();
      if (lane == 0) { part[wid] = s; bar_arrive(bar); }
    };
    T acc = T(0), zm = T(0);
#pragma unroll
    for (int j = 0; j < RPT; ++j) {
      const int slot = j * ROW_THREADS + t0;
      q[j] = qm[j] = ql[j] = d1[j] = d2[j] = x[j] = m[j] = mi[j] = dg[j] = T(0);
      cnt[j] = 0;
      if (owned(j)) {
        const uint32_t i = (uint32_t)row[j];
        T am;
        int naf;
        clu_row<T>(g, i, s_blk[0], s_blk[1], job.sigma, am, naf, [&](uint32_t r) {
          nbr[cnt[j] * SLOTS + slot] = r;
          ++cnt[j];
        });
        const T mm = pc == 0 ? precond_t<0, T>(am, naf)
                   : pc == 1 ? precond_t<1, T>(am, naf) : precond_t<2, T>(am, naf);
        const T b = reinterpret_cast<const T*>(job.b)[i];
        zm += mm == T(0) ? T(1) : T(0);
        const T im = mm == T(0) ? T(0) : T(1) / mm;
        q[j] = b * im;
        m[j] = mm;
        mi[j] = T(0.5) * im;                     // p is kept doubled
        dg[j] = T(2) * am;
        acc += q[j] * b;
        q_glob[i] = q[j];
      }
    }
    send(sh.partB, &sh.barB, acc);
    send(sh.partA, &sh.barA, zm);
    bool ok = row_wait(sh.fail, &sh.barD[0], pd[0]);
    pd[0] ^= 1u;
    bool run = ok && sh.d[0].stop == 0;
    unsigned pq = 0, pcb = 0;
    for (int k = 1; run; ++k) {
      if (!(ok = row_wait(sh.fail, &sh.barQ, pq))) break;   // q_k is complete
      pq ^= 1u;
      acc = T(0);
      T p[RPT];
#pragma unroll
      for (int j = 0; j < RPT; ++j) {
        // 2 (H - sigma) q = (2 a_ii - 2 sigma) q_i + sum over neighbours
        const uint32_t* nl = nbr + j * ROW_THREADS + t0;
        T s = T(0);
        const int most = __reduce_max_sync(0xffffffffu, cnt[j]);
        for (int c0 = 0; c0 < most; c0 += ROW_BATCH) {
          T v[ROW_BATCH];
#pragma unroll
          for (int c = 0; c < ROW_BATCH; ++c)
            v[c] = c0 + c < cnt[j] ? __ldcg(q_glob + nl[(c0 + c) * SLOTS]) : T(0);
#pragma unroll
          for (int c = 0; c < ROW_BATCH; ++c)
            if (c0 + c < most) s += v[c];
        }
        p[j] = dg[j] * q[j] + s;
        acc += q[j] * p[j];
      }
      send(sh.partA, &sh.barA, acc);
      // d_{k-2} and x_{k-2} while alpha_k is summed
      if (k > 2) {
        const int t = k & 1;
        if (!(ok = row_wait(sh.fail, &sh.barD[t], pd[t]))) break;
        pd[t] ^= 1u;
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
      if (!(ok = row_wait(sh.fail, &sh.barC, pcb))) break;
      pcb ^= 1u;
      const T* co = reinterpret_cast<const T*>(sh.c);
      const T c1 = co[0], c2 = co[1], c3 = co[2];
      acc = T(0);
#pragma unroll
      for (int j = 0; j < RPT; ++j) {
        const T qn = p[j] * mi[j] * c1 - c2 * q[j] - c3 * qm[j];
        ql[j] = qm[j];
        qm[j] = q[j];
        q[j] = qn;
        if (row[j] >= 0) q_glob[row[j]] = qn;
        acc += m[j] * qn * qn;
      }
      send(sh.partB, &sh.barB, acc);
    }
    if (!ok) row_fail(sh.fail, ra.err);
    T* xo = reinterpret_cast<T*>(job.x);
#pragma unroll
    for (int j = 0; j < RPT; ++j)
      if (row[j] >= 0) xo[row[j]] = x[j];
  } else if (wid == -1) {
    // ---- beta warp (the schedule of minres_clu.cuh, the sums over the grid)
    double ib = 1.0;
    bool ok = true;
    unsigned pb = 0;
    for (int k = 1;; ++k) {
      if (nwa > 0) {
        if (!(ok = row_wait(sh.fail, &sh.barB, pb))) break;
        pb ^= 1u;
      }
      double sum;
      if (!(ok = grid_total<true>(slotB, G, cta, (unsigned long long)k, row_parts(sh.partB, nwa), sum,
                           ra.limit, ra.err)))
        break;
      if (lane == 0) bar_arrive(&sh.barQ);                   // every CTA has stored its q_k
      const double ibp = ib;
      ib = sum > 0.0 ? rsqrt(sum) : 0.0;
      const double u = (lane & 1 ? 0.5 * ib : (sum >= 0.0 ? sum : NAN)) * ib;
      const double w = u * (lane & 1 ? ib : ibp);
      const int t = k & 1;
      if (lane < 2) {
        sh.f[t][lane ? 4 : 1] = u;
        sh.f[t][lane ? 5 : 6] = w;
        if (lane == 0) { sh.f[t][0] = sum; sh.f[t][2] = ibp; sh.f[t][3] = ib; }
      }
      __syncwarp();
      if (lane == 0) bar_arrive(&sh.barF[t]);
      if (k == 1 || k > 2) {
        const int v = k == 1 ? 0 : t;
        if (!(ok = row_wait(sh.fail, &sh.barD[v], pd[v]))) break;
        pd[v] ^= 1u;
        if (sh.d[v].stop) break;
      }
    }
    if (!ok) row_fail(sh.fail, ra.err);
  } else if (wid == -CLU_CW) {
    // ---- alpha warp
    bool ok = true;
    unsigned pa = 0, pf[2] = {0, 0};
    for (int k = 0;; ++k) {
      const int t = k & 1;
      if (nwa > 0) {
        if (!(ok = row_wait(sh.fail, &sh.barA, pa))) break;
        pa ^= 1u;
      }
      double tot;
      if (!(ok = grid_total<false>(slotA, G, cta, (unsigned long long)k + 1, row_parts(sh.partA, nwa), tot,
                           ra.limit, ra.err)))
        break;
      if (k > 0) {
        if (!(ok = row_wait(sh.fail, &sh.barF[t], pf[t]))) break;
        pf[t] ^= 1u;
      }
      if (k > 2) {
        if (!(ok = row_wait(sh.fail, &sh.barD[t], pd[t]))) break;
        pd[t] ^= 1u;
        if (sh.d[t].stop) break;
      }
      if (k == 0) {
        if (lane == 0) { sh.alpha[0] = tot; bar_arrive(&sh.barE[0]); }
        if (!(ok = row_wait(sh.fail, &sh.barD[0], pd[0]))) break;
        pd[0] ^= 1u;
        if (sh.d[0].stop) break;
        continue;
      }
      const double al = clu_alpha(sh.f[t], k, tot);
      if (lane == 0) {
        T* co = reinterpret_cast<T*>(sh.c);
        co[0] = (T)sh.f[t][3]; co[1] = (T)al; co[2] = (T)sh.f[t][6];
        bar_arrive(&sh.barC);
      }
      if (lane == 1) { sh.alpha[t] = al; bar_arrive(&sh.barE[t]); }
    }
    if (!ok) row_fail(sh.fail, ra.err);
  } else if (wid == 1 - CLU_CW) {
    // ---- rotation warp
    MinresState S{};
    S.k = 1;
    bool ok = true;
    unsigned pf[2] = {0, 0}, pe[2] = {0, 0};
    for (int k = 1;; ++k) {
      const int t = k & 1, u = t ^ 1;
      if (!(ok = row_wait(sh.fail, &sh.barF[t], pf[t]))) break;
      pf[t] ^= 1u;
      if (!(ok = row_wait(sh.fail, &sh.barE[u], pe[u]))) break;
      pe[u] ^= 1u;
      if (S.done != 0) break;                    // an iteration begun past the last step
      const double al = sh.alpha[u];
      if (k == 1) {
        init_state(S, sh.f[t][0], al, job.tol, job.kmax, job.sigma);
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
    if (!ok) row_fail(sh.fail, ra.err);
    S.pending = 0;
    S.done = 2;
    if (!ok) S.status = HS_TIMEOUT;
    if (lane == 0 && cta == 0) *job.st = S;
  }
}

template <typename T, int RPT>
hs_status launch_row_t(hs_handle* hd, const RowArgs& ra, int pc, int G) {
  const size_t sm = sizeof(uint32_t) * (size_t)hd->L * ROW_THREADS * RPT;
  auto kern = k_minres_row<T, RPT>;
  RowArgs a = ra;
  int p = pc;
  void* args[] = {&a, &p};
  return row_launch(hd, (const void*)kern, G, ROW_NT, sm, 4 * ROW_THREADS * RPT + 1024, args);
}

template <typename T>
hs_status launch_row(hs_handle* hd, const RowArgs& ra, int pc, int G) {
  const int rpc = ((int)hd->n + G - 1) / G;
  switch ((rpc + ROW_THREADS - 1) / ROW_THREADS) {
    case 1: return launch_row_t<T, 1>(hd, ra, pc, G);
    case 2: return launch_row_t<T, 2>(hd, ra, pc, G);
    case 3: return launch_row_t<T, 3>(hd, ra, pc, G);
    default: return HS_CUDA;
  }
}

}  // namespace

hs_status row_launch(hs_handle* hd, const void* kern, int G, int nt, size_t smem, size_t fixed,
                     void** args) {
  int optin = 0;
  cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, hd->device);
  if (smem + fixed > (size_t)optin) return HS_CUDA;
  if (!allow_smem(kern, smem) ||
      cudaLaunchCooperativeKernel(kern, dim3(G), dim3(nt), args, smem, hd->stream) != cudaSuccess) {
    cudaGetLastError();
    return HS_CUDA;
  }
  count_launches(1);
  return HS_OK;
}

hs_status row_args(hs_handle* hd, const void* b, const MinresVecs& v, double tol, long long kmax,
                   int exchanges, RowArgs* ra, int* G) {
  const int bud = hd->sm_budget.load(std::memory_order_relaxed);
  *G = std::max(1, std::min(hd->num_sms, bud > 0 ? bud : hd->num_sms));
  if (*G > 256) return HS_CUDA;
  ra->job = SmemJob{hd->geo(), b, v.x, hd->d_state, hd->sigma, tol, kmax};
  ra->slots = reinterpret_cast<GridWord*>(hd->d_partial);
  ra->err = reinterpret_cast<int*>(hd->d_counter + 10);
  ra->limit = 1ull << 22;
  if (const char* e = getenv("HS_BARRIER_LIMIT")) ra->limit = strtoull(e, nullptr, 10);
  ra->q = v.q0;
  ra->w0 = v.q1;
  ra->w1 = v.p;
  HS_CUDA_TRY(hd, cudaMemsetAsync(hd->d_counter + 10, 0, sizeof(unsigned), hd->stream));
  HS_CUDA_TRY(hd, cudaMemsetAsync(hd->d_partial, 0, exchanges * GRID_WORDS * sizeof(GridWord) * *G,
                                  hd->stream));
  return HS_OK;
}

hs_status grid_finish(hs_handle* hd) {
  int* gave_up = reinterpret_cast<int*>(hd->h_pinned);
  HS_CUDA_TRY(hd, cudaMemcpyAsync(hd->h_state, hd->d_state, sizeof(MinresState),
                                  cudaMemcpyDeviceToHost, hd->stream));
  HS_CUDA_TRY(hd, cudaMemcpyAsync(gave_up, hd->d_counter + 10, sizeof(int), cudaMemcpyDeviceToHost,
                                  hd->stream));
  HS_CUDA_TRY(hd, cudaStreamSynchronize(hd->stream));
  if (*gave_up) hd->h_state->status = HS_TIMEOUT;
  return HS_OK;
}

hs_status solve_row(hs_handle* hd, const void* b, const MinresVecs& v, hs_dtype dt, int pc,
                    double tol, long long kmax) {
  RowArgs ra{};
  int G = 0;
  hs_status st = row_args(hd, b, v, tol, kmax, 2, &ra, &G);
  if (st != HS_OK) return st;
  st = dt == HS_F64 ? launch_row<double>(hd, ra, pc, G) : launch_row<float>(hd, ra, pc, G);
  return st != HS_OK ? st : grid_finish(hd);
}

}  // namespace hs
