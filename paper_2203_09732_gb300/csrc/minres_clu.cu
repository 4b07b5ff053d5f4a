// Preconditioned MINRES of Algorithm 2 (Appendix A) in one thread-block
// cluster, for chains of up to 16384 rows (minres_clu.cuh): the kernel of a
// single solve and the choice of the cluster size.
#include <algorithm>
#include <cstdlib>

#include "minres_clu.cuh"

namespace hs {

namespace {

template <typename T, int RPT>
__global__ void __launch_bounds__(CLU_NT, 1) k_minres_clu(SmemJob job, int pc, unsigned limit) {
  extern __shared__ __align__(16) char dyn[];
  __shared__ CluShared sh;
  clu_setup(sh);
  CluPhase ph{limit};
  clu_solve<T, RPT>(job, pc, sh, dyn, ph);
  clu_sync();   // no CTA leaves while another may still write to it
}

// One FP64 solve per cluster: jobs[blockIdx.x / cs] (all of one L), the
// Lanczos scalars in trace + cluster * tstride where trace is set.
__global__ void __launch_bounds__(CLU_NT, 1) k_minres_clu_many(const SmemJob* jobs, int pc,
                                                               double* trace, long long tstride,
                                                               unsigned limit) {
  extern __shared__ __align__(16) char dyn[];
  __shared__ CluShared sh;
  __shared__ SmemJob sj;
  clu_setup(sh);
  CluPhase ph{limit};
  const int cs = (int)clu_size(), id = (int)blockIdx.x / cs;
  if (threadIdx.x == 0) sj = jobs[id];
  __syncthreads();
  clu_solve64(clu_rpt((int)sj.g.n, cs), sj, pc, sh, dyn, ph, trace ? trace + id * tstride : nullptr);
  clu_sync();
}

template <typename T, int RPT>
hs_status launch_t(hs_handle* hd, const SmemJob& job, int pc, int cs) {
  return clu_launch(k_minres_clu<T, RPT>, cs, cs, clu_bytes<T>((int)hd->n, hd->L, cs, RPT),
                    hd->stream, job, pc, clu_limit())
             ? HS_OK : HS_CUDA;
}

template <typename T>
hs_status launch_rpt(hs_handle* hd, const SmemJob& job, int pc, int cs) {
  const int rpt = clu_rpt((int)hd->n, cs);
  // rows per thread: as few as hold the rows in FP64 (each row is FP64 work on
  // the critical path); two at least in FP32, where half the warps make half
  // the partials and messages (n = 924, 8 CTAs: 1.72 -> 1.59 us per iteration;
  // FP64 there 2.38 -> 3.00)
  if constexpr (sizeof(T) == 8)
    if (rpt == 1) return launch_t<T, 1>(hd, job, pc, cs);
  switch (rpt) {
    case 1:
    case 2: return launch_t<T, 2>(hd, job, pc, cs);
    case 4: return launch_t<T, 4>(hd, job, pc, cs);
    case CLU_RPT_MAX: return launch_t<T, CLU_RPT_MAX>(hd, job, pc, cs);
    default: return HS_CUDA;
  }
}

}  // namespace

// CTAs per cluster. More CTAs share the FP64 work but make every exchange
// longer. Measured per iteration (us, row norm, FP64 / FP32; the grid forms
// that took these solves before in brackets):
//   n = 70     1 CTA 1.92 / 1.25, 8 CTAs 1.99 / 1.48                    (12.2 / 15.2)
//   n = 252    1 CTA 2.74 / 1.35, 2 CTAs 2.16 / 1.35, 8 CTAs 2.09 / 1.48  (11.4 / 15.6)
//   n = 924    4 CTAs 3.09 / 1.60, 8 CTAs 2.43 / 1.60, 16 CTAs 2.45 / 1.69 (11.7 / 15.6)
//   n = 3432   8 CTAs 5.46 / 2.29, 16 CTAs 4.04 / 2.19                     (12.2 / 17.1)
//   n = 12870  16 CTAs FP32 4.78                                            (17.8)
// FP64 at n = 12870 stays with the grid forms where the one-reduction recurrence
// serves (cluster_choice: Jacobi, 16 CTAs, 12.5 us). HS_MINRES_CLUSTER
// sets the number of CTAs (a power of two, at most 16; 0: off).
int clu_choice(long long n, int sms) {
  if (n > CLU_ROWS) return 0;
  int cs = n <= 128 ? 1 : n <= 512 ? 2 : n <= 1024 ? 8 : 16;
  if (const char* e = getenv("HS_MINRES_CLUSTER")) cs = atoi(e);
  while (cs > sms) cs >>= 1;
  return cs;
}

unsigned clu_limit() {
  const char* e = getenv("HS_BARRIER_LIMIT");
  return e ? (unsigned)std::min<unsigned long long>(strtoull(e, nullptr, 10), CLU_WAIT_LIMIT)
           : CLU_WAIT_LIMIT;
}

hs_status solve_clu(hs_handle* hd, const void* b, void* x, hs_dtype dt, int pc, double tol,
                    long long kmax, int cs) {
  const SmemJob job{hd->geo(), b, x, hd->d_state, hd->sigma, tol, kmax};
  const hs_status st = dt == HS_F64 ? launch_rpt<double>(hd, job, pc, cs)
                                    : launch_rpt<float>(hd, job, pc, cs);
  if (st != HS_OK) return st;
  HS_CUDA_TRY(hd, cudaMemcpyAsync(hd->h_state, hd->d_state, sizeof(MinresState),
                                  cudaMemcpyDeviceToHost, hd->stream));
  HS_CUDA_TRY(hd, cudaStreamSynchronize(hd->stream));
  return HS_OK;
}

hs_status launch_clu_many(const SmemJob* jobs, int count, int n, int L, int pc, int cs,
                          cudaStream_t s, double* trace, long long tstride, unsigned limit) {
  const int rpt = clu_rpt(n, cs);
  if (!rpt) return HS_CUDA;
  return clu_launch(k_minres_clu_many, count * cs, cs, clu_bytes<double>(n, L, cs, rpt), s, jobs, pc,
                    trace, tstride, limit)
             ? HS_OK : HS_CUDA;
}

}  // namespace hs
