// Twist overlap z = <psi| U_twist |psi>, U_twist = exp[i 2pi/L sum_j j Sz_j]
// (Sec. III). In the Sz basis U is diagonal with u_alpha = exp(i 2pi/L (t - L(L+1)/4)),
// t = sum of the (1-based) sites that are up, so
//   z = exp(-i pi (L+1)/2) sum_{r=0}^{L-1} W_r exp(i 2pi r / L),
//   W_r = sum_{alpha: t_alpha = r mod L} c_alpha^2   (Appendix B's z = sum c^2 u).
// The kernel accumulates the L bins W_r in FP64; t = tlow(p) + thigh(H).
#include <algorithm>
#include <cmath>

#include "rows.cuh"

namespace hs {

namespace {

// One FP64 operation per entry (acc = c c + acc) is what the sum needs: 2.0 ps an
// entry on 152 SMs at the FP64 pipe's 19 cycles per warp and SM, against 1.2 ps for
// reading its 8 bytes (ten vectors of L = 24, 27 M entries: 53 and 32 us). So each lane of each warp has its
// own L accumulators in shared memory ([bin][lane], no bank conflicts, no
// atomics: FP64 atomics in shared memory are compare-and-swap loops), all
// vectors go in one launch, each on its own CTAs, and one small kernel adds the
// CTAs' bins in a fixed order. L = 24, 10 vectors: 870 -> 112 us a call.
constexpr int TW_NT = 256;
constexpr int TW_WARPS = TW_NT / 32;
constexpr int TW_LOW = 1 << KLO_MAX;

size_t tw_smem(int L) { return sizeof(double) * (size_t)TW_WARPS * 32 * L; }

// Vector q = blockIdx.y, this CTA's blocks of the chain: part[(q gridDim.x +
// blockIdx.x) 32 + r] = W_r of its rows (r < L).
__global__ void __launch_bounds__(TW_NT) k_twist(Geo g, const double* __restrict__ psi,
                                                 double* __restrict__ part) {
  extern __shared__ double bins[];                // [warp][bin][lane]
  __shared__ uint8_t tl[TW_LOW];                  // tlow mod L of the low patterns
  const int L = g.L;
  for (int i = threadIdx.x; i < g.nlow; i += TW_NT)
    tl[i] = (uint8_t)(le_tlow(__ldg(&g.low[i].packed)) % (uint32_t)L);
  const int wid = threadIdx.x >> 5, lane = threadIdx.x & 31;
  double* mine = bins + (size_t)wid * L * 32 + lane;
  for (int b = 0; b < L; ++b) mine[b * 32] = 0.0;
  __syncthreads();
  const double* v = psi + (size_t)blockIdx.y * g.n;
  const int stride = gridDim.x * TW_WARPS;
  for (int bi = blockIdx.x * TW_WARPS + wid; bi < g.nblocks; bi += stride) {
    const uint32_t* w = reinterpret_cast<const uint32_t*>(g.blocks + bi);
    const uint32_t R = __ldg(w), meta = __ldg(w + 3);
    const int cls = meta & 0xFF, C = g.cls_C[cls], th = (int)(meta >> 24);
    const uint8_t* t = tl + g.cls_off[cls];
    double c[JMAX];
#pragma unroll
    for (int j = 0; j < JMAX; ++j) {
      const int r = lane + 32 * j;
      c[j] = r < C ? __ldg(v + R + r) : 0.0;
    }
#pragma unroll
    for (int j = 0; j < JMAX; ++j) {
      if (32 * j >= C) break;
      const int r = lane + 32 * j;
      int b = th + (int)t[r < C ? r : 0];
      if (b >= L) b -= L;
      mine[b * 32] = fma(c[j], c[j], mine[b * 32]);
    }
  }
  __syncthreads();
  // warp b adds bin b over the lanes of all warps
  for (int b = wid; b < L; b += TW_WARPS) {
    double s = 0.0;
    for (int q = 0; q < TW_WARPS; ++q) s += bins[((size_t)q * L + b) * 32 + lane];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
    if (lane == 0) part[((size_t)blockIdx.y * gridDim.x + blockIdx.x) * 32 + b] = s;
  }
}

// W[q][r] = sum over the CTAs of vector q, in a fixed order.
__global__ void __launch_bounds__(128) k_twist_sum(const double* __restrict__ part, int ncta, int L,
                                                   double* __restrict__ W) {
  __shared__ double s[4][32];
  const int wid = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const double* p = part + (size_t)blockIdx.x * ncta * 32 + lane;
  double t = 0.0;
  if (lane < L)
    for (int c = wid; c < ncta; c += 4) t += p[(size_t)c * 32];
  s[wid][lane] = t;
  __syncthreads();
  if (wid == 0) W[(size_t)blockIdx.x * 32 + lane] = (s[0][lane] + s[1][lane]) + (s[2][lane] + s[3][lane]);
}

}  // namespace

hs_status launch_twist(hs_handle* hd, const double* psi, int K, double* z_host) {
  hs_status st = ensure_reduce(hd);
  if (st != HS_OK) return st;
  const int L = hd->L;
  const size_t sm = tw_smem(L);
  if (!allow_smem(k_twist, sm)) return fail(hd, HS_CUDA, "hs_twist: shared memory");
  // CTAs per vector: about three per SM in all, at least four blocks a warp; the
  // sums of a launch's vectors first in the scratch, then the CTAs' bins
  constexpr int KB = 64;
  const int most = std::max(1, (int)hd->blocks.size() / (4 * TW_WARPS));
  for (int q0 = 0; q0 < K; q0 += KB) {
    const int kb = std::min(KB, K - q0);
    const int ncta = std::max(1, std::min(most, 3 * hd->num_sms / kb));
    double* W = hd->d_partial;
    double* part = W + KB * 32;
    k_twist<<<dim3(ncta, kb), TW_NT, sm, hd->stream>>>(hd->geo(), psi + (long long)q0 * hd->n, part);
    k_twist_sum<<<kb, 128, 0, hd->stream>>>(part, ncta, L, W);
    count_launches(2);
    HS_CUDA_TRY(hd, cudaGetLastError());
    HS_CUDA_TRY(hd, cudaMemcpyAsync(hd->h_pinned, W, sizeof(double) * kb * 32,
                                    cudaMemcpyDeviceToHost, hd->stream));
    HS_CUDA_TRY(hd, cudaStreamSynchronize(hd->stream));
    for (int q = 0; q < kb; ++q) {
      double re = 0, im = 0;
      for (int r = 0; r < L; ++r) {
        const double a = 2.0 * M_PI * r / L;
        re += hd->h_pinned[32 * q + r] * std::cos(a);
        im += hd->h_pinned[32 * q + r] * std::sin(a);
      }
      // global phase exp(-i pi (L+1)/2): L even, so (L+1)/2 is a half-integer
      const double ph = -M_PI * (L + 1) / 2.0;
      const double cr = std::cos(ph), ci = std::sin(ph);
      z_host[2 * (q0 + q)] = re * cr - im * ci;
      z_host[2 * (q0 + q) + 1] = re * ci + im * cr;
    }
  }
  return HS_OK;
}

}  // namespace hs
