// Matrix-free H x (Eq. (1)), the basis ranking (Sec. I: Sz = 0 sector in
// ascending integer order), the diagonal / preconditioner export (Sec. II) and
// the FP64 refinement residual r = b - (H - sigma) x.
#include <algorithm>
#include <cstdlib>

#include "hv_cls.cuh"

namespace hs {

// ---------------------------------------------------------------------------
// v / 2. FP64: by the exponent where that is exact in every lane of the warp (a few
// integer instructions instead of one on the FP64 pipe).
__device__ __forceinline__ float half_of(float v) { return 0.5f * v; }
__device__ __forceinline__ double half_of(double v) {
  const int hi = __double2hiint(v), lo = __double2loint(v);
  const uint32_t e = ((uint32_t)hi >> 20) & 0x7FFu;
  const bool zero = ((uint32_t)(hi << 1) | (uint32_t)lo) == 0u;
  if (!__all_sync(0xffffffffu, zero || e - 2u < 2045u)) return 0.5 * v;
  return __hiloint2double(zero ? hi : hi - 0x100000, lo);
}

// y = (H - sigma * shifted) x, one thread per row and one CTA per block (as many
// threads as the longest block has rows). Every load of a row but the low
// neighbours (from the block's x segment in shared memory) goes out at once, so
// a short chain costs a launch and three trips to L2; in FP64 the FP64 pipe
// bounds the long ones (about 16 instructions a row at L = 24, 19 cycles per warp
// and SM: 90 us), so nothing adds zeros, the low neighbours are summed by the
// threads in the order of LowSorted (5 adds in a warp instead of 8) and the halving
// is done on the exponent (without that and the votes on c1, c2: 119 and 469 us at
// L = 24 and 26). A form with one warp per block and up to eight rows per lane added
// zeros for rows and bonds that were not there and copied the low table to each
// CTA. us, that form -> this (L = 24, 26 FP64: the six-low-bit superblock form ->
// this; L = 24 before both 176):
//   FP64  L = 12 8.2 -> 4.1  16 10.8 -> 5.2  20 31.1 -> 14.4  22 55 -> 35  24 137 -> 116  26 528 -> 445
//   FP32  L = 12 6.2 -> 4.1  16 6.2 -> 4.1  20 8.2 -> 6.2  22 14.4 -> 12.3
// 40 warps per SM in FP64 (48 registers): with 32 and 48 119 and 121 us at L = 24.
template <typename T>
__global__ void __launch_bounds__(32 * JMAX, sizeof(T) == 8 ? 5 : 6) k_rows(Geo g, const T* __restrict__ x,
                                                    T* __restrict__ y, const double* d_sigma,
                                                    int shifted) {
  __shared__ T xs[32 * JMAX], ls[32 * JMAX], ds[4];
  constexpr int HB = 10;                        // high bonds gathered at once
  const uint4* hw = reinterpret_cast<const uint4*>(g.blocks + blockIdx.x);
  const uint4 h0 = __ldg(hw), h1 = __ldg(hw + 1), h2 = __ldg(hw + 2), h3 = __ldg(hw + 3);
  const int w = h0.w & 0xFF, nh = (h0.w >> 8) & 0xFF, code = (h0.w >> 16) & 3;
  const int r = threadIdx.x, C = g.cls_C[w];
  const bool on = r < C;
  if (r < 4) {
    // what a_ii - sigma has besides the entry's dlow, by cut bonds that flip
    const double dhs = __hiloint2double((int)h1.y, (int)h1.x) - (shifted ? __ldg(d_sigma) : 0.0);
    ds[r] = (T)dhs + (T(0.5) - T(0.5) * T(__popc(r)));
  }
  T xi = T(0), c1 = T(0), c2 = T(0), dlow = T(0);
  uint4 so = make_uint4(0, 0, 0, 0);
  uint32_t xc = 0;
  const T* xr = x + h0.x + r;
  T v[HB];
  if (on) {
    const LowEntry* le = g.low + g.cls_off[w] + r;
    const uint2 e = __ldg(reinterpret_cast<const uint2*>(le));
    so = __ldg(reinterpret_cast<const uint4*>(g.low + g.nlow) + g.cls_off[w] + r);
    if constexpr (sizeof(T) == 8) dlow = __ldg(&le->dlow);
    else dlow = __ldg(&le->dlow_f);
    xi = __ldg(xr);
    const uint32_t hd[HB] = {h1.z, h1.w, h2.x, h2.y, h2.z, h2.w, h3.x, h3.y, h3.z, h3.w};
#pragma unroll
    for (int m = 0; m < HB; ++m)
      if (m < nh) v[m] = __ldg(xr + (int32_t)hd[m]);
    xc = le_code(e.x) ^ code;
    if (xc & 1u) c1 = __ldg(xr + (int32_t)h0.z);
    if (xc & 2u) c2 = __ldg(x + (h0.y + (e.y & 0xFFFFu)));
  }
  xs[r] = xi;
  __syncthreads();
  // the low neighbours of the row that so names
  const int cnt = so.w >> 8;
  const int most = __reduce_max_sync(0xffffffffu, cnt);
  T acc = T(0);
#pragma unroll
  for (int m = 0; m < NB_MAX; ++m) {
    if (m >= most) break;
    const uint32_t wd = m < 4 ? so.x : m < 8 ? so.y : so.z;
    const uint32_t q = (wd >> (8 * (m & 3))) & 0xFFu;
    if (m == 0) acc = cnt > 0 ? xs[q] : T(0);
    else if (m < cnt) acc += xs[q];
  }
  if (on) ls[so.w & 0xFFu] = acc;
  __syncthreads();
  if ((r & ~31) >= C) return;
  acc = on ? ls[r] : T(0);
  for (int m0 = HB; m0 < nh; m0 += 4) {
    const uint4 hh = __ldg(hw + 4 + ((m0 - HB) >> 2));
    const uint32_t hd[4] = {hh.x, hh.y, hh.z, hh.w};
    T u[4];
#pragma unroll
    for (int m = 0; m < 4; ++m)
      u[m] = on && m0 + m < nh ? __ldg(xr + (int32_t)hd[m]) : T(0);
#pragma unroll
    for (int m = 0; m < 4; ++m)
      if (m0 + m < nh) acc += u[m];
  }
#pragma unroll
  for (int m = 0; m < HB; ++m)
    if (m < nh) acc += v[m];
  if (__any_sync(0xffffffffu, xc & 1u)) acc += c1;
  if (__any_sync(0xffffffffu, xc & 2u)) acc += c2;
  const T half = half_of(acc);
  if (on) __stcs(y + h0.x + r, (dlow + ds[xc]) * xi + half);
}

// ---------------------------------------------------------------------------
// Ranking: colex rank of the popcount-N word s = sum_i C(p_i, i) over its set
// bits p_1 < p_2 < ... (equal to the ascending-integer rank of the sector).
__global__ void k_unrank(const uint32_t* __restrict__ binom, int L, int N, long long first,
                         long long count, unsigned int* __restrict__ out) {
  const int W = LMAX / 2 + 2;
  for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < count;
       t += (long long)gridDim.x * blockDim.x) {
    uint32_t r = (uint32_t)(first + t);
    uint32_t s = 0;
    int p = L - 1;
    for (int c = N; c >= 1; --c) {
      while (binom[p * W + c] > r) --p;
      s |= 1u << p;
      r -= binom[p * W + c];
      --p;
    }
    out[t] = s;
  }
}

__global__ void k_rank(const uint32_t* __restrict__ binom, int L, int N,
                       const unsigned int* __restrict__ st, long long count,
                       long long* __restrict__ out) {
  const int W = LMAX / 2 + 2;
  for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < count;
       t += (long long)gridDim.x * blockDim.x) {
    uint32_t s = st[t];
    if ((L < 32 && (s >> L) != 0u) || __popc(s) != N) { out[t] = -1; continue; }
    long long r = 0;
    int c = 1;
    while (s) {
      const int p = __ffs(s) - 1;
      r += binom[p * W + c];
      ++c;
      s &= s - 1u;
    }
    out[t] = r;
  }
}

// ---------------------------------------------------------------------------
// diag[i] = a_ii, minv[i] = 1 / M_ii (FP64).
__global__ void __launch_bounds__(HV_THREADS) k_diag(Geo g, double* diag, double* minv, int pc,
                                                     const double* d_sigma) {
  extern __shared__ __align__(16) char smem[];
  const RowSmem<double> s = row_smem_setup<double>(smem, g);
  const double sigma = *d_sigma;
  const int lane = threadIdx.x & 31;
  for_blocks(g, sigma, [&](const Hdr& h) {
    for (int r = lane; r < h.C; r += 32) {
      const LowEntry& e = s.low[h.off + r];
      const uint32_t xc = cut_mask(e.packed, h);
      const double am = diag_d(e, h, xc);
      const uint32_t i = h.R + r;
      if (diag) diag[i] = am + sigma;
      if (minv) {
        const int naf = naf_row(e.packed, h, xc);
        const double m = pc == 0 ? 1.0 : (pc == 1 ? fabs(am) : sqrt(am * am + 0.25 * naf));
        minv[i] = 1.0 / m;
      }
    }
  });
}

// ---------------------------------------------------------------------------
// FP64 residual r = b - (H - sigma) x with per-CTA partial sums
// [sum r^2 / M, sum r^2, sum b^2 / M, sum b^2] (host adds them in order).
// MODE: RES_PRODUCT forms the product here; RES_ZERO: x is zero (the first
// refinement sweep), so r = b and x is not read; RES_GIVEN: rv already holds
// (H - sigma) x (from a faster product kernel) and is overwritten in place.
constexpr int RES_PRODUCT = 0, RES_ZERO = 1, RES_GIVEN = 2;
template <int PC, int MODE>
__global__ void __launch_bounds__(HV_THREADS) k_resid64(Geo g, const double* __restrict__ bv,
                                                        const double* __restrict__ x,
                                                        double* __restrict__ rv,
                                                        const double* d_sigma,
                                                        double* partial) {
  extern __shared__ __align__(16) char smem[];
  const RowSmem<double> s = row_smem_setup<double>(smem, g);
  const double sigma = *d_sigma;
  const int lane = threadIdx.x & 31;
  double acc[4] = {0.0, 0.0, 0.0, 0.0};
  for_blocks(g, sigma, [&](const Hdr& h) {
    double xi[JMAX], hx[JMAX];
    if constexpr (MODE == RES_PRODUCT) {
      block_hv<double>(x, s, h, xi, hx);
    } else {
#pragma unroll
      for (int j = 0; j < JMAX; ++j) hx[j] = 0.0;
    }
#pragma unroll
    for (int j = 0; j < JMAX; ++j) {
      const int r = lane + 32 * j;
      if (j < h.J && r < h.C) {
        const LowEntry& e = s.low[h.off + r];
        const uint32_t xc = cut_mask(e.packed, h);
        const double m = precond_t<PC, double>(diag_d(e, h, xc), naf_row(e.packed, h, xc));
        const uint32_t i = h.R + r;
        const double bi_ = bv[i];
        const double ri = bi_ - (MODE == RES_GIVEN ? rv[i] : hx[j]);
        rv[i] = ri;
        acc[0] += ri * ri / m;
        acc[1] += ri * ri;
        acc[2] += bi_ * bi_ / m;
        acc[3] += bi_ * bi_;
      }
    }
  });
  block_sum<4>(acc, s.red);
  if (threadIdx.x == 0)
    for (int j = 0; j < 4; ++j) partial[blockIdx.x * 4 + j] = acc[j];
}

// ---------------------------------------------------------------------------
template <typename T>
static size_t smem_of(const hs_handle* hd) {
  return row_smem_bytes<T>((int)hd->low.size());
}

template <typename K>
static hs_status prep_smem(hs_handle* hd, K kern, size_t bytes) {
  return allow_smem(kern, bytes) ? HS_OK : fail(hd, HS_CUDA, "shared memory refused");
}

hs_status launch_matvec(hs_handle* hd, const void* x, void* y, hs_dtype dt, int shifted) {
  // FP64: one thread per row at every L (the six-low-bit superblock form takes
  // 49, 137, 528 and 2084 us at L = 22 .. 28, this 35, 116, 445 and 1776). FP32:
  // the class form from L = 24 on (22.7, 65.7 and 257 us at L = 24, 26, 28; the
  // ten-low-bit superblock form 27, 82 and 333, one thread per row 31, 123 and
  // 600; at L = 22 12.3 against 12.3 with one thread per row). HS_HV_SB=1 uses the
  // superblock forms wherever a plan was built; HS_HV_CLS=0 / 1: the class form
  // off, or wherever the blocks have ten low bits.
  const char* e = getenv("HS_HV_SB");
  if (e && e[0] == '1') {
    bool used = false;
    hs_status st = launch_matvec_sb(hd, x, y, dt, shifted, &used);
    if (st != HS_OK || used) return st;
  }
  const Geo g = hd->geo();
  const int nt = (*std::max_element(g.cls_C, g.cls_C + g.k + 1) + 31) / 32 * 32;
  const char* c = getenv("HS_HV_CLS");
  if (dt == HS_F64) {
    k_rows<double><<<g.nblocks, nt, 0, hd->stream>>>(
        g, static_cast<const double*>(x), static_cast<double*>(y), hd->d_sigma, shifted);
  } else if (hd->d_order && (c ? c[0] == '1' : hd->L >= 24)) {
    const int grid = CLS_MB * hd->num_sms;
    k_cls<sb::MODE_HV><<<grid, CLS_NT, 0, hd->stream>>>(g, cls_work(hd, grid),
        static_cast<const float*>(x), static_cast<float*>(y), hd->d_sigma, shifted,
        sb::MinresArgs{});
  } else {
    k_rows<float><<<g.nblocks, nt, 0, hd->stream>>>(
        g, static_cast<const float*>(x), static_cast<float*>(y), hd->d_sigma, shifted);
  }
  count_launches(1);
  HS_CUDA_TRY(hd, cudaGetLastError());
  return HS_OK;
}

hs_status launch_unrank(hs_handle* hd, long long first, long long count, unsigned int* out) {
  if (count <= 0) return HS_OK;
  const int grid = (int)std::min<long long>((count + 255) / 256, hd->num_sms * 8LL);
  k_unrank<<<grid, 256, 0, hd->stream>>>(hd->d_binom, hd->L, hd->N, first, count, out); count_launches(1);
  HS_CUDA_TRY(hd, cudaGetLastError());
  return HS_OK;
}

hs_status launch_rank(hs_handle* hd, const unsigned int* st, long long count, long long* out) {
  if (count <= 0) return HS_OK;
  const int grid = (int)std::min<long long>((count + 255) / 256, hd->num_sms * 8LL);
  k_rank<<<grid, 256, 0, hd->stream>>>(hd->d_binom, hd->L, hd->N, st, count, out); count_launches(1);
  HS_CUDA_TRY(hd, cudaGetLastError());
  return HS_OK;
}

hs_status launch_diag(hs_handle* hd, double* diag, hs_precond pc, double* minv) {
  const size_t sm = smem_of<double>(hd);
  if (prep_smem(hd, k_diag, sm) != HS_OK) return HS_CUDA;
  k_diag<<<row_grid(hd), HV_THREADS, sm, hd->stream>>>(hd->geo(), diag, minv, (int)pc,
                                                       hd->d_sigma); count_launches(1);
  HS_CUDA_TRY(hd, cudaGetLastError());
  return HS_OK;
}

template <int MODE>
static hs_status resid64_t(hs_handle* hd, const double* b, const double* x, double* r,
                           hs_precond pc, int grid, size_t sm) {
  const Geo g = hd->geo();
  switch (pc) {
    case HS_PC_ID:
      if (prep_smem(hd, k_resid64<0, MODE>, sm) != HS_OK) return HS_CUDA;
      k_resid64<0, MODE><<<grid, HV_THREADS, sm, hd->stream>>>(g, b, x, r, hd->d_sigma, hd->d_partial); count_launches(1);
      break;
    case HS_PC_JACOBI:
      if (prep_smem(hd, k_resid64<1, MODE>, sm) != HS_OK) return HS_CUDA;
      k_resid64<1, MODE><<<grid, HV_THREADS, sm, hd->stream>>>(g, b, x, r, hd->d_sigma, hd->d_partial); count_launches(1);
      break;
    default:
      if (prep_smem(hd, k_resid64<2, MODE>, sm) != HS_OK) return HS_CUDA;
      k_resid64<2, MODE><<<grid, HV_THREADS, sm, hd->stream>>>(g, b, x, r, hd->d_sigma, hd->d_partial); count_launches(1);
      break;
  }
  HS_CUDA_TRY(hd, cudaGetLastError());
  return HS_OK;
}

hs_status resid64(hs_handle* hd, const double* b, const double* x, double* r, hs_precond pc,
                  double sums_out[4], bool x_zero) {
  hs_status st = ensure_reduce(hd);
  if (st != HS_OK) return st;
  const size_t sm = smem_of<double>(hd);
  const int grid = row_grid(hd);
  if (x_zero) {
    st = resid64_t<RES_ZERO>(hd, b, x, r, pc, grid, sm);
  } else {
    // from L = 22 on the product kernel and a pass over its result are faster
    // than both in the block form: form (H - sigma) x in r, then r = b - r with
    // the sums
    const char* e = getenv("HS_HV_SB");
    bool used = !e && hd->L >= 22;
    if (used)
      st = launch_matvec(hd, x, r, HS_F64, 1);
    else if (e && e[0] == '1')
      st = launch_matvec_sb(hd, x, r, HS_F64, 1, &used);
    if (st != HS_OK) return st;
    st = used ? resid64_t<RES_GIVEN>(hd, b, x, r, pc, grid, sm)
              : resid64_t<RES_PRODUCT>(hd, b, x, r, pc, grid, sm);
  }
  if (st != HS_OK) return st;
  return sum_partials(hd, grid, 4, sums_out);
}

}  // namespace hs
