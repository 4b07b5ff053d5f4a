// The element-wise passes of the FP32 MINRES of long chains: the initial pass
// (ROWS_INIT) and pass B (ROWS_B), with M formed per row from the low table and the
// block header (nothing of size n is stored for it).
//
// Pass B reads six vectors and writes three (1.44 GB at L = 28, 214 us at the copy
// rate), so memory should bound it. On the superblock layout (k_sbrows) it took 305
// us: a warp came to each of a superblock's sub-blocks through three dependent
// tables. Here the warps walk the blocks in rank order, the next header loaded
// meanwhile, with the 24 loads of four rows per lane in flight: 262 us. CTAs by
// class (hv_cls.cuh), whose warps read 1 KB pieces far apart, took 400; two rows per
// lane and 48 warps per SM 270. An iteration at L = 24, 26, 28: 58, 183 and 562 ->
// 50, 149 and 522 us.
#pragma once
#include "rows.cuh"
#include "sb_kern.cuh"

namespace hs {

constexpr int BLK_ROWS_MB = 4;                   // CTAs per SM (64 registers)

struct BlkRows {
  const float* b;                // ROWS_INIT: the right-hand side
  sb::MinresArgs ma;
  double tol;
  long long kmax;
  const double* d_sigma;
  double dscale;                 // bound of the terms of a_ii
};

template <int PC, int MODE>
__global__ void __launch_bounds__(HV_THREADS, BLK_ROWS_MB) k_blk_rows(Geo g, BlkRows a) {
  __shared__ uint2 tab[1 << KLO_MAX];
  constexpr int JH = 4;
  const int lane = threadIdx.x & 31;
  __shared__ double s_red[32 * 4];
  __shared__ float cf[8];
  __shared__ double s_sigma;
  __shared__ long long s_k;
  __shared__ int s_done, s_pending;
  for (int r = threadIdx.x; r < g.nlow; r += HV_THREADS) {
    const LowEntry& e = g.low[r];
    tab[r] = make_uint2(e.packed, __float_as_uint(e.dlow_f));
  }
  if (threadIdx.x == 0) {
    s_done = 0; s_pending = 0; s_k = 0;
    if constexpr (MODE == sb::ROWS_B) {
      const MinresState* st = a.ma.st;
      s_done = st->done; s_pending = st->pending; s_k = st->k;
      s_sigma = st->sigma;
      const double bk = st->beta;
      cf[0] = (float)(1.0 / bk); cf[1] = (float)(st->alpha / bk); cf[2] = (float)(bk / st->beta_prev);
      cf[3] = (float)st->cq; cf[4] = (float)st->cd1; cf[5] = (float)st->cd2; cf[6] = (float)st->tau;
    } else {
      s_sigma = *a.d_sigma;
    }
    // rounding bound of a_ii - sigma as assembled from the tables (a few
    // additions of terms up to dscale + |sigma|)
    cf[7] = (float)(8.0 * 1.1920928955078125e-7 * (a.dscale + fabs(s_sigma)));
  }
  __syncthreads();
  if (s_done == 2) return;
  const bool doQ = s_done == 0;        // done == 1: only the last d/x update is left
  const bool doC = s_pending != 0, odd = (s_k & 1) != 0;
  const double sigma = s_sigma;
  float acc = 0.0f, zm = 0.0f;
  const MinresVecs& v = a.ma.v;
  const float* qc = (const float*)(odd ? v.q1 : v.q0);   // q_k
  float* qn = (float*)(odd ? v.q0 : v.q1);               // q_{k-1} -> q_{k+1}
  const float* pv = (const float*)v.p;
  const float* dA = (const float*)(odd ? v.d1 : v.d0);   // d_{k-2}
  float* dB = (float*)(odd ? v.d0 : v.d1);               // d_{k-3} -> d_{k-1}
  float* xv = (float*)v.x;
  const float c1 = cf[0], c2 = cf[1], c3 = cf[2], cq = cf[3], cd1 = cf[4], cd2 = cf[5], tau = cf[6];
  const float mtiny = cf[7];
  for_blocks(g, sigma, [&](const Hdr& h) {
    // JH rows per lane at a time: every load before any arithmetic or store
    for (int j0 = 0; j0 < h.J; j0 += JH) {
      float va[JH], vb[JH], vc[JH], vd[JH], ve[JH], vf[JH];
#pragma unroll
      for (int j = 0; j < JH; ++j) {
        const int r = lane + 32 * (j0 + j);
        const bool ok = r < h.C;
        const uint32_t i = h.R + (uint32_t)r;
        if constexpr (MODE == sb::ROWS_INIT) {
          va[j] = ok ? a.b[i] : 0.0f;
        } else {
          va[j] = ok ? qn[i] : 0.0f;                             // q_{k-1}
          vb[j] = ok && doC ? dA[i] : 0.0f;                      // d_{k-2}
          vc[j] = ok && doC ? dB[i] : 0.0f;                      // d_{k-3}
          vd[j] = ok && doC ? xv[i] : 0.0f;                      // x
          ve[j] = ok && doQ ? pv[i] : 0.0f;                      // p
          vf[j] = ok && doQ ? qc[i] : 0.0f;                      // q_k
        }
      }
#pragma unroll
      for (int j = 0; j < JH; ++j) {
        const int r = lane + 32 * (j0 + j);
        if (r >= h.C) continue;
        const uint2 e = tab[h.off + r];
        const uint32_t xc = le_code(e.x) ^ (uint32_t)h.code;
        const float am = __uint_as_float(e.y) + (h.dhs_f + (0.5f - 0.5f * (float)__popc(xc)));
        const float mm = precond_t<PC, float>(am, naf_row(e.x, h, xc));
        const uint32_t i = h.R + (uint32_t)r;
        if constexpr (MODE == sb::ROWS_INIT) {
          // a Jacobi entry at the rounding level of a_ii - sigma counts as
          // a_ii = sigma (Sec. II assumes a_ii != sigma)
          const bool zero = !(mm > mtiny);
          zm += zero ? 1.0f : 0.0f;
          const float q = zero ? 0.0f : va[j] / mm;
          ((float*)v.q1)[i] = q;
          ((float*)v.q0)[i] = 0.0f;
          ((float*)v.d0)[i] = 0.0f;
          ((float*)v.d1)[i] = 0.0f;
          xv[i] = 0.0f;
          acc += q * va[j];
        } else {
          if (doC) {
            // d_{k-1} = (q_{k-1} / beta_{k-1} - delta d_{k-2} - eps d_{k-3}) / gamma_{k-1};
            // x_{k-1} = x_{k-2} + tau_{k-1} d_{k-1}
            const float d = cq * va[j] + cd1 * vb[j] + cd2 * vc[j];
            dB[i] = d;
            xv[i] = vd[j] + tau * d;
          }
          if (doQ) {
            // q_{k+1} = M^-1 p / beta_k - (alpha_k / beta_k) q_k - (beta_k / beta_{k-1}) q_{k-1}
            const float q = (ve[j] / mm) * c1 - c2 * vf[j] - c3 * va[j];
            qn[i] = q;
            acc += mm * q * q;                                   // beta_{k+1}^2 = q . M q
          }
        }
      }
    }
  });
  double vv[2] = {(double)acc, (double)zm}, tot[2];
  if (last_cta_sum<2>(vv, s_red, a.ma.partial, a.ma.counter, tot) && threadIdx.x == 0) {
    MinresState S;
    if constexpr (MODE == sb::ROWS_INIT) {
      init_state(S, tot[0], tot[1], a.tol, a.kmax, sigma);
    } else {
      S = *a.ma.st;
      if (doQ) {
        givens_update(S, tot[0]);     // sets the pending update of iteration k
      } else {
        S.pending = 0;                // the last update is applied
        S.done = 2;
      }
    }
    *a.ma.st = S;
  }
}

}  // namespace hs
