// FP32 products of long chains, one warp per block: y = (H - sigma) x (hv.cu) and
// pass A of the FP32 MINRES (minres_sb.cu).
//
// Every CTA keeps to blocks of one class (low popcount): the low part of its rows
// (neighbour and wrap ranks, diagonal) is laid out once in shared memory, one
// 16-byte word a row, and the rows per lane J and the neighbours per row are
// compile-time constants; ranks past a row's neighbours name a zero. The classes
// share the grid in proportion to their work and each walks its blocks in rank
// order, so all warps gather from one window of x.
// The ten-low-bit superblock form (sb_kern.cuh) issued 193 thread instructions a
// row at L = 28 (333 us, issue 60 %); here 138, and the wavefronts of loads and
// shared memory bound it (77 % of their peak; waits on gathers come next). us,
// that form -> this: L = 24 27 -> 22.7, L = 26 82 -> 65.7, L = 28 333 -> 257. With the low part in registers (16 warps per SM, 228 bytes
// spilled) 357; with equal shares by rows 511.
#pragma once
#include "rows.cuh"
#include "sb_kern.cuh"

namespace hs {

// Four CTAs of eight warps per SM (64 registers; us at L = 28: 32 warps per SM 257,
// 20, 24, 40 and 48 warps 311, 295, 258 and 273).
constexpr int CLS_NT = 256, CLS_NW = CLS_NT / 32, CLS_MB = 4;
constexpr int CLS_CTAS_MIN = 2 * (KLO_MAX + 1);
constexpr int CLS_HG = 2;                       // high bonds gathered at once for four rows per lane

// The blocks by class: order[first[w] .. first[w + 1]) are those of class w, in
// rank order; CTAs cstart[w] .. cstart[w + 1] - 1 take them.
struct ClsWork {
  const uint32_t* order;
  int first[KLO_MAX + 2];
  int cstart[KLO_MAX + 2];
};

template <int J, int NB, int MODE>
__device__ __forceinline__ float cls_run(const Geo& g, const ClsWork& cw, int w, int me,
                                         const float* __restrict__ x, float* __restrict__ y,
                                         double sigma, float* xs_all, uint4* tab) {
  constexpr int HG = J > 2 ? CLS_HG : 8;
  const int lane = threadIdx.x & 31;
  const int C = g.cls_C[w];
  const uint32_t wb = (uint32_t)(threadIdx.x >> 5) << 8;   // this warp's buffer in xs_all
  float* xs = xs_all + wb;
  // the class's rows: nine neighbour ranks, code, wrap rank, diagonal
  for (int r = threadIdx.x; r < 32 * J; r += CLS_NT) {
    const LowEntry e = g.low[g.cls_off[w] + min(r, C - 1)];
    const int cnt = le_cnt(e.packed);
    uint32_t n3[3];
#pragma unroll
    for (int i = 0; i < 3; ++i) {
      // ranks past cnt name slot 255, which is zero
      const int have = cnt - 4 * i;
      const uint32_t keep = have >= 4 ? ~0u : have <= 0 ? 0u : (1u << (8 * have)) - 1u;
      n3[i] = (e.nbw[i] & keep) | ~keep;
    }
    tab[r] = make_uint4(n3[0], n3[1],
                        (n3[2] & 0xFFu) | le_code(e.packed) << 8 | (uint32_t)e.wrap_r << 16,
                        __float_as_uint(e.dlow_f));
  }
  __syncthreads();
  const uint4* tl = tab + lane;
  if (lane == 31) xs[255] = 0.0f;
  const bool last = lane + 32 * (J - 1) < C;
  float qp = 0.0f;
  const int end = cw.first[w + 1], stride = (cw.cstart[w + 1] - cw.cstart[w]) * CLS_NW;
  int at = cw.first[w] + me;
  if (at >= end) return qp;
  uint32_t word = hdr_word(g, (int)__ldg(cw.order + at));
  uint32_t nid = at + stride < end ? __ldg(cw.order + at + stride) : 0u;
  while (true) {
    const Hdr h = make_hdr(g, word, sigma);
    at += stride;
    const bool more = at < end;
    if (more) word = hdr_word(g, (int)nid);
    if (at + stride < end) nid = __ldg(cw.order + at + stride);
    const float* xb = x + h.R + lane;
    const float* x1 = xb + h.bdelta;
    const float* x2 = x + h.Rwrap;
    // what a_ii - sigma has besides dlow: both cut bonds parallel, one, none
    const float d0 = h.dhs_f + 0.5f, d2 = h.dhs_f - 0.5f;
    auto on = [&](int j) { return j < J - 1 || last; };
    float xi[J];
#pragma unroll
    for (int j = 0; j < J; ++j) xi[j] = on(j) ? __ldg(xb + 32 * j) : 0.0f;
    // the rows in one or two groups of up to four per lane
#pragma unroll
    for (int j0 = 0; j0 < J; j0 += 4) {
      constexpr int JH = J < 4 ? J : 4;
      float acc[JH], v[HG][JH];
      auto highs = [&](int m0) {
#pragma unroll
        for (int mm = 0; mm < HG; ++mm)
          if (m0 + mm < h.nh) {
            const float* xh = xb + (int32_t)__shfl_sync(0xffffffffu, h.word, 6 + m0 + mm);
#pragma unroll
            for (int j = 0; j < JH; ++j)
              if (j0 + j < J) v[mm][j] = on(j0 + j) ? __ldg(xh + 32 * (j0 + j)) : 0.0f;
          }
      };
      highs(0);
#pragma unroll
      for (int j = 0; j < JH; ++j)
        if (j0 + j < J) {
          const uint32_t en = tl[32 * (j0 + j)].z, xc = (en >> 8) ^ (uint32_t)h.code;
          const float c1 = (xc & 1u) && on(j0 + j) ? __ldg(x1 + 32 * (j0 + j)) : 0.0f;
          const float c2 = (xc & 2u) && on(j0 + j) ? __ldg(x2 + (en >> 16)) : 0.0f;
          acc[j] = c1 + c2;
        }
      if (j0 == 0) {
#pragma unroll
        for (int j = 0; j < J; ++j) xs[lane + 32 * j] = xi[j];
        __syncwarp();
      }
#pragma unroll
      for (int j = 0; j < JH; ++j)
        if (j0 + j < J) {
          const uint4 e = tl[32 * (j0 + j)];
          float low = 0.0f;
#pragma unroll
          for (int m = 0; m < NB; ++m)
            low += xs_all[__byte_perm(m < 4 ? e.x : m < 8 ? e.y : e.z, wb, 0x7650 | (m & 3))];
          acc[j] += low;
        }
      for (int m0 = 0;;) {
#pragma unroll
        for (int mm = 0; mm < HG; ++mm)
          if (m0 + mm < h.nh) {
#pragma unroll
            for (int j = 0; j < JH; ++j)
              if (j0 + j < J) acc[j] += v[mm][j];
          }
        m0 += HG;
        if (m0 >= h.nh) break;
        highs(m0);
      }
      float* yb = y + h.R + lane + 32 * j0;
#pragma unroll
      for (int j = 0; j < JH; ++j)
        if (j0 + j < J) {
          const uint4 e = tl[32 * (j0 + j)];
          const uint32_t xc = ((e.z >> 8) ^ (uint32_t)h.code) & 3u;
          const float am = __uint_as_float(e.w) + (xc == 0u ? d0 : xc == 3u ? d2 : h.dhs_f);
          const float xo = xs[lane + 32 * (j0 + j)];
          const float p = am * xo + 0.5f * acc[j];
          if (on(j0 + j)) {
            if constexpr (MODE == sb::MODE_MINRES) {
              yb[32 * j] = p;
              qp += xo * p;
            } else {
              __stcs(yb + 32 * j, p);
            }
          }
        }
    }
    __syncwarp();
    if (!more) break;
  }
  return qp;
}

template <int MODE>
__global__ void __launch_bounds__(CLS_NT, CLS_MB)
    k_cls(Geo g, ClsWork cw, const float* __restrict__ x, float* __restrict__ y,
          const double* d_sigma, int shifted, sb::MinresArgs ma) {
  __shared__ float xs[32 * JMAX * CLS_NW];
  __shared__ uint4 tab[32 * JMAX];
  double sigma = 0.0;
  if constexpr (MODE == sb::MODE_MINRES) {
    const MinresState* st = ma.st;
    if (st->done != 0) return;   // finished, or only the last d/x update is left (pass B)
    x = (const float*)((st->k & 1) ? ma.v.q1 : ma.v.q0);   // q_k
    y = (float*)ma.v.p;
    sigma = st->sigma;
  } else if (shifted) {
    sigma = *d_sigma;
  }
  int w = 0;
  while (w < g.k && (int)blockIdx.x >= cw.cstart[w + 1]) ++w;
  const int me = ((int)blockIdx.x - cw.cstart[w]) * CLS_NW + (int)(threadIdx.x >> 5);
  float qp = 0.0f;
  switch ((g.cls_C[w] + 31) >> 5) {
    case 8: qp = cls_run<8, 9, MODE>(g, cw, w, me, x, y, sigma, xs, tab); break;
    case 7: qp = cls_run<7, 8, MODE>(g, cw, w, me, x, y, sigma, xs, tab); break;
    case 4: qp = cls_run<4, 6, MODE>(g, cw, w, me, x, y, sigma, xs, tab); break;
    case 2: qp = cls_run<2, 4, MODE>(g, cw, w, me, x, y, sigma, xs, tab); break;
    default: qp = cls_run<1, 2, MODE>(g, cw, w, me, x, y, sigma, xs, tab); break;
  }
  if constexpr (MODE == sb::MODE_MINRES) {
    __shared__ double s_red[32 * 4];
    double vv[1] = {(double)qp}, tot[1];
    if (last_cta_sum<1>(vv, s_red, ma.partial, ma.counter, tot) && threadIdx.x == 0) {
      MinresState* st = ma.st;
      const double bk = st->beta;
      st->alpha = tot[0] / (bk * bk);                  // alpha_k = q_k . p_k / beta_k^2
      if (!isfinite(st->alpha)) { st->status = HS_NONFINITE; st->done = 2; st->pending = 0; }
    }
  }
}

// The classes' shares of a grid of at least CLS_CTAS_MIN: a block costs about 1.3 + J (cycles at L = 28:
// J = 8 13300, 7 12300, 4 6800, 2 4400, 1 3300).
inline ClsWork cls_work(const hs_handle* hd, int grid) {
  ClsWork cw{};
  cw.order = hd->d_order;
  const Geo g = hd->geo();
  double cost[KLO_MAX + 1], tot = 0.0, run = 0.0;
  for (int w = 0; w <= KLO_MAX; ++w) {
    cw.first[w] = hd->cls_first[w];
    cost[w] = (hd->cls_first[w + 1] - hd->cls_first[w]) * (1.3 + (g.cls_C[w] + 31) / 32);
    tot += cost[w];
  }
  cw.first[KLO_MAX + 1] = hd->cls_first[KLO_MAX + 1];
  for (int w = 0; w <= KLO_MAX; ++w) {
    cw.cstart[w] = (int)(run / tot * (grid - KLO_MAX - 1)) + w;
    run += cost[w];
  }
  cw.cstart[KLO_MAX + 1] = grid;
  return cw;
}

}  // namespace hs
