// Kernel of the six-low-bit superblock product (sb6.cuh): y = (H - sigma) x
// (Eq. (1)), one CTA per superblock pair, or, in MINRES mode, pass A of
// Algorithm 2 (p = (H - sigma) q_k and alpha_k = q_k . p / beta_k^2 by a
// last-CTA reduction).
//
// Per pair: (1) every thread takes flat rows of the pair: x of each row goes
// asynchronously into its slot element, the whole-superblock shifts of the row
// are summed into the same element of G; (2) one lane per sub-block computes its
// rows from shared memory and writes them over their sums; (3) the pair's rows
// are stored from G in rank order, coalesced.
#pragma once
#include "minres_scalar.cuh"
#include "rows.cuh"
#include "sb6.cuh"
#include "sb_kern.cuh"

namespace hs {
namespace sb6 {

// Shared memory: X [2][2^km slots], the zero slots, G [2][2^km slots], dl, dmid,
// uT [2][2], Sup [2].
template <typename T>
__host__ __device__ inline size_t smem_bytes6(int km) {
  return sizeof(T) * ((size_t)((4 << km) + ZSLOTS) * ST<T> + 2 * 2 * (K + 1) * DL + (1 << km) + 4) +
         2 * sizeof(sb::Sup);
}

template <typename T, int NT, int MINB, int U, int MODE>
__global__ void __launch_bounds__(NT, MINB) k_sb6(Geo6 g, const T* __restrict__ x,
                                                  T* __restrict__ y, const double* d_sigma,
                                                  int shifted, sb::MinresArgs ma) {
  extern __shared__ __align__(16) char smem[];
  __shared__ double s_red[32 * 4];
  __shared__ double s_sig;
  __shared__ long long s_k;
  __shared__ int s_done;
  if constexpr (MODE == sb::MODE_MINRES) {
    if (threadIdx.x == 0) {
      const MinresState* st = ma.st;
      s_done = st->done; s_k = st->k; s_sig = st->sigma;
    }
    __syncthreads();
    if (s_done != 0) return;   // finished, or only the last d/x update is left (pass B)
    const bool odd = (s_k & 1) != 0;
    x = (const T*)(odd ? ma.v.q1 : ma.v.q0);   // q_k
    y = (T*)ma.v.p;
  } else {
    if (threadIdx.x == 0) s_sig = shifted ? *d_sigma : 0.0;
    __syncthreads();
  }
  const double sigma = s_sig;
  const int km = g.km, tile = ST<T> << km;
  T* X = reinterpret_cast<T*>(smem);
  T* Z = X + 2 * tile;
  T* G = Z + ZSLOTS * ST<T>;
  T* dl = G + 2 * tile;
  T* dmid = dl + 2 * 2 * (K + 1) * DL;
  T* uT = dmid + (1 << km);                          // dT - sigma +- 1/4 (bond (KS-1, KS))
  sb::Sup* sh = reinterpret_cast<sb::Sup*>(uT + 4);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  for (int i = tid; i < (1 << km); i += NT) dmid[i] = __ldg((const T*)g.dmid + i);
  for (int i = tid; i < 2 * 2 * (K + 1) * DL; i += NT) dl[i] = __ldg((const T*)g.dl + i);
  for (int i = tid; i < ZSLOTS * ST<T>; i += NT) Z[i] = T(0);
  T acc = T(0);
  // a pair's headers are loaded while the pair before it is computed
  const int hs = tid / sb::SUP_WORDS, hw = tid % sb::SUP_WORDS;   // header word of this thread
  auto header = [&](const int4& p) {
    const int id = hs ? p.y : p.x;
    return tid < 2 * sb::SUP_WORDS && id >= 0
               ? __ldg(reinterpret_cast<const uint32_t*>(g.sup + id) + hw) : 0u;
  };
  int4 pr = __ldg(g.pairs + min((int)blockIdx.x, g.npairs - 1));
  uint32_t hword = header(pr);
  for (int pi = blockIdx.x; pi < g.npairs; pi += gridDim.x) {
    __syncthreads();  // the previous pair is done with sh, X, G and uT
    if (tid < 2 * sb::SUP_WORDS) reinterpret_cast<uint32_t*>(sh + hs)[hw] = hword;
    const int nx = pi + (int)gridDim.x;
    const int4 prn = nx < g.npairs ? __ldg(g.pairs + nx) : pr;
    int e = warp < pr.w ? __ldg(g.tasks + (size_t)(pr.z + warp) * 32 + lane) : NO_TASK;
    __syncthreads();
    if (tid < 4) {
      // the superblock's share of every diagonal: dT - sigma and the Ising
      // term of bond (KS-1, KS), by the top mid bit (tid & 1)
      const int s = tid >> 1;
      const uint32_t tb0 = (sh[s].meta >> 16) & 1u;   // bit 0 of T
      const double ks = ((uint32_t)(tid & 1) == tb0) ? 0.25 : -0.25;
      uT[tid] = (T)(sh[s].dT - sigma + ks);
    }
#pragma unroll 1
    for (int s = 0; s < 2; ++s)
      if (sh[s].C)
        sb6_flat<T>(x + sh[s].R, sh[s], g.slotmap + g.slot_off[sh[s].meta & 0xFF], X + s * tile,
                       G + s * tile, tid, NT);
    hword = header(prn);
    sb::cp_async_wait_all();
    __syncthreads();
    for (int wt = warp; wt < pr.w; wt += NT / 32) {
      if (wt != warp) e = __ldg(g.tasks + (size_t)(pr.z + wt) * 32 + lane);
      const int s = (e >> 15) & 1, m = e & 0x7FFF;
      const uint32_t hm = sh[s].meta;
      // one class per warp: lane 0 always has a task
      const int w = __shfl_sync(0xffffffffu, (int)(hm & 0xFF) - __popc((unsigned)m), 0);
      if (e != NO_TASK) {
        const uint32_t top = (hm >> 17) & 1u;
        const T u = dmid[m] + uT[s * 2 + ((m >> (km - 1)) & 1)];
        acc += sb6_rows_any<T>(w, m, km, top, X + s * tile, sh[1 - s].C ? X + (1 - s) * tile : nullptr,
                               Z, G + s * tile + swz(m) * ST<T>,
                               dl + (((int)top * 2 + (m & 1)) * (K + 1) + w) * DL, u);
      }
    }
    __syncthreads();
    // the pair's rows in rank order
#pragma unroll 1
    for (int s = 0; s < 2; ++s) {
      const int C = (int)sh[s].C;
      const uint16_t* map = g.slotmap + g.slot_off[sh[s].meta & 0xFF];
      const T* Gs = G + s * tile;
      T* ys = y + sh[s].R;
      int i = tid;
      for (; i + (U - 1) * NT < C; i += U * NT) {
        int e[U];
#pragma unroll
        for (int u = 0; u < U; ++u) e[u] = __ldg(map + i + u * NT);
#pragma unroll
        for (int u = 0; u < U; ++u) ys[i + u * NT] = Gs[e[u]];
      }
      for (; i < C; i += NT) ys[i] = Gs[__ldg(map + i)];
    }
    pr = prn;
  }
  if constexpr (MODE == sb::MODE_MINRES) {
    double vv[1] = {(double)acc}, tot[1];
    if (last_cta_sum<1>(vv, s_red, ma.partial, ma.counter, tot) && threadIdx.x == 0) {
      MinresState* st = ma.st;
      const double bk = st->beta;
      st->alpha = tot[0] / (bk * bk);                        // alpha_k = q_k . p_k / beta_k^2
      if (!isfinite(st->alpha)) { st->status = HS_NONFINITE; st->done = 2; st->pending = 0; }
    }
  }
}

// Device copy of one plan.
struct DevPlan6 {
  Geo6 geo{};
  void* mem = nullptr;
  int grid = 0;
  size_t smem = 0;
  int ok = 0;
};

// Two CTAs of 256 threads per SM (122 registers; three of 128 or one of 384
// threads: 4 to 15 % slower).
constexpr int NT6 = 256;
template <typename T, int MODE>
constexpr auto kernel6() { return k_sb6<T, NT6, 2, 4, MODE>; }

}  // namespace sb6
}  // namespace hs
