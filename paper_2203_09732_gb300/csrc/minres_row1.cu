// The one-reduction recurrence of minres_pipe.cu on the row form's layout
// (minres_row.cu): one thread per row (up to three), neighbour lists in shared
// memory, vectors in registers, one grid exchange per iteration.
//
// k_minres_smem1 took 9.5 us per FP64 iteration at n = 12870: after the exchange
// (3 us) the scalars of the step (1 us), then the product's three trips to L2 and
// the sums, one after the other. Here the exchange is followed by the product at
// once; the coefficients that the vectors need, two multiplications from the
// sums, arrive meanwhile, and the rest of the step's scalars (beta_{k+1}, the
// Givens rotation) run on a control warp under the product and the next sums.
// Five control warps add the five sums. n = 12870: 6.3 us per iteration, n =
// 48620: 8.9 (two reductions in this layout: 9.6 and 12.4). The exchange is about
// 2.5 us of it, the rest a chain of L2 trips, FP64 instructions and CTA barriers.
#include <algorithm>
#include <cstdlib>

#include "minres_row.cuh"

namespace hs {

namespace {

constexpr int ONE_CW = PIPE_NV;                  // control warps: one per sum
constexpr int ONE_NW = 11;                       // compute warps
constexpr int ONE_NT = 32 * (ONE_NW + ONE_CW);
constexpr int ONE_THREADS = 32 * ONE_NW;

struct OneShared {
  double s[PIPE_NV];                             // S1..S5 of the step
  unsigned long long barP, barR, barQ, barS, barC, barD[2];
  double c[4];                                   // 1/beta_k, a, c, 1/(2 beta_k) (of type T)
  struct { double co[4]; int apply, stop; } d[2];
  int fail;
};

template <typename T, int RPT>
__global__ void __launch_bounds__(ONE_NT, 1) k_minres_row1(RowArgs ra, int pc, int rperiod) {
  extern __shared__ __align__(16) char dyn[];
  __shared__ OneShared sh;
  const SmemJob& job = ra.job;
  const Geo& g = job.g;
  const int n = (int)g.n;
  const int G = gridDim.x, cta = blockIdx.x;
  const int lane = threadIdx.x & 31;
  const int wid = (int)(threadIdx.x >> 5) - ONE_CW;
  constexpr int SLOTS = ONE_THREADS * RPT;
  double* stage = reinterpret_cast<double*>(dyn);             // [sum][thread]
  uint32_t* nbr = reinterpret_cast<uint32_t*>(dyn + sizeof(double) * PIPE_NV * ONE_THREADS);
  __shared__ uint16_t order[SLOTS];
  __shared__ uint8_t bonds[SLOTS];
  __shared__ int s_blk[2];
  __shared__ int s_class[LMAX / 2];
  static_assert(ONE_NT / 32 >= LMAX / 2, "one warp per number of neighbours");
  const int rpc = (n + G - 1) / G;
  const int r0 = min(n, cta * rpc), rows = min(n, r0 + rpc) - r0;
  const int nwa = rows > ONE_THREADS ? ONE_NW : (rows + 31) / 32;
  // q_1 and q_{k+1} of a replacement step; v_k and v_{k+1} by turns
  T* qg = reinterpret_cast<T*>(ra.q);
  T* vg[2] = {reinterpret_cast<T*>(ra.w0), reinterpret_cast<T*>(ra.w1)};
  if (threadIdx.x == 0) {
    bar_init(&sh.barP, max(1, nwa));
    bar_init(&sh.barR, max(1, nwa));
    bar_init(&sh.barQ, 1);
    bar_init(&sh.barS, ONE_CW - 1);
    bar_init(&sh.barC, 1);
    bar_init(&sh.barD[0], 1);
    bar_init(&sh.barD[1], 1);
    sh.fail = 0;
  }
  row_deal<T>(g, r0, rows, order, bonds, s_blk, s_class);
  auto replaced = [&](int k) { return k > 0 && rperiod > 0 && k % rperiod == 0; };
  unsigned pd[2] = {0, 0};
  if (wid >= 0 && wid < nwa) {
    // ---- compute warps
    T q[RPT], qm[RPT], p[RPT], pm[RPT], v[RPT];  // q_k, q_{k-1}, p_k, p_{k-1}, v_k
    T d1[RPT], d2[RPT], x[RPT], m[RPT], mi[RPT], dg[RPT];
    int cnt[RPT], row[RPT];
    const int t0 = wid * 32 + lane;
    auto place = [&](int j) { return j * ONE_THREADS + (j ? ONE_THREADS - 1 - t0 : t0); };
    auto send = [&](const T (&a)[PIPE_NV]) {
#pragma unroll
      for (int i = 0; i < PIPE_NV; ++i) stage[i * ONE_THREADS + t0] = (double)a[i];
      __syncwarp();
      if (lane == 0) bar_arrive(&sh.barP);
    };
    // 2 (H - sigma) u, u = own[] here and src[] elsewhere
    auto product = [&](const T* src, const T (&own)[RPT], T (&out)[RPT]) {
#pragma unroll
      for (int j = 0; j < RPT; ++j) {
        const uint32_t* nl = nbr + j * ONE_THREADS + t0;
        T s = T(0);
        const int most = __reduce_max_sync(0xffffffffu, cnt[j]);
        for (int c0 = 0; c0 < most; c0 += ROW_BATCH) {
          T w[ROW_BATCH];
#pragma unroll
          for (int c = 0; c < ROW_BATCH; ++c)
            w[c] = c0 + c < cnt[j] ? __ldcg(src + nl[(c0 + c) * SLOTS]) : T(0);
#pragma unroll
          for (int c = 0; c < ROW_BATCH; ++c)
            if (c0 + c < most) s += w[c];
        }
        out[j] = dg[j] * own[j] + s;
      }
    };
    T a[PIPE_NV] = {};
#pragma unroll
    for (int j = 0; j < RPT; ++j) {
      const int slot = j * ONE_THREADS + t0;
      row[j] = place(j) < rows ? r0 + order[place(j)] : -1;
      q[j] = qm[j] = p[j] = pm[j] = v[j] = d1[j] = d2[j] = x[j] = m[j] = mi[j] = dg[j] = T(0);
      cnt[j] = 0;
      if (row[j] >= 0) {
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
        a[1] += mm == T(0) ? T(1) : T(0);
        m[j] = mm;
        mi[j] = mm == T(0) ? T(0) : T(1) / mm;
        dg[j] = T(2) * am;
        q[j] = b * mi[j];
        a[0] += q[j] * b;
        qg[i] = q[j];
      }
    }
    send(a);
    unsigned pq = 0, pcb = 0;
    bool ok = row_wait(sh.fail, &sh.barQ, pq);   // q_1 is complete
    pq ^= 1u;
    ok = ok && row_wait(sh.fail, &sh.barD[0], pd[0]);
    pd[0] ^= 1u;
    bool run = ok && sh.d[0].stop == 0;
    if (run) {
      // p_1 = (H - sigma) q_1, v_1 and the sums of step 1 (q_0 = p_0 = 0)
      T hv[RPT];
      product(qg, q, hv);
#pragma unroll
      for (int i = 0; i < PIPE_NV; ++i) a[i] = T(0);
#pragma unroll
      for (int j = 0; j < RPT; ++j) {
        p[j] = T(0.5) * hv[j];
        v[j] = mi[j] * p[j];
        if (row[j] >= 0) vg[1][row[j]] = v[j];
        a[0] += q[j] * p[j];
        a[1] += p[j] * v[j];
        a[3] += m[j] * q[j] * q[j];
      }
      send(a);
    }
    for (int k = 1; run; ++k) {
      if (!(ok = row_wait(sh.fail, &sh.barQ, pq))) break;    // v_k is complete
      pq ^= 1u;
      const bool repl = replaced(k);
      T hv[RPT];
      if (!repl) product(vg[k & 1], v, hv);
      if (!(ok = row_wait(sh.fail, &sh.barC, pcb))) break;
      pcb ^= 1u;
      const T* co = reinterpret_cast<const T*>(sh.c);
      const T c1 = co[0], c2 = co[1], c3 = co[2], c1h = co[3];
      T* vn = vg[(k + 1) & 1];
#pragma unroll
      for (int i = 0; i < PIPE_NV; ++i) a[i] = T(0);
      T qo[RPT];
#pragma unroll
      for (int j = 0; j < RPT; ++j) {
        qo[j] = q[j];
        q[j] = c1 * v[j] - c2 * q[j] - c3 * qm[j];
        qm[j] = qo[j];
      }
      // the sums of step k + 1 from q_{k+1}, p_{k+1}, v_{k+1}
      auto sums = [&](int j) {
        v[j] = mi[j] * p[j];
        if (row[j] >= 0) vn[row[j]] = v[j];
        const T mq = m[j] * q[j];
        a[0] += q[j] * p[j];
        a[1] += p[j] * v[j];
        a[2] += p[j] * qo[j];
        a[3] += mq * q[j];
        a[4] += mq * qo[j];
      };
      if (!repl) {
#pragma unroll
        for (int j = 0; j < RPT; ++j) {
          const T pn = c1h * hv[j] - c2 * p[j] - c3 * pm[j];
          pm[j] = p[j];
          p[j] = pn;
          sums(j);
        }
      } else {
#pragma unroll
        for (int j = 0; j < RPT; ++j)
          if (row[j] >= 0) qg[row[j]] = q[j];
        __syncwarp();
        if (lane == 0) bar_arrive(&sh.barR);
      }
      if (!repl) send(a);
      // d_k = (q_k / beta_k - delta_k d_{k-1} - eps_k d_{k-2}) / gamma_k and x_k
      const int t = k & 1;
      if (!(ok = row_wait(sh.fail, &sh.barD[t], pd[t]))) break;
      pd[t] ^= 1u;
      if (sh.d[t].apply) {
        const T* dc = reinterpret_cast<const T*>(sh.d[t].co);
        const T cq = dc[0], e1 = dc[1], e2 = dc[2], tau = dc[3];
#pragma unroll
        for (int j = 0; j < RPT; ++j) {
          const T d = cq * qo[j] + e1 * d1[j] + e2 * d2[j];
          d2[j] = d1[j];
          d1[j] = d;
          x[j] += tau * d;
        }
      }
      if (sh.d[t].stop) break;
      if (repl) {
        // p_{k+1} as a product with q_{k+1}, once that is complete
        if (!(ok = row_wait(sh.fail, &sh.barQ, pq))) break;
        pq ^= 1u;
        product(qg, q, hv);
#pragma unroll
        for (int j = 0; j < RPT; ++j) {
          pm[j] = p[j];
          p[j] = T(0.5) * hv[j];
          sums(j);
        }
        send(a);
      }
    }
    if (!ok) row_fail(sh.fail, ra.err);
    T* xo = reinterpret_cast<T*>(job.x);
#pragma unroll
    for (int j = 0; j < RPT; ++j)
      if (row[j] >= 0) xo[row[j]] = x[j];
  } else if (wid < 0) {
    // ---- control warps: warp j adds value j; warp 0 runs the scalars
    const int j = wid + ONE_CW;
    GridWord* words = ra.slots + (size_t)j * GRID_WORDS * G;
    unsigned pp = 0, pr = 0, ps = 0;
    unsigned long long gen = 0;
    bool ok = true;
    auto wait_sums = [&]() {                     // the compute warps' values are staged
      if (nwa == 0) return true;
      const bool got = row_wait(sh.fail, &sh.barP, pp);
      pp ^= 1u;
      return got;
    };
    auto exchange = [&](double t, double& tot) {
      ++gen;
      return j == 0 ? grid_total<true>(words, G, cta, gen, t, tot, ra.limit, ra.err)
                    : grid_total<false>(words, G, cta, gen, t, tot, ra.limit, ra.err);
    };
    auto total = [&]() {                         // this warp's sum over the grid, into sh.s
      if (!wait_sums()) return false;
      double t = 0.0;
      for (int i = lane; i < nwa * 32; i += 32) t += stage[j * ONE_THREADS + i];
      t = warp_sum_all(t);
      double tot = 0.0;
      if (!exchange(t, tot)) return false;
      if (lane == 0) {
        sh.s[j] = tot;
        bar_arrive(j == 0 ? &sh.barQ : &sh.barS);
      }
      __syncwarp();                              // warp 0 reads sh.s[0] in every lane
      return true;
    };
    if (j > 0) {
      ok = total();
      for (int k = 0; ok; ++k) {
        const int t = k & 1;
        if (!(ok = row_wait(sh.fail, &sh.barD[t], pd[t]))) break;
        pd[t] ^= 1u;
        if (sh.d[t].stop) break;
        ok = total();
      }
    } else {
      MinresState S{};
      S.k = 1;
      double ib = 0.0, ibp = 1.0, S6 = 0.0;
      auto others = [&]() {
        const bool got = row_wait(sh.fail, &sh.barS, ps);
        ps ^= 1u;
        return got;
      };
      ok = total() && others();
      if (ok) {
        init_state(S, sh.s[0], sh.s[1], job.tol, job.kmax, job.sigma);
        ib = S.beta > 0.0 ? 1.0 / S.beta : 0.0;
        if (lane == 0) { sh.d[0].apply = 0; sh.d[0].stop = S.done != 0; bar_arrive(&sh.barD[0]); }
      }
      for (int k = 0; ok && S.done == 0; ++k) {
        if (replaced(k)) {                       // q_{k+1} complete, no sums
          double none;
          if (nwa > 0) {
            if (!(ok = row_wait(sh.fail, &sh.barR, pr))) break;
            pr ^= 1u;
          }
          if (!(ok = exchange(0.0, none))) break;
          if (lane == 0) bar_arrive(&sh.barQ);
        }
        const double ib2 = ib * ib, c = S.beta * ibp;
        if (!(ok = total() && others())) break;
        // the coefficients of q_{k+1} first: 1 / beta, a = alpha / beta, c
        const double S1 = sh.s[0];
        const double alpha = S1 * ib2, a = alpha * ib;
        if (lane == 0) {
          T* co = reinterpret_cast<T*>(sh.c);
          co[0] = (T)ib; co[1] = (T)a; co[2] = (T)c; co[3] = (T)(0.5 * ib);
          bar_arrive(&sh.barC);
        }
        const double S4 = sh.s[3];
        pipe_scalars<T>(S, sh.s[0], sh.s[1], sh.s[2], S4, sh.s[4], S6, alpha, a, c, ib, ib2, ibp);
        S6 = S4;
        const int t = (k + 1) & 1;
        if (lane == 0) {
          T* co = reinterpret_cast<T*>(sh.d[t].co);
          co[0] = (T)S.cq; co[1] = (T)S.cd1; co[2] = (T)S.cd2; co[3] = (T)S.tau;
          sh.d[t].apply = S.pending;
          sh.d[t].stop = S.done != 0;
          bar_arrive(&sh.barD[t]);
        }
      }
      S.pending = 0;
      S.done = 2;
      if (!ok) S.status = HS_TIMEOUT;
      if (lane == 0 && cta == 0) *job.st = S;
    }
    if (!ok) row_fail(sh.fail, ra.err);
  }
}

template <typename T, int RPT>
hs_status launch_t(hs_handle* hd, const RowArgs& ra, int pc, int G, int rperiod) {
  const size_t sm = sizeof(double) * PIPE_NV * ONE_THREADS +
                    sizeof(uint32_t) * (size_t)hd->L * ONE_THREADS * RPT;
  auto kern = k_minres_row1<T, RPT>;
  RowArgs a = ra;
  int p = pc, r = rperiod;
  void* args[] = {&a, &p, &r};
  return row_launch(hd, (const void*)kern, G, ONE_NT, sm, 4 * ONE_THREADS * RPT + 1024, args);
}

template <typename T>
hs_status launch_rpt(hs_handle* hd, const RowArgs& ra, int pc, int G, int rperiod) {
  const int rpc = ((int)hd->n + G - 1) / G;
  switch ((rpc + ONE_THREADS - 1) / ONE_THREADS) {
    case 1: return launch_t<T, 1>(hd, ra, pc, G, rperiod);
    case 2: return launch_t<T, 2>(hd, ra, pc, G, rperiod);
    case 3: return launch_t<T, 3>(hd, ra, pc, G, rperiod);
    default: return HS_CUDA;
  }
}

}  // namespace

hs_status solve_row1(hs_handle* hd, const void* b, const MinresVecs& v, hs_dtype dt, int pc,
                     double tol, long long kmax, bool* broke) {
  RowArgs ra{};
  int G = 0;
  *broke = false;
  hs_status st = row_args(hd, b, v, tol, kmax, PIPE_NV, &ra, &G);
  if (st != HS_OK) return st;
  const int r = pipe_replace_period();
  st = dt == HS_F64 ? launch_rpt<double>(hd, ra, pc, G, r) : launch_rpt<float>(hd, ra, pc, G, r);
  if (st != HS_OK) return st;
  if ((st = grid_finish(hd)) != HS_OK) return st;
  const MinresState& S = *hd->h_state;
  *broke = S.status == HS_BREAKDOWN && S.pad == PIPE_EXPANSION;
  return *broke ? HS_CUDA : HS_OK;
}

}  // namespace hs
