// Host check of the six-low-bit superblock product (test infrastructure).
//
// Runs the kernel's own code from sb6.cuh on the CPU: the plan (build_plan6),
// the flat pass (slot copies and whole-superblock sums, sb6_flat) and the
// per-lane row code (sb6_rows_any) over the pair's work list, pair by pair in the
// kernel's order. Every slot element that the copies do not fill, G and the guard
// regions around x hold NaN, so that a read of anything not staged shows up in y;
// a wrong neighbour or diagonal term shows up against the oracle's explicit H.
//   sb6_host_check L KS sigma dir
// reads dir/h.bin (L doubles) and dir/x.bin (n doubles), writes dir/y64.bin and
// dir/y32.bin (the FP32 result widened).
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <string>
#include <vector>

#include "../../paper_2203_09732_gb300/csrc/sb6.cuh"

using namespace hs;
using namespace hs::sb6;

template <typename T>
static bool run(int L, const double* h, int KS, const T* x, T* y, double sigma) {
  HostPlan6<T> P;
  if (!build_plan6<T>(L, h, KS, &P)) return false;
  const sb::HostPlan& B = P.base;
  const int km = B.km, tile = ST<T> << km;
  std::vector<T> X(2 * (size_t)tile + ZSLOTS * ST<T>), G(2 * (size_t)tile);
  T* Z = X.data() + 2 * tile;
  const int NT = 96;  // emulated threads of the flat pass (any count)
  for (const int4 pr : P.pairs) {
    sb::Sup sh[2];
    sh[0] = pr.x >= 0 ? B.sup[pr.x] : sb::Sup{};
    sh[1] = pr.y >= 0 ? B.sup[pr.y] : sb::Sup{};
    for (T& v : X) v = (T)NAN;
    for (int e = 0; e < ZSLOTS * ST<T>; ++e) Z[e] = T(0);
    for (T& v : G) v = (T)NAN;
    T uT[4];
    for (int t = 0; t < 4; ++t) {
      const int s = t >> 1;
      const uint32_t tb0 = (sh[s].meta >> 16) & 1u;
      uT[t] = (T)(sh[s].dT - sigma + (((uint32_t)(t & 1) == tb0) ? 0.25 : -0.25));
    }
    for (int s = 0; s < 2; ++s)
      if (sh[s].C)
        for (int t = 0; t < NT; ++t)
          sb6_flat<T>(x + sh[s].R, sh[s], P.slotmap.data() + P.slot_off[sh[s].meta & 0xFF],
                         X.data() + s * tile, G.data() + s * tile, t, NT);
    for (int wt = 0; wt < pr.w; ++wt) {
      const uint16_t* e = &P.tasks[(size_t)(pr.z + wt) * 32];
      if (e[0] == NO_TASK) return false;      // lane 0 gives the warp's class
      int wc = -1;
      for (int lane = 0; lane < 32; ++lane) {
        if (e[lane] == NO_TASK) continue;
        const int s = e[lane] >> 15, m = e[lane] & 0x7FFF;
        const uint32_t hm = sh[s].meta;
        const int w = (int)(hm & 0xFF) - sb::popc_host((uint32_t)m);
        if (wc < 0) wc = w;
        if (w != wc) return false;            // one class per warp
        const uint32_t top = (hm >> 17) & 1u;
        sb6_rows_any<T>(w, m, km, top, X.data() + s * tile,
                        sh[1 - s].C ? X.data() + (1 - s) * tile : nullptr, Z,
                        G.data() + s * tile + swz(m) * ST<T>,
                        &P.dl[(((int)top * 2 + (m & 1)) * (K + 1) + w) * DL],
                        P.dmid[m] + uT[s * 2 + ((m >> (km - 1)) & 1)]);
      }
    }
    for (int s = 0; s < 2; ++s)
      for (uint32_t i = 0; i < sh[s].C; ++i)
        y[sh[s].R + i] = G[s * tile + P.slotmap[P.slot_off[sh[s].meta & 0xFF] + i]];
  }
  return true;
}

static bool io(const char* fn, void* p, size_t bytes, const char* mode) {
  FILE* f = fopen(fn, mode);
  if (!f) return false;
  const size_t got = mode[0] == 'r' ? fread(p, 1, bytes, f) : fwrite(p, 1, bytes, f);
  fclose(f);
  return got == bytes;
}

int main(int argc, char** argv) {
  if (argc != 5) {
    fprintf(stderr, "usage: sb6_host_check L KS sigma dir\n");
    return 2;
  }
  const int L = atoi(argv[1]), KS = atoi(argv[2]);
  const double sigma = atof(argv[3]);
  const std::string dir = argv[4];
  std::vector<double> h(L);
  if (!io((dir + "/h.bin").c_str(), h.data(), sizeof(double) * L, "rb")) return 3;
  HostPlan6<double> probe;
  if (!build_plan6<double>(L, h.data(), KS, &probe)) {
    printf("plan does not apply\n");
    return 4;
  }
  const size_t n = (size_t)sb::binom64(L, L / 2);
  std::vector<double> xs(n);
  if (!io((dir + "/x.bin").c_str(), xs.data(), sizeof(double) * n, "rb")) return 3;
  const size_t guard = 1 << 20;
  std::vector<double> xb(n + 2 * guard, NAN), yb(n + 2 * guard, NAN);
  for (size_t i = 0; i < n; ++i) xb[guard + i] = xs[i];
  if (!run<double>(L, h.data(), KS, xb.data() + guard, yb.data() + guard, sigma)) return 6;
  if (!io((dir + "/y64.bin").c_str(), yb.data() + guard, sizeof(double) * n, "wb")) return 5;
  std::vector<float> xf(n + 2 * guard, NAN), yf(n + 2 * guard, NAN);
  for (size_t i = 0; i < n; ++i) xf[guard + i] = (float)xs[i];
  if (!run<float>(L, h.data(), KS, xf.data() + guard, yf.data() + guard, sigma)) return 6;
  std::vector<double> y32(n);
  for (size_t i = 0; i < n; ++i) y32[i] = yf[guard + i];
  if (!io((dir + "/y32.bin").c_str(), y32.data(), sizeof(double) * n, "wb")) return 5;
  printf("ok n=%zu pairs=%zu warps=%zu\n", n, probe.pairs.size(), probe.tasks.size() / 32);
  return 0;
}
