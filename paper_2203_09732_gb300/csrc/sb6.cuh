// Superblock product (H - sigma) x of Eq. (1) with six low bits: one lane per
// sub-block, its rows in registers.
//
// The split of a state word is that of sb.cuh with k = 6: p = bits 0..5,
// m = the km = KS - 6 mid bits, T = the top L - KS bits. A sub-block (T, m) holds
// the C(6, w) <= 20 rows whose low pattern p has popcount w = L/2 - popcount(T)
// - popcount(m), in ascending p. A lane owns a whole sub-block: with the rows of
// a class known at compile time,
//   low interior  (j, j+1), j < 5        : register additions;
//   mid interior  (j, j+1), 6 <= j < KS-1 : slot m ^ (3 << (j-6)), same rows: 16-byte
//                                          loads of whole slots;
//   cut (5, 6)                           : slot m ^ 1, a contiguous run of rows (the
//                                          rows with bit 5 clear come first);
//   wrap (L-1, 0)                        : the partner superblock's slot m, row of
//                                          p ^ 1 (fixed per class);
//   bond (KS-1, KS) and high interior    : whole-superblock shifts in rank order,
//                                          summed by a flat coalesced pass into G.
// Why six: each neighbour run costs a few instructions of addressing however
// many rows it has, so more rows per lane mean fewer instructions per row (11
// rows on average here, 3.4 with four low bits), until registers run out (20
// rows of x and of sums; seven low bits would need 70).
//
// x of the pair {T, T ^ top} and G lie in shared memory in slots of ST elements
// at the swizzled index swz(m); ST is an odd number of 16-byte entries, so lanes
// whose slots differ mod 8 read distinct bank groups, and swz is linear over XOR,
// so the neighbour slots of such lanes do too. The work list of a pair is cut
// into warps of one class each, dealt so that aligned groups of 8 lanes have
// distinct swz(m) mod 8 where the class allows it.
#pragma once
#include <map>
#include <utility>

#include "sb.cuh"

namespace hs {
namespace sb6 {

constexpr int K = 6;            // low bits
constexpr int CMAX = 20;        // rows of the largest sub-block
constexpr int KM_MAX = 8;       // mid bits: 256 slots per superblock
constexpr int DL = 20;          // diagonal entries per (top, bit 0 of m, class)
constexpr uint16_t NO_TASK = 0xFFFFu;
// slot length in elements: 5 (FP32) or 11 (FP64) 16-byte entries
template <typename T> constexpr int ST = sizeof(T) == 8 ? 22 : 20;
constexpr int ZSLOTS = 8;       // zero slots behind the tile, one per bank group

__host__ __device__ constexpr int swz(int m) { return m ^ ((m >> 2) & 7) ^ ((m >> 5) & 7); }

__host__ __device__ constexpr int choose(int n, int r) {
  if (r < 0 || r > n) return 0;
  int v = 1;
  for (int i = 1; i <= r; ++i) v = v * (n - r + i) / i;
  return v;
}
__host__ __device__ constexpr int popc6(int p) {
  int c = 0;
  for (int b = 0; b < K; ++b) c += (p >> b) & 1;
  return c;
}
// r-th pattern of class w in ascending order, and the rank of p in its class
__host__ __device__ constexpr int pat6(int w, int r) {
  int seen = 0;
  for (int p = 0; p < (1 << K); ++p)
    if (popc6(p) == w && seen++ == r) return p;
  return 0;
}
__host__ __device__ constexpr int rank6(int p) {
  int r = 0;
  for (int q = 0; q < p; ++q) r += popc6(q) == popc6(p);
  return r;
}
template <int W, int R> struct Pat { static constexpr int v = pat6(W, R); };
template <int P> struct Rank { static constexpr int v = rank6(P); };

// Device copy of the tables.
struct Geo6 {
  const sb::Sup* sup;          // superblock headers, ascending T
  const int4* pairs;           // {T0, T0 | top} superblock indices (-1: absent), first warp of
                               // the work list, its warps
  const uint16_t* slotmap;     // per class wq: flat row -> element of superblock 0's slots
  const uint16_t* tasks;       // 32 lanes a warp: s << 15 | m, or NO_TASK
  const void* dmid;            // [2^km] mid Ising + fields (T)
  const void* dl;              // [top][bit 0 of m][w][DL]: low, cut and wrap Ising + low fields (T)
  int npairs, km;
  int slot_off[sb::WQ_MAX + 1];
};

// Host tables for element type T (the slot stride differs).
template <typename T>
struct HostPlan6 {
  sb::HostPlan base;           // superblocks, pairs, Sub with k = 6
  std::vector<int4> pairs;
  std::vector<uint16_t> slotmap, tasks;
  std::vector<T> dmid, dl;
  int slot_off[sb::WQ_MAX + 1] = {0};
};

// Build the plan for chain length L, fields h[0..L-1] and a KS-bit window.
// False where the split does not apply (km = KS - 6 must be 1..8, and the top
// field must have 2..17 bits).
template <typename T>
inline bool build_plan6(int L, const double* h, int KS, HostPlan6<T>* P) {
  *P = HostPlan6<T>{};
  const int km = KS - K;
  if (km < 1 || km > KM_MAX || !sb::build_plan(L, h, K, KS, &P->base, KM_MAX)) return false;
  const sb::HostPlan& B = P->base;
  const int nm = 1 << km;
  P->dmid.assign(nm, T(0));
  for (int wq = 0; wq <= KS; ++wq) {
    P->slot_off[wq] = (int)P->slotmap.size();
    for (int m = 0; m < nm; ++m) {
      const int w = wq - sb::popc_host((uint32_t)m);
      if (w < 0 || w > K) continue;
      P->dmid[m] = (T)B.sub[(size_t)wq * nm + m].dmid;
      for (int r = 0; r < choose(K, w); ++r)
        P->slotmap.push_back((uint16_t)(swz(m) * ST<T> + r));
    }
  }
  // work lists, one per pair of classes (wq of T0, of T0 | top)
  std::map<std::pair<int, int>, std::pair<int, int>> lists;
  auto list_of = [&](int wq0, int wq1) {
    const auto key = std::make_pair(wq0, wq1);
    auto it = lists.find(key);
    if (it != lists.end()) return it->second;
    const int first = (int)P->tasks.size() / 32;
    const int by_size[K + 1] = {3, 2, 4, 1, 5, 0, 6};     // largest classes first
    for (int w : by_size) {
      std::vector<uint16_t> lane;
      for (int s = 0; s < 2; ++s)
        for (int b0 = 0; b0 < 2; ++b0) {
          const int wq = s ? wq1 : wq0;
          if (wq < 0) continue;
          std::vector<std::vector<int>> bk(8);
          int left = 0;
          for (int m = b0; m < nm; m += 2)
            if (wq - sb::popc_host((uint32_t)m) == w) {
              bk[swz(m) & 7].push_back(m);
              ++left;
            }
          // rounds over the bank groups, the fullest first
          while (left) {
            int ord[8] = {0, 1, 2, 3, 4, 5, 6, 7};
            std::stable_sort(ord, ord + 8,
                             [&](int a, int b) { return bk[a].size() > bk[b].size(); });
            for (int q = 0; q < 8; ++q)
              if (!bk[ord[q]].empty()) {
                lane.push_back((uint16_t)(s << 15 | bk[ord[q]].back()));
                bk[ord[q]].pop_back();
                --left;
              }
          }
        }
      while (lane.size() % 32) lane.push_back(NO_TASK);
      P->tasks.insert(P->tasks.end(), lane.begin(), lane.end());
    }
    const auto v = std::make_pair(first, (int)P->tasks.size() / 32 - first);
    lists[key] = v;
    return v;
  };
  for (const int2 pr : B.pairs) {
    const auto l = list_of(pr.x >= 0 ? (int)(B.sup[pr.x].meta & 0xFF) : -1,
                           pr.y >= 0 ? (int)(B.sup[pr.y].meta & 0xFF) : -1);
    P->pairs.push_back(make_int4(pr.x, pr.y, l.first, l.second));
  }
  P->dl.assign(2 * 2 * (K + 1) * DL, T(0));
  for (int top = 0; top < 2; ++top)
    for (int b0 = 0; b0 < 2; ++b0)
      for (int w = 0; w <= K; ++w)
        for (int r = 0; r < choose(K, w); ++r) {
          const int p = pat6(w, r);
          double d = B.dlow[B.cls_off[w] + r];
          d += (((p >> (K - 1)) & 1) == b0) ? 0.25 : -0.25;
          d += ((p & 1) == top) ? 0.25 : -0.25;
          P->dl[(((size_t)top * 2 + b0) * (K + 1) + w) * DL + r] = (T)d;
        }
  return true;
}

// ---------------------------------------------------------------------------
// Row code shared by the kernel and the host check.
#ifdef __CUDA_ARCH__
#define SB6_HD __device__ __forceinline__
#else
#define SB6_HD inline
#endif

template <int I> struct Int { static constexpr int v = I; };
template <int... I, class F>
SB6_HD void for_seq(std::integer_sequence<int, I...>, F&& f) {
  (f(Int<I>{}), ...);
}
template <int N, class F>
SB6_HD void static_for(F&& f) {
  for_seq(std::make_integer_sequence<int, N>{}, f);
}

// v[0..N) = p[0..N), in 16-byte loads (p 16-byte aligned; N a multiple of E).
template <typename T> constexpr int E = 16 / sizeof(T);
constexpr int up(int n, int e) { return (n + e - 1) / e * e; }
template <typename T, int N>
SB6_HD void ldv(const T* p, T* v) {
#ifdef __CUDA_ARCH__
#pragma unroll
  for (int c = 0; c < N; c += E<T>) {
    if constexpr (sizeof(T) == 4) {
      const float4 a = *reinterpret_cast<const float4*>(p + c);
      v[c] = a.x; v[c + 1] = a.y; v[c + 2] = a.z; v[c + 3] = a.w;
    } else {
      const double2 a = *reinterpret_cast<const double2*>(p + c);
      v[c] = a.x; v[c + 1] = a.y;
    }
  }
#else
  for (int c = 0; c < N; ++c) v[c] = p[c];
#endif
}
template <typename T, int N>
SB6_HD void stv(T* p, const T* v) {
#ifdef __CUDA_ARCH__
#pragma unroll
  for (int c = 0; c < N; c += E<T>) {
    if constexpr (sizeof(T) == 4)
      *reinterpret_cast<float4*>(p + c) = make_float4(v[c], v[c + 1], v[c + 2], v[c + 3]);
    else
      *reinterpret_cast<double2*>(p + c) = make_double2(v[c], v[c + 1]);
  }
#else
  for (int c = 0; c < N; ++c) p[c] = v[c];
#endif
}
// a[0..N) += p[0..N): 16-byte loads, in FP32 two additions per instruction.
template <typename T, int N>
SB6_HD void addv(const T* p, T* a) {
#ifdef __CUDA_ARCH__
#pragma unroll
  for (int c = 0; c < N; c += E<T>) {
    if constexpr (sizeof(T) == 4) {
      const float4 v = *reinterpret_cast<const float4*>(p + c);
      asm("{\n.reg .b64 x, y, z;\n"
          "mov.b64 x, {%0, %1};\nmov.b64 y, {%2, %3};\nadd.rn.f32x2 z, x, y;\n"
          "mov.b64 {%0, %1}, z;\n}" : "+f"(a[c]), "+f"(a[c + 1]) : "f"(v.x), "f"(v.y));
      asm("{\n.reg .b64 x, y, z;\n"
          "mov.b64 x, {%0, %1};\nmov.b64 y, {%2, %3};\nadd.rn.f32x2 z, x, y;\n"
          "mov.b64 {%0, %1}, z;\n}" : "+f"(a[c + 2]), "+f"(a[c + 3]) : "f"(v.z), "f"(v.w));
    } else {
      const double2 v = *reinterpret_cast<const double2*>(p + c);
      a[c] += v.x;
      if (c + 1 < N) a[c + 1] += v.y;
    }
  }
#else
  for (int c = 0; c < N; ++c) a[c] += p[c];
#endif
}

// y = (H - sigma) x for the rows of sub-block m (class W), written over its sums
// in g. X: this superblock's slots; Xp: the partner's (nullptr: none); Z: the zero
// slots; g: the sub-block's slot of G; dl: the class's diagonal terms for (top,
// bit 0 of m); u = dmid + dT - sigma + Ising of bond (KS-1, KS). Returns
// sum_r x_r y_r. N rows are computed where W has C: the entries between are not
// rows (their slots hold whatever was there) and nothing reads them.
template <typename T, int W>
SB6_HD T sb6_rows(int m, int km, uint32_t top, const T* X, const T* Xp, const T* Z, T* g,
                  const T* dl, T u) {
  constexpr int C = choose(K, W), N = up(C, E<T>);
  const int pm = swz(m);
  T x[N], a[N];
  ldv<T, N>(X + pm * ST<T>, x);
  ldv<T, N>(g, a);
  // low interior bonds
  static_for<C>([&](auto r) {
    static_for<K - 1>([&](auto j) {
      constexpr int p = Pat<W, decltype(r)::v>::v;
      if constexpr (((p >> decltype(j)::v) & 1) != ((p >> (decltype(j)::v + 1)) & 1))
        a[decltype(r)::v] += x[Rank<p ^ (3 << decltype(j)::v)>::v];
    });
  });
  // mid interior bonds. FP32: a parallel bond reads the zero slot of the bank
  // group the antiparallel one would use (no branches, no bank conflicts); FP64:
  // only the antiparallel ones (an addition of zeros costs as much as any)
  int t = (m ^ (m >> 1)) & ((1 << (km - 1)) - 1);
  if constexpr (sizeof(T) == 4) {
#pragma unroll
    for (int j = 0; j < KM_MAX - 1; ++j)
      if (j < km - 1) {
        const int idx = pm ^ swz(3 << j);
        addv<T, N>(((t >> j) & 1) ? X + idx * ST<T> : Z + (idx & 7) * ST<T>, a);
      }
  } else {
    while (t) {
#ifdef __CUDA_ARCH__
      const int j = __ffs(t) - 1;
#else
      int j = 0;
      while (!((t >> j) & 1)) ++j;
#endif
      t &= t - 1;
      addv<T, N>(X + swz(m ^ (3 << j)) * ST<T>, a);
    }
  }
  // cut bond (5, 6): the rows with bit 5 set (bit 0 of m clear) or clear (set)
  {
    const T* s = X + (pm ^ swz(1)) * ST<T>;
    constexpr int c0 = choose(5, W - 1), a0 = choose(5, W), c1 = choose(5, W), s1 = choose(5, W + 1);
    if (!(m & 1)) {
      if constexpr (c0 > 0) {
        T v[up(c0, E<T>)];
        ldv<T, up(c0, E<T>)>(s, v);
        static_for<c0>([&](auto i) { a[a0 + decltype(i)::v] += v[decltype(i)::v]; });
      }
    } else {
      if constexpr (c1 > 0 && W < K) {
        constexpr int b = s1 / E<T> * E<T>;             // aligned start
        T v[up(s1 - b + c1, E<T>)];
        ldv<T, up(s1 - b + c1, E<T>)>(s + b, v);
        static_for<c1>([&](auto i) { a[decltype(i)::v] += v[s1 - b + decltype(i)::v]; });
      }
    }
  }
  // wrap bond (L-1, 0)
  if (Xp) {
    const T* s = Xp + pm * ST<T>;
    if (!top) {
      if constexpr (W > 0) {
        constexpr int CS = choose(K, W - 1);
        T v[up(CS, E<T>)];
        ldv<T, up(CS, E<T>)>(s, v);
        static_for<C>([&](auto r) {
          constexpr int p = Pat<W, decltype(r)::v>::v;
          if constexpr (p & 1) a[decltype(r)::v] += v[Rank<p ^ 1>::v];
        });
      }
    } else {
      if constexpr (W < K) {
        constexpr int CS = choose(K, W + 1);
        T v[up(CS, E<T>)];
        ldv<T, up(CS, E<T>)>(s, v);
        static_for<C>([&](auto r) {
          constexpr int p = Pat<W, decltype(r)::v>::v;
          if constexpr (!(p & 1)) a[decltype(r)::v] += v[Rank<p ^ 1>::v];
        });
      }
    }
  }
  T dot = T(0);
  {
    T d[N];
    ldv<T, N>(dl, d);
#pragma unroll
    for (int r = 0; r < C; ++r) {
      const T y = (d[r] + u) * x[r] + T(0.5) * a[r];
      a[r] = y;
      dot += x[r] * y;
    }
  }
  stv<T, N>(g, a);
  return dot;
}

template <typename T>
SB6_HD T sb6_rows_any(int w, int m, int km, uint32_t top, const T* X, const T* Xp, const T* Z, T* g,
                      const T* dl, T u) {
  switch (w) {
    case 0: return sb6_rows<T, 0>(m, km, top, X, Xp, Z, g, dl, u);
    case 1: return sb6_rows<T, 1>(m, km, top, X, Xp, Z, g, dl, u);
    case 2: return sb6_rows<T, 2>(m, km, top, X, Xp, Z, g, dl, u);
    case 3: return sb6_rows<T, 3>(m, km, top, X, Xp, Z, g, dl, u);
    case 4: return sb6_rows<T, 4>(m, km, top, X, Xp, Z, g, dl, u);
    case 5: return sb6_rows<T, 5>(m, km, top, X, Xp, Z, g, dl, u);
    default: return sb6_rows<T, 6>(m, km, top, X, Xp, Z, g, dl, u);
  }
}

// Rows i0 + u nt, u < U, of one superblock H (x rows xs[0, C)): copies x of the row
// into its slot element and sums x over its high interior flips and its (KS-1,
// KS) flip into the same element of G; four bonds of loads in flight.
template <typename T, int U>
SB6_HD void sb6_flat_rows(const T* xs, const sb::Sup& H, const uint16_t* map, T* X, T* G, int i0,
                          int nt) {
  const int nh = (int)((H.meta >> 8) & 0xFF);
  const int ka = (int)H.ka, kb = (int)H.kb;
  const T* xk = xs + H.kd;
  int e[U];
  T g[U];
#pragma unroll
  for (int u = 0; u < U; ++u) {
    const int i = i0 + u * nt;
    e[u] = sb::sb_ldg(map + i);
    g[u] = (i >= ka && i < kb) ? xk[i] : T(0);
  }
#pragma unroll
  for (int u = 0; u < U; ++u) sb::sb_copy(X + e[u], xs + i0 + u * nt);
  int q = 0;
  for (; q + 4 <= nh; q += 4) {
    T v[4][U];
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      const T* b = xs + H.hd[q + c] + i0;
#pragma unroll
      for (int u = 0; u < U; ++u) v[c][u] = b[u * nt];
    }
#pragma unroll
    for (int c = 0; c < 4; ++c)
#pragma unroll
      for (int u = 0; u < U; ++u) g[u] += v[c][u];
  }
  for (; q < nh; ++q) {
    const T* b = xs + H.hd[q] + i0;
#pragma unroll
    for (int u = 0; u < U; ++u) g[u] += b[u * nt];
  }
#pragma unroll
  for (int u = 0; u < U; ++u) G[e[u]] = g[u];
}

// All rows of a superblock: thread t of nt takes rows t, t + nt, ..., four at a
// time, then two, then one.
template <typename T>
SB6_HD void sb6_flat(const T* xs, const sb::Sup& H, const uint16_t* map, T* X, T* G, int t, int nt) {
  const int C = (int)H.C;
  int i0 = t;
  for (; i0 + 3 * nt < C; i0 += 4 * nt) sb6_flat_rows<T, 4>(xs, H, map, X, G, i0, nt);
  if (i0 + nt < C) {
    sb6_flat_rows<T, 2>(xs, H, map, X, G, i0, nt);
    i0 += 2 * nt;
  }
  if (i0 < C) sb6_flat_rows<T, 1>(xs, H, map, X, G, i0, nt);
}

#undef SB6_HD

}  // namespace sb6
}  // namespace hs
