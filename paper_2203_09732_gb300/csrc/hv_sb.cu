// Superblock form of y = (H - sigma) x (Eq. (1)) for long chains: one CTA per
// superblock pair {T, T ^ top}. Phase 1 stages x of the pair into shared
// memory by asynchronous copies while it sums the high-bit and (KS-1, KS)
// flips of every row from global memory (coalesced shifted streams); phase 2
// walks the sub-blocks and reads shared memory only. Layout and bond kinds:
// sb.cuh; the kernel (shared with MINRES pass A): sb_kern.cuh. This file
// builds the plans and launches the product.
#include <cstdlib>
#include <cstring>

#include "common.cuh"
#include "sb.cuh"
#include "sb4_kern.cuh"
#include "sb6_kern.cuh"
#include "sb_kern.cuh"

namespace hs {
namespace sb {

constexpr int NT_SB = 512;

// The product kernel for a plan with km mid bits: the mid-bond count as a
// compile-time constant for the windows the library uses (km = 4), else read
// from the plan.
template <typename T>
static auto kernel_of(int km) {
  return km == 4 ? k_sbhv<T, NT_SB, 2, 4, MODE_HV, 3> : k_sbhv<T, NT_SB, 2, 4, MODE_HV, 0>;
}

template <typename T>
static hs_status make_dev(hs_handle* hd, int KS, DevPlan** out) {
  *out = nullptr;
  HostPlan P;
  if (!build_plan(hd->L, hd->h, std::min(hd->k, K_MAX), KS, &P)) return HS_OK;
  auto al = [](size_t b) { return (b + 255) & ~(size_t)255; };
  const size_t s_low = al(P.low.size() * sizeof(Low16)), s_dlow = al(P.dlow.size() * sizeof(double)),
               s_sub = al(P.sub.size() * sizeof(Sub)), s_ord = al(P.order.size() * sizeof(uint16_t)),
               s_sup = al(P.sup.size() * sizeof(Sup)), s_pr = al(P.pairs.size() * sizeof(int2));
  const size_t total = s_low + s_dlow + s_sub + s_ord + s_sup + s_pr;
  std::vector<char> host(total, 0);
  size_t o = 0;
  auto put = [&](const void* src, size_t bytes, size_t slot) {
    std::memcpy(host.data() + o, src, bytes);
    const size_t at = o;
    o += slot;
    return at;
  };
  const size_t o_low = put(P.low.data(), P.low.size() * sizeof(Low16), s_low);
  const size_t o_dlow = put(P.dlow.data(), P.dlow.size() * sizeof(double), s_dlow);
  const size_t o_sub = put(P.sub.data(), P.sub.size() * sizeof(Sub), s_sub);
  const size_t o_ord = put(P.order.data(), P.order.size() * sizeof(uint16_t), s_ord);
  const size_t o_sup = put(P.sup.data(), P.sup.size() * sizeof(Sup), s_sup);
  const size_t o_pr = put(P.pairs.data(), P.pairs.size() * sizeof(int2), s_pr);
  DevPlan* d = new DevPlan();
  if (dev_alloc(hd, &d->mem, total) != HS_OK) {
    delete d;
    return fail(hd, HS_OOM, "superblock table allocation failed");
  }
  // pageable source: the copy is staged before the call returns
  if (cudaMemcpyAsync(d->mem, host.data(), total, cudaMemcpyHostToDevice, hd->stream) != cudaSuccess) {
    cudaGetLastError();
    dev_free(hd, d->mem);
    delete d;
    return fail(hd, HS_CUDA, "superblock table upload failed");
  }
  char* base = static_cast<char*>(d->mem);
  Geo& g = d->geo;
  g.low = reinterpret_cast<const Low16*>(base + o_low);
  g.dlow = reinterpret_cast<const double*>(base + o_dlow);
  g.sub = reinterpret_cast<const Sub*>(base + o_sub);
  g.order = reinterpret_cast<const uint16_t*>(base + o_ord);
  g.sup = reinterpret_cast<const Sup*>(base + o_sup);
  g.pairs = reinterpret_cast<const int2*>(base + o_pr);
  g.npairs = (int)P.pairs.size();
  g.k = P.k;
  g.km = P.km;
  g.KS = P.KS;
  for (int i = 0; i < K_MAX + 2; ++i) {
    g.cls_off[i] = P.cls_off[i];
    g.cls_C[i] = P.cls_C[i];
  }
  for (int i = 0; i <= WQ_MAX; ++i) g.nvalid[i] = P.nvalid[i];
  g.dscale = P.dscale;
  d->smem = smem_bytes<T>((int)P.low.size(), P.km);
  auto kern = kernel_of<T>(P.km);
  int nb = 0;
  if (allow_smem(kern, d->smem) &&
      cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, kern, NT_SB, d->smem) == cudaSuccess &&
      nb > 0) {
    d->grid = std::min(g.npairs, nb * hd->num_sms);
    d->ok = 1;
  } else {
    cudaGetLastError();  // the tile does not fit: the plan stays unused
  }
  *out = d;
  return HS_OK;
}

}  // namespace sb

namespace sb4 {

constexpr int NT4_F = 512;   // FP32: two CTAs of 512 threads per SM
constexpr int NT4_D = 256;   // FP64: more registers per thread

// The kernel for a plan: the mid loop unrolled for the library's windows
// (10 mid bits in FP32, 9 in FP64), a run-time loop for other windows.
template <typename T, int MODE>
using K4 = void (*)(Geo4, const T*, T*, const double*, int, sb::MinresArgs);
template <typename T, int MODE>
K4<T, MODE> kernel4_for(int km) {
  if constexpr (sizeof(T) == 8) {
    if (km == 9) return k_sb4<double, NT4_D, 2, 4, MODE, 9>;
    return k_sb4<double, NT4_D, 2, 4, MODE, 0>;
  } else {
    if (km == 10) return k_sb4<float, NT4_F, 2, 4, MODE, 10>;
    return k_sb4<float, NT4_F, 2, 4, MODE, 0>;
  }
}

template <typename T>
static hs_status make_dev4(hs_handle* hd, int KS, DevPlan4** out) {
  *out = nullptr;
  HostPlan4 P;
  if (!build_plan4(hd->L, hd->h, KS, &P)) return HS_OK;
  const sb::HostPlan& B = P.base;
  auto al = [](size_t b) { return (b + 255) & ~(size_t)255; };
  struct Part { const void* src; size_t bytes; size_t at; };
  std::vector<Part> parts = {
      {B.sup.data(), B.sup.size() * sizeof(sb::Sup), 0},
      {B.pairs.data(), B.pairs.size() * sizeof(int2), 0},
      {P.slotmap.data(), P.slotmap.size() * sizeof(uint16_t), 0},
      {P.order.data(), P.order.size() * sizeof(uint16_t), 0},
      {P.lo.data(), P.lo.size() * sizeof(uint16_t), 0},
      {P.dmid_f.data(), P.dmid_f.size() * sizeof(float), 0},
      {P.dmid_d.data(), P.dmid_d.size() * sizeof(double), 0},
      {P.dl_f.data(), P.dl_f.size() * sizeof(float), 0},
      {P.dl_d.data(), P.dl_d.size() * sizeof(double), 0}};
  size_t total = 0;
  for (Part& q : parts) {
    q.at = total;
    total += al(q.bytes);
  }
  std::vector<char> host(total, 0);
  for (const Part& q : parts) std::memcpy(host.data() + q.at, q.src, q.bytes);
  DevPlan4* d = new DevPlan4();
  if (dev_alloc(hd, &d->mem, total) != HS_OK) {
    delete d;
    return fail(hd, HS_OOM, "superblock table allocation failed");
  }
  // pageable source: the copy is staged before the call returns
  if (cudaMemcpyAsync(d->mem, host.data(), total, cudaMemcpyHostToDevice, hd->stream) != cudaSuccess) {
    cudaGetLastError();
    dev_free(hd, d->mem);
    delete d;
    return fail(hd, HS_CUDA, "superblock table upload failed");
  }
  char* base = static_cast<char*>(d->mem);
  Geo4& g = d->geo;
  g.sup = reinterpret_cast<const sb::Sup*>(base + parts[0].at);
  g.pairs = reinterpret_cast<const int2*>(base + parts[1].at);
  g.slotmap = reinterpret_cast<const uint16_t*>(base + parts[2].at);
  g.order = reinterpret_cast<const uint16_t*>(base + parts[3].at);
  g.lo = reinterpret_cast<const uint16_t*>(base + parts[4].at);
  g.dmid_f = reinterpret_cast<const float*>(base + parts[5].at);
  g.dmid_d = reinterpret_cast<const double*>(base + parts[6].at);
  g.dl_f = reinterpret_cast<const float*>(base + parts[7].at);
  g.dl_d = reinterpret_cast<const double*>(base + parts[8].at);
  g.npairs = (int)B.pairs.size();
  g.km = B.km;
  g.KS = B.KS;
  g.cmax = P.cmax;
  for (int i = 0; i <= WQ_MAX; ++i) {
    g.slot_off[i] = P.slot_off[i];
    g.order_off[i] = P.order_off[i];
    g.nvalid[i] = P.nvalid[i];
  }
  g.dscale = B.dscale;
  d->smem = smem_bytes4<T>(g.km, g.cmax);
  auto kern = kernel4_for<T, sb::MODE_HV>(g.km);
  const int nt = sizeof(T) == 8 ? NT4_D : NT4_F;
  int nb = 0;
  if (allow_smem(kern, d->smem) &&
      cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, kern, nt, d->smem) == cudaSuccess &&
      nb > 0) {
    d->grid = std::min(g.npairs, nb * hd->num_sms);
    d->ok = 1;
  } else {
    cudaGetLastError();
  }
  *out = d;
  return HS_OK;
}

}  // namespace sb4

namespace sb6 {

template <typename T>
static hs_status make_dev6(hs_handle* hd, int KS, DevPlan6** out) {
  *out = nullptr;
  HostPlan6<T> P;
  if (!build_plan6<T>(hd->L, hd->h, KS, &P)) return HS_OK;
  const sb::HostPlan& B = P.base;
  auto al = [](size_t b) { return (b + 255) & ~(size_t)255; };
  struct Part { const void* src; size_t bytes; size_t at; };
  std::vector<Part> parts = {{B.sup.data(), B.sup.size() * sizeof(sb::Sup), 0},
                             {P.pairs.data(), P.pairs.size() * sizeof(int4), 0},
                             {P.slotmap.data(), P.slotmap.size() * sizeof(uint16_t), 0},
                             {P.tasks.data(), P.tasks.size() * sizeof(uint16_t), 0},
                             {P.dmid.data(), P.dmid.size() * sizeof(T), 0},
                             {P.dl.data(), P.dl.size() * sizeof(T), 0}};
  size_t total = 0;
  for (Part& q : parts) {
    q.at = total;
    total += al(q.bytes);
  }
  std::vector<char> host(total, 0);
  for (const Part& q : parts) std::memcpy(host.data() + q.at, q.src, q.bytes);
  DevPlan6* d = new DevPlan6();
  if (dev_alloc(hd, &d->mem, total) != HS_OK) {
    delete d;
    return fail(hd, HS_OOM, "superblock table allocation failed");
  }
  // pageable source: the copy is staged before the call returns
  if (cudaMemcpyAsync(d->mem, host.data(), total, cudaMemcpyHostToDevice, hd->stream) != cudaSuccess) {
    cudaGetLastError();
    dev_free(hd, d->mem);
    delete d;
    return fail(hd, HS_CUDA, "superblock table upload failed");
  }
  char* base = static_cast<char*>(d->mem);
  Geo6& g = d->geo;
  g.sup = reinterpret_cast<const sb::Sup*>(base + parts[0].at);
  g.pairs = reinterpret_cast<const int4*>(base + parts[1].at);
  g.slotmap = reinterpret_cast<const uint16_t*>(base + parts[2].at);
  g.tasks = reinterpret_cast<const uint16_t*>(base + parts[3].at);
  g.dmid = base + parts[4].at;
  g.dl = base + parts[5].at;
  g.npairs = (int)P.pairs.size();
  g.km = B.km;
  for (int i = 0; i <= sb::WQ_MAX; ++i) g.slot_off[i] = P.slot_off[i];
  d->smem = smem_bytes6<T>(g.km);
  auto kern = kernel6<T, sb::MODE_HV>();
  int nb = 0;
  if (allow_smem(kern, d->smem) &&
      cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, kern, NT6, d->smem) == cudaSuccess &&
      nb > 0) {
    d->grid = std::min(g.npairs, nb * hd->num_sms);
    d->ok = 1;
  } else {
    cudaGetLastError();
  }
  *out = d;
  return HS_OK;
}

}  // namespace sb6

// Superblock windows of k + 4 bits (16 slots of 256 rows per superblock: x
// slots and sums of a pair take 65 KB in FP32, two CTAs per SM) and at most
// L - 10 bits, so that a chain has at least 512 superblock pairs to spread
// over the GPU. HS_SB_KS32 and HS_SB_KS64 override the window (tuning).
// The defaults need the FP64 plans of ten bits (initial pass) and of six (pass A)
// only; the others are made here if the environment asks for their forms now (a
// capture then finds them), else at their first use (hs_create at L = 24 and 28: 5.8
// and 73.2 ms with all made here, 3.7 and 65.2 so).
hs_status sb_setup(hs_handle* hd) {
  hd->sb_on = true;
  hd->sb_ks[0] = std::min(hd->k + 4, hd->L - 10);
  hd->sb_ks[1] = std::min(hd->k + 3, hd->L - 10);
  if (const char* e = getenv("HS_SB_KS32")) hd->sb_ks[0] = atoi(e);
  if (const char* e = getenv("HS_SB_KS64")) hd->sb_ks[1] = atoi(e);
  // four-low-bit plans (sb4.cuh): 14-bit windows in FP32, 13 in FP64 (the
  // slots and sums of a pair take about 96 KB either way); HS_SB4_KS32 and
  // HS_SB4_KS64 override them (tests of small chains)
  hd->sb4_ks[0] = std::min(14, hd->L - 6);
  hd->sb4_ks[1] = std::min(13, hd->L - 6);
  if (const char* e = getenv("HS_SB4_KS32")) hd->sb4_ks[0] = atoi(e);
  if (const char* e = getenv("HS_SB4_KS64")) hd->sb4_ks[1] = atoi(e);
  sb::DevPlan* d = nullptr;
  hs_status st = sb::make_dev<double>(hd, hd->sb_ks[1], &d);
  hd->sb_ks[1] = -1;
  if (st != HS_OK) return st;
  hd->sb_plan[1] = d;
  // six-low-bit plan (sb6.cuh, FP64): 13-bit windows (the slots and sums of a
  // pair take 97 KB; 12 and 11 bits leave more whole-superblock bonds to global
  // memory, L = 28: 2084 -> 2811 -> 3682 us); HS_SB6_KS overrides it (tests of
  // small chains)
  int j64 = std::min(13, hd->L - 6);
  if (const char* e = getenv("HS_SB6_KS")) j64 = atoi(e);
  sb6::DevPlan6* d6 = nullptr;
  if ((st = sb6::make_dev6<double>(hd, j64, &d6)) != HS_OK) return st;
  hd->sb6_plan = d6;
  if (getenv("HS_HV_SB") || getenv("HS_SB4")) sb_ten(hd, 0);
  if (getenv("HS_SB4")) {
    sb_four(hd, 0);
    sb_four(hd, 1);
  }
  return HS_OK;
}

// Whether plans can be made now (not while the stream is being captured).
static bool can_make(hs_handle* hd) {
  cudaStreamCaptureStatus c = cudaStreamCaptureStatusNone;
  return cudaStreamIsCapturing(hd->stream, &c) == cudaSuccess && c == cudaStreamCaptureStatusNone;
}

void* sb_ten(hs_handle* hd, int ti) {
  if (!hd->sb_plan[ti] && hd->sb_ks[ti] >= 0 && can_make(hd)) {
    sb::DevPlan* d = nullptr;
    const hs_status st = ti ? sb::make_dev<double>(hd, hd->sb_ks[ti], &d)
                            : sb::make_dev<float>(hd, hd->sb_ks[ti], &d);
    if (st != HS_OK) hd->err.clear();   // no room: another form
    hd->sb_ks[ti] = -1;
    hd->sb_plan[ti] = d;
  }
  return hd->sb_plan[ti];
}

void* sb_four(hs_handle* hd, int ti) {
  if (!hd->sb4_plan[ti] && hd->sb4_ks[ti] >= 0 && can_make(hd)) {
    sb4::DevPlan4* d = nullptr;
    const hs_status st = ti ? sb4::make_dev4<double>(hd, hd->sb4_ks[ti], &d)
                            : sb4::make_dev4<float>(hd, hd->sb4_ks[ti], &d);
    if (st != HS_OK) hd->err.clear();
    hd->sb4_ks[ti] = -1;
    hd->sb4_plan[ti] = d;
  }
  return hd->sb4_plan[ti];
}

void sb_release(hs_handle* hd) {
  for (int i = 0; i < 2; ++i) {
    auto* d = static_cast<sb::DevPlan*>(hd->sb_plan[i]);
    if (d) {
      dev_free(hd, d->mem);
      delete d;
    }
    hd->sb_plan[i] = nullptr;
    auto* d4 = static_cast<sb4::DevPlan4*>(hd->sb4_plan[i]);
    if (d4) {
      dev_free(hd, d4->mem);
      delete d4;
    }
    hd->sb4_plan[i] = nullptr;
  }
  if (auto* d6 = static_cast<sb6::DevPlan6*>(hd->sb6_plan)) {
    dev_free(hd, d6->mem);
    delete d6;
  }
  hd->sb6_plan = nullptr;
}

}  // namespace hs

// The superblock form of MINRES pass A, and of products under HS_HV_SB=1: six low
// bits in FP64, whose additions bound every form (no zeros for parallel mid bonds,
// and the fewest instructions around them; a product at L = 24: 137 us, four bits
// 172; L = 28: 2.08 ms and 2.50); in FP32 0: the class form (hv_cls.cuh; L = 28:
// 257 us against 333 with ten bits, 344 with six, 392 with four), or ten bits
// where it does not apply. HS_SB4=1 / 0 selects four or ten bits for both (tests
// compare forms).
int hs_want_sb(hs_dtype dt) {
  const char* e = getenv("HS_SB4");
  if (e) return e[0] == '1' ? 4 : 10;
  return dt == HS_F64 ? 6 : 0;
}

namespace hs {

hs_status launch_matvec_sb(hs_handle* hd, const void* x, void* y, hs_dtype dt, int shifted,
                           bool* used) {
  *used = false;
  const int want = hs_want_sb(dt);
  {
    auto* d6 = static_cast<sb6::DevPlan6*>(hd->sb6_plan);
    if (want == 6 && d6 && d6->ok && ((uintptr_t)x % 8) == 0 && ((uintptr_t)y % 8) == 0) {
      const sb::MinresArgs none{};
      sb6::kernel6<double, sb::MODE_HV>()<<<d6->grid, sb6::NT6, d6->smem, hd->stream>>>(
          d6->geo, static_cast<const double*>(x), static_cast<double*>(y), hd->d_sigma, shifted,
          none);
      count_launches(1);
      HS_CUDA_TRY(hd, cudaGetLastError());
      *used = true;
      return HS_OK;
    }
  }
  {
    auto* d4 = static_cast<sb4::DevPlan4*>(want == 4 ? sb_four(hd, dt == HS_F32 ? 0 : 1) : nullptr);
    const size_t es = dt == HS_F32 ? sizeof(float) : sizeof(double);
    if (d4 && d4->ok && ((uintptr_t)x % es) == 0 && ((uintptr_t)y % es) == 0) {
      const sb::MinresArgs none{};
      if (dt == HS_F32)
        sb4::kernel4_for<float, sb::MODE_HV>(d4->geo.km)<<<d4->grid, sb4::NT4_F, d4->smem,
                                                            hd->stream>>>(
            d4->geo, static_cast<const float*>(x), static_cast<float*>(y), hd->d_sigma, shifted,
            none);
      else
        sb4::kernel4_for<double, sb::MODE_HV>(d4->geo.km)<<<d4->grid, sb4::NT4_D, d4->smem,
                                                             hd->stream>>>(
            d4->geo, static_cast<const double*>(x), static_cast<double*>(y), hd->d_sigma, shifted,
            none);
      count_launches(1);
      HS_CUDA_TRY(hd, cudaGetLastError());
      *used = true;
      return HS_OK;
    }
  }
  auto* d = static_cast<sb::DevPlan*>(sb_ten(hd, dt == HS_F32 ? 0 : 1));
  if (!d || !d->ok) return HS_OK;
  const size_t es = dt == HS_F32 ? sizeof(float) : sizeof(double);
  if (((uintptr_t)x % es) != 0 || ((uintptr_t)y % es) != 0) return HS_OK;
  const sb::MinresArgs none{};
  if (dt == HS_F32) {
    sb::kernel_of<float>(d->geo.km)<<<d->grid, sb::NT_SB, d->smem, hd->stream>>>(
        d->geo, static_cast<const float*>(x), static_cast<float*>(y), hd->d_sigma, shifted, none);
  } else {
    sb::kernel_of<double>(d->geo.km)<<<d->grid, sb::NT_SB, d->smem, hd->stream>>>(
        d->geo, static_cast<const double*>(x), static_cast<double*>(y), hd->d_sigma, shifted, none);
  }
  count_launches(1);
  HS_CUDA_TRY(hd, cudaGetLastError());
  *used = true;
  return HS_OK;
}

}  // namespace hs
