// Pieces shared by the row forms of MINRES (minres_row.cu: two reductions per
// iteration; minres_row1.cu: one): the arguments, the bounded wait on a barrier of
// the CTA, the dealing of a CTA's rows to its threads.
#pragma once
#include "minres_clu.cuh"

namespace hs {

constexpr int ROW_BATCH = 16;                   // neighbour loads in flight per thread

struct RowArgs {
  SmemJob job;
  GridWord* slots;               // GRID_WORDS G words per exchange
  int* err;
  unsigned long long limit;
  void* q;                       // gather vectors, n elements each
  void* w0;
  void* w1;
};

// Wait for a barrier of this CTA (whole warps); false in every lane once a warp has
// set fail.
__device__ __forceinline__ bool row_wait(int& fail, unsigned long long* b, unsigned parity) {
  const uint32_t a = smem_u32(b);
  for (unsigned it = 0; it != CLU_WAIT_LIMIT; ++it) {
    uint32_t done;
    asm volatile("{\n.reg .pred p;\n"
                 "mbarrier.try_wait.parity.acquire.cta.shared::cta.b64 p, [%1], %2;\n"
                 "selp.u32 %0, 1, 0, p;\n}"
                 : "=r"(done) : "r"(a), "r"(parity) : "memory");
    if (__all_sync(0xffffffffu, done)) return true;
    if ((it & 15u) == 15u && __any_sync(0xffffffffu, *(volatile int*)&fail)) return false;
  }
  return false;
}

// A wait of this warp gave up: the CTA's other warps stop waiting, and the host
// reports HS_TIMEOUT whatever the state says (grid_finish): its writer may have
// been past its own last wait.
__device__ __forceinline__ void row_fail(int& fail, int* err) {
  fail = 1;
  if ((threadIdx.x & 31) == 0) atomicExch(err, 1);
}

// Deals rows r0 .. r0 + rows - 1 (all threads): order = their places sorted by
// falling number of neighbours; s_blk = their first and last block.
template <typename T>
__device__ __forceinline__ void row_deal(const Geo& g, int r0, int rows, uint16_t* order,
                                         uint8_t* bonds, int* s_blk, int* s_class) {
  const int lane = threadIdx.x & 31;
  if (threadIdx.x < 2 && rows > 0)
    s_blk[threadIdx.x] = clu_block(g, (uint32_t)(r0 + (threadIdx.x ? rows - 1 : 0)), 0, g.nblocks - 1);
  __syncthreads();
  // deal the rows: a stable counting sort by number of neighbours (even, 2..L)
  for (int r = threadIdx.x; r < rows; r += blockDim.x) {
    T am;
    int naf;
    clu_row<T>(g, (uint32_t)(r0 + r), s_blk[0], s_blk[1], 0.0, am, naf, [](uint32_t) {});
    bonds[r] = (uint8_t)naf;
  }
  __syncthreads();
  // warp c takes the rows with L - 2 c neighbours: how many, then where
  for (int pass = 0; pass < 2; ++pass) {
    const int c = threadIdx.x >> 5;
    if (c < g.L / 2) {
      int at = 0;
      if (pass)
        for (int d = 0; d < c; ++d) at += s_class[d];
      for (int b = 0; b < rows; b += 32) {
        const bool is = b + lane < rows && bonds[b + lane] == g.L - 2 * c;
        const unsigned m = __ballot_sync(0xffffffffu, is);
        if (pass && is) order[at + __popc(m & ((1u << lane) - 1u))] = (uint16_t)(b + lane);
        at += __popc(m);
      }
      if (!pass && lane == 0) s_class[c] = at;
    }
    __syncthreads();
  }
}

// Host side (minres_row.cu): the arguments of a solve on the handle's SMs with
// its exchange words cleared; a cooperative launch (HS_CUDA without a message
// when it does not fit or is refused; fixed: static shared memory).
hs_status row_args(hs_handle* hd, const void* b, const MinresVecs& v, double tol, long long kmax,
                   int exchanges, RowArgs* ra, int* G);
hs_status row_launch(hs_handle* hd, const void* kern, int G, int nt, size_t smem, size_t fixed,
                     void** args);

}  // namespace hs
