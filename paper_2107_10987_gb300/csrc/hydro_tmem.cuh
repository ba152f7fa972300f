// hydro_tmem.cuh -- tensor memory, where a row of the row sweep keeps its
// plus-states.
//
// The sweep carries the nine plus-states of its row, 90 floats a thread, from
// one cell to the next: too many for registers, and indexed by the loop over
// the points.  As a local array they went to L2 and back (two CTAs'
// 110 KB of primitives leave 26 KB of first-level cache, and 0.2 % of the reads
// hit): 40 % of the kernel's L2 traffic and a latency in every point.  Tensor
// memory (256 KB per SM, otherwise idle here) holds a 32-bit word
// per thread and column: a warp reads and writes the 32 lanes of its quarter
// (warp index mod 4), the column is a register.  4,096 sub-grids: 2.06 ->
// 1.84 ms.
//
// A CTA of 6 warps takes kTmemCols = 256 of the SM's 512 columns (180 are
// used: warps 0-3 the first 90, warps 4 and 5 the next), so that the two CTAs
// that share an SM both have theirs; no third fits beside their shared memory.
// The allocation waits where other work on the SM holds the columns, until
// that work's CTA ends; a CTA of these kernels holds its own from start to end
// and waits at most for CTAs that hold theirs.
#pragma once
#include "hydro_common.cuh"

namespace hyd {

constexpr int kTmemCols = 256;
constexpr int kTmemThread = 90;  // columns of a thread: nine records of F floats
static_assert(9 * F <= kTmemThread && 2 * kTmemThread <= kTmemCols, "two warps to a quarter of the lanes");

// Start of a CTA (all threads; sh: a word of shared memory): the thread's first
// column, in its warp's lanes.
__device__ __forceinline__ uint32_t tmem_alloc(uint32_t* sh) {
  if (threadIdx.x < 32) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                     (uint32_t)__cvta_generic_to_shared(sh)),
                 "n"(kTmemCols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  return *(volatile uint32_t*)sh + ((threadIdx.x & 96u) << 16) + (threadIdx.x >> 7) * kTmemThread;
}

// End of the CTA (all threads), t: what tmem_alloc returned.  The fences order
// every thread's accesses before the barrier and the deallocation after it.
__device__ __forceinline__ void tmem_free(uint32_t t) {
  __syncwarp();
  asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  if (threadIdx.x < 32) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(t), "n"(kTmemCols));
}

// Record r of this thread; next: the stores so far are visible to the reads that
// follow.  The warp's threads call together: each access is one instruction of
// the whole warp, so each reconverges it first (the row sweep branches per
// thread before them: the smooth cells' lines, the contact test, the spin's cap,
// conversions outside FP32's normal range).
struct RowPlusTmem {
  uint32_t t;  // tmem_alloc's
  __device__ __forceinline__ void next() {
    __syncwarp();
    asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
  }
  struct Rec {
    float q[F];
    __device__ __forceinline__ operator const float*() const { return q; }
  };
  __device__ __forceinline__ Rec record(int r) const {
    static_assert(F == 10, "a record is 8 + 2 columns");
    Rec v;
    float* q = v.q;
    __syncwarp();
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%10];\n\t"
        "tcgen05.ld.sync.aligned.32x32b.x2.b32 {%8, %9}, [%11];\n\t"
        "tcgen05.wait::ld.sync.aligned;"
        : "=f"(q[0]), "=f"(q[1]), "=f"(q[2]), "=f"(q[3]), "=f"(q[4]), "=f"(q[5]), "=f"(q[6]), "=f"(q[7]),
          "=f"(q[8]), "=f"(q[9])
        : "r"(t + F * r), "r"(t + F * r + 8)
        : "memory");
    return v;
  }
  __device__ __forceinline__ void store(int r, const float q[F]) {
    __syncwarp();
    asm volatile(
        "tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%2, %3, %4, %5, %6, %7, %8, %9};\n\t"
        "tcgen05.st.sync.aligned.32x32b.x2.b32 [%1], {%10, %11};" ::"r"(t + F * r),
        "r"(t + F * r + 8), "f"(q[0]), "f"(q[1]), "f"(q[2]), "f"(q[3]), "f"(q[4]), "f"(q[5]), "f"(q[6]), "f"(q[7]),
        "f"(q[8]), "f"(q[9])
        : "memory");
  }
};
}  // namespace hyd
