// tcgen05 and mbarrier pieces shared by the emulator network's fused kernels.
#ifndef CPM_MLP_TC_CUH
#define CPM_MLP_TC_CUH

#include <cuda_runtime.h>

#include <cstdint>

#include "cpm_mlp_internal.h"

namespace cpmmlp {

constexpr int kRows = 128, kSlab = 32;  // M of an MMA; K of a packed slab
constexpr int kStageBytes = 16 * 1024;  // of the weight rings: a slab of 256 rows, or a first or last layer

__device__ __forceinline__ void bar_init(uint64_t *b, uint32_t count)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(b)), "r"(count) : "memory");
}
__device__ __forceinline__ void bar_arrive(uint64_t *b)
{
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(b)) : "memory");
}
// programmatic dependent launch: the launches before this one are done; the next one may start
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void pdl_next() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
template <typename K, typename A>
cudaError_t pdl_launch(K kernel, const A &args, int grid, int threads, int smem, bool chained, cudaStream_t st)
{
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t c{};
    c.gridDim = dim3((unsigned)grid);
    c.blockDim = dim3((unsigned)threads);
    c.dynamicSmemBytes = (size_t)smem;
    c.stream = st;
    c.attrs = &at;
    c.numAttrs = chained ? 1 : 0;
    return cudaLaunchKernelEx(&c, kernel, args);
}

// whether the phase `parity` of b is over, without waiting
__device__ __forceinline__ bool bar_over(uint64_t *b, uint32_t parity)
{
    uint32_t done;
    asm volatile("{\n .reg .pred p;\n mbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n"
                 " selp.u32 %0, 1, 0, p;\n}"
                 : "=r"(done)
                 : "r"(smem_u32(b)), "r"(parity)
                 : "memory");
    return done != 0;
}
// s.abort: set once a wait of the CTA ran out
// bounded wait for the phase `parity` of b; false once a wait of the CTA ran out (this one or another)
template <typename Barriers>
__device__ __forceinline__ bool bar_wait(Barriers &s, uint64_t *b, uint32_t parity)
{
    const uint32_t addr = smem_u32(b);
    for (uint32_t it = 0; it < kTcSpinLimit; ++it) {
        uint32_t done;
        asm volatile("{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n"
                     " selp.u32 %0, 1, 0, p;\n}"
                     : "=r"(done)
                     : "r"(addr), "r"(parity)
                     : "memory");
        if (done) return true;
        if (s.abort) return false;
    }
    s.abort = 1;
    return false;
}
// Issued by a whole warp, for one elected thread of it: the operands are then known to be uniform.  (An MMA of
// 128 x 48 x 16 issues every 46 cycles so, every 56 from one thread's branch, and every 100 from a loop that is
// not unrolled.)
__device__ __forceinline__ void tc_commit(uint64_t *b)
{
    asm volatile("{\n .reg .pred one;\n elect.sync _|one, 0xffffffff;\n"
                 " @one tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n}" ::"r"(smem_u32(b))
                 : "memory");
}
__device__ __forceinline__ void tc_mma(uint32_t d, uint64_t ad, uint64_t bd, uint32_t idesc, bool accumulate)
{
    asm volatile("{\n .reg .pred acc, one;\n setp.ne.b32 acc, %4, 0;\n elect.sync _|one, 0xffffffff;\n"
                 " @one tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, acc;\n}" ::"r"(d),
                 "l"(ad), "l"(bd), "r"(idesc), "r"(accumulate ? 1 : 0)
                 : "memory");
}
__device__ __forceinline__ uint32_t tc_idesc(int n)
{
    return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(n >> 3) << 17) | ((uint32_t)(kRows >> 4) << 24);
}

// the same for a whole warp, which stays together whichever way it goes
template <typename Barriers>
__device__ __forceinline__ bool warp_wait(Barriers &s, uint64_t *b, uint32_t parity)
{
    return __all_sync(0xffffffffu, bar_wait(s, b, parity));
}

// the accumulator's 16 columns from `addr` of this warp's 32 lanes; complete after tcgen05.wait::ld
__device__ __forceinline__ void tc_load16(uint32_t (&v)[16], uint32_t addr)
{
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, "
                 "%14, %15}, [%16];"
                 : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]),
                   "=r"(v[8]), "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15])
                 : "r"(addr)
                 : "memory");
}
// and 8
__device__ __forceinline__ void tc_load8(uint32_t (&v)[8], uint32_t addr)
{
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                 : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7])
                 : "r"(addr)
                 : "memory");
}
// the loads of v have landed (v is an operand, so that no use of it moves before the wait)
__device__ __forceinline__ void tc_loaded(uint32_t (&v)[8])
{
    asm volatile("tcgen05.wait::ld.sync.aligned;"
                 : "+r"(v[0]), "+r"(v[1]), "+r"(v[2]), "+r"(v[3]), "+r"(v[4]), "+r"(v[5]), "+r"(v[6]), "+r"(v[7])
                 :
                 : "memory");
}
template <int N>
__device__ __forceinline__ void tc_loaded(uint32_t (&v)[N])
{
#pragma unroll
    for (int j = 0; j < N; j += 16)
        asm volatile("tcgen05.wait::ld.sync.aligned;"
                     : "+r"(v[j]), "+r"(v[j + 1]), "+r"(v[j + 2]), "+r"(v[j + 3]), "+r"(v[j + 4]), "+r"(v[j + 5]),
                       "+r"(v[j + 6]), "+r"(v[j + 7]), "+r"(v[j + 8]), "+r"(v[j + 9]), "+r"(v[j + 10]), "+r"(v[j + 11]),
                       "+r"(v[j + 12]), "+r"(v[j + 13]), "+r"(v[j + 14]), "+r"(v[j + 15])
                     :
                     : "memory");
}
// bytes of the packed weights: layer 0, a slab of a hidden layer, the last layer (slabs too)
__host__ __device__ __forceinline__ int first_bytes(int k0p, int width) { return width * k0p * 2; }
__host__ __device__ __forceinline__ int slab_bytes(int width) { return width * kSlab * 2; }
__host__ __device__ __forceinline__ int last_bytes(int width, int n_out) { return n_out * width * 2; }

}  // namespace cpmmlp

#endif
