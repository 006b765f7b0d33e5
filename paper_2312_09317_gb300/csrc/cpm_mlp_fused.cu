// The forward pass of the emulator network, all layers of all members in one kernel, on the
// fifth-generation tensor cores.
//
// A CTA takes (member, 128-row tile) items.  The activations of a tile never leave the SM: a layer's
// accumulator (128 x width, FP32) lies in tensor memory, its epilogue writes GELU(acc + b), rounded to
// bf16, over the layer's input in shared memory, and the next layer reads it there.  Three roles:
//   loader (one thread)  the weights, packed as the MMAs read them, by bulk copies into a ring of
//                        two stages, a 32-deep K slab of a layer each;
//   issuer (one warp)    a layer's MMAs, slab by slab, once its input is written;
//   epilogue (8 warps)   warp w reads tensor-memory lanes 32 (w % 4) .. and every other 32 columns; it also
//                        converts an item's inputs to bf16.
// Two CTAs share an SM (100 KB of shared memory, half the tensor memory each), so that one's MMAs, copies
// and waits run behind the other's epilogue.  Every element is summed over K in the order of the
// layer-by-layer kernel (ascending, 16 at a time): the same bits.
//
// What bounds it: the instructions of the epilogue (about 18 issue slots per 32 outputs, 55% of all slots
// used) and, beside them, the ring: a hidden layer's MMAs take 5,300 cycles, of which 2,200 are the MMAs.
// 65,536 rows of 5 members of 7-256x4-16: 312 us; with a launch per layer, whose activations go through HBM,
// 700 us.  One CTA per SM with 16 epilogue warps that the next layer's MMAs follow in chunks of 64 or 128
// columns: 338 and 326 us.
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <cstdint>

#include "cpm_mlp_internal.h"
#include "cpm_mlp_tc.cuh"

namespace cpmmlp {
namespace {

constexpr int kStages = 2;
constexpr int kEpiWarps = 8, kThreads = (kEpiWarps + 2) * 32;

struct FusedArgs {
    FusedNet net;
    const float *X;
    int64_t rows;
    float *out;
    int64_t s_member;
    int *err;
    int report_timeout;
    int k0p;              // inputs padded to a multiple of 16
    int64_t member_bytes; // packed weights per member
    int mtiles, items;
};

struct Barriers {
    uint64_t wfull[kStages], wempty[kStages];
    uint64_t hready, dfull;  // a hidden layer: output written (the next input), accumulator complete
    uint64_t ofull, oread;   // the outputs: accumulator complete, read out
    uint64_t xready;         // the item's inputs written
    uint64_t drain;
    volatile int abort;      // a wait ran out: every role leaves its loop
};

__global__ void __launch_bounds__(kThreads, 2) fused_forward_kernel(const FusedArgs p)
{
    extern __shared__ __align__(1024) unsigned char fused_smem[];
    __shared__ __align__(8) Barriers bars;
    __shared__ uint32_t tmem_slot;
    const int width = p.net.width, slabs = width / kSlab, n_hidden = p.net.n_hidden, n_out = p.net.n_out;
    unsigned char *Ws = fused_smem;                                  // kStages stages
    unsigned char *As = Ws + kStages * kStageBytes;                  // 128 x width
    unsigned char *Xs = As + kRows * width * 2;                      // 128 x k0p
    float *bias_s = reinterpret_cast<float *>(Xs + kRows * p.k0p * 2);  // two items' biases, layer after layer
    const int n_bias = n_hidden * width + n_out;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 256;" ::"r"(smem_u32(&tmem_slot))
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    if (threadIdx.x == 0) {
        for (int k = 0; k < kStages; ++k) {
            bar_init(&bars.wfull[k], 1);
            bar_init(&bars.wempty[k], 1);
        }
        bar_init(&bars.hready, kEpiWarps);
        bar_init(&bars.dfull, 1);
        bar_init(&bars.ofull, 1);
        bar_init(&bars.oread, kEpiWarps);
        bar_init(&bars.xready, kEpiWarps);
        bar_init(&bars.drain, 1);
        bars.abort = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem = __shfl_sync(0xffffffffu, tmem_slot, 0);
    const int i0 = (int)((int64_t)p.items * blockIdx.x / gridDim.x);
    const int i1 = (int)((int64_t)p.items * (blockIdx.x + 1) / gridDim.x);

    if (warp == 1) {
        // ---- loader
        if (lane == 0) {
            uint32_t stage = 0, parity = 1;  // of the stage's last use; 1: none yet
            uint32_t n_slab = 0;
            const auto load = [&](const unsigned char *src, int bytes) {
                if (n_slab >= kStages && !bar_wait(bars, &bars.wempty[stage], parity)) return false;
                const uint32_t full = smem_u32(&bars.wfull[stage]);
                asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(full), "r"(bytes) : "memory");
                asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                                 smem_u32(Ws + stage * kStageBytes)),
                             "l"(src), "r"(bytes), "r"(full)
                             : "memory");
                ++n_slab;
                if (++stage == kStages) {
                    stage = 0;
                    parity ^= 1u;
                }
                return true;
            };
            bool ok = true;
            for (int i = i0; i < i1 && ok; ++i) {
                const unsigned char *src = p.net.packed + i / p.mtiles * p.member_bytes;
                ok = load(src, first_bytes(p.k0p, width));
                src += first_bytes(p.k0p, width);
                for (int k = 0; k < (n_hidden - 1) * slabs && ok; ++k, src += slab_bytes(width))
                    ok = load(src, slab_bytes(width));
                if (ok) ok = load(src, last_bytes(width, n_out));
            }
            // (after an abort) the copies in flight land before the CTA's shared memory is given up
            for (uint32_t k = n_slab > kStages ? n_slab - kStages : 0; k < n_slab; ++k)
                tc_wait(&bars.wfull[k % kStages], (k / kStages) & 1u);
        }
        __syncwarp();
    } else if (warp == 0) {
        // ---- issuer
        uint32_t n_h = 0;                // hidden epilogues waited for
        uint32_t stage = 0, parity = 0;  // of the next slab
        // matrix descriptors: the address, in 16-byte units, is their low field
        const uint64_t da = tc_desc(smem_u32(As), 128u, (uint32_t)(width / 8) * 128u);
        const uint64_t dx = tc_desc(smem_u32(Xs), 128u, (uint32_t)(p.k0p / 8) * 128u);
        const uint64_t dw = tc_desc(smem_u32(Ws), 128u, (uint32_t)(kSlab / 8) * 128u);
        const uint64_t dw_x = tc_desc(smem_u32(Ws), 128u, (uint32_t)(p.k0p / 8) * 128u);
        const uint32_t idesc = tc_idesc(width), idesc_out = tc_idesc(n_out);
        const auto slab = [&]() { return warp_wait(bars, &bars.wfull[stage], parity); };
        const auto at = [&](uint64_t d) { return d + stage * (kStageBytes / 16); };
        const auto slab_done = [&]() {
            tc_commit(&bars.wempty[stage]);
            if (++stage == kStages) {
                stage = 0;
                parity ^= 1u;
            }
        };
        bool ok = true;
        for (int i = i0; i < i1 && ok; ++i) {
            ok = slab() && warp_wait(bars, &bars.xready, (uint32_t)(i - i0) & 1u);
            if (ok && i > i0) ok = warp_wait(bars, &bars.oread, (uint32_t)(i - i0 - 1) & 1u);
            if (!ok) break;
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            for (int ks = 0; ks < p.k0p / 16; ++ks) tc_mma(tmem, dx + ks * 16, at(dw_x) + ks * 16, idesc, ks > 0);
            slab_done();
            tc_commit(&bars.dfull);
            for (int l = 1; l <= n_hidden && ok; ++l, ++n_h) {
                ok = slab() && warp_wait(bars, &bars.hready, n_h & 1u);
                if (!ok) break;
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                if (l < n_hidden) {
                    uint64_t d = da;
                    for (int kc = 0; kc < slabs; ++kc) {
                        if (kc > 0) ok = slab();
                        if (!ok) break;
#pragma unroll
                        for (int ks = 0; ks < kSlab / 16; ++ks, d += 16)
                            tc_mma(tmem, d, at(dw) + ks * 16, idesc, kc + ks > 0);
                        slab_done();
                    }
                    if (ok) tc_commit(&bars.dfull);
                } else {
                    // the outputs: every slab of K from one stage
                    for (int kc = 0; kc < slabs; ++kc)
#pragma unroll
                        for (int ks = 0; ks < kSlab / 16; ++ks)
                            tc_mma(tmem, da + kc * 32 + ks * 16, at(dw) + kc * (n_out * 4) + ks * 16, idesc_out, kc + ks > 0);
                    slab_done();
                    tc_commit(&bars.ofull);
                }
            }
        }
        if (!ok) {
            // the MMAs issued so far end before tensor memory is given up
            tc_commit(&bars.drain);
            tc_wait(&bars.drain, 0);
        }
    } else {
        // ---- epilogue
        const int q = warp & 3, part = (warp - 2) >> 2, tid = threadIdx.x - 64, r = q * 32 + lane;
        const uint32_t lanes = tmem + ((uint32_t)(q * 32) << 16);
        unsigned char *arow = As + (size_t)(r >> 3) * (width / 8) * 128 + (r & 7) * 16;
        uint32_t n_d = 0;  // hidden layers done
        bool ok = true;
        for (int i = i0; i < i1 && ok; ++i) {
            const int e = i / p.mtiles;
            const int64_t row = (int64_t)(i % p.mtiles) * kRows + r;
            // the member's biases, into the half that the item before the last used (this warp is past the xready
            // of the last item, so every warp is past the one before); the inputs: the last item's were read before
            // its first hidden layer came through
            float *bias = bias_s + ((i - i0) & 1) * n_bias;
            const float *w = p.net.w + e * p.net.P;
            for (int g = tid; g < n_bias; g += kEpiWarps * 32) {
                const int l = g / width, k = g - l * width;  // b_l follows W_l
                bias[g] = __ldg(w + (int64_t)p.net.n_in * width + (l > 0 ? width : 0) +
                                (l > 1 ? (int64_t)(l - 1) * width : 0) +
                                (l < n_hidden ? (int64_t)l * width * width
                                              : (int64_t)(n_hidden - 1) * width * width + (int64_t)n_out * width) + k);
            }
            const int kc = p.k0p / 8, n_in = p.net.n_in;
            for (int g = tid; g < kRows * kc; g += kEpiWarps * 32) {
                const int rr = g & 7, k8 = (g >> 3) % kc, r8 = (g >> 3) / kc;
                const int64_t xrow = (int64_t)(i % p.mtiles) * kRows + r8 * 8 + rr;
                __align__(16) __nv_bfloat16 h[8];
#pragma unroll
                for (int j = 0; j < 8; ++j) {
                    const int k = k8 * 8 + j;
                    h[j] = __float2bfloat16(xrow < p.rows && k < n_in ? p.X[xrow * n_in + k] : 0.0f);
                }
                *reinterpret_cast<uint4 *>(Xs + (size_t)g * 16) = *reinterpret_cast<const uint4 *>(h);
            }
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            __syncwarp();
            if (lane == 0) bar_arrive(&bars.xready);
            ok = warp_wait(bars, &bars.xready, (uint32_t)(i - i0) & 1u);
            for (int l = 0; l < n_hidden && ok; ++l, ++n_d) {
                ok = warp_wait(bars, &bars.dfull, n_d & 1u);
                if (ok && p.report_timeout) {  // as if this wait had run out, once it has completed
                    bars.abort = 1;
                    ok = false;
                }
                if (!ok) break;
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                // sixteen columns at a time, the next ones on their way while these are worked on
                uint32_t v[2][16];
                tc_load16(v[0], lanes + (uint32_t)(part * 32));
                for (int n0 = part * 32; n0 < width; n0 += 64) {
#pragma unroll
                    for (int half = 0; half < 2; ++half) {
                        float4 bv[4];
#pragma unroll
                        for (int j = 0; j < 4; ++j)
                            bv[j] = reinterpret_cast<const float4 *>(bias + n0 + 16 * half)[j];
                        tc_loaded(v[half]);
                        if (half == 0) tc_load16(v[1], lanes + (uint32_t)(n0 + 16));
                        else if (n0 + 64 < width) tc_load16(v[0], lanes + (uint32_t)(n0 + 64));
                        __align__(16) __nv_bfloat162 h[8];
                        uint64_t z[8];
                        float zmax = 0.0f;
#pragma unroll
                        for (int j = 0; j < 8; ++j) {
                            z[j] = add2(pack2(__uint_as_float(v[half][2 * j]), __uint_as_float(v[half][2 * j + 1])),
                                        j % 2 == 0 ? pack2(bv[j / 2].x, bv[j / 2].y) : pack2(bv[j / 2].z, bv[j / 2].w));
                            const float2 zj = unpack2(z[j]);
                            zmax = fmaxf(zmax, fmaxf(fabsf(zj.x), fabsf(zj.y)));
                            const float2 g = unpack2(gelu2_f(z[j]));
                            h[j] = __floats2bfloat162_rn(g.x, g.y);
                        }
                        if (!(zmax <= kGelu2Max)) {  // (a NaN is ignored by fmaxf and propagates through either form)
#pragma unroll
                            for (int j = 0; j < 8; ++j) {
                                const float2 zj = unpack2(z[j]);
                                h[j] = __floats2bfloat162_rn(gelu_f(zj.x), gelu_f(zj.y));
                            }
                        }
                        unsigned char *o = arow + (n0 / 8 + 2 * half) * 128;
                        *reinterpret_cast<uint4 *>(o) = reinterpret_cast<const uint4 *>(h)[0];
                        *reinterpret_cast<uint4 *>(o + 128) = reinterpret_cast<const uint4 *>(h)[1];
                    }
                }
                asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
                __syncwarp();
                if (lane == 0) bar_arrive(&bars.hready);
                bias += width;
            }
            if (!ok) break;
            // outputs
            ok = warp_wait(bars, &bars.ofull, (uint32_t)(i - i0) & 1u);
            if (!ok) break;
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            const int n0 = part * 16;
            if (n0 < n_out) {
                uint32_t v[16];
                tc_load16(v, lanes + (uint32_t)n0);
                tc_loaded(v);
                if (row < p.rows) {
                    float *o = p.out + e * p.s_member + row * n_out + n0;
#pragma unroll
                    for (int j = 0; j < 16; ++j) o[j] = __uint_as_float(v[j]) + bias[n0 + j];
                }
            }
            asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
            __syncwarp();
            if (lane == 0) bar_arrive(&bars.oread);
        }
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (threadIdx.x == 0 && bars.abort && p.err) atomicExch(p.err, 1);
    if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 256;" ::"r"(tmem) : "memory");
}

// One 16-byte piece of a packed layer per thread: 8 consecutive inputs of one output, in the canonical
// no-swizzle K-major layout (8 x 16-byte core matrices, K-adjacent ones 128 bytes apart).
__global__ void fused_pack_kernel(const FusedNet n, const __nv_bfloat16 *wb, unsigned char *packed, int k0p,
                                  int64_t member_bytes)
{
    const int slabs = n.width / kSlab;
    const int64_t pieces = member_bytes / 16;
    for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < pieces * n.n_members;
         t += (int64_t)gridDim.x * blockDim.x) {
        const int e = (int)(t / pieces);
        int64_t at = (t % pieces) * 16;
        const __nv_bfloat16 *W = wb + e * n.P;
        int K = n.n_in, kc = k0p / 8, k_first = 0;  // of the packed block: the layer's inputs, 8-wide columns, first input
        if (at >= first_bytes(k0p, n.width)) {
            at -= first_bytes(k0p, n.width);
            W += (int64_t)n.n_in * n.width + n.width;
            K = n.width;
            const int64_t layer = (int64_t)slabs * slab_bytes(n.width);
            if (at < layer * (n.n_hidden - 1)) {
                W += at / layer * ((int64_t)n.width * n.width + n.width);
                at %= layer;
                k_first = (int)(at / slab_bytes(n.width)) * kSlab;
                at %= slab_bytes(n.width);
            } else {
                at -= layer * (n.n_hidden - 1);
                W += (int64_t)(n.n_hidden - 1) * ((int64_t)n.width * n.width + n.width);
                k_first = (int)(at / slab_bytes(n.n_out)) * kSlab;
                at %= slab_bytes(n.n_out);
            }
            kc = kSlab / 8;
        }
        const int q = (int)(at / 16), rr = q & 7, k8 = (q >> 3) % kc, r8 = (q >> 3) / kc;
        const __nv_bfloat16 *src = W + (int64_t)(r8 * 8 + rr) * K + k_first + k8 * 8;
        __align__(16) __nv_bfloat16 h[8];
#pragma unroll
        for (int j = 0; j < 8; ++j) h[j] = k_first + k8 * 8 + j < K ? src[j] : __float2bfloat16(0.0f);
        *reinterpret_cast<uint4 *>(packed + t * 16) = *reinterpret_cast<const uint4 *>(h);
    }
}

}  // namespace

bool fused_fits(int n_in, int width, int n_out)
{
    return n_in <= 32 && width % 64 == 0 && width <= 256 && n_out % 16 == 0 && n_out <= 32;
}

int64_t fused_packed_bytes(int n_in, int width, int n_hidden, int n_out)
{
    return first_bytes(padded_inputs(n_in), width) + (int64_t)(n_hidden - 1) * (width / kSlab) * slab_bytes(width) +
           last_bytes(width, n_out);
}

cudaError_t fused_pack(const FusedNet &n, const __nv_bfloat16 *wb, unsigned char *packed, cudaStream_t st)
{
    const int64_t bytes = fused_packed_bytes(n.n_in, n.width, n.n_hidden, n.n_out);
    const int64_t blocks = (bytes / 16 * n.n_members + 255) / 256;
    fused_pack_kernel<<<(unsigned)(blocks < 2432 ? blocks : 2432), 256, 0, st>>>(n, wb, packed, padded_inputs(n.n_in),
                                                                                bytes);
    return cudaPeekAtLastError();
}

cudaError_t fused_forward(const FusedNet &n, const float *X, int64_t rows, float *out, int64_t s_member, int *err,
                          int report_timeout, cudaStream_t st)
{
    if (rows <= 0) return cudaSuccess;
    FusedArgs p{};
    p.net = n;
    p.X = X;
    p.rows = rows;
    p.out = out;
    p.s_member = s_member;
    p.err = err;
    p.report_timeout = report_timeout;
    p.k0p = padded_inputs(n.n_in);
    p.member_bytes = fused_packed_bytes(n.n_in, n.width, n.n_hidden, n.n_out);
    p.mtiles = (int)((rows + kRows - 1) / kRows);
    p.items = p.mtiles * n.n_members;
    const int smem = kStages * kStageBytes + kRows * n.width * 2 + kRows * p.k0p * 2 +
                     2 * 4 * (n.n_hidden * n.width + n.n_out);
    int dev = 0, sms = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(fused_forward_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                      200 * 1024);
    if (e != cudaSuccess) return e;
    fused_forward_kernel<<<p.items < 2 * sms ? p.items : 2 * sms, kThreads, smem, st>>>(p);
    return cudaPeekAtLastError();
}

}  // namespace cpmmlp
