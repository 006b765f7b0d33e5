// The forward pass of the emulator network, all layers of all members in one kernel, on the
// fifth-generation tensor cores.
//
// A CTA, one per SM, takes (member, 128-row tile) items, two at a time.  The activations of a tile never
// leave the SM: a layer's accumulator (128 x width, FP32) lies in tensor memory, its epilogue writes
// GELU(acc + b), rounded to bf16, over the layer's input in shared memory, and the next layer reads it there.
// Three roles:
//   loader (one thread)  the weights, packed as the MMAs read them, by bulk copies into a ring of up to
//                        four stages, a 32-deep K slab of a layer each;
//   issuer (one warp)    a layer's MMAs, slab by slab, once its input is written: one tile's, then the
//                        other's;
//   epilogue (8 warps a tile)  a warp reads tensor-memory lanes 32 (warp % 4) .. and every other 16 columns;
//                        it also converts an item's inputs to bf16.
// The two tiles are a phase apart: one's MMAs run behind the other's epilogue.  Every element is summed over K
// in the order of the layer-by-layer kernel (ascending, 16 at a time): the same bits.
//
// What bounds it: the epilogue, 26 instructions for a pair of outputs of which the four to the special-function
// units take 32 of a scheduler's cycles, 8,200 a layer of two tiles; and the 3,500 of a tile's MMAs, which read
// 74% of what shared memory gives, as far as the other tile's epilogue does not cover them: 13,200 together.
// A prediction of 65,536 rows by 5 members of 7-256x4-16, with mean and deviation: 286 us.  Two CTAs on an SM, a
// tile and 32 KB of ring each, so that a slab's copy (1,200 cycles) was waited for: 330.  A launch per layer,
// whose activations go through HBM: 765.  Tried beside it: 12 and 16 epilogue warps a tile (336, 347), stages of
// 32 KB, slabs asked for ahead (no change).
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <cstdint>

#include "cpm_mlp_internal.h"
#include "cpm_mlp_tc.cuh"

namespace cpmmlp {
namespace {

constexpr int kMaxStages = 4, kTiles = 2;  // stages of the ring; tiles of a CTA
constexpr int kFusedSmem = 224 * 1024;             // of a CTA, at most
constexpr int kEpiWarps = 8, kThreads = (kTiles * kEpiWarps + 2) * 32;  // epilogue warps of a tile

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
    int mtiles, items, stages;
};

struct Barriers {
    uint64_t wfull[kMaxStages], wempty[kMaxStages];
    // of each tile
    uint64_t hready[kTiles], dfull[kTiles];  // a hidden layer: output written (the next input), accumulator complete
    uint64_t ofull[kTiles], oread[kTiles];   // the outputs: accumulator complete, read out
    uint64_t xready[kTiles];                 // the item's inputs written
    uint64_t drain;
    volatile int abort;                      // a wait ran out: every role leaves its loop
};

__global__ void __launch_bounds__(kThreads, 1) fused_forward_kernel(const FusedArgs p)
{
    extern __shared__ __align__(1024) unsigned char fused_smem[];
    __shared__ __align__(8) Barriers bars;
    __shared__ uint32_t tmem_slot;
    const int width = p.net.width, slabs = width / kSlab, n_hidden = p.net.n_hidden, n_out = p.net.n_out;
    const int n_bias = n_hidden * width + n_out, stages = p.stages;
    const int a_bytes = kRows * width * 2, x_bytes = kRows * p.k0p * 2;
    unsigned char *Ws = fused_smem;                 // the ring
    unsigned char *As = Ws + stages * kStageBytes;  // a tile's 128 x width
    unsigned char *Xs = As + kTiles * a_bytes;      // a tile's 128 x k0p
    float *bias_s = reinterpret_cast<float *>(Xs + kTiles * x_bytes);  // a tile's biases, layer after layer
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 512;" ::"r"(smem_u32(&tmem_slot))
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    if (threadIdx.x == 0) {
        for (int k = 0; k < stages; ++k) {
            bar_init(&bars.wfull[k], 1);
            bar_init(&bars.wempty[k], 1);
        }
        for (int c = 0; c < kTiles; ++c) {
            bar_init(&bars.hready[c], kEpiWarps);
            bar_init(&bars.dfull[c], 1);
            bar_init(&bars.ofull[c], 1);
            bar_init(&bars.oread[c], kEpiWarps);
            bar_init(&bars.xready[c], kEpiWarps);
        }
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
                if (n_slab >= (uint32_t)stages && !bar_wait(bars, &bars.wempty[stage], parity)) return false;
                const uint32_t full = smem_u32(&bars.wfull[stage]);
                asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(full), "r"(bytes) : "memory");
                asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                                 smem_u32(Ws + stage * kStageBytes)),
                             "l"(src), "r"(bytes), "r"(full)
                             : "memory");
                ++n_slab;
                if (++stage == (uint32_t)stages) {
                    stage = 0;
                    parity ^= 1u;
                }
                return true;
            };
            bool ok = true;
            for (int i = i0; i < i1 && ok; i += kTiles) {
                const int tiles = i1 - i < kTiles ? i1 - i : kTiles;
                int64_t at = 0;  // of the layer in a member's weights
                for (int l = 0; l <= n_hidden && ok; ++l) {
                    const int slab = l == 0 ? first_bytes(p.k0p, width)
                                     : l < n_hidden ? slab_bytes(width) : last_bytes(width, n_out);
                    const int n = l > 0 && l < n_hidden ? slabs : 1;
                    for (int c = 0; c < tiles && ok; ++c) {
                        const unsigned char *src = p.net.packed + (i + c) / p.mtiles * p.member_bytes + at;
                        for (int k = 0; k < n && ok; ++k, src += slab) ok = load(src, slab);
                    }
                    at += (int64_t)n * slab;
                }
            }
            // (after an abort) the copies in flight land before the CTA's shared memory is given up
            for (uint32_t k = n_slab > (uint32_t)stages ? n_slab - stages : 0; k < n_slab; ++k)
                tc_wait(&bars.wfull[k % stages], (k / stages) & 1u);
        }
        __syncwarp();
    } else if (warp == 0) {
        // ---- issuer
        uint32_t h_phase = 0;            // a bit per tile: of the next hidden epilogue to wait for
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
            if (++stage == (uint32_t)stages) {
                stage = 0;
                parity ^= 1u;
            }
        };
        bool ok = true;
        for (int i = i0; i < i1 && ok; i += kTiles) {
            const int tiles = i1 - i < kTiles ? i1 - i : kTiles;
            const uint32_t n = (uint32_t)(i - i0) / kTiles;  // items of a tile before
            for (int l = 0; l <= n_hidden && ok; ++l)
                for (int c = 0; c < tiles && ok; ++c) {
                    const uint32_t d = tmem + c * 256;
                    uint64_t act = da + c * (a_bytes / 16);
                    ok = slab();
                    if (ok && l == 0) {
                        ok = warp_wait(bars, &bars.xready[c], n & 1u);
                        if (ok && n > 0) ok = warp_wait(bars, &bars.oread[c], (n - 1) & 1u);
                    } else if (ok) {
                        ok = warp_wait(bars, &bars.hready[c], h_phase >> c & 1u);
                        h_phase ^= 1u << c;
                    }
                    if (!ok) break;
                    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                    if (l == 0) {
                        for (int ks = 0; ks < p.k0p / 16; ++ks)
                            tc_mma(d, dx + c * (x_bytes / 16) + ks * 16, at(dw_x) + ks * 16, idesc, ks > 0);
                        slab_done();
                        tc_commit(&bars.dfull[c]);
                    } else if (l < n_hidden) {
                        for (int kc = 0; kc < slabs; ++kc) {
                            if (kc > 0) ok = slab();
                            if (!ok) break;
#pragma unroll
                            for (int ks = 0; ks < kSlab / 16; ++ks, act += 16)
                                tc_mma(d, act, at(dw) + ks * 16, idesc, kc + ks > 0);
                            slab_done();
                        }
                        if (ok) tc_commit(&bars.dfull[c]);
                    } else {
                        // the outputs: every slab of K from one stage
                        for (int kc = 0; kc < slabs; ++kc)
#pragma unroll
                            for (int ks = 0; ks < kSlab / 16; ++ks, act += 16)
                                tc_mma(d, act, at(dw) + kc * (n_out * 4) + ks * 16, idesc_out, kc + ks > 0);
                        slab_done();
                        tc_commit(&bars.ofull[c]);
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
        const int c = (warp - 2) / kEpiWarps;  // this warp's tile
        const int q = warp & 3, part = (warp - 2) % kEpiWarps >> 2, tid = (threadIdx.x - 64) % (kEpiWarps * 32);
        const int r = q * 32 + lane;
        const uint32_t lanes = tmem + c * 256 + ((uint32_t)(q * 32) << 16);
        unsigned char *arow = As + c * a_bytes + (size_t)(r >> 3) * (width / 8) * 128 + (r & 7) * 16;
        unsigned char *xs = Xs + c * x_bytes;
        float *const biases = bias_s + c * n_bias;
        uint32_t n_d = 0, n = 0;  // hidden layers done, items done
        bool ok = true;
        for (int i = i0 + c; i < i1 && ok; i += kTiles, ++n) {
            const int e = i / p.mtiles;
            const int64_t row = (int64_t)(i % p.mtiles) * kRows + r;
            // the inputs, over those of the last item, which were read before its first hidden layer came through
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
                *reinterpret_cast<uint4 *>(xs + (size_t)g * 16) = *reinterpret_cast<const uint4 *>(h);
            }
            // the biases of a new member, once every warp of the tile is done with the last one's
            if (n > 0) ok = warp_wait(bars, &bars.oread[c], (n - 1) & 1u);
            if (!ok) break;
            if (n == 0 || e != (i - kTiles) / p.mtiles) {
                const float *w = p.net.w + e * p.net.P;
                for (int g = tid; g < n_bias; g += kEpiWarps * 32) {
                    const int l = g / width, k = g - l * width;  // b_l follows W_l
                    biases[g] = __ldg(w + (int64_t)p.net.n_in * width + (l > 0 ? width : 0) +
                                      (l > 1 ? (int64_t)(l - 1) * width : 0) +
                                      (l < n_hidden ? (int64_t)l * width * width
                                                    : (int64_t)(n_hidden - 1) * width * width + (int64_t)n_out * width) +
                                      k);
                }
            }
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            __syncwarp();
            if (lane == 0) bar_arrive(&bars.xready[c]);
            ok = warp_wait(bars, &bars.xready[c], n & 1u);
            const float *bias = biases;
            for (int l = 0; l < n_hidden && ok; ++l, ++n_d) {
                ok = warp_wait(bars, &bars.dfull[c], n_d & 1u);
                if (ok && p.report_timeout) {  // as if this wait had run out, once it has completed
                    bars.abort = 1;
                    ok = false;
                }
                if (!ok) break;
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                for (int n0 = part * 16; n0 < width; n0 += kEpiWarps / 4 * 16) {
                    uint32_t v[16];
                    tc_load16(v, lanes + (uint32_t)n0);
                    float4 bv[4];
#pragma unroll
                    for (int j = 0; j < 4; ++j) bv[j] = reinterpret_cast<const float4 *>(bias + n0)[j];
                    tc_loaded(v);
                    __align__(16) __nv_bfloat162 h[8];
                    float zmax = 0.0f;
#pragma unroll
                    for (int j = 0; j < 8; ++j) {
                        const uint64_t z = add2(pack2(__uint_as_float(v[2 * j]), __uint_as_float(v[2 * j + 1])),
                                                j % 2 == 0 ? pack2(bv[j / 2].x, bv[j / 2].y) : pack2(bv[j / 2].z, bv[j / 2].w));
                        const float2 zj = unpack2(z);
                        v[2 * j] = __float_as_uint(zj.x);
                        v[2 * j + 1] = __float_as_uint(zj.y);
                        zmax = fmaxf(zmax, fmaxf(fabsf(zj.x), fabsf(zj.y)));
                        const float2 g = unpack2(gelu2_f(z));
                        h[j] = __floats2bfloat162_rn(g.x, g.y);
                    }
                    if (!(zmax <= kGelu2Max)) {  // (a NaN is ignored by fmaxf and propagates through either form)
#pragma unroll
                        for (int j = 0; j < 8; ++j)
                            h[j] = __floats2bfloat162_rn(gelu_f(__uint_as_float(v[2 * j])), gelu_f(__uint_as_float(v[2 * j + 1])));
                    }
                    unsigned char *o = arow + n0 / 8 * 128;
#pragma unroll
                    for (int j = 0; j < 2; ++j)
                        *reinterpret_cast<uint4 *>(o + j * 128) = reinterpret_cast<const uint4 *>(h)[j];
                }
                asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
                __syncwarp();
                if (lane == 0) bar_arrive(&bars.hready[c]);
                bias += width;
            }
            if (!ok) break;
            // outputs
            ok = warp_wait(bars, &bars.ofull[c], n & 1u);
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
            if (lane == 0) bar_arrive(&bars.oread[c]);
        }
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (threadIdx.x == 0 && bars.abort && p.err) atomicExch(p.err, 1);
    if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 512;" ::"r"(tmem) : "memory");
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
    // as much of a ring as fits beside the tiles (four stages for 7-256x4-16; two always do)
    const int rest = kTiles * (kRows * (n.width + p.k0p) * 2 + 4 * (n.n_hidden * n.width + n.n_out));
    p.stages = kMaxStages;
    while (p.stages > 2 && p.stages * kStageBytes + rest > kFusedSmem) --p.stages;
    int smem = p.stages * kStageBytes + rest;
    if (smem < kFusedSmem / 2 + 1024) smem = kFusedSmem / 2 + 1024;  // one CTA per SM: it takes all of tensor memory
    int dev = 0, sms = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    // the limit belongs to the kernel, not to the launch: every thread sets the same
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(fused_forward_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kFusedSmem);
    if (e != cudaSuccess) return e;
    fused_forward_kernel<<<p.items < sms ? p.items : sms, kThreads, smem, st>>>(p);
    return cudaPeekAtLastError();
}

}  // namespace cpmmlp
