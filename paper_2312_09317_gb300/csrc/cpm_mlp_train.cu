// One training batch of the emulator network, forward and back, all members in one kernel.
//
// A CTA takes (member, N-row tile) items; the tile's activations and gradients never leave the SM but for
// what the weight gradients need.  A batch has few rows (1,024 rows of 5 members: 40 tiles of 128), so what
// counts is the time of a tile's chain of 2 (hidden layers + 1) products, and the products are turned
// around: a layer's weights are the MMA's A operand, 128 outputs in the lanes of tensor memory, and the
// tile's rows are its N, as few as give every SM one tile (48 at 1,024 rows).  A layer is then
//   weights  streamed from L2 through a ring of three 32 KB stages, independent of the chain;
//   MMAs     32 of 128 x N x 16 from shared memory, 2,100 cycles with the waits for the ring;
//   epilogue a lane per output and 8 rows at a time: 24 elements a thread with 16 warps.
// What bounds it is the latency of that chain: 8,300 cycles a layer forward (4,500 of them the epilogue), 5,500
// back, and 8,000 to gather the rows, of 66,000.  With 128 rows in the lanes on 40 SMs it was 100,000.
// GELU' is kept from the way forward in FP32, where its exponential is at hand.  Every element is summed over K
// in ascending order, 16 at a time, as by the single-layer kernels.
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <cstdint>

#include "cpm_mlp_internal.h"
#include "cpm_mlp_tc.cuh"

namespace cpmmlp {
namespace {

constexpr int kTrainWarps = 16, kTrainThreads = (kTrainWarps + 2) * 32;
constexpr int kTrainStages = 3, kStage2 = 2 * kStageBytes;  // of the ring: two slabs of a hidden layer
constexpr int kMaxTile = 128;
constexpr int kTrainSmem = 224 * 1024;  // of a CTA, at most
// The activations lie with the rows innermost (MN-major): core matrices of 8 K indices x 8 rows, K-adjacent ones
// next to each other, so that a lane's 8 rows of an output are one 16-byte store, a warp's contiguous.
constexpr uint32_t kRowsInner = 1u << 16;  // of the instruction descriptor, for the B operand

struct TrainKernelArgs {
    FusedNet net;
    TrainArgs tr;
    const float *X;
    int64_t rows;
    int *err;
    int report_timeout;
    int k0p;               // inputs padded to a multiple of 16
    int64_t member_bytes;  // packed weights per member
    int tile, mtiles, items;
};

struct TrainBarriers {
    uint64_t wfull[kTrainStages], wempty[kTrainStages];
    uint64_t hready, dfull;  // a hidden layer (or its gradient): output written (the next input), accumulator complete
    uint64_t ofull, oread;   // the outputs: accumulator complete; the item's last accumulator read out
    uint64_t sready, xready; // the item: data rows of the tile known, inputs written
    uint64_t pready;         // the gradient of its outputs written
    uint64_t drain;
    volatile int abort;      // a wait ran out: every role leaves its loop
};

// the data row of a batch's row, -1 (and the flag) where order[] points outside the data
__device__ __forceinline__ int64_t batch_row(const TrainArgs &t, int64_t r)
{
    const int64_t src = t.order ? (int64_t)__ldg(t.order + t.off + r) : t.off + r;
    if (src >= 0 && src < t.n_total) return src;
    *t.bad = 1;
    return -1;
}

// blocks: of 128 outputs of a hidden layer
template <int blocks>
__global__ void __launch_bounds__(kTrainThreads, 1) fused_train_kernel(const TrainKernelArgs p)
{
    extern __shared__ __align__(1024) unsigned char train_smem[];
    __shared__ __align__(8) TrainBarriers bars;
    __shared__ uint32_t tmem_slot;
    __shared__ int64_t src_s[kMaxTile];  // data rows of the tile
    const int width = p.net.width, slabs = width / kSlab, pairs = slabs / 2, n_hidden = p.net.n_hidden, n_out = p.net.n_out, tile = p.tile;
    unsigned char *Ws = train_smem;                                 // kTrainStages stages
    unsigned char *As = Ws + kTrainStages * kStage2;                // tile x width
    unsigned char *Ps = As + tile * width * 2;                      // tile x n_out
    unsigned char *Xs = Ps + tile * n_out * 2;                      // tile x k0p
    float *Ys = reinterpret_cast<float *>(Xs + tile * p.k0p * 2);   // tile x n_out
    float *bias_s = Ys + tile * n_out;                              // layer after layer
    const int n_bias = n_hidden * width + n_out;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 256;" ::"r"(smem_u32(&tmem_slot))
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    if (threadIdx.x == 0) {
        for (int k = 0; k < kTrainStages; ++k) {
            bar_init(&bars.wfull[k], 1);
            bar_init(&bars.wempty[k], 1);
        }
        bar_init(&bars.hready, kTrainWarps);
        bar_init(&bars.dfull, 1);
        bar_init(&bars.ofull, 1);
        bar_init(&bars.oread, kTrainWarps);
        bar_init(&bars.sready, kTrainWarps);
        bar_init(&bars.xready, kTrainWarps);
        bar_init(&bars.pready, kTrainWarps);
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
            pdl_wait();  // the weights
            const auto load = [&](const unsigned char *src, int bytes) {
                if (n_slab >= kTrainStages && !bar_wait(bars, &bars.wempty[stage], parity)) return false;
                const uint32_t full = smem_u32(&bars.wfull[stage]);
                asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(full), "r"(bytes) : "memory");
                asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                                 smem_u32(Ws + stage * kStage2)),
                             "l"(src), "r"(bytes), "r"(full)
                             : "memory");
                ++n_slab;
                if (++stage == kTrainStages) {
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
                for (int k = 0; k < (n_hidden - 1) * pairs && ok; ++k, src += 2 * slab_bytes(width))
                    ok = load(src, 2 * slab_bytes(width));
                if (ok) ok = load(src, last_bytes(width, n_out));
                const unsigned char *t = p.tr.packed_t + i / p.mtiles * p.tr.member_bytes_t;
                if (ok) ok = load(t, last_bytes(width, n_out));
                t += last_bytes(width, n_out);
                for (int k = 0; k < (n_hidden - 1) * pairs && ok; ++k, t += 2 * slab_bytes(width))
                    ok = load(t, 2 * slab_bytes(width));
            }
            // (after an abort) the copies in flight land before the CTA's shared memory is given up
            for (uint32_t k = n_slab > kTrainStages ? n_slab - kTrainStages : 0; k < n_slab; ++k)
                tc_wait(&bars.wfull[k % kTrainStages], (k / kTrainStages) & 1u);
        }
        __syncwarp();
    } else if (warp == 0) {
        // ---- issuer
        uint32_t n_h = 0;                // hidden epilogues waited for
        uint32_t stage = 0, parity = 0;  // of the next slab
        // Matrix descriptors: the address, in 16-byte units, is their low field.  Weights are read in blocks of
        // 128 rows; where a block has fewer (or a last layer n_out), the lanes past them hold whatever follows in
        // the stage, and are not used.
        const uint64_t da = tc_desc(smem_u32(As), 128u, (uint32_t)(width / 8) * 128u);
        const uint64_t dp = tc_desc(smem_u32(Ps), 128u, (uint32_t)(n_out / 8) * 128u);
        const uint64_t dx = tc_desc(smem_u32(Xs), 128u, (uint32_t)(p.k0p / 8) * 128u);
        const uint64_t dw = tc_desc(smem_u32(Ws), 128u, (uint32_t)(kSlab / 8) * 128u);
        const uint64_t dw_x = tc_desc(smem_u32(Ws), 128u, (uint32_t)(p.k0p / 8) * 128u);
        const uint64_t dw_p = tc_desc(smem_u32(Ws), 128u, (uint32_t)(n_out / 8) * 128u);
        const uint32_t idesc_x = tc_idesc(tile), idesc = idesc_x | kRowsInner;
        // a slab is asked for before the MMAs of the one before it are issued (a wait costs 170 cycles also where
        // it is over)
        bool here = false;
        const auto slab = [&]() {
            const bool ok = __all_sync(0xffffffffu, here) || warp_wait(bars, &bars.wfull[stage], parity);
            const uint32_t next = stage + 1 == kTrainStages ? 0 : stage + 1;
            here = bar_over(&bars.wfull[next], next == 0 ? parity ^ 1u : parity);
            return ok;
        };
        const auto at = [&](uint64_t d) { return d + stage * (kStage2 / 16); };
        const auto slab_done = [&]() {
            tc_commit(&bars.wempty[stage]);
            if (++stage == kTrainStages) {
                stage = 0;
                parity ^= 1u;
            }
        };
        // a layer whose K (16 k_steps) lies in one stage
        const auto small = [&](uint64_t w, int w_block, uint64_t b, uint32_t id, int k_steps) {
#pragma unroll
            for (int k = 0; k < blocks; ++k)
                for (int ks = 0; ks < k_steps; ++ks)
                    tc_mma(tmem + k * kRows, at(w) + k * w_block + ks * 16, b + ks * 16, id, ks > 0);
            slab_done();
            tc_commit(&bars.dfull);
        };
        // a hidden layer, or a gradient's way through one: K = width, slab by slab
        const auto hidden = [&]() {
            uint64_t b = da;
            const uint32_t second = (uint32_t)slab_bytes(width) / 16;
            for (int kc = 0; kc < pairs; ++kc) {
                if (kc > 0 && !slab()) return false;
#pragma unroll
                for (int ks = 0; ks < 2 * kSlab / 16; ++ks, b += 16)
#pragma unroll
                    for (int k = 0; k < blocks; ++k)
                        tc_mma(tmem + k * kRows, at(dw) + ks / 2 * second + k * (kRows * kSlab * 2 / 16) + ks % 2 * 16, b,
                               idesc, kc + ks > 0);
                slab_done();
            }
            tc_commit(&bars.dfull);
            return true;
        };
        bool ok = true;
        for (int i = i0; i < i1 && ok; ++i) {
            ok = slab() && warp_wait(bars, &bars.xready, (uint32_t)(i - i0) & 1u);
            if (ok && i > i0) ok = warp_wait(bars, &bars.oread, (uint32_t)(i - i0 - 1) & 1u);
            if (!ok) break;
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            small(dw_x, kRows * p.k0p * 2 / 16, dx, idesc_x, p.k0p / 16);
            for (int l = 1; l <= n_hidden && ok; ++l, ++n_h) {
                ok = slab() && warp_wait(bars, &bars.hready, n_h & 1u);
                if (!ok) break;
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                if (l < n_hidden) {
                    ok = hidden();
                } else {
                    // the outputs: every slab of K from one stage
                    for (int kc = 0; kc < slabs; ++kc)
#pragma unroll
                        for (int ks = 0; ks < kSlab / 16; ++ks)
                            tc_mma(tmem, at(dw) + kc * (n_out * 4) + ks * 16, da + kc * 32 + ks * 16, idesc, kc + ks > 0);
                    slab_done();
                    tc_commit(&bars.ofull);
                }
            }
            if (ok) ok = slab() && warp_wait(bars, &bars.pready, (uint32_t)(i - i0) & 1u);
            if (!ok) break;
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            small(dw_p, kRows * n_out * 2 / 16, dp, idesc, n_out / 16);
            for (int l = n_hidden - 1; l >= 1 && ok; --l, ++n_h) {
                ok = slab() && warp_wait(bars, &bars.hready, n_h & 1u);
                if (!ok) break;
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                ok = hidden();
            }
        }
        if (!ok) {
            // the MMAs issued so far end before tensor memory is given up
            tc_commit(&bars.drain);
            tc_wait(&bars.drain, 0);
        }
    } else {
        // ---- epilogue: units of 8 rows of 32 outputs, every fourth to a warp
        constexpr int kAhead = 3;  // units whose loads are under way together
        const int q = warp & 3, part = (warp - 2) >> 2, tid = threadIdx.x - 64;
        const int chunks = tile / 8, units = blocks * chunks;
        const int64_t R = (p.rows + 7) / 8;
        uint32_t n_d = 0;  // hidden layers done
        bool ok = true;
        for (int i = i0; i < i1 && ok; ++i) {
            const int e = i / p.mtiles;
            const int64_t row0 = (int64_t)(i % p.mtiles) * tile, rb0 = row0 / 8;
            // The item's biases, inputs and targets, over those of the last item: every warp was past their last
            // use before that item's gradients came through.
            const int n_in = p.net.n_in, k0p = p.k0p;
            for (int r = tid; r < tile; r += kTrainWarps * 32)
                src_s[r] = row0 + r < p.rows ? batch_row(p.tr, row0 + r) : -1;
            __syncwarp();
            if (lane == 0) bar_arrive(&bars.sready);
            ok = warp_wait(bars, &bars.sready, (uint32_t)(i - i0) & 1u);
            if (!ok) break;
#pragma unroll 2
            for (int g = tid; g < tile * k0p; g += kTrainWarps * 32) {
                const int k = g % k0p, r = g / k0p;
                const int64_t src = src_s[r];
                const __nv_bfloat16 h = __float2bfloat16(src >= 0 && k < n_in ? __ldg(p.X + src * n_in + k) : 0.0f);
                *reinterpret_cast<__nv_bfloat16 *>(Xs + ((r >> 3) * (k0p / 8) + (k >> 3)) * 128 + (r & 7) * 16 + (k & 7) * 2) = h;
            }
#pragma unroll 2
            for (int g = tid; g < tile * n_out; g += kTrainWarps * 32) {
                const int64_t src = src_s[g / n_out];
                Ys[g] = src >= 0 ? __ldg(p.tr.Y + src * n_out + g % n_out) : 0.0f;
            }
            if (i == i0) {  // from here on what the last update wrote, or read
                pdl_wait();
                pdl_next();
            }
            const float *w = p.net.w + e * p.net.P;
#pragma unroll 4
            for (int g = tid; g < n_bias; g += kTrainWarps * 32) {
                const int l = g / width, k = g - l * width;  // b_l follows W_l
                bias_s[g] = w[(int64_t)p.net.n_in * width + (l > 0 ? width : 0) + (l > 1 ? (int64_t)(l - 1) * width : 0) +
                              (l < n_hidden ? (int64_t)l * width * width
                                            : (int64_t)(n_hidden - 1) * width * width + (int64_t)n_out * width) + k];
            }
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            __syncwarp();
            if (lane == 0) bar_arrive(&bars.xready);
            ok = warp_wait(bars, &bars.xready, (uint32_t)(i - i0) & 1u);
            if (e == 0)
                for (int g = tid; g < tile * k0p; g += kTrainWarps * 32) {
                    const int k = g / 8 % k0p, r = g / 8 / k0p * 8 + g % 8;
                    if (row0 + r < R * 8)
                        p.tr.xb[rb0 * k0p * 8 + g] = *reinterpret_cast<const __nv_bfloat16 *>(
                            Xs + ((r >> 3) * (k0p / 8) + (k >> 3)) * 128 + (r & 7) * 16 + (k & 7) * 2);
                }
            // unit u: block of outputs, rows 8 c ..; this lane's output f
            const auto block = [&](int u) { return u >= chunks ? 1 : 0; };
            const auto chunk = [&](int u) { return u >= chunks ? u - chunks : u; };
            const auto valid = [&](int u) { return u < units && block(u) * kRows + q * 32 < width; };
            const auto column = [&](int u) { return tmem + ((uint32_t)(q * 32) << 16) + (uint32_t)(block(u) * kRows + chunk(u) * 8); };
            // its 8 rows to the tile's image S
            const auto put = [&](unsigned char *S, int k_width, int u, int f, const uint4 &h) {
                *reinterpret_cast<uint4 *>(S + (chunk(u) * k_width + f) * 16) = h;
            };
            // the first n of 8 rows, the others zero
            const auto mask = [&](uint4 h, int n) {
                uint32_t *x = reinterpret_cast<uint32_t *>(&h);
#pragma unroll
                for (int j = 0; j < 4; ++j) x[j] &= n > 2 * j + 1 ? 0xffffffffu : n > 2 * j ? 0xffffu : 0u;
                return h;
            };
            const int64_t tile0 = (e * R + rb0) * width;  // of the tile in H, in pieces of 8 rows
            const auto done = [&](uint64_t *b) {
                asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
                __syncwarp();
                if (lane == 0) bar_arrive(b);
            };
            for (int l = 0; l < n_hidden && ok; ++l, ++n_d) {
                ok = warp_wait(bars, &bars.dfull, n_d & 1u);
                if (ok && p.report_timeout) {  // as if this wait had run out, once it has completed
                    bars.abort = 1;
                    ok = false;
                }
                if (!ok) break;
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                uint4 *Hl = reinterpret_cast<uint4 *>(p.tr.H[l]) + tile0;
                float4 *Gl = reinterpret_cast<float4 *>(p.tr.G[l]) + 2 * tile0;
                for (int u0 = part; u0 < units; u0 += 4 * kAhead) {
                    uint32_t v[kAhead][8];
#pragma unroll
                    for (int t = 0; t < kAhead; ++t)
                        if (valid(u0 + 4 * t)) tc_load8(v[t], column(u0 + 4 * t));
#pragma unroll
                    for (int t = 0; t < kAhead; ++t) {
                        const int u = u0 + 4 * t, f = block(u) * kRows + q * 32 + lane;
                        if (!valid(u)) continue;
                        tc_loaded(v[t]);
                        const float b = bias_s[l * width + f];
                        __align__(16) __nv_bfloat162 h[4];
                        float g[8], zmax = 0.0f;
#pragma unroll
                        for (int j = 0; j < 4; ++j) {
                            const uint64_t z = add2(pack2(__uint_as_float(v[t][2 * j]), __uint_as_float(v[t][2 * j + 1])), both(b));
                            const float2 zj = unpack2(z);
                            zmax = fmaxf(zmax, fmaxf(fabsf(zj.x), fabsf(zj.y)));
                            uint64_t grad;
                            const float2 y = unpack2(gelu2_f<true>(z, grad)), d = unpack2(grad);
                            h[j] = __floats2bfloat162_rn(y.x, y.y);
                            g[2 * j] = d.x;
                            g[2 * j + 1] = d.y;
                        }
                        if (!(zmax <= kGelu2Max)) {  // (a NaN is ignored by fmaxf and propagates through either form)
#pragma unroll
                            for (int j = 0; j < 4; ++j) {
                                const float z0 = __uint_as_float(v[t][2 * j]) + b, z1 = __uint_as_float(v[t][2 * j + 1]) + b;
                                h[j] = __floats2bfloat162_rn(gelu_f(z0), gelu_f(z1));
                                g[2 * j] = gelu_grad_f(z0);
                                g[2 * j + 1] = gelu_grad_f(z1);
                            }
                        }
                        uint4 hv = *reinterpret_cast<const uint4 *>(h);
                        put(As, width, u, f, hv);
                        const int64_t rb = rb0 + chunk(u);
                        if (rb >= R) continue;
                        if (rb * 8 + 8 > p.rows) hv = mask(hv, (int)(p.rows - rb * 8));
                        Hl[chunk(u) * width + f] = hv;
                        float4 *go = Gl + chunk(u) * 2 * width + f;
                        go[0] = make_float4(g[0], g[1], g[2], g[3]);
                        go[width] = make_float4(g[4], g[5], g[6], g[7]);
                    }
                }
                done(&bars.hready);
            }
            if (!ok) break;
            // outputs: their loss, and their gradient, the first input of the way back
            ok = warp_wait(bars, &bars.ofull, (uint32_t)(i - i0) & 1u);
            if (!ok) break;
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            if (q == 0) {
                const float b = lane < n_out ? bias_s[n_hidden * width + lane] : 0.0f;
                float sq = 0.0f;
                for (int c = part; c < chunks; c += 4) {
                    uint32_t v[8];
                    tc_load8(v, column(c));
                    tc_loaded(v);
                    __align__(16) __nv_bfloat16 h[8];
                    const uint4 &hv = *reinterpret_cast<const uint4 *>(h);
#pragma unroll
                    for (int j = 0; j < 8; ++j) {
                        const int r = c * 8 + j;
                        const float d = lane < n_out && row0 + r < p.rows ? __uint_as_float(v[j]) + b - Ys[r * n_out + lane] : 0.0f;
                        h[j] = __float2bfloat16(2.0f * d * p.tr.inv);
                        sq += d * d;
                    }
                    if (lane < n_out) {
                        put(Ps, n_out, c, lane, hv);
                        if (rb0 + c < R) reinterpret_cast<uint4 *>(p.tr.dP)[(e * R + rb0 + c) * n_out + lane] = hv;
                    }
                }
#pragma unroll
                for (int d = 16; d > 0; d >>= 1) sq += __shfl_xor_sync(0xffffffffu, sq, d);
                if (lane == 0) atomicAdd(p.tr.loss + e, sq * p.tr.inv);
            }
            done(&bars.pready);
            // the way back: dZ_l = (dZ_{l+1} W_{l+1}) GELU'(Z_l), over the activations of its last input
            for (int l = n_hidden - 1; l >= 0; --l, ++n_d) {
                float4 *Gl = reinterpret_cast<float4 *>(p.tr.G[l]) + 2 * tile0;
                float4 g[kAhead][2];
                const auto load_g = [&](int u0) {
#pragma unroll
                    for (int t = 0; t < kAhead; ++t) {
                        const int u = u0 + 4 * t, f = block(u) * kRows + q * 32 + lane;
                        const int64_t rb = rb0 + chunk(u);
                        g[t][0] = g[t][1] = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
                        if (valid(u) && rb < R) {
                            const float4 *go = Gl + chunk(u) * 2 * width + f;
                            g[t][0] = go[0];
                            g[t][1] = go[width];
                        }
                    }
                };
                load_g(part);
                ok = warp_wait(bars, &bars.dfull, n_d & 1u);
                if (!ok) break;
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                for (int u0 = part; u0 < units; u0 += 4 * kAhead) {
                    if (u0 > part) load_g(u0);
                    uint32_t v[kAhead][8];
#pragma unroll
                    for (int t = 0; t < kAhead; ++t)
                        if (valid(u0 + 4 * t)) tc_load8(v[t], column(u0 + 4 * t));
#pragma unroll
                    for (int t = 0; t < kAhead; ++t) {
                        const int u = u0 + 4 * t, f = block(u) * kRows + q * 32 + lane;
                        if (!valid(u)) continue;
                        tc_loaded(v[t]);
                        const float gj[8] = {g[t][0].x, g[t][0].y, g[t][0].z, g[t][0].w,
                                             g[t][1].x, g[t][1].y, g[t][1].z, g[t][1].w};
                        const int64_t rb = rb0 + chunk(u);
                        __align__(16) __nv_bfloat162 h[4];
#pragma unroll
                        for (int j = 0; j < 4; ++j)
                            h[j] = __floats2bfloat162_rn(__uint_as_float(v[t][2 * j]) * gj[2 * j],
                                                         __uint_as_float(v[t][2 * j + 1]) * gj[2 * j + 1]);
                        uint4 hv = *reinterpret_cast<const uint4 *>(h);
                        if (rb * 8 + 8 > p.rows) hv = mask(hv, (int)max(p.rows - rb * 8, (int64_t)0));
                        put(As, width, u, f, hv);
                        if (rb < R) reinterpret_cast<uint4 *>(Gl)[chunk(u) * 2 * width + f] = hv;  // over the GELU' just read
                    }
                }
                if (l > 0) done(&bars.hready);
            }
            if (!ok) break;
            asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
            __syncwarp();
            if (lane == 0) bar_arrive(&bars.oread);
        }
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (threadIdx.x == 0 && bars.abort && p.err) atomicExch(p.err, 1);
    if (warp == 0)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 256;" ::"r"(tmem) : "memory");
}

// The transposed weights as the way back reads them: B[n][k] = W[k][n], the last layer first.
__global__ void fused_pack_t_kernel(const FusedNet n, const __nv_bfloat16 *wb, unsigned char *packed, int64_t member_bytes)
{
    const int slabs = n.width / kSlab;
    const int64_t pieces = member_bytes / 16;
    for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < pieces * n.n_members;
         t += (int64_t)gridDim.x * blockDim.x) {
        const int e = (int)(t / pieces);
        int64_t at = (t % pieces) * 16;
        const int64_t hidden = (int64_t)n.width * n.width + n.width, layer = (int64_t)slabs * slab_bytes(n.width);
        const __nv_bfloat16 *W = wb + e * n.P + (int64_t)n.n_in * n.width + n.width;  // layer 1
        int kc = n.n_out / 8, k_first = 0;
        if (at < last_bytes(n.width, n.n_out)) {
            W += (n.n_hidden - 1) * hidden;
        } else {
            at -= last_bytes(n.width, n.n_out);
            W += (n.n_hidden - 2 - at / layer) * hidden;
            at %= layer;
            k_first = (int)(at / slab_bytes(n.width)) * kSlab;
            at %= slab_bytes(n.width);
            kc = kSlab / 8;
        }
        const int q = (int)(at / 16), rr = q & 7, k8 = (q >> 3) % kc, r8 = (q >> 3) / kc;
        __align__(16) __nv_bfloat16 h[8];
#pragma unroll
        for (int j = 0; j < 8; ++j) h[j] = W[(int64_t)(k_first + k8 * 8 + j) * n.width + r8 * 8 + rr];
        *reinterpret_cast<uint4 *>(packed + t * 16) = *reinterpret_cast<const uint4 *>(h);
    }
}

}  // namespace

int64_t fused_packed_t_bytes(int width, int n_hidden, int n_out)
{
    return last_bytes(width, n_out) + (int64_t)(n_hidden - 1) * (width / kSlab) * slab_bytes(width);
}

cudaError_t fused_pack_t(const FusedNet &n, const __nv_bfloat16 *wb, unsigned char *packed_t, cudaStream_t st)
{
    const int64_t bytes = fused_packed_t_bytes(n.width, n.n_hidden, n.n_out);
    const int64_t blocks = (bytes / 16 * n.n_members + 255) / 256;
    fused_pack_t_kernel<<<(unsigned)(blocks < 2432 ? blocks : 2432), 256, 0, st>>>(n, wb, packed_t, bytes);
    return cudaPeekAtLastError();
}

cudaError_t fused_train(const FusedNet &n, const TrainArgs &tr, const float *X, int64_t rows, int *err,
                        int report_timeout, cudaStream_t st)
{
    if (rows <= 0) return cudaSuccess;
    int dev = 0, sms = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return e;
    TrainKernelArgs p{};
    p.net = n;
    p.tr = tr;
    p.tr.member_bytes_t = fused_packed_t_bytes(n.width, n.n_hidden, n.n_out);
    p.X = X;
    p.rows = rows;
    p.err = err;
    p.report_timeout = report_timeout;
    p.k0p = padded_inputs(n.n_in);
    p.member_bytes = fused_packed_bytes(n.n_in, n.width, n.n_hidden, n.n_out);
    // the smallest tile that leaves every SM at most one; past 128 rows SMs take several tiles
    p.tile = 16;
    while (p.tile < kMaxTile && (rows + p.tile - 1) / p.tile * n.n_members > sms) p.tile += 16;
    p.mtiles = (int)((rows + p.tile - 1) / p.tile);
    p.items = p.mtiles * n.n_members;
    // (212,096 bytes for the largest shape that fused_fits takes: 32 inputs and outputs, 15 layers of 256, tiles of 128)
    const int smem = kTrainStages * kStage2 + p.tile * (n.width + n.n_out + p.k0p) * 2 + p.tile * n.n_out * 4 +
               4 * (n.n_hidden * n.width + n.n_out);
    const auto kernel = n.width > kRows ? fused_train_kernel<2> : fused_train_kernel<1>;
    // the limit belongs to the kernel, not to the launch: every thread sets the same
    e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kTrainSmem);
    if (e != cudaSuccess) return e;
    return pdl_launch(kernel, p, p.items < sms ? p.items : sms, kTrainThreads, smem, tr.chained, st);
}

}  // namespace cpmmlp
