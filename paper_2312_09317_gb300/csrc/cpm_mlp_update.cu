// The weight gradients of a training batch and their Adam step, all layers of all members in one launch.
//
// dW_l = dZ_l^T H_{l-1} over the batch's rows, db_l = the sums of dZ_l.  A CTA takes a 64 (outputs) x 128
// (inputs) tile of one layer of one member: five members of 7-256x4-16 are 150 tiles, one per SM, whose
// operands (192 bf16 a row) come from L2 through a cp.async ring of 32-row slabs, read by ldmatrix with
// a transpose, since both lie with the summed index outermost.  Rows are summed in ascending order, 16 at a
// time, by one accumulator per element.  The tile's owner then has the whole gradient of its weights, so it
// applies their Adam step from its registers and writes the weights back, in FP32 and in the two bf16
// layouts that the next forward and backward read: the gradients never reach memory.
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <cstdint>

#include "cpm_mlp_internal.h"

namespace cpmmlp {
namespace {

constexpr int kTM = 64, kTN = 128, kTK = 32, kRing = 6, kUpdThreads = 256;
constexpr int kPitchA = kTM + 8, kPitchB = kTN + 8;  // halves: rows 9 and 17 x 16 B apart, ldmatrix without conflicts
constexpr int kSlabHalves = kTK * (kPitchA + kPitchB);
constexpr int kUpdSmem = kRing * kSlabHalves * 2;

struct Update {
    FusedNet net;
    TrainArgs tr;
    UpdateArgs u;
    int64_t rows;
    int k0p, tiles;  // tiles of a member
    int64_t member_bytes, member_bytes_t;
};

__device__ __forceinline__ void cp16(uint32_t dst, const void *src, bool in)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;\n" ::"r"(dst), "l"(src), "r"(in ? 16 : 0) : "memory");
}
__device__ __forceinline__ void ldsm_t(uint32_t (&v)[4], uint32_t addr)
{
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0, %1, %2, %3}, [%4];"
                 : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3])
                 : "r"(addr)
                 : "memory");
}
// a weight and its moments, read before the gradient is summed: their latency is behind the sum
struct State {
    float w, m, v;
};
__device__ __forceinline__ State state(const UpdateArgs &u, int64_t at) { return {u.w[at], u.m[at], u.v[at]}; }
// its Adam step, returning its new value (rounded as adam_kernel's is)
__device__ __forceinline__ float adam(const UpdateArgs &u, int64_t at, const State &s, float gr)
{
    const float mm = fmaf(1.0f - u.b1, gr, u.b1 * s.m);
    const float vv = fmaf((1.0f - u.b2) * gr, gr, u.b2 * s.v);
    u.m[at] = mm;
    u.v[at] = vv;
    const float wn = s.w - u.lr * (mm / u.c1) / (sqrtf(vv / u.c2) + u.eps);
    u.w[at] = wn;
    return wn;
}

__global__ void __launch_bounds__(kUpdThreads, 1) fused_update_kernel(const Update p)
{
    extern __shared__ __align__(128) __nv_bfloat16 ring[];
    __shared__ float part[8][kTM + 1];
    const int width = p.net.width, n_hidden = p.net.n_hidden, n_out = p.net.n_out, n_in = p.net.n_in;
    const int e = blockIdx.x / p.tiles;
    // the tile: layer l, outputs m0 .., inputs n0 ..
    const int mt = width / kTM, nt = (width + kTN - 1) / kTN;
    int t = blockIdx.x % p.tiles, l, fo, fi, m0, n0;
    if (t < (n_hidden - 1) * mt * nt) {  // the layers with the most work first
        l = 1 + t / (mt * nt);
        t %= mt * nt;
        fo = width, fi = width, m0 = t / nt * kTM, n0 = t % nt * kTN;
    } else if ((t -= (n_hidden - 1) * mt * nt) < nt) {
        l = n_hidden, fo = n_out, fi = width, m0 = 0, n0 = t * kTN;
    } else {
        l = 0, fo = width, fi = n_in, m0 = (t - nt) * kTM, n0 = 0;
    }
    const int M = min(fo - m0, kTM), N = l == 0 ? p.k0p : min(fi - n0, kTN);  // of the staged tile, multiples of 16
    // operands: 16-byte pieces, by row and by 8 columns
    const bool last = l == n_hidden, first = l == 0;
    const unsigned char *A = last ? reinterpret_cast<const unsigned char *>(p.tr.dP + e * p.rows * n_out)
                                  : reinterpret_cast<const unsigned char *>(p.tr.G[l] + (e * width + m0) * p.rows);
    const int64_t a_row = last ? n_out * 2 : 16, a_col = last ? 16 : 32 * p.rows;
    const unsigned char *B = reinterpret_cast<const unsigned char *>(
        first ? p.tr.xb : p.tr.H[l - 1] + (e * width + n0) * p.rows);
    const int64_t b_row = first ? p.k0p * 2 : 16, b_col = first ? 16 : 16 * p.rows;
    const uint32_t ring0 = smem_u32(ring);
    const int slabs = (int)((p.rows + kTK - 1) / kTK);
    const auto load = [&](int s) {
        if (s < slabs) {
            const uint32_t a = ring0 + (s % kRing) * kSlabHalves * 2, b = a + kTK * kPitchA * 2;
            const int64_t r0 = (int64_t)s * kTK;
            const int r = threadIdx.x & (kTK - 1);
            const bool in = r0 + r < p.rows;
            const int64_t src = in ? r0 + r : 0;
#pragma unroll
            for (int c = threadIdx.x / kTK; c < kTM / 8; c += kUpdThreads / kTK)
                if (c * 8 < M) cp16(a + (r * kPitchA + c * 8) * 2, A + src * a_row + c * a_col, in);
#pragma unroll
            for (int c = threadIdx.x / kTK; c < kTN / 8; c += kUpdThreads / kTK)
                if (c * 8 < N) cp16(b + (r * kPitchB + c * 8) * 2, B + src * b_row + c * b_col, in);
        }
        asm volatile("cp.async.commit_group;\n" ::: "memory");
    };

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int wm = (warp >> 2) * 32, wn = (warp & 3) * 32;
    const bool work = wm < M && wn < N;  // (a half of a warp's 32 x 32 may lie outside: staged by nobody, never stored)
    const bool bias = n0 == 0;
    // ldmatrix rows of this lane: matrix lane / 8, row lane % 8 of it
    const int a_off = ((lane >> 4) * 8 + (lane & 7)) * kPitchA + wm + ((lane >> 3) & 1) * 8;
    const int b_off = (((lane >> 3) & 1) * 8 + (lane & 7)) * kPitchB + wn + (lane >> 4) * 8;
    const int64_t off_w = l == 0 ? 0 : (int64_t)n_in * width + width + (int64_t)(l - 1) * ((int64_t)width * width + width);
    const int64_t off_b = off_w + (int64_t)fi * fo, at_b = e * p.net.P + off_b + m0 + threadIdx.x;
    float acc[2][4][4] = {};
    float2 db = make_float2(0.0f, 0.0f);  // of outputs 2 (lane), + 1, over the rows = warp mod 8
    for (int s = 0; s < kRing - 1; ++s) load(s);
    // accumulator element r of block (i, j): row +8 for r >= 2, column +1 for odd r
    const auto row = [&](int i, int r) { return wm + i * 16 + (lane >> 2) + (r >= 2 ? 8 : 0); };
    const auto col = [&](int j, int r) { return n0 + wn + j * 8 + 2 * (lane & 3) + (r & 1); };
    const auto at_w = [&](int lm, int gn) { return e * p.net.P + off_w + (int64_t)(m0 + lm) * fi + gn; };
    State st[2][4][4], st_b{};
    if (p.u.update) {
        if (work) {
#pragma unroll
            for (int i = 0; i < 2; ++i)
#pragma unroll
                for (int j = 0; j < 4; ++j)
#pragma unroll
                    for (int r = 0; r < 4; ++r) {
                        const int lm = row(i, r), gn = col(j, r);
                        if (lm < M && gn < fi) st[i][j][r] = state(p.u, at_w(lm, gn));
                    }
        }
        if (bias && threadIdx.x < M) st_b = state(p.u, at_b);
    }
    for (int s = 0; s < slabs; ++s) {
        asm volatile("cp.async.wait_group %0;\n" ::"n"(kRing - 2) : "memory");
        __syncthreads();  // slab s has landed for all, and all are done with slab s - 1, whose place is filled next
        load(s + kRing - 1);
        const uint32_t a = ring0 + (s % kRing) * kSlabHalves * 2, b = a + kTK * kPitchA * 2;
        if (work) {
#pragma unroll
            for (int ks = 0; ks < kTK; ks += 16) {
                uint32_t af[2][4], bf[2][4];
#pragma unroll
                for (int i = 0; i < 2; ++i) ldsm_t(af[i], a + (ks * kPitchA + a_off + i * 16) * 2);
#pragma unroll
                for (int j = 0; j < 2; ++j) ldsm_t(bf[j], b + (ks * kPitchB + b_off + j * 16) * 2);
#pragma unroll
                for (int i = 0; i < 2; ++i)
#pragma unroll
                    for (int j = 0; j < 4; ++j)
                        asm volatile(
                            "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 "
                            "{%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};\n"
                            : "+f"(acc[i][j][0]), "+f"(acc[i][j][1]), "+f"(acc[i][j][2]), "+f"(acc[i][j][3])
                            : "r"(af[i][0]), "r"(af[i][1]), "r"(af[i][2]), "r"(af[i][3]), "r"(bf[j / 2][j % 2 * 2]),
                              "r"(bf[j / 2][j % 2 * 2 + 1]));
            }
        }
        if (bias && lane * 2 < M) {
            const __nv_bfloat16 *z = ring + (s % kRing) * kSlabHalves + lane * 2;
#pragma unroll
            for (int r = warp; r < kTK; r += 8) {  // (rows past the batch are zero)
                const float2 v = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162 *>(z + r * kPitchA));
                db.x += v.x;
                db.y += v.y;
            }
        }
    }
    asm volatile("cp.async.wait_all;\n" ::: "memory");

    if (bias) {
        if (lane * 2 < M) {
            part[warp][lane * 2] = db.x;
            part[warp][lane * 2 + 1] = db.y;
        }
        __syncthreads();
        if (threadIdx.x < M) {
            float g = 0.0f;
#pragma unroll
            for (int k = 0; k < 8; ++k) g += part[k][threadIdx.x];
            if (p.u.update) adam(p.u, at_b, st_b, g);
            else p.u.g[at_b] = g;
        }
    }
    if (!work) return;
    // packed forms: W[o][k] at 128 B core matrices of 8 outputs x 8 inputs, K-adjacent ones next to each other
    unsigned char *pk = p.u.packed + e * p.member_bytes, *pt = p.u.packed_t + e * p.member_bytes_t;
    const int hidden_bytes = width * width * 2;
    int kc = kFusedSlab / 8, kc_t = kFusedSlab / 8;
    if (l == 0) {
        kc = p.k0p / 8;
    } else {
        pk += width * p.k0p * 2 + (int64_t)(l - 1) * hidden_bytes;
        pt += l == n_hidden ? 0 : n_out * width * 2 + (int64_t)(n_hidden - 1 - l) * hidden_bytes;
        if (l == n_hidden) {
            kc = width / 8;
            kc_t = n_out / 8;
        }
    }
    const auto place = [&](int r, int k, int chunks, int rows) {  // of row r, K index k: slab, core matrix, byte
        const int k8 = k >> 3;
        return (int64_t)(k8 / chunks) * rows * chunks * 16 + ((r >> 3) * chunks + k8 % chunks) * 128 + (r & 7) * 16 +
               (k & 7) * 2;
    };
#pragma unroll
    for (int i = 0; i < 2; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j)
#pragma unroll
            for (int r = 0; r < 4; ++r) {
                const int lm = row(i, r), gn = col(j, r), gm = m0 + lm;
                if (lm >= M || gn >= fi) continue;
                if (!p.u.update) {
                    p.u.g[at_w(lm, gn)] = acc[i][j][r];
                    continue;
                }
                const __nv_bfloat16 wb = __float2bfloat16(adam(p.u, at_w(lm, gn), st[i][j][r], acc[i][j][r]));
                *reinterpret_cast<__nv_bfloat16 *>(pk + place(gm, gn, kc, fo)) = wb;
                if (l > 0) *reinterpret_cast<__nv_bfloat16 *>(pt + place(gn, gm, kc_t, fi)) = wb;
            }
}

}  // namespace

cudaError_t fused_update(const FusedNet &n, const TrainArgs &tr, const UpdateArgs &u, int64_t rows, cudaStream_t st)
{
    Update p{};
    p.net = n;
    p.tr = tr;
    p.u = u;
    p.rows = rows;
    p.k0p = (n.n_in + 15) / 16 * 16;
    const int mt = n.width / kTM, nt = (n.width + kTN - 1) / kTN;
    p.tiles = (n.n_hidden - 1) * mt * nt + nt + mt;
    p.member_bytes = fused_packed_bytes(n.n_in, n.width, n.n_hidden, n.n_out);
    p.member_bytes_t = fused_packed_t_bytes(n.width, n.n_hidden, n.n_out);
    const cudaError_t e = cudaFuncSetAttribute(fused_update_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kUpdSmem);
    if (e != cudaSuccess) return e;
    fused_update_kernel<<<p.tiles * n.n_members, kUpdThreads, kUpdSmem, st>>>(p);
    return cudaPeekAtLastError();
}

}  // namespace cpmmlp
