// The weight gradients of a training batch and their Adam step, all layers of all members in one launch.
//
// dW_l = dZ_l^T H_{l-1} over the batch's rows, db_l = the sums of dZ_l.  A CTA takes a 64 (outputs) x 128
// (inputs) tile of one layer of one member: five members of 7-256x4-16 are 150 tiles, one per SM.  Its
// operands come from L2 through a cp.async ring of 32-row slabs, in 16-byte pieces of 8 rows of a column,
// contiguous in memory, in shared memory and for ldmatrix.  Rows are summed in ascending order, 16 at a
// time, by one accumulator per element.  The tile's owner then has the whole gradient of its weights, so it
// applies their Adam step and writes the weights back, in FP32 and in the two bf16 layouts that the next
// forward and backward read: the gradients never reach memory, and the weights' state, fetched behind the
// products, goes through it once.  1,024 rows: about 22 us, half of it the sums; with the accumulators' own
// threads stepping their scattered weights 36 us.
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <cstdint>

#include "cpm_mlp_internal.h"
#include "cpm_mlp_tc.cuh"

namespace cpmmlp {
namespace {

constexpr int kTM = 64, kTN = 128, kTK = 32, kRing = 6, kUpdThreads = 512;
constexpr int kBytesA = kTM * kTK * 2, kBytesB = kTN * kTK * 2, kRingBytes = kRing * (kBytesA + kBytesB);
constexpr int kStateBytes = kTM * kTN * 4;                // each of w, m and v
constexpr int kPitchG = kTN + 4, kPitchW = kTN + 8;       // of the gradients (floats) and new weights (halves)
constexpr int kUpdSmem = kRingBytes + 3 * kStateBytes;
static_assert(kTM * kPitchG * 4 + kTM * kPitchW * 2 <= kRingBytes, "the ring's place takes gradients and new weights");

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
__device__ __forceinline__ void ldsm(uint32_t (&v)[4], uint32_t addr)
{
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0, %1, %2, %3}, [%4];"
                 : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3])
                 : "r"(addr)
                 : "memory");
}
// one weight's Adam step on its moments; its new value (rounded as adam_kernel's is)
__device__ __forceinline__ float adam(const UpdateArgs &u, float w, float &m, float &v, float gr)
{
    m = fmaf(1.0f - u.b1, gr, u.b1 * m);
    v = fmaf((1.0f - u.b2) * gr, gr, u.b2 * v);
    return w - u.lr * (m / u.c1) / (sqrtf(v / u.c2) + u.eps);
}
__device__ __forceinline__ float adam_at(const UpdateArgs &u, int64_t at, float gr)
{
    float m = u.m[at], v = u.v[at];
    const float w = adam(u, u.w[at], m, v, gr);
    u.m[at] = m;
    u.v[at] = v;
    u.w[at] = w;
    return w;
}
// byte of (row, K index k) in a packed layer of `rows` rows and `chunks` core matrices of 8 x 8 to a slab
__device__ __forceinline__ int place(int r, int k, int rows, int chunks)
{
    const int k8 = k >> 3;
    return k8 / chunks * rows * chunks * 16 + ((r >> 3) * chunks + k8 % chunks) * 128 + (r & 7) * 16 + (k & 7) * 2;
}

__global__ void __launch_bounds__(kUpdThreads, 1) fused_update_kernel(const Update p)
{
    extern __shared__ __align__(128) unsigned char upd_smem[];
    __shared__ float part[8][kTM + 1];
    const int width = p.net.width, n_hidden = p.net.n_hidden, n_out = p.net.n_out, n_in = p.net.n_in;
    const int e = blockIdx.x / p.tiles;
    // the tile: layer l, outputs m0 .., inputs n0 ..
    const int mt = width / kTM, nt = (width + kTN - 1) / kTN;
    int t = blockIdx.x % p.tiles, l, fo, fi, m0, n0;
    if (t < (n_hidden - 1) * mt * nt) {
        l = 1 + t / (mt * nt);
        t %= mt * nt;
        fo = width, fi = width, m0 = t / nt * kTM, n0 = t % nt * kTN;
    } else if ((t -= (n_hidden - 1) * mt * nt) < nt) {
        l = n_hidden, fo = n_out, fi = width, m0 = 0, n0 = t * kTN;
    } else {
        l = 0, fo = width, fi = n_in, m0 = (t - nt) * kTM, n0 = 0;
    }
    const bool last = l == n_hidden, first = l == 0;
    const int M = min(fo - m0, kTM), N = first ? p.k0p : min(fi - n0, kTN);  // of the tile, multiples of 16
    // operands: 16-byte pieces of 8 rows of a column, a's and b's columns to 8 rows
    const int64_t R = (p.rows + 7) / 8;
    const uint4 *A = last ? reinterpret_cast<const uint4 *>(p.tr.dP) + e * R * n_out
                          : reinterpret_cast<const uint4 *>(p.tr.G[l]) + e * R * 2 * width + m0;
    const uint4 *B = first ? reinterpret_cast<const uint4 *>(p.tr.xb)
                           : reinterpret_cast<const uint4 *>(p.tr.H[l - 1]) + e * R * width + n0;
    const int a_cols = last ? n_out : 2 * width, b_cols = first ? p.k0p : width;
    const uint32_t ring = smem_u32(upd_smem);
    unsigned char *state = upd_smem + kRingBytes;
    const int slabs = (int)((p.rows + kTK - 1) / kTK);
    const int64_t at0 = e * p.net.P +
                        (first ? 0 : (int64_t)n_in * width + width + (int64_t)(l - 1) * ((int64_t)width * width + width));
    const auto load = [&](int s) {
        if (s >= slabs) return;
        const uint32_t a = ring + (s % kRing) * (kBytesA + kBytesB), b = a + kBytesA;
        {
            const int c = threadIdx.x % kTN, k = threadIdx.x / kTN;
            const int64_t rb = (int64_t)s * (kTK / 8) + k;
            if (c < N) cp16(b + (k * kTN + c) * 16, B + (rb < R ? rb : 0) * b_cols + c, rb < R);
        }
        const int c = threadIdx.x % kTM, k = threadIdx.x / kTM;
        const int64_t rb = (int64_t)s * (kTK / 8) + k;
        if (k < kTK / 8 && c < M) cp16(a + (k * kTM + c) * 16, A + (rb < R ? rb : 0) * a_cols + c, rb < R);
    };
    const auto commit = [] { asm volatile("cp.async.commit_group;\n" ::: "memory"); };

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int wm = (warp >> 2) * 16, wn = (warp & 3) * 32;
    const bool work = wm < M && wn < N;  // (half of a warp's 16 x 32 may lie outside: staged by nobody, never used)
    const bool bias = n0 == 0, db_here = bias && threadIdx.x < 4 * M;
    // ldmatrix: this lane's row of the four 8 x 8 matrices
    const int a_off = ((lane >> 4) * kTM + wm + ((lane >> 3) & 1) * 8 + (lane & 7)) * 16;
    const int b_off = (((lane >> 3) & 1) * kTN + wn + (lane >> 4) * 8 + (lane & 7)) * 16;
    const int db_f = threadIdx.x >> 2, db_r = threadIdx.x & 3;  // bias gradients: output, rows 2 db_r and the next, mod 8
    float acc[4][4] = {};
    float2 db = make_float2(0.0f, 0.0f);
    // the weights' state was last written before the launch before this one
    if (p.u.update && !first) {
        const uint32_t dst = smem_u32(state);
        for (int q = threadIdx.x; q < M * (N / 4); q += kUpdThreads) {
            const int r = q / (N / 4), c = q % (N / 4) * 4;
            const int64_t at = at0 + (int64_t)(m0 + r) * fi + n0 + c;
            const uint32_t d = dst + (r * kTN + c) * 4;
            cp16(d, p.u.w + at, true);
            cp16(d + kStateBytes, p.u.m + at, true);
            cp16(d + 2 * kStateBytes, p.u.v + at, true);
        }
    }
    pdl_wait();
    pdl_next();
    for (int s = 0; s < kRing - 1; ++s) {
        load(s);
        commit();
    }
    for (int s = 0; s < slabs; ++s) {
        asm volatile("cp.async.wait_group %0;\n" ::"n"(kRing - 2) : "memory");
        __syncthreads();  // slab s has landed for all, and all are done with slab s - 1, whose place is filled next
        load(s + kRing - 1);
        commit();
        const uint32_t a = ring + (s % kRing) * (kBytesA + kBytesB), b = a + kBytesA;
        if (work) {
#pragma unroll
            for (int ks = 0; ks < kTK / 8; ks += 2) {
                uint32_t af[4], bf[2][4];
                ldsm(af, a + ks * kTM * 16 + a_off);
#pragma unroll
                for (int j = 0; j < 2; ++j) ldsm(bf[j], b + (ks * kTN + j * 16) * 16 + b_off);
#pragma unroll
                for (int j = 0; j < 4; ++j)
                    asm volatile(
                        "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 "
                        "{%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};\n"
                        : "+f"(acc[j][0]), "+f"(acc[j][1]), "+f"(acc[j][2]), "+f"(acc[j][3])
                        : "r"(af[0]), "r"(af[1]), "r"(af[2]), "r"(af[3]), "r"(bf[j / 2][j % 2 * 2]),
                          "r"(bf[j / 2][j % 2 * 2 + 1]));
            }
        }
        if (db_here) {
            const unsigned char *z = upd_smem + (s % kRing) * (kBytesA + kBytesB) + db_f * 16 + db_r * 4;
#pragma unroll
            for (int k = 0; k < kTK / 8; ++k) {  // (rows past the batch are zero)
                const float2 v = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162 *>(z + k * kTM * 16));
                db.x += v.x;
                db.y += v.y;
            }
        }
    }
    asm volatile("cp.async.wait_all;\n" ::: "memory");
    __syncthreads();

    // the gradients, over the ring: each weight's step then reads and writes rows of the matrix in order
    float *G = reinterpret_cast<float *>(upd_smem);
    unsigned char *W = upd_smem + kTM * kPitchG * 4;
    if (work) {
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            float *g = G + (wm + (lane >> 2)) * kPitchG + wn + j * 8 + 2 * (lane & 3);
            *reinterpret_cast<float2 *>(g) = make_float2(acc[j][0], acc[j][1]);
            *reinterpret_cast<float2 *>(g + 8 * kPitchG) = make_float2(acc[j][2], acc[j][3]);
        }
    }
    if (db_here) {
        part[2 * db_r][db_f] = db.x;
        part[2 * db_r + 1][db_f] = db.y;
    }
    __syncthreads();
    if (bias && threadIdx.x < M) {
        float g = 0.0f;
#pragma unroll
        for (int k = 0; k < 8; ++k) g += part[k][threadIdx.x];
        const int64_t at = at0 + (int64_t)fi * fo + m0 + threadIdx.x;
        if (p.u.update) adam_at(p.u, at, g);
        else p.u.g[at] = g;
    }
    unsigned char *pk = p.u.packed + e * p.member_bytes;
    if (first) {
        for (int q = threadIdx.x; q < M * fi; q += kUpdThreads) {
            const int r = q / fi, c = q % fi;
            const int64_t at = at0 + (int64_t)m0 * fi + q;
            if (p.u.update)
                *reinterpret_cast<__nv_bfloat16 *>(pk + place(m0 + r, c, fo, p.k0p / 8)) =
                    __float2bfloat16(adam_at(p.u, at, G[r * kPitchG + c]));
            else
                p.u.g[at] = G[r * kPitchG + c];
        }
        return;
    }
    pk += first_bytes(p.k0p, width) + (int64_t)(l - 1) * width * width * 2;
    const int per_row = N / 4;
    for (int q = threadIdx.x; q < M * per_row; q += kUpdThreads) {
        const int r = q / per_row, c = q % per_row * 4;
        const int64_t at = at0 + (int64_t)(m0 + r) * fi + n0 + c;
        const float4 g = *reinterpret_cast<const float4 *>(G + r * kPitchG + c);
        if (!p.u.update) {
            *reinterpret_cast<float4 *>(p.u.g + at) = g;
            continue;
        }
        const unsigned char *s = state + (r * kTN + c) * 4;
        float4 w = *reinterpret_cast<const float4 *>(s), m = *reinterpret_cast<const float4 *>(s + kStateBytes),
               v = *reinterpret_cast<const float4 *>(s + 2 * kStateBytes);
        w.x = adam(p.u, w.x, m.x, v.x, g.x);
        w.y = adam(p.u, w.y, m.y, v.y, g.y);
        w.z = adam(p.u, w.z, m.z, v.z, g.z);
        w.w = adam(p.u, w.w, m.w, v.w, g.w);
        *reinterpret_cast<float4 *>(p.u.w + at) = w;
        *reinterpret_cast<float4 *>(p.u.m + at) = m;
        *reinterpret_cast<float4 *>(p.u.v + at) = v;
        __align__(8) __nv_bfloat162 h[2] = {__floats2bfloat162_rn(w.x, w.y), __floats2bfloat162_rn(w.z, w.w)};
        const uint2 hh = *reinterpret_cast<const uint2 *>(h);
        *reinterpret_cast<uint2 *>(pk + place(m0 + r, n0 + c, fo, kSlab / 8)) = hh;
        *reinterpret_cast<uint2 *>(W + (r * kPitchW + c) * 2) = hh;
    }
    if (!p.u.update) return;
    // the transpose, from the tile's new weights: 8 outputs of an input in 16 bytes
    __syncthreads();
    unsigned char *pt = p.u.packed_t + e * p.member_bytes_t;
    if (!last) pt += last_bytes(width, n_out) + (int64_t)(n_hidden - 1 - l) * width * width * 2;
    for (int q = threadIdx.x; q < M / 8 * N; q += kUpdThreads) {
        const int c = q % N, r = q / N * 8;
        __align__(16) __nv_bfloat16 h[8];
#pragma unroll
        for (int j = 0; j < 8; ++j) h[j] = *reinterpret_cast<const __nv_bfloat16 *>(W + ((r + j) * kPitchW + c) * 2);
        *reinterpret_cast<uint4 *>(pt + place(n0 + c, m0 + r, fi, last ? n_out / 8 : kSlab / 8)) =
            *reinterpret_cast<const uint4 *>(h);
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
    p.k0p = padded_inputs(n.n_in);
    const int mt = n.width / kTM, nt = (n.width + kTN - 1) / kTN;
    p.tiles = (n.n_hidden - 1) * mt * nt + nt + mt;
    p.member_bytes = fused_packed_bytes(n.n_in, n.width, n.n_hidden, n.n_out);
    p.member_bytes_t = fused_packed_t_bytes(n.width, n.n_hidden, n.n_out);
    const cudaError_t e = cudaFuncSetAttribute(fused_update_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kUpdSmem);
    if (e != cudaSuccess) return e;
    return pdl_launch(fused_update_kernel, p, p.tiles * n.n_members, kUpdThreads, kUpdSmem, true, st);
}

}  // namespace cpmmlp
