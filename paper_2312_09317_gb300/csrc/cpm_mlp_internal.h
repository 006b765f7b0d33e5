// Shared by the translation units of the emulator network.  Not part of the public C ABI.
#pragma once

#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <cstdint>

namespace cpmmlp {

// The whole forward pass of every member in one kernel (cpm_mlp_fused.cu): networks of n_hidden layers of
// `width` units, a multiple of 64 up to 256, at most 32 inputs, 16 or 32 outputs.
struct FusedNet {
    int n_members, n_in, width, n_hidden, n_out;
    const float *w;              // parameters, FP32 (biases)
    int64_t P;                   // per member
    const unsigned char *packed; // weights as fused_pack lays them out
};
constexpr int kFusedMaxHidden = 16;
inline int padded_inputs(int n_in) { return (n_in + 15) / 16 * 16; }  // K of the first layer
bool fused_fits(int n_in, int width, int n_out);
int64_t fused_packed_bytes(int n_in, int width, int n_hidden, int n_out);  // per member
cudaError_t fused_pack(const FusedNet &n, const __nv_bfloat16 *wb, unsigned char *packed, cudaStream_t st);
// out[e s_member + row n_out + k] of rows [0, rows) of X; err: set where a wait ran out; report_timeout: test hook
cudaError_t fused_forward(const FusedNet &n, const float *X, int64_t rows, float *out, int64_t s_member, int *err,
                          int report_timeout, cudaStream_t st);

// A training batch: rows order[off ..] (or off ..) of X and Y, its activations and gradients.
struct TrainArgs {
    const float *Y;
    const int32_t *order;
    int64_t off, n_total;
    // Operands of the weight gradients, 8 rows of a column in 16 bytes (R = rows / 8, rounded up; rows past the
    // batch are zero):
    __nv_bfloat16 *xb;                  // [R][inputs padded to 16][8]
    __nv_bfloat16 *H[kFusedMaxHidden];  // per hidden layer [member][R][width][8]: outputs
    float *G[kFusedMaxHidden];          // [member][R][2][width][4]: GELU'; the way back puts the bf16 gradients of
                                        // the pre-activations over the first half, [width][8]
    __nv_bfloat16 *dP;                  // [member][R][n_out][8]: gradient of the outputs
    float *loss;                        // per member, added to
    float inv;                          // 1 / (rows n_out)
    int *bad;                           // set where order[] points outside the data
    const unsigned char *packed_t;      // transposed weights (fused_pack_t)
    int64_t member_bytes_t;
    bool chained;                       // the launch before this one in the stream is a fused_update
};
int64_t fused_packed_t_bytes(int width, int n_hidden, int n_out);  // per member
cudaError_t fused_pack_t(const FusedNet &n, const __nv_bfloat16 *wb, unsigned char *packed_t, cudaStream_t st);
// forward and backward over a batch: xb, H, the gradients in G, dP and the losses
cudaError_t fused_train(const FusedNet &n, const TrainArgs &tr, const float *X, int64_t rows, int *err,
                        int report_timeout, cudaStream_t st);

// Where the gradients of a batch go: to g as they are, or (update) through an Adam step into the weights and
// both of their packed forms.
struct UpdateArgs {
    int update;
    float *g;
    float *w, *m, *v;
    unsigned char *packed, *packed_t;
    float lr, b1, b2, eps, c1, c2;
};
cudaError_t fused_update(const FusedNet &n, const TrainArgs &tr, const UpdateArgs &u, int64_t rows, cudaStream_t st);

#ifdef __CUDACC__

// Standard normal CDF Phi(z) = (1 + erf(z / sqrt 2)) / 2 and the density
// term exp(-z^2 / 2), with erf from the rational approximation of
// Abramowitz & Stegun, Handbook of Mathematical Functions, formula 7.1.26
// (after Hastings): for x >= 0,
//   erf(x) = 1 - (a1 t + a2 t^2 + a3 t^3 + a4 t^4 + a5 t^5) exp(-x^2) + e(x),
//   t = 1 / (1 + p x),  |e(x)| <= 1.5e-7,
// p = 0.3275911, a1..a5 = 0.254829592, -0.284496736, 1.421413741,
// -1.453152027, 1.061405429.  The reciprocal and the exponential are the
// fast hardware approximations.  With float32 rounding the |Phi error| stays
// below 4e-7 (the tests pin it on a dense grid against float64), far under
// the bf16 rounding (2^-9) of the activations that the epilogue stores.  The
// GELU epilogue is issue-bound, and this form is shorter than erff.
__device__ __forceinline__ float phi_f(float z, float &dens)
{
    const float x = fabsf(z) * 0.70710678118654752f;
    dens = __expf(-x * x);  // exp(-z^2 / 2)
    const float t = __fdividef(1.0f, fmaf(0.3275911f, x, 1.0f));
    float poly = 1.061405429f;
    poly = fmaf(poly, t, -1.453152027f);
    poly = fmaf(poly, t, 1.421413741f);
    poly = fmaf(poly, t, -0.284496736f);
    poly = fmaf(poly, t, 0.254829592f);
    const float half_tail = 0.5f * poly * t * dens;  // (1 - erf(x)) / 2
    return z >= 0.0f ? 1.0f - half_tail : half_tail;
}

__device__ __forceinline__ float gelu_f(float z)
{
    float dens;
    return z * phi_f(z, dens);
}

// Two GELUs at a time in packed FP32 (Blackwell's f32x2 instructions, half the issue slots).  The value is that of
// gelu_f, operation by operation, so that each result has its bits for |z| <= kGelu2Max (the tests compare all floats of
// that range); there exp(-z^2 / 2) is a normal number, so that exp2 and the reciprocal need none of the scaling that
// a subnormal result or a huge argument would.  The sign enters by two multiplications instead of a comparison and a
// selection: Phi = b - sigma h with (b, sigma) = (1, 1) for z >= 0 and (0, -1) below, exactly.
constexpr float kGelu2Max = 13.0f;
__device__ __forceinline__ uint64_t pack2(float a, float b)
{
    uint64_t r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
    return r;
}
__device__ __forceinline__ float2 unpack2(uint64_t r)
{
    float2 v;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(v.x), "=f"(v.y) : "l"(r));
    return v;
}
__device__ __forceinline__ uint64_t fma2(uint64_t a, uint64_t b, uint64_t c)
{
    uint64_t r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}
__device__ __forceinline__ uint64_t mul2(uint64_t a, uint64_t b)
{
    uint64_t r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ uint64_t add2(uint64_t a, uint64_t b)
{
    uint64_t r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ uint64_t both(float a) { return pack2(a, a); }
__device__ __forceinline__ float exp2_approx(float a)
{
    float r;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(a));
    return r;
}
__device__ __forceinline__ float rcp_approx(float a)
{
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(a));
    return r;
}
__device__ __forceinline__ float gelu_grad_f(float z)
{
    float dens;
    const float cdf = phi_f(z, dens);
    return cdf + z * 0.39894228040143268f * dens;
}

// with GRAD also the derivative, as gelu_grad_f
template <bool GRAD>
__device__ __forceinline__ uint64_t gelu2_f(uint64_t z, uint64_t &grad)
{
    constexpr uint64_t kAbs = 0x7fffffff7fffffffull, kSign = ~kAbs;
    const uint64_t xs = mul2(z, both(0.70710678118654752f));
    const float2 u = unpack2(fma2(both(0.3275911f), xs & kAbs, both(1.0f)));
    const float2 w = unpack2(mul2(mul2(xs, xs), both(-1.4426950408889634f)));  // log2 of exp(-z^2 / 2)
    const uint64_t dens = pack2(exp2_approx(w.x), exp2_approx(w.y)), t = pack2(rcp_approx(u.x), rcp_approx(u.y));
    uint64_t poly = fma2(both(1.061405429f), t, both(-1.453152027f));
    poly = fma2(poly, t, both(1.421413741f));
    poly = fma2(poly, t, both(-0.284496736f));
    poly = fma2(poly, t, both(0.254829592f));
    const uint64_t minus_h = mul2(mul2(mul2(both(-0.5f), poly), t), dens);
    const uint64_t one = (z & kSign) | 0x3f8000003f800000ull;  // +-1, the sign of z
    const uint64_t cdf = fma2(one, minus_h, fma2(one, both(0.5f), both(0.5f)));
    if (GRAD) grad = fma2(mul2(z, both(0.39894228040143268f)), dens, cdf);
    return mul2(z, cdf);
}
__device__ __forceinline__ uint64_t gelu2_f(uint64_t z)
{
    uint64_t grad;
    return gelu2_f<false>(z, grad);
}

constexpr uint32_t kTcSpinLimit = 1u << 22;

__device__ __forceinline__ uint32_t smem_u32(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ uint64_t tc_desc(uint32_t saddr, uint32_t lbo, uint32_t sbo)
{
    return (uint64_t)((saddr & 0x3FFFFu) >> 4) | ((uint64_t)((lbo >> 4) & 0x3FFFu) << 16) |
           ((uint64_t)((sbo >> 4) & 0x3FFFu) << 32) | (1ull << 46);
}

__device__ __forceinline__ bool tc_wait(uint64_t *mbar, uint32_t parity)
{
    const uint32_t addr = smem_u32(mbar);
    for (uint32_t it = 0; it < kTcSpinLimit; ++it) {
        uint32_t done;
        asm volatile("{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n"
                     " selp.u32 %0, 1, 0, p;\n}"
                     : "=r"(done)
                     : "r"(addr), "r"(parity)
                     : "memory");
        if (done) return true;
    }
    return false;
}

#endif

}  // namespace cpmmlp
