// One round of copy attempts, as a warp runs it: shared by the single-lattice and the batched
// round kernels.
//
// The energy change follows the paper's Methods: Eq. 1 (adhesion over the Moore neighbourhood,
// each pair counted once; volume term), Eq. 3 (perimeter term) and Eq. 8/Eq. 9 (Act term,
// geometric mean), all in integers; Eq. 2 acceptance through the integer threshold table.
#pragma once

#include <cstdint>

#include "cpm_internal.h"

namespace cpmgb {
namespace {

// What the energy change needs of a type, in the order it is read (four 16-byte loads).
struct __align__(16) TypeRow {
    int32_t Ju, J0, Jf, lv2;  // adhesion with the cells' one type, the medium, obstacles; 2 lambda_V
    int64_t cvi, cvj;         // lambda_V (1 - 2 V_t) for the gaining cell, lambda_V (1 + 2 V_t) for the losing one
    int32_t lp, at2, la, ma;  // lambda_P, 2 A_t, lambda_Act, Max_Act
    uint32_t div_m, div_s;    // floor(u / Max_Act) = u div_m >> div_s for u < 2^30
    int32_t act_lo, gm_max;   // TypeParams::act_lo, gm_max
};
constexpr int kNoCell = kMaxTypes;  // the row of the medium: no volume, perimeter or Act term
constexpr int kMaxCount = 27;       // sites of a 3^3 window

struct SmemTables {
    TypeRow row[kMaxTypes + 1];
    int32_t J[kMaxTypes * kMaxTypes];
    int32_t act_hi[kMaxTypes * kMaxTypes];
    int32_t ln[kLnEntries];
    uint32_t inv[kMaxCount + 1];    // floor(n / d) = mulhi(2 n, inv[d]) for n < 2^31 / 27
};

__device__ __forceinline__ void load_tables(SmemTables &sm, const RoundArgs &a, bool with_act)
{
    for (int k = threadIdx.x; k < kMaxTypes * kMaxTypes; k += blockDim.x) {
        sm.J[k] = a.tp.J[k / kMaxTypes][k % kMaxTypes];
        if (with_act) sm.act_hi[k] = (int32_t)a.tp.act_hi[k / kMaxTypes][k % kMaxTypes];
    }
    if (threadIdx.x <= kNoCell) {
        const int k = threadIdx.x, t = k == kNoCell ? 0 : k;
        TypeRow r{};
        r.Ju = a.tp.J[t][a.uni];
        r.J0 = a.tp.J[t][0];
        r.Jf = a.tp.J[t][a.tp.obstacle_type];
        if (k != kNoCell) {
            const int64_t lv = a.tp.lambda_v[k], vt = a.tp.v_target[k];
            r.lv2 = (int32_t)(2u * (uint32_t)a.tp.lambda_v[k]);
            r.cvi = lv * (1 - 2 * vt);
            r.cvj = lv * (1 + 2 * vt);
            r.lp = a.tp.lambda_p[k];
            r.at2 = (int32_t)(2u * (uint32_t)a.tp.a_target[k]);
            if (with_act) {  // (Max_act in 0 .. 127: without Act it is any number, which nothing reads)
                r.la = a.tp.lambda_act[k];
                r.ma = a.tp.max_act[k];
                r.act_lo = (int32_t)a.tp.act_lo[k];
                r.gm_max = a.tp.gm_max[k];
                // M = ceil(2^(30+l) / Max) <= 2^31 with 2^l >= Max: the error u (M Max - 2^(30+l)) stays below 2^(30+l)
                uint32_t l = 0;
                while ((1 << l) < r.ma) ++l;
                r.div_s = 30 + l;
                r.div_m = r.ma > 0 ? (uint32_t)(((1ull << r.div_s) + r.ma - 1) / (uint32_t)r.ma) : 0u;
            }
        }
        sm.row[k] = r;
    }
    if (with_act) {
        for (int k = threadIdx.x; k < kLnEntries; k += blockDim.x) sm.ln[k] = a.ln_tab[k];
        // M = ceil(2^31 / d): the error 2 n (M d - 2^31) stays below 2^32 for n < 2^31 / 27
        for (uint32_t d = 1 + threadIdx.x; d <= kMaxCount; d += blockDim.x) sm.inv[d] = (0x80000000u + d - 1) / d;
    }
}

// Type of a lattice id.  When every cell has the same type (a.uni), it follows from the id alone,
// which takes the type table's load out of the chain of dependent loads of an attempt.
__device__ __forceinline__ int type_of(const RoundArgs &a, int32_t sigma)
{
    if (a.uni) return sigma > 0 ? (int)a.uni : (sigma < 0 ? a.tp.obstacle_type : 0);
    return sigma < 0 ? a.tp.obstacle_type : (int)__ldg(a.cell_type + sigma);
}

// x + d (d in -1, 0, 1) on a periodic axis of extent n, for x in [0, n)
__device__ __forceinline__ uint32_t wrap_step(uint32_t x, int d, uint32_t n)
{
    return d < 0 ? (x == 0 ? n - 1 : x - 1) : (d > 0 ? (x + 1 == n ? 0 : x + 1) : x);
}

// A lattice word of the round kernels.  With Act and areas of edge 8 or
// more, through the streaming cache path (ld.global.cs, evict first): the
// active blocks of a round are then 8 sites apart, a round touches each
// line of its stencils about once, and the tallies and type tables it also
// reads stay in L2 longer (4% faster on the 1024^3 tissue with a = 8).  With
// smaller areas the stencils of neighbouring blocks share lines and plain
// loads are faster (6% on the same tissue with a = 4).
template <bool ACT>
__device__ __forceinline__ int32_t lat_word(const RoundArgs &a, const RoundBufs &b, uint32_t site)
{
    return ACT && a.stream_loads ? __ldcs(b.lat + site) : b.lat[site];
}

// Act value of a site from its stamp: Max - age, clipped at 0.
__device__ __forceinline__ int act_value(uint32_t stamp, uint32_t t8, int max_act)
{
    const int age = (int)((t8 - stamp) & 255u);
    const int v = max_act - age;
    return v > 0 ? v : 0;
}

__device__ __noinline__ int64_t floor_div_pos(int64_t num, int64_t den)
{
    int64_t q = num / den;
    if (num % den != 0 && num < 0) q -= 1;
    return q;
}

// Energies in 64 bits, for any parameters; and in 32 bits with weights that RoundArgs::narrow admits, where a sum is
// clamped to +-2^30 once before the Act term is added.  With lambda_Act < 2^19 that term is at least -16 lambda_Act >
// -2^23 (the gaining cell's mean over its own Max_act) and at most 16 lambda_Act Max_j / Max_i, so with Max_act 1 and
// 127 at most 2032 lambda_Act <= 2^30 - 2^23 - 2032: no sum reaches 2^31, one clamped from above stays above 2^30 - 2^23
// and so above every threshold (below 2^22), and one clamped from below stays below 0, as the sums themselves do.
static_assert(16ll * 127 * ((1 << 19) - 1) < (1 << 30) - (1 << 23), "the Act term stays clear of a clamped sum");
struct Wide {
    using E = int64_t;
    __device__ __forceinline__ static E energy(int64_t h) { return h; }
    // floor(lambda_Act g / (4096 Max_Act))
    __device__ __forceinline__ static E act(const TypeRow &r, int32_t g)
    {
        return floor_div_pos((int64_t)r.la * g, (int64_t)r.ma * 4096);
    }
    __device__ __forceinline__ static E act_lo(const RoundArgs &a, const SmemTables &, int t) { return a.tp.act_lo[t]; }
    __device__ __forceinline__ static E act_hi(const RoundArgs &a, const SmemTables &, int t, int tj)
    {
        return a.tp.act_hi[t][tj];
    }
};
struct Narrow {
    using E = int32_t;
    __device__ __forceinline__ static E energy(int64_t h)
    {
        const int64_t m = 1 << 30;
        return (int32_t)(h > m ? m : (h < -m ? -m : h));
    }
    // floor(floor(lambda_Act g / 4096) / Max_Act): the inner quotient is below 2^30 in magnitude, a negative one is
    // divided as its complement
    __device__ __forceinline__ static E act(const TypeRow &r, int32_t g)
    {
        const int32_t q = (int32_t)(((int64_t)r.la * g) >> 12), s = q >> 31;
        return (int32_t)((uint64_t)(uint32_t)(q ^ s) * r.div_m >> r.div_s) ^ s;
    }
    __device__ __forceinline__ static E act_lo(const RoundArgs &, const SmemTables &sm, int t) { return sm.row[t].act_lo; }
    __device__ __forceinline__ static E act_hi(const RoundArgs &, const SmemTables &sm, int t, int tj)
    {
        return sm.act_hi[t * kMaxTypes + tj];
    }
};
// floor(sum / count) of an Act log-sum, as an index of EXPQ
__device__ __forceinline__ uint32_t mean_index(const SmemTables &sm, int32_t sum, int32_t count)
{
    return __umulhi(2u * (uint32_t)sum, sm.inv[count]) >> 6;
}

// the previous round's tracked change (see round_cta) into the other buffer
template <int DIM>
__device__ __noinline__ void track_carry(const RoundArgs &a, const RoundBufs &b, int32_t si, int32_t sj, int2 e)
{
    const uint32_t j = (uint32_t)e.x, bits = (uint32_t)e.y;
    const uint32_t jx = j % a.nx, jy = (j / a.nx) % a.ny, jz = j / (a.nx * a.ny);
#pragma unroll
    for (int d = 0; d < DIM; ++d) {
        const int64_t x = d == 0 ? jx : (d == 1 ? jy : jz);
        const int64_t n = d == 0 ? a.nx : (d == 1 ? a.ny : a.nz);
        if (si > 0) {
            const int64_t k = (int64_t)((bits >> (3 * d)) & 7u) - 3;
            atomicAdd((unsigned long long *)(b.Sn + 3 * si + d), (unsigned long long)(x + n * k));
        }
        if (sj > 0) {
            const int64_t k = (int64_t)((bits >> (9 + 3 * d)) & 7u) - 3;
            atomicAdd((unsigned long long *)(b.Sn + 3 * sj + d), (unsigned long long)(-(x + n * k)));
        }
    }
}

// An attempt that survived the early reject, handed from the lane that drew it to the group of four
// lanes that evaluates it.
struct __align__(16) Survivor {
    uint32_t i_dir;  // active index, and the stencil index (0..26) of the source above bit kDirShift
    uint32_t off;    // storage offset of the target
    uint32_t x, y, z;
    uint32_t w2;     // acceptance draw
    int32_t wi, wj;  // lattice words of source and target
};
constexpr uint32_t kRoundThreads = 256;  // most threads of a CTA, one attempt each
struct Survivors {
    Survivor at[kRoundThreads];
    uint32_t n[2];   // survivors so far; a loop over rounds clears one count while the other is in use
};
// n_active <= 2^31 / 27 in 3D and 2^31 / 9 in 2D, so the index and the direction share a word
template <int DIM>
constexpr int kDirShift = DIM == 3 ? 27 : 28;

// Storage offset of a site, and the step in it from coordinate v to v + d (d in -1, 0, 1) on an axis.
// CUBED (3D, extents multiples of 8): 8 x 8 x 8 cubes of 2 KB one after the other, x fastest, in each 4 x 2 x 2
// boxes of 64 bytes, so that a window lies in a few boxes of mostly one cube (see cpm_api.cu, run_cubed).
template <int AXIS>
__device__ __forceinline__ uint32_t cubed_off(const RoundArgs &a, uint32_t v)
{
    if (AXIS == 0) return (v & 3u) | (v & 4u) << 2 | (v >> 3) << 9;
    if (AXIS == 1) return ((v & 1u) << 2 | (v & 6u) << 4) + (v >> 3) * (64u * a.nx);
    return ((v & 1u) << 3 | (v & 6u) << 6) + (v >> 3) * (8u * a.nx * a.ny);
}
template <bool CUBED>
__device__ __forceinline__ uint32_t site_off(const RoundArgs &a, uint32_t x, uint32_t y, uint32_t z)
{
    if (CUBED) return cubed_off<0>(a, x) + cubed_off<1>(a, y) + cubed_off<2>(a, z);
    return x + a.nx * (y + a.ny * z);
}
template <int AXIS, bool CUBED>
__device__ __forceinline__ uint32_t axis_step(const RoundArgs &a, uint32_t v, int d)
{
    const uint32_t to = wrap_step(v, d, AXIS == 0 ? a.nx : (AXIS == 1 ? a.ny : a.nz));
    if (CUBED) return cubed_off<AXIS>(a, to) - cubed_off<AXIS>(a, v);
    return (to - v) * (AXIS == 0 ? 1u : (AXIS == 1 ? a.nx : a.nx * a.ny));
}

// The share of one lane (sub, of G = 4 or 8) in the 3^d window around a site without its centre:
// the eight columns (dx, dy) != (0, 0) are dealt out 8 / G to a lane, and in 3D lanes 0 and 1 also
// take the sites below and above the centre.  The columns are the lane's for good, so an offset is
// one addition of a column's and a plane's step, with no division and no shuffle per neighbour.
template <int DIM, int G, bool CUBED>
struct Window {
    static constexpr int COLS = 8 / G, K = DIM == 3 ? 3 * COLS + 1 : COLS;
    uint32_t col[COLS], below, above;  // steps of the columns and the planes
    __device__ __forceinline__ Window(const RoundArgs &a, uint32_t sub, uint32_t x, uint32_t y, uint32_t z)
    {
#pragma unroll
        for (int c = 0; c < COLS; ++c) {
            const uint32_t m = sub + (uint32_t)(G * c), idx = m + (m >= 4 ? 1u : 0u);  // skip the centre column
            const int dy = idx < 3 ? -1 : (idx < 6 ? 0 : 1), dx = (int)idx - 3 * dy - 4;
            col[c] = axis_step<0, CUBED>(a, x, dx) + axis_step<1, CUBED>(a, y, dy);
        }
        below = DIM == 3 ? axis_step<2, CUBED>(a, z, -1) : 0;
        above = DIM == 3 ? axis_step<2, CUBED>(a, z, 1) : 0;
    }
    // whether the lane has a k-th neighbour, and its offset from the centre
    __device__ __forceinline__ static bool has(int k, uint32_t sub) { return DIM == 2 || k < 3 * COLS || sub < 2; }
    __device__ __forceinline__ uint32_t step(int k, uint32_t sub) const
    {
        if (DIM == 2) return col[k];
        if (k == 3 * COLS) return sub == 0 ? below : above;
        return col[k / 3] + (k % 3 == 0 ? below : (k % 3 == 2 ? above : 0u));
    }
};

// sum over the G lanes of a group
template <int G>
__device__ __forceinline__ int32_t group_sum(int32_t v)
{
#pragma unroll
    for (int d = 1; d < G; d *= 2) v += __shfl_xor_sync(0xffffffffu, v, d);
    return v;
}

// The draws of one attempt: active block (ix, iy, iz), active index i, in the round p.
// Depends on the launch arguments only.
struct Draw {
    uint32_t i_dir, off, src, x, y, z, w2;
};
template <int DIM, bool CUBED = false>
__device__ __forceinline__ Draw round_draw(const RoundArgs &a, const RoundPos &p, uint32_t ix, uint32_t iy, uint32_t iz,
                                           uint32_t i)
{
    constexpr uint32_t NB = DIM == 3 ? 26 : 8;
    Draw d;
    const uint32_t bx = ix * a.c + p.cx, by = iy * a.c + p.cy, bz = DIM == 3 ? iz * a.c + p.cz : 0;
    const Philox4 w = philox4x32_10(bx + a.nbx * (by + a.nby * bz), p.r, p.t, p.sp, a.key0, a.key1);
    const uint32_t jl = draw_below(w.v[0], a.sd);
    if (a.s_log2 < 32) {
        d.x = (bx << a.s_log2) + (jl & (a.s - 1));
        d.y = (by << a.s_log2) + ((jl >> a.s_log2) & (a.s - 1));
        d.z = DIM == 3 ? (bz << a.s_log2) + (jl >> (2 * a.s_log2)) : 0;
    } else {
        d.x = bx * a.s + jl % a.s;
        d.y = by * a.s + (jl / a.s) % a.s;
        d.z = DIM == 3 ? bz * a.s + jl / (a.s * a.s) : 0;
    }
    const uint32_t n = draw_below(w.v[1], NB);
    const uint32_t idx = n + (n >= NB / 2 ? 1u : 0u);  // skip the centre of the 3^d stencil
    const int ox = (int)(idx % 3), oy = (int)((idx / 3) % 3), oz = DIM == 3 ? (int)(idx / 9) : 1;
    d.i_dir = i | (idx << kDirShift<DIM>);
    d.off = site_off<CUBED>(a, d.x, d.y, d.z);
    d.src = d.off + axis_step<0, CUBED>(a, d.x, ox - 1) + axis_step<1, CUBED>(a, d.y, oy - 1) +
            (DIM == 3 ? axis_step<2, CUBED>(a, d.z, oz - 1) : 0u);
    d.w2 = w.v[2];
    return d;
}

// One round's attempts of a CTA, one per thread with `valid` set.  Every thread of the CTA calls
// it; n_queue, a count in shared memory (one of q.n), is 0 on entry.
//
// Phase 1, one lane per attempt: the target's and source's words, the carry of the previous
// round's change, the early reject.  About a fifth of the attempts on a tissue survive.
// Phase 2, G lanes per survivor, 32 / G survivors per warp, dealt out over the warps of the CTA.
// With G = 4 a lane holds two of a window's eight columns, so that its loads (two in 2D, seven in
// 3D) are issued together, a survivor's sums are two shuffles, and the scalar part of the energy is
// paid once for eight survivors; G = 8 makes the chain of one survivor shorter where a CTA has
// warps to spare.  With one lane per attempt throughout, the window's loads wait for one
// another (registers), and a warp's instructions run for the fifth of its lanes that survived:
// 82 warp instructions per attempt on the 3D tissue, 10 of 32 lanes active.
// Measured against that (ms per MCS): 256^3 cube cells 0.911 -> 0.597, 1024^3 fibre tissue
// 189.2 -> 143.3 (in rows), 64 uneven lattices of a sweep 5.00 -> 2.90.  Eight lanes per survivor and a queue
// per warp: 0.976 and 180.7; two attempts per lane (half the warps): 1.46 and 336.
template <int DIM, bool PERIM, bool ACT, bool EXTRA, int G, bool CUBED = false>
__device__ __forceinline__ void round_cta(const RoundArgs &a, const RoundBufs &b, uint32_t t, const SmemTables &sm,
                                          Survivors &q, uint32_t &n_queue, bool valid, const Draw &d,
                                          uint32_t first_warp = 0)
{
    using Win = Window<DIM, G, CUBED>;
    static_assert(G == 4 || G == 8, "the four tallies take four lanes");
    constexpr int NB = DIM == 3 ? 26 : 8, K = Win::K;
    constexpr uint32_t kIndexMask = (1u << kDirShift<DIM>) - 1u;
    const uint32_t lane = threadIdx.x & 31u;
    // the warps take the survivors in turn, from first_warp on
    const uint32_t warp = (threadIdx.x >> 5) + (threadIdx.x >> 5 >= first_warp ? 0u : blockDim.x >> 5) - first_warp;
    const uint32_t t8 = t & 255u;

    // the lattice, flags and tallies read from here on are the previous round's output, so a round
    // launched as a programmatic dependent of the previous one waits for it here
    if (a.pdl) asm volatile("griddepcontrol.wait;" ::: "memory");
    {
        int32_t wj = 0, wi = 0;
        bool alive = false;
        if (valid) {
            const uint32_t i = d.i_dir & kIndexMask;
            const uint8_t flag = b.flag_prev[i];
            wj = lat_word<ACT>(a, b, d.off);
            wi = lat_word<ACT>(a, b, d.src);
            // the previous round's accepted change goes into the next tallies; its flag is cleared here, so that
            // the buffer is all 0 when the next round sets its own (most flags are never written)
            if (flag) {
                b.flag_prev[i] = 0;
                const int4 e = b.pend_prev[i];
                if (e.x > 0) { atomicAdd(b.Vn + e.x, 1); atomicAdd(b.An + e.x, e.z); }
                if (e.y > 0) { atomicAdd(b.Vn + e.y, -1); atomicAdd(b.An + e.y, e.w); }
                if (EXTRA && b.Sc) track_carry<DIM>(a, b, e.x, e.y, b.tpend_prev[i]);
            }
            const int32_t sj = cell_id(wj), si = cell_id(wi);
            alive = si != sj && si >= 0 && sj >= 0;
        }
        const unsigned m = __ballot_sync(0xffffffffu, alive);
        uint32_t first = 0;
        if (lane == 0 && m) first = atomicAdd(&n_queue, (uint32_t)__popc(m));
        first = __shfl_sync(0xffffffffu, first, 0);
        if (alive) {
            Survivor &s = q.at[first + (uint32_t)__popc(m & ((1u << lane) - 1u))];
            s.i_dir = d.i_dir;
            s.off = d.off;
            s.x = d.x;
            s.y = d.y;
            s.z = d.z;
            s.w2 = d.w2;
            s.wi = wi;
            s.wj = wj;
        }
    }
    __syncthreads();

    const uint32_t cnt = n_queue, sub = lane & (G - 1u);
    uint32_t accepted = 0;
    for (uint32_t base = (32 / G) * warp; base < cnt; base += blockDim.x / G) {
        const uint32_t e = base + lane / G;
        const bool on = e < cnt;
        const Survivor s = q.at[on ? e : base];  // a group without a survivor repeats a valid one, without effect
        const int32_t si = cell_id(s.wi), sj = cell_id(s.wj);
        // tallies of both cells: one load, a lane each
        int32_t tal = 0;
        if (sub < (PERIM ? 4u : 2u)) {
            const int32_t cell = sub & 1u ? sj : si;
            if (cell > 0) tal = (sub & 2u ? b.Ac : b.Vc)[cell];
        }
        const uint32_t dir = s.i_dir >> kDirShift<DIM>;
        const int ox = (int)(dir % 3), oy = (int)((dir / 3) % 3), oz = DIM == 3 ? (int)(dir / 9) : 1;
        // Motility (Eq. 4, Eq. 5) and tracked centroids (Eq. 11), read with the tallies: the field at the source by
        // lane 0, the moving cell's persistence direction by lane 1, the tracked sums of both cells by a lane per
        // cell and axis.
        constexpr int kSums = EXTRA ? (2 * DIM + G - 1) / G : 0;
        int32_t fx = 0, fy = 0, fz = 0;
        double hx = 0.0, hy = 0.0, hz = 0.0;
        int64_t sums[kSums > 0 ? kSums : 1];
        if (EXTRA) {
            const int32_t moving = si > 0 ? si : sj;
            if (a.chem && sub == 0) {
                const uint32_t isite = wrap_step(s.x, ox - 1, a.nx) +
                                       a.nx * (wrap_step(s.y, oy - 1, a.ny) +
                                               a.ny * (DIM == 3 ? wrap_step(s.z, oz - 1, a.nz) : 0));
                const int16_t *c = a.chem + (size_t)isite * DIM;
                fx = c[0];
                fy = c[1];
                if (DIM == 3) fz = c[2];
            }
            if (a.pers_dir && sub == 1 && moving > 0) {
                const double *p = a.pers_dir + 3 * (size_t)moving;
                hx = p[0];
                hy = p[1];
                if (DIM == 3) hz = p[2];
            }
#pragma unroll
            for (int k = 0; k < kSums; ++k) {
                const int at = (int)sub + k * G;  // cell at / DIM, axis at % DIM
                const int32_t cell = at < DIM ? si : sj;
                sums[k] = b.Sc && at < 2 * DIM && cell > 0 ? b.Sc[3 * cell + at % DIM] : 0;
            }
        }
        const Win win(a, sub, s.x, s.y, s.z);
        int32_t wn[K];
#pragma unroll
        for (int k = 0; k < K; ++k) wn[k] = Win::has(k, sub) ? lat_word<ACT>(a, b, s.off + win.step(k, sub)) : 0;
        const int ti = type_of(a, si), tj = type_of(a, sj);
        const TypeRow &ri = sm.row[si > 0 ? ti : kNoCell], &rj = sm.row[sj > 0 ? tj : kNoCell];
        // Counts of the neighbours in sigma_i, in sigma_j, in the medium and on obstacles, a byte each.
        // Target's Act log-sum over its same-cell window: 24 bits (at most 26 x LN[127]), the number of
        // zero Act values above them.
        const int maxj = ACT ? rj.ma : 0;
        int32_t counts = 0, lsj = 0;
#pragma unroll
        for (int k = 0; k < K; ++k) {
            const int32_t sn = cell_id(wn[k]);
            int32_t c = sn == si ? 1 : 0;
            if (sn == sj) c += 1 << 8;
            if (sn == 0) c += 1 << 16;
            if (sn < 0) c += 1 << 24;
            if (ACT && sn == sj && Win::has(k, sub)) {
                const int av = act_value(word_stamp(wn[k]), t8, maxj);
                lsj += av == 0 ? 1 << 24 : sm.ln[av];
            }
            counts += Win::has(k, sub) ? c : 0;
        }
        counts = group_sum<G>(counts);
        const int mi = counts & 255, mj = (counts >> 8) & 255;
        int32_t adhesion;
        if (a.uni) {
            // every cell has one type: the adhesion follows from the counts
            const int n0 = (counts >> 16) & 255, nf = (counts >> 24) & 255, nc = NB - n0 - nf;
            const TypeRow &Ji = sm.row[ti], &Jj = sm.row[tj];
            adhesion = Ji.Ju * (nc - (si > 0 ? mi : 0)) + Ji.J0 * (n0 - (si > 0 ? 0 : mi)) + Ji.Jf * nf;
            adhesion -= Jj.Ju * (nc - (sj > 0 ? mj : 0)) + Jj.J0 * (n0 - (sj > 0 ? 0 : mj)) + Jj.Jf * nf;
        } else {
            adhesion = 0;
#pragma unroll
            for (int k = 0; k < K; ++k)
                if (Win::has(k, sub)) {
                    const int32_t sn = cell_id(wn[k]);
                    const int tn = type_of(a, sn);
                    if (sn != si) adhesion += sm.J[ti * kMaxTypes + tn];
                    if (sn != sj) adhesion -= sm.J[tj * kMaxTypes + tn];
                }
            adhesion = group_sum<G>(adhesion);
        }
        const int32_t Vi = __shfl_sync(0xffffffffu, tal, 0, G), Vj = __shfl_sync(0xffffffffu, tal, 1, G);
        const int32_t Ai = PERIM ? __shfl_sync(0xffffffffu, tal, 2, G) : 0;
        const int32_t Aj = PERIM ? __shfl_sync(0xffffffffu, tal, 3, G) : 0;
        if (ACT) lsj = group_sum<G>(lsj);
        const int dAi = NB - 2 * mi, dAj = 2 * mj - NB;
        // a cell of type t that grows by a site: lambda_V (2 (V - V_t) + 1), that shrinks: lambda_V (1 - 2 (V - V_t));
        // its interfaces change by d: lambda_P d (2 (A - A_t) + d).  Products of 32-bit factors (RoundArgs::narrow
        // says that they are), sums in 64 bits.
        int64_t dh = adhesion;
        if (a.narrow) {
            dh += (int64_t)ri.lv2 * Vi + ri.cvi + rj.cvj - (int64_t)rj.lv2 * Vj;
            if (PERIM) {
                const int32_t pi = ri.lp * dAi, pj = rj.lp * dAj;
                dh += (int64_t)pi * (dAi - ri.at2) + (int64_t)(2 * pi) * Ai + (int64_t)pj * (dAj - rj.at2) +
                      (int64_t)(2 * pj) * Aj;
            }
        } else {
            if (si > 0) dh += (int64_t)a.tp.lambda_v[ti] * (2 * ((int64_t)Vi - a.tp.v_target[ti]) + 1);
            if (sj > 0) dh += (int64_t)a.tp.lambda_v[tj] * (1 - 2 * ((int64_t)Vj - a.tp.v_target[tj]));
            if (PERIM && si > 0)
                dh += (int64_t)a.tp.lambda_p[ti] * dAi * (2 * ((int64_t)Ai - a.tp.a_target[ti]) + dAi);
            if (PERIM && sj > 0)
                dh += (int64_t)a.tp.lambda_p[tj] * dAj * (2 * ((int64_t)Aj - a.tp.a_target[tj]) + dAj);
        }
        int64_t dhq = 16 * dh;
        if (EXTRA && (a.chem || a.pers_dir)) {
            // Each term, in 1/16 energy units, is floor(e) with e formed by the rounded double operations of the
            // replay, d = target - source: chemotaxis e = ((double)(-16 lambda (d . C)) / 16384) * (1/|d|),
            // persistence e = ((d_x p_x + d_y p_y + d_z p_z) * (double)(-16 lambda)) * (1/|d|).  Double precision is
            // what a round of motile cells waits for (64 results a warp instruction take an SM 16 cycles), so both
            // terms go through the same operations, lane 0's chemotaxis and lane 1's persistence; products with
            // d = -1, 0, 1 and the division by a power of two are exact (256^2 motile cells: 6.2 us a
            // round with each lane computing both in turn, 4.3 so).
            const int tp = si > 0 ? ti : tj;
            const int dx = 1 - ox, dy = 1 - oy, dz = DIM == 3 ? 1 - oz : 0;
            const bool chem = sub == 0;
            const auto times = [](int d, double x) { return d == 0 ? 0.0 : (d < 0 ? -x : x); };
            double v = __dadd_rn(times(dx, hx), times(dy, hy));
            if (DIM == 3) v = __dadd_rn(v, times(dz, hz));
            const int64_t along = (int64_t)dx * fx + (int64_t)dy * fy + (int64_t)dz * fz;
            const double w = (double)(chem ? -16 * (int64_t)a.tp.lambda_chem[tp] * along
                                           : -16 * (int64_t)a.tp.lambda_pers[tp]);
            const double e = __dmul_rn(__dmul_rn(chem ? 1.0 / 16384.0 : v, w), a.tp.inv_len[dx * dx + dy * dy + dz * dz]);
            const int64_t term = (int64_t)floor(e);
            dhq += __shfl_sync(0xffffffffu, term, 0, G) + __shfl_sync(0xffffffffu, term, 1, G);
        }
        // the test of Eq. 2 at an energy h > 0 (w2 < THR[h]): THR[h] = floor(2^32 exp(-h / 16T)), so it
        // holds exactly for h <= 16 T ln(2^32 / (w2 + 1)).  The logarithm in single precision decides all
        // h but the few within a.h_eps (over ten times its error bound) of that value, for which the
        // table is read; a test thus mostly ends without another dependent load.
        const float hs = a.h_scale * (32.0f - __log2f((float)s.w2 + 1.0f));
        const int32_t h_lo = (int32_t)floorf(hs - a.h_eps), h_hi = (int32_t)ceilf(hs + a.h_eps);
        const auto below = [&](auto h) {
            if (h <= h_lo) return true;
            if (h > h_hi) return false;
            return h < a.L && s.w2 < __ldg(a.thr + h);
        };
        const bool barred = !on || (sj > 0 && Vj <= 1);  // no survivor, or a cell's last site
        const auto test = [&](auto arith) {
            using Ar = decltype(arith);
            using E = typename Ar::E;
            E h = Ar::energy(dhq);
            int decided = barred ? 0 : -1;  // 1 accept, 0 reject, -1 open
            if (ACT) {
                const int tp = si > 0 ? ti : tj;
                const TypeRow &rm = sm.row[tp];  // of the moving cell
                bool window = false;             // the source's window is needed
                int32_t gj = 0;
                if (decided < 0 && rm.la != 0 && rm.ma != 0) {
                    // the Act term lies in [act_lo, act_hi] = [floor(-lam Gmax_i / (Max 4096)), floor(lam Gmax_j /
                    // (Max 4096))] (GM in [0, Gmax] per cell, lambda >= 0); when every value in that range gives the
                    // same outcome of the test (THR is non-increasing), the geometric means are not needed
                    const E lo = h + (si > 0 ? Ar::act_lo(a, sm, ti) : 0), hi = h + (sj > 0 ? Ar::act_hi(a, sm, tp, tj) : 0);
                    if (hi <= 0) decided = 1;
                    else if (lo > 0 && !below(lo)) decided = 0;
                    else if (below(hi)) decided = 1;
                    else {
                        // target: the log-sum gathered above (the centre and the mj same-cell neighbours; 0 when any
                        // of their Act values is 0)
                        if (sj > 0) {
                            const int cv = act_value(word_stamp(s.wj), t8, maxj);
                            if (cv != 0 && lsj < 1 << 24) gj = __ldg(a.expq + mean_index(sm, lsj + sm.ln[cv], mj + 1));
                        }
                        // the same with the target's mean known: [floor(lam (G_j - Gmax_i) / ..), floor(lam G_j / ..)]
                        const E hi1 = h + Ar::act(rm, gj), lo1 = h + Ar::act(rm, gj - ri.gm_max);
                        if (hi1 <= 0 || below(hi1)) decided = 1;
                        else if (lo1 > 0 && !below(lo1)) decided = 0;
                        else window = true;  // si > 0: otherwise lo1 = hi1, and one of the two holds
                    }
                }
                if (__any_sync(0xffffffffu, window)) {
                    const uint32_t xi = wrap_step(s.x, ox - 1, a.nx), yi = wrap_step(s.y, oy - 1, a.ny);
                    const uint32_t zi = DIM == 3 ? wrap_step(s.z, oz - 1, a.nz) : 0;
                    const uint32_t src = site_off<CUBED>(a, xi, yi, zi);
                    const Win win_i(a, sub, xi, yi, zi);
#pragma unroll
                    for (int k = 0; k < K; ++k)
                        wn[k] = window && Win::has(k, sub) ? lat_word<ACT>(a, b, src + win_i.step(k, sub)) : 0;
                    int32_t ci = 0, lsi = 0;
#pragma unroll
                    for (int k = 0; k < K; ++k)
                        if (Win::has(k, sub) && cell_id(wn[k]) == si) {
                            const int av = act_value(word_stamp(wn[k]), t8, ri.ma);
                            ci += 1;
                            lsi += av == 0 ? 1 << 24 : sm.ln[av];
                        }
                    ci = group_sum<G>(ci);
                    lsi = group_sum<G>(lsi);
                    if (window) {
                        int32_t gi = 0;
                        const int cv = act_value(word_stamp(s.wi), t8, ri.ma);
                        if (cv != 0 && lsi < 1 << 24) gi = __ldg(a.expq + mean_index(sm, lsi + sm.ln[cv], ci + 1));
                        h += Ar::act(rm, gj - gi);
                    }
                }
            }
            return decided >= 0 ? decided == 1 : (h <= 0 || below(h));
        };
        const bool ok = a.narrow ? test(Narrow{}) : test(Wide{});
        const bool leader = sub == 0 && ok;
        int32_t shifts = 0;
        if (EXTRA && b.Sc) {
            // The copy adds its site to sigma_i's sums and removes it from sigma_j's, at the periodic image nearest
            // that cell's centroid as the round began; the image shifts (-3..3 per axis, 3 bits each: sigma_i's in
            // bits 0..8, sigma_j's in bits 9..17) travel with the pending change, so that the next round adds the
            // same amounts to the other buffer.
#pragma unroll
            for (int k = 0; k < kSums; ++k) {
                const int at = (int)sub + k * G, d = at % DIM;
                const bool of_i = at < DIM;
                const int32_t cell = of_i ? si : sj;
                if (!ok || at >= 2 * DIM || cell <= 0) continue;
                const int64_t x = d == 0 ? s.x : (d == 1 ? s.y : s.z), n = d == 0 ? a.nx : (d == 1 ? a.ny : a.nz);
                const int64_t shift = track_image_shift(x, sums[k], of_i ? Vi : Vj, n), image = x + n * shift;
                atomicAdd((unsigned long long *)(b.Sn + 3 * cell + d), (unsigned long long)(of_i ? image : -image));
                shifts |= (int32_t)(shift + 3) << ((of_i ? 0 : 9) + 3 * d);
            }
            shifts = group_sum<G>(shifts);
        }
        if (leader) {
            const uint32_t i = s.i_dir & kIndexMask;
            // a copy stamps the site with this MCS (a medium copy: age 128, no activity)
            b.lat[s.off] = ACT && a.packed ? pack_word(si, si > 0 ? t8 : ((t - 128u) & 255u)) : si;
            if (si > 0) { atomicAdd(b.Vn + si, 1); atomicAdd(b.An + si, dAi); }
            if (sj > 0) { atomicAdd(b.Vn + sj, -1); atomicAdd(b.An + sj, dAj); }
            b.pend_cur[i] = make_int4(si, sj, dAi, dAj);
            b.flag_cur[i] = 1;
            if (EXTRA && b.Sc) b.tpend_cur[i] = make_int2((int32_t)(s.x + a.nx * (s.y + a.ny * s.z)), shifts);
        }
        accepted += (uint32_t)__popc(__ballot_sync(0xffffffffu, leader));
    }
    if (lane == 0 && accepted != 0) atomicAdd(a.accepts, (unsigned long long)accepted);
}

// Stamps whose age is 128 or more are reset to age exactly 128, so that ages
// stay below 256 until the next clamp (run every 64 MCS).  Obstacle words are
// left as they are (their stamp is never read).
__device__ __forceinline__ void clamp_word(int32_t *p, uint32_t t8)
{
    const int32_t w = *p;
    if (cell_id(w) < 0) return;
    const uint32_t age = (t8 - word_stamp(w)) & 255u;
    if (age >= 128u) *p = pack_word(cell_id(w), (t8 - 128u) & 255u);
}

}  // namespace
}  // namespace cpmgb
