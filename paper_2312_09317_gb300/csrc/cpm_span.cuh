// Many rounds of one small lattice in one launch, by one thread-block cluster.
//
// A round of a small lattice is a few thousand attempts, far less than the GPU holds; what it costs
// is the chain from one round to the next.  With a launch per round that chain holds the launch, the
// fill of the SMs and the drain at the kernel's end.  Here a cluster of up to 16 CTAs stays on its
// SMs, the rounds are separated by the cluster's hardware barrier, and each thread draws its next
// attempt while it waits there.  A lattice whose attempts one CTA holds needs no cluster, and its
// words, tallies and flags stay in that CTA's shared memory from the first round to the last.
// us per round, with a launch each / in spans: 200^2 points 3.03 / 2.82, the same on areas of 40^2
// (25 attempts, resident) 2.20 / 1.25, motile cells of 256^2 5.3 / 4.3, 3D Act tissue of 256^3 on areas of
// 16^3 7.1 / 5.9, 3D Act cells of 64^3 on areas of 8^3 3.9 / 2.7.
// What is left of a round on a cluster is the release at its barrier (about 1,000 cycles until L2 has
// acknowledged the writes), two dependent L2 loads (the words of an attempt, then its window) and some
// 1,500 cycles of instructions.
#pragma once

#include "cpm_internal.h"
#include "cpm_round.cuh"

namespace cpmgb {
namespace {

constexpr uint32_t kSpanColours = 1024;  // sub-passes whose colours a CTA holds at a time

__device__ __forceinline__ uint32_t cluster_rank()
{
    uint32_t r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}

// The rounds p.sp, ... of n_sub sub-passes on the buffers l, by the nc CTAs of a cluster.
template <int DIM, bool PERIM, bool ACT, bool EXTRA, int G>
__device__ __forceinline__ void span_run(const RoundArgs &a, const LatticeBufs &l, const SpanPos &p, uint32_t nc,
                                         const SmemTables &sm, Survivors &q, uint16_t *colours)
{
    const uint32_t tid = threadIdx.x, rank = nc > 1 ? cluster_rank() : 0;
    const auto arrive = [&]() {
        __syncwarp();
        if (nc > 1) asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
    };
    const auto wait = [&]() {
        __syncwarp();
        if (nc > 1) asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
        else __syncthreads();
    };
    // colours of whole cycles from relative cycle c0 on (cycle 0: the one that holds sub-pass p.sp of MCS p.t)
    const uint32_t per_chunk = kSpanColours / p.C, cycles = p.per_mcs / p.C;
    const auto fill_colours = [&](uint32_t c0) {
        for (uint32_t j = tid; j < per_chunk; j += blockDim.x) {
            const uint32_t m = p.sp / p.C + c0 + j;
            uint16_t *out = colours + j * p.C;
            for (uint32_t c = 0; c < p.C; ++c)
                out[c] = (uint16_t)(c % a.c | (c / a.c % a.c) << 4 | (c / (a.c * a.c)) << 8);
            for (uint32_t i = p.C - 1; i >= 1; --i) {
                const Philox4 w = philox4x32_10(i, m % cycles, p.t + m / cycles, 1u << 24, a.key0, a.key1);
                const uint32_t o = draw_below(w.v[0], i + 1);
                const uint16_t tmp = out[i];
                out[i] = out[o];
                out[o] = tmp;
            }
        }
        __syncthreads();
    };

    uint32_t chunk = 0, at_chunk = 0, in_cycle = p.sp % p.C;  // cycle of the current sub-pass, place in it
    fill_colours(0);
    RoundPos pos;
    const auto set_colour = [&]() {
        const uint32_t col = colours[at_chunk * p.C + in_cycle];
        pos.cx = col & 15u;
        pos.cy = col >> 4 & 15u;
        pos.cz = col >> 8;
    };
    pos.t = p.t;
    pos.sp = p.sp;
    pos.r = 0;
    set_colour();

    // attempts: stripes of nc * p.lanes; a thread's block of the first stripe is the same in every round
    const uint32_t stripe = nc * p.lanes;
    const uint32_t i0 = rank * p.lanes + tid, x0 = i0 % a.nax, y0 = i0 / a.nax % a.nay, z0 = i0 / (a.nax * a.nay);
    bool valid = tid < p.lanes && i0 < a.n_active;
    Draw d{};
    if (valid) d = round_draw<DIM>(a, pos, x0, y0, z0, i0);
    uint32_t par = p.par, stage = 0;
    for (uint32_t left = p.n_sub; left > 0;) {
        // (a batch's kernel has ACT where any member has the term; the words of a member without it are plain ids)
        if (ACT && a.packed && pos.sp == 0 && pos.r == 0 && pos.t % 64 == 0) {
            const uint32_t n = a.nx * a.ny * a.nz;
            for (uint32_t x = rank * blockDim.x + tid; x < n; x += nc * blockDim.x) clamp_word(l.lat + x, pos.t & 255u);
            arrive();
            wait();
        }
        const RoundBufs b = round_bufs(l, par);
        for (uint32_t first = 0; first < a.n_active; first += stripe, ++stage) {
            if (first > 0) {
                __syncthreads();  // the previous stripe's survivors are done with
                const uint32_t i = first + i0;
                valid = tid < p.lanes && i < a.n_active;
                if (valid) d = round_draw<DIM>(a, pos, i % a.nax, i / a.nax % a.nay, i / (a.nax * a.nay), i);
            }
            // the warps without attempts of their own are the first to evaluate; the others draw their next ones
            round_cta<DIM, PERIM, ACT, EXTRA, G>(a, b, pos.t, sm, q, q.n[stage & 1u], valid, d, p.lanes / 32);
            if (tid == 0) q.n[(stage & 1u) ^ 1u] = 0;  // last read in the previous stage, used in the next
        }
        arrive();
        par ^= 1u;
        if (++pos.r == p.k) {
            pos.r = 0;
            --left;
            if (++pos.sp == p.per_mcs) {
                pos.sp = 0;
                ++pos.t;
            }
            if (++in_cycle == p.C) {
                in_cycle = 0;
                if (++at_chunk == per_chunk) {
                    at_chunk = 0;
                    chunk += per_chunk;
                    __syncthreads();  // every thread is done with the old colours
                    fill_colours(chunk);
                }
            }
            set_colour();
        }
        valid = tid < p.lanes && i0 < a.n_active;
        if (valid) d = round_draw<DIM>(a, pos, x0, y0, z0, i0);
        wait();
    }
}

// The lattice's words, tallies and flags in a CTA's shared memory: bytes, and the two copies.
struct SpanResident {
    int32_t *lat, *tal;
    uint8_t *flag;
};
__device__ __forceinline__ SpanResident span_resident(unsigned char *smem, uint32_t n_sites, uint32_t n_ids)
{
    SpanResident r;
    r.lat = reinterpret_cast<int32_t *>(smem);
    r.tal = r.lat + n_sites;
    r.flag = reinterpret_cast<uint8_t *>(r.tal + 4 * (size_t)n_ids);
    return r;
}
__device__ __forceinline__ void span_load(const SpanResident &r, const LatticeBufs &l, uint32_t n_sites, uint32_t n_ids,
                                          uint32_t n_active)
{
    for (uint32_t x = threadIdx.x; x < n_sites; x += blockDim.x) r.lat[x] = l.lat[x];
    for (uint32_t x = threadIdx.x; x < n_ids; x += blockDim.x) {
        r.tal[x] = l.V[0][x];
        r.tal[n_ids + x] = l.A[0][x];
        r.tal[2 * n_ids + x] = l.V[1][x];
        r.tal[3 * n_ids + x] = l.A[1][x];
    }
    for (uint32_t x = threadIdx.x; x < n_active; x += blockDim.x) {
        r.flag[x] = l.flag[0][x];
        r.flag[n_active + x] = l.flag[1][x];
    }
}
__device__ __forceinline__ void span_store(const SpanResident &r, const LatticeBufs &l, uint32_t n_sites, uint32_t n_ids,
                                           uint32_t n_active)
{
    for (uint32_t x = threadIdx.x; x < n_sites; x += blockDim.x) l.lat[x] = r.lat[x];
    for (uint32_t x = threadIdx.x; x < n_ids; x += blockDim.x) {
        l.V[0][x] = r.tal[x];
        l.A[0][x] = r.tal[n_ids + x];
        l.V[1][x] = r.tal[2 * n_ids + x];
        l.A[1][x] = r.tal[3 * n_ids + x];
    }
    for (uint32_t x = threadIdx.x; x < n_active; x += blockDim.x) {
        l.flag[0][x] = r.flag[x];
        l.flag[1][x] = r.flag[n_active + x];
    }
}
// the resident view of a lattice's buffers (pending changes and tracked sums stay in global memory)
__device__ __forceinline__ LatticeBufs span_view(const SpanResident &r, const LatticeBufs &l, uint32_t n_ids,
                                                 uint32_t n_active)
{
    LatticeBufs v = l;
    v.lat = r.lat;
    v.V[0] = r.tal;
    v.A[0] = r.tal + n_ids;
    v.V[1] = r.tal + 2 * n_ids;
    v.A[1] = r.tal + 3 * n_ids;
    v.flag[0] = r.flag;
    v.flag[1] = r.flag + n_active;
    return v;
}

// One lattice, a cluster of p.nc CTAs.
template <int DIM, bool PERIM, bool ACT, bool EXTRA>
__global__ void __launch_bounds__(kSpanThreads, 1) span_kernel(const RoundArgs a, const LatticeBufs l, const SpanPos p)
{
    extern __shared__ __align__(16) unsigned char span_smem[];
    __shared__ SmemTables sm;
    __shared__ Survivors q;
    __shared__ uint16_t colours[kSpanColours];
    __shared__ LatticeBufs view;
    load_tables(sm, a, ACT);
    if (threadIdx.x < 2) q.n[threadIdx.x] = 0;
    const uint32_t n_sites = a.nx * a.ny * a.nz, n_ids = (uint32_t)p.n_cells + 1;
    const SpanResident res = span_resident(span_smem, n_sites, n_ids);
    if (p.resident) span_load(res, l, n_sites, n_ids, a.n_active);
    if (threadIdx.x == 0) view = p.resident ? span_view(res, l, n_ids, a.n_active) : l;
    __syncthreads();
    span_run<DIM, PERIM, ACT, EXTRA, 8>(a, view, p, p.nc, sm, q, colours);
    if (p.resident) span_store(res, l, n_sites, n_ids, a.n_active);
}

template <int DIM, bool PERIM, bool ACT, bool EXTRA>
cudaError_t span_limits()
{
    auto kern = span_kernel<DIM, PERIM, ACT, EXTRA>;
    const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, kSpanMaxSmem);
    return e == cudaSuccess ? cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) : e;
}

inline void span_config(cudaLaunchConfig_t &cfg, cudaLaunchAttribute &attr, uint32_t nc, uint32_t threads)
{
    cfg.gridDim = dim3(nc);
    cfg.blockDim = dim3(threads);
    attr.id = cudaLaunchAttributeClusterDimension;
    attr.val.clusterDim.x = nc;
    attr.val.clusterDim.y = 1;
    attr.val.clusterDim.z = 1;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
}

// A cluster's CTAs share one of the GPU's SM groups; whether one has room for 16 is the GPU's affair, or that of the
// share of it that the process has.
template <int DIM, bool PERIM, bool ACT, bool EXTRA>
uint32_t span_cluster_t()
{
    uint32_t nc = span_limits<DIM, PERIM, ACT, EXTRA>() == cudaSuccess ? 16 : 1;
    for (; nc > 1; nc /= 2) {
        cudaLaunchConfig_t cfg = {};
        cudaLaunchAttribute attr = {};
        span_config(cfg, attr, nc, kSpanThreads);
        int n = 0;
        if (cudaOccupancyMaxActiveClusters(&n, span_kernel<DIM, PERIM, ACT, EXTRA>, &cfg) == cudaSuccess && n > 0) break;
    }
    if (nc < 16) cudaGetLastError();  // a refusal is an answer
    return nc;
}

template <int DIM, bool PERIM, bool ACT, bool EXTRA>
cudaError_t launch_span_t(const RoundArgs &a, const LatticeBufs &l, SpanPos p, cudaStream_t st)
{
    const cudaError_t e = span_limits<DIM, PERIM, ACT, EXTRA>();
    if (e != cudaSuccess) return e;
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute attr = {};
    span_config(cfg, attr, p.nc, p.threads);
    cfg.dynamicSmemBytes = p.resident;
    cfg.stream = st;
    return cudaLaunchKernelEx(&cfg, span_kernel<DIM, PERIM, ACT, EXTRA>, a, l, p);
}

// Members of a batch, a CTA each, n_mcs MCS of every member; the lattices are resident in shared memory.
// Members do not wait for one another, and a round costs its own chain instead of a launch. Registers:
// three CTAs of 256 per SM (80); with four (64) the spills cost more than the warps give, with two (128)
// too few members share an SM. us for 5 MCS of runs of 64 x 64 sites (80 rounds), 8 / 300 / 1,024 / 2,048
// members: 257 / 418 / 972 / 1,571; with a launch per round 403 / 664 / 1,239 / 1,987.
template <int DIM, bool PERIM, bool ACT, bool EXTRA>
__global__ void __launch_bounds__(kBatchSpanThreads, 3) batch_span_kernel(BatchLattice *lats, uint32_t n_mcs)
{
    extern __shared__ __align__(16) unsigned char span_smem[];
    __shared__ RoundArgs ra;
    __shared__ SmemTables sm;
    __shared__ Survivors q;
    __shared__ uint16_t colours[kSpanColours];
    __shared__ LatticeBufs view;
    BatchLattice &L = lats[blockIdx.x];
    for (uint32_t k = threadIdx.x; k < sizeof(RoundArgs) / sizeof(uint32_t); k += blockDim.x)
        reinterpret_cast<uint32_t *>(&ra)[k] = reinterpret_cast<const uint32_t *>(&L.base)[k];
    if (threadIdx.x < 2) q.n[threadIdx.x] = 0;
    __syncthreads();
    load_tables(sm, ra, ACT);
    const uint32_t n_sites = ra.nx * ra.ny * ra.nz, n_ids = (uint32_t)L.n_cells + 1;
    const SpanResident res = span_resident(span_smem, n_sites, n_ids);
    span_load(res, L.bufs, n_sites, n_ids, ra.n_active);
    if (threadIdx.x == 0) {
        view = span_view(res, L.bufs, n_ids, ra.n_active);
        ra.stream_loads = 0;  // the words are in shared memory
    }
    SpanPos p{};
    p.t = (uint32_t)L.t_start;
    p.per_mcs = L.R / L.k;
    p.C = L.C;
    p.k = L.k;
    p.n_sub = n_mcs * p.per_mcs;
    p.par = (uint32_t)(L.g_start & 1u);
    p.nc = 1;
    p.lanes = blockDim.x;
    __syncthreads();
    span_run<DIM, PERIM, ACT, EXTRA, 4>(ra, view, p, 1, sm, q, colours);
    span_store(res, L.bufs, n_sites, n_ids, ra.n_active);
    if (threadIdx.x == 0) {
        L.t_start += n_mcs;
        L.g_start += (uint64_t)n_mcs * L.R;
    }
}

template <int DIM, bool PERIM, bool ACT, bool EXTRA>
cudaError_t launch_batch_span_t(BatchLattice *lats, uint32_t n, uint32_t n_mcs, uint32_t threads, uint32_t smem,
                                cudaStream_t st)
{
    auto kern = batch_span_kernel<DIM, PERIM, ACT, EXTRA>;
    const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, kSpanMaxSmem);
    if (e != cudaSuccess) return e;
    kern<<<n, threads, smem, st>>>(lats, n_mcs);
    return cudaGetLastError();
}

template <int DIM>
cudaError_t launch_batch_span_d(bool perim, bool act, bool motile, BatchLattice *lats, uint32_t n, uint32_t n_mcs,
                                uint32_t threads, uint32_t smem, cudaStream_t st)
{
#define CPM_SPAN(PE, AC)                                                                     \
    (motile ? launch_batch_span_t<DIM, PE, AC, true>(lats, n, n_mcs, threads, smem, st)      \
            : launch_batch_span_t<DIM, PE, AC, false>(lats, n, n_mcs, threads, smem, st))
    if (act) return perim ? CPM_SPAN(true, true) : CPM_SPAN(false, true);
    return perim ? CPM_SPAN(true, false) : CPM_SPAN(false, false);
#undef CPM_SPAN
}

template <int DIM>
uint32_t span_cluster_d(bool perim, bool act, bool extra)
{
#define CPM_SPAN(PE, AC) (extra ? span_cluster_t<DIM, PE, AC, true>() : span_cluster_t<DIM, PE, AC, false>())
    if (act) return perim ? CPM_SPAN(true, true) : CPM_SPAN(false, true);
    return perim ? CPM_SPAN(true, false) : CPM_SPAN(false, false);
#undef CPM_SPAN
}

template <int DIM>
cudaError_t launch_span_d(bool perim, bool act, const RoundArgs &a, const LatticeBufs &l, const SpanPos &p,
                          cudaStream_t st)
{
    const bool extra = l.S[0] || a.chem || a.pers_dir;
#define CPM_SPAN(PE, AC) \
    (extra ? launch_span_t<DIM, PE, AC, true>(a, l, p, st) : launch_span_t<DIM, PE, AC, false>(a, l, p, st))
    if (act) return perim ? CPM_SPAN(true, true) : CPM_SPAN(false, true);
    return perim ? CPM_SPAN(true, false) : CPM_SPAN(false, false);
#undef CPM_SPAN
}

}  // namespace
}  // namespace cpmgb
