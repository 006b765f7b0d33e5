// Device kernels of the GB300 CPM sweep: one round of copy attempts over the
// blocks of the active checkerboard colour, plus the bookkeeping kernels
// (tally recount and comparison, Act stamp clamp, Act read-out).
//
// Every active block makes one copy attempt per round (Results, Fig. 3A: a
// barrier after every attempt; here the kernel boundary); cpm_round.cuh holds
// the attempt itself.
//
// Tallies are double-buffered so that every attempt of a round sees the
// tallies as they stood when the round began (deterministic form of the
// paper's atomic updates, Fig. 2B): round g reads buffer g&1 and adds both its
// own accepted changes and those of round g-1 into buffer (g+1)&1, which then
// equals the state after round g.  The change of round g-1 is carried in
// pend_prev, indexed by active-block number (equal for every colour); a
// one-byte flag per active block says whether it holds a change, so that
// only accepted copies (a few per cent) move a 16-byte entry.
#include <cstdint>

#include "cpm_internal.h"
#include "cpm_round.cuh"

namespace cpmgb {
namespace {

constexpr int kThreads = (int)kRoundThreads;
static_assert(kBatchMaxThreads == kRoundThreads, "the queue of survivors holds a CTA's attempts");

// wrapped coordinates x-1, x, x+1 along an axis of extent n
__device__ __forceinline__ void around(uint32_t x, uint32_t n, uint32_t out[3])
{
    out[0] = x == 0 ? n - 1 : x - 1;
    out[1] = x;
    out[2] = x + 1 == n ? 0 : x + 1;
}

// The attempts of one brick (kx, ky, kz) of active blocks by one CTA, a thread each (x fastest).
template <int DIM, bool PERIM, bool ACT, bool EXTRA, bool CUBED = false>
__device__ __forceinline__ void round_brick(const RoundArgs &a, const RoundBufs &b, const RoundPos &p,
                                            const SmemTables &sm, Survivors &q, uint32_t kx, uint32_t ky, uint32_t kz)
{
    const uint32_t lx = a.brick_lx, ly = a.brick_ly, slot = threadIdx.x;
    const uint32_t ix = (kx << lx) + (slot & ((1u << lx) - 1u));
    const uint32_t iy = (ky << ly) + ((slot >> lx) & ((1u << ly) - 1u));
    const uint32_t iz = DIM == 3 ? (kz << a.brick_lz) + (slot >> (lx + ly)) : 0;
    const bool valid = ix < a.nax && iy < a.nay && iz < a.naz;
    Draw d{};
    if (valid) d = round_draw<DIM, CUBED>(a, p, ix, iy, iz, ix + a.nax * (iy + a.nay * iz));
    round_cta<DIM, PERIM, ACT, EXTRA, 4, CUBED>(a, b, p.t, sm, q, q.n[0], valid, d);
}

// Resident CTAs per SM (register budget).  A round is bound by the instructions of its attempts and by
// the chain of dependent loads, so registers that hold a window's loads in flight are worth more than
// the warps they cost: 48 registers (five CTAs of 256) against 40 (six): 1024^3 fibre tissue in rows 145.5 /
// 165.0 ms per MCS, 256^3 cube cells 0.61 / 0.63 ms.
constexpr int kRoundMinBlocks = 5;

// EXTRA: composite variable tracking (b.Sc, b.Sn, b.tpend_* set), a field or persistence directions, a
// kernel of its own so that the sweep without them carries none of their code
template <int DIM, bool PERIM, bool ACT, bool EXTRA, bool CUBED>
__global__ void __launch_bounds__(kThreads, kRoundMinBlocks)
    round_kernel(const RoundArgs a, const RoundBufs b, const RoundPos p)
{
    __shared__ SmemTables sm;
    __shared__ Survivors queue;
    // the next round may place its CTAs on free SM slots from now on; they compute
    // their sites and random numbers, then wait for this round to finish
    if (a.pdl) asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    load_tables(sm, a, ACT);
    if (threadIdx.x == 0) queue.n[0] = 0;
    __syncthreads();
    uint32_t kx = blockIdx.x, ky = blockIdx.y, kz = blockIdx.z;
    if (a.nbr_x) {  // a linear grid (more bricks along y or z than a grid has blocks)
        kz = kx / (a.nbr_x * a.nbr_y);
        ky = kx / a.nbr_x % a.nbr_y;
        kx %= a.nbr_x;
    }
    round_brick<DIM, PERIM, ACT, EXTRA, CUBED>(a, b, p, sm, queue, kx, ky, kz);
}

// One (lattice, brick) item of batch round q: lattice it.x's round number
// g_start + q, exactly as the single-lattice round kernel would run it (same
// colour, counters and tallies).  ra, rb, rp, sm and queue are the CTA's shared set-up.
template <int DIM, bool PERIM, bool ACT, bool EXTRA>
__device__ __forceinline__ void batch_round_item(RoundArgs &ra, RoundBufs &rb, RoundPos &rp, SmemTables &sm,
                                                 Survivors &queue,
                                                 const BatchLattice *lats, int4 it, uint32_t q, uint32_t pdl)
{
    const BatchLattice &L = lats[it.x];
    __syncthreads();  // the previous item of this CTA is done with ra and sm
    static_assert(sizeof(RoundArgs) % sizeof(uint32_t) == 0, "copied in words");
    for (uint32_t k = threadIdx.x; k < sizeof(RoundArgs) / sizeof(uint32_t); k += blockDim.x)
        reinterpret_cast<uint32_t *>(&ra)[k] = reinterpret_cast<const uint32_t *>(&L.base)[k];
    __syncthreads();
    if (threadIdx.x == 0) {
        queue.n[0] = 0;
        // q is below R: the members of the round's items have that many rounds
        const uint32_t sp = q / L.k, r = q % L.k;
        const uint32_t col = L.colours[sp];
        rp.cx = col % ra.c;
        rp.cy = (col / ra.c) % ra.c;
        rp.cz = col / (ra.c * ra.c);
        rp.t = (uint32_t)L.t_start;
        rp.sp = sp;
        rp.r = r;
        ra.pdl = pdl;
        rb = round_bufs(L.bufs, (uint32_t)((L.g_start + q) & 1u));
    }
    load_tables(sm, ra, ACT);
    __syncthreads();
    round_brick<DIM, PERIM, ACT, EXTRA>(ra, rb, rp, sm, queue, (uint32_t)it.y, (uint32_t)it.z, (uint32_t)it.w);
}

// Batched round: every CTA takes one (lattice, brick) item.
// EXTRA: members keep tracked centroid sums (LatticeBufs::S), or have a field or persistence directions
template <int DIM, bool PERIM, bool ACT, bool EXTRA>
__global__ void __launch_bounds__(kBatchMaxThreads, kRoundMinBlocks)
    batch_round_kernel(const BatchLattice *lats, const int4 *items, uint32_t q)
{
    // the next round's CTAs may set up on free SM slots from now on; they wait before they read what a round writes
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    __shared__ RoundArgs ra;
    __shared__ RoundBufs rb;
    __shared__ RoundPos rp;
    __shared__ SmemTables sm;
    __shared__ Survivors queue;
    batch_round_item<DIM, PERIM, ACT, EXTRA>(ra, rb, rp, sm, queue, lats, items[blockIdx.x], q, 1);
}

// Colours of the sub-passes of one member's current MCS, one cycle per thread: a Fisher-Yates shuffle of
// the C colours per cycle, swap i (C-1 down to 1) drawn from counter (i, cycle, MCS, 1<<24).  Once per MCS,
// because the shuffle is a chain of C - 1 Philox calls that every CTA of every round would otherwise repeat
// before its first attempt.
__device__ __forceinline__ void batch_colours_member(const BatchLattice &L)
{
    const uint32_t cycles = L.R / (L.k * L.C);
    for (uint32_t cycle = threadIdx.x; cycle < cycles; cycle += blockDim.x) {
        uint8_t *out = L.colours + (size_t)cycle * L.C;
        for (uint32_t c = 0; c < L.C; ++c) out[c] = (uint8_t)c;
        for (uint32_t i = L.C - 1; i >= 1; --i) {
            const Philox4 w = philox4x32_10(i, cycle, (uint32_t)L.t_start, 1u << 24, L.base.key0, L.base.key1);
            const uint32_t j = draw_below(w.v[0], i + 1);
            const uint8_t tmp = out[i];
            out[i] = out[j];
            out[j] = tmp;
        }
    }
}

// Act stamp clamp of one (member, chunk of 65,536 sites) item, for a member
// whose MCS t_start is a multiple of 64 (run at the start of its MCS).
__device__ __forceinline__ void batch_clamp_item(const BatchLattice *lats, int2 it)
{
    const BatchLattice &L = lats[it.x];
    if (!L.base.packed || (L.t_start % 64) != 0) return;
    const uint64_t n = (uint64_t)L.base.nx * L.base.ny * L.base.nz;
    const uint32_t t8 = (uint32_t)L.t_start & 255u;
    const uint64_t lo = (uint64_t)it.y * 65536u, hi = lo + 65536u < n ? lo + 65536u : n;
    for (uint64_t x = lo + threadIdx.x; x < hi; x += blockDim.x) clamp_word(L.bufs.lat + x, t8);
}


__device__ __forceinline__ unsigned long long ld_acquire_gpu(const unsigned long long *p)
{
    unsigned long long v;
    asm volatile("ld.acquire.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
    return v;
}

// Grid-wide barrier of a co-resident (cooperative) grid on a 64-bit counter
// that starts at 0 (a call may pass billions of arrivals): the k-th barrier
// waits for k * gridDim.x arrivals.  The wait is bounded: after max_polls
// polls (about 100 ns apart) the CTA records the timeout in *err and the
// barrier returns false; the caller then returns.
__device__ __forceinline__ bool grid_barrier(unsigned long long *bar, unsigned long long target, long long max_polls,
                                             int *err, int &ok_s)
{
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();
        atomicAdd(bar, 1ull);
        int ok = 1;
        long long polls = 0;
        while (ld_acquire_gpu(bar) < target) {
            if (polls++ >= max_polls) {
                ok = 0;
                atomicExch(err, 1);
                break;
            }
            __nanosleep(100);
        }
        __threadfence();
        ok_s = ok;
    }
    __syncthreads();
    return ok_s != 0;
}

// The persistent batched MCS loop: n_mcs MCS of every member in one
// cooperative launch.  Per MCS: the colours and the Act clamp items, then rounds q = 0 ..
// r_max - 1 over the items of the members that still have rounds
// (upto_q[q] items), then the advance of every member's MCS and round
// counters, each phase closed by a grid barrier.  The work and its order
// within a phase are those of the per-round launches, so the result is the
// same bit for bit.
template <int DIM, bool PERIM, bool ACT, bool EXTRA>
__global__ void __launch_bounds__(kBatchMaxThreads, kRoundMinBlocks)
    batch_loop_kernel(BatchLattice *lats, uint32_t n_lats, const int4 *items, const uint32_t *upto_q, uint32_t r_max,
                      const int2 *clamp, uint32_t n_clamp, uint32_t n_mcs, unsigned long long *bar, unsigned *next,
                      long long max_polls, int *err, int test_absent)
{
    __shared__ RoundArgs ra;
    __shared__ RoundBufs rb;
    __shared__ RoundPos rp;
    __shared__ SmemTables sm;
    __shared__ Survivors queue;
    __shared__ int ok_s;
    __shared__ uint32_t claim_s;
    // test of the timeout path: the first CTA never arrives, so the others' first barrier wait runs out
    if (test_absent && blockIdx.x == 0) return;
    unsigned long long target = 0;
    for (uint32_t m = 0; m < n_mcs; ++m) {
        for (uint32_t l = blockIdx.x; l < n_lats; l += gridDim.x) batch_colours_member(lats[l]);
        if (ACT)
            for (uint32_t c = blockIdx.x; c < n_clamp; c += gridDim.x) batch_clamp_item(lats, clamp[c]);
        target += gridDim.x;
        if (!grid_barrier(bar, target, max_polls, err, ok_s)) return;
        for (uint32_t q = 0; q < r_max; ++q) {
            const uint32_t n_items = upto_q[q];
            // items are claimed one at a time from the round's counter, so that CTAs that drew cheap items
            // take more of them (a fixed grid-stride split leaves the round waiting for the unluckiest CTA)
            for (;;) {
                __syncthreads();
                if (threadIdx.x == 0) claim_s = atomicAdd(next + q, 1u);
                __syncthreads();
                const uint32_t k = claim_s;
                if (k >= n_items) break;
                batch_round_item<DIM, PERIM, ACT, EXTRA>(ra, rb, rp, sm, queue, lats, items[k], q, 0);
            }
            target += gridDim.x;
            if (!grid_barrier(bar, target, max_polls, err, ok_s)) return;
        }
        if (blockIdx.x == 0) {
            for (uint32_t l = threadIdx.x; l < n_lats; l += blockDim.x) {
                lats[l].t_start += 1;
                lats[l].g_start += lats[l].R;
            }
            for (uint32_t q = threadIdx.x; q < r_max; q += blockDim.x) next[q] = 0;  // the next MCS claims anew
        }
        target += gridDim.x;
        if (!grid_barrier(bar, target, max_polls, err, ok_s)) return;
    }
}

template <int DIM>
__global__ void recount_kernel(const int32_t *__restrict__ lat, int32_t *V, int32_t *A, uint32_t nx, uint32_t ny,
                               uint32_t nz, uint64_t n)
{
    for (uint64_t x = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; x < n; x += (uint64_t)gridDim.x * blockDim.x) {
        const int32_t s = cell_id(lat[x]);
        if (s <= 0) continue;
        const uint32_t px = (uint32_t)(x % nx), py = (uint32_t)((x / nx) % ny), pz = (uint32_t)(x / ((uint64_t)nx * ny));
        uint32_t xs[3], ys[3], zs[3];
        around(px, nx, xs);
        around(py, ny, ys);
        if (DIM == 3) around(pz, nz, zs); else zs[0] = zs[1] = zs[2] = 0;
        int cnt = 0;
        for (int dz = (DIM == 3 ? 0 : 1); dz < (DIM == 3 ? 3 : 2); ++dz)
            for (int dy = 0; dy < 3; ++dy)
                for (int dx = 0; dx < 3; ++dx) {
                    if (dx == 1 && dy == 1 && dz == 1) continue;
                    cnt += cell_id(lat[xs[dx] + nx * (ys[dy] + ny * zs[dz])]) != s;
                }
        atomicAdd(V + s, 1);
        atomicAdd(A + s, cnt);
    }
}

__global__ void compare_kernel(const int32_t *V, const int32_t *A, const int32_t *V2, const int32_t *A2, int32_t n,
                               unsigned long long *n_bad)
{
    for (int32_t k = blockIdx.x * blockDim.x + threadIdx.x; k < n; k += gridDim.x * blockDim.x)
        if (k > 0 && (V[k] != V2[k] || A[k] != A2[k])) atomicAdd(n_bad, 1ull);
}

__global__ void clamp_kernel(int32_t *lat, uint64_t n, uint32_t t)
{
    const uint32_t t8 = t & 255u;
    for (uint64_t x = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; x < n; x += (uint64_t)gridDim.x * blockDim.x)
        clamp_word(lat + x, t8);
}

__global__ void act_values_kernel(const int32_t *lat, const uint8_t *cell_type, TypeParams tp, uint64_t n,
                                  uint32_t t_last, uint8_t *out)
{
    for (uint64_t x = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; x < n; x += (uint64_t)gridDim.x * blockDim.x) {
        const int32_t w = lat[x];
        const int32_t s = cell_id(w);
        int v = 0;
        if (s > 0) v = act_value(word_stamp(w), t_last & 255u, tp.max_act[cell_type[s]]);
        out[x] = (uint8_t)v;
    }
}

__global__ void unpack_ids_kernel(const int32_t *lat, int32_t *ids, uint64_t n)
{
    for (uint64_t x = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; x < n; x += (uint64_t)gridDim.x * blockDim.x)
        ids[x] = cell_id(lat[x]);
}

__global__ void pack_ids_kernel(int32_t *lat, const int32_t *ids, const uint8_t *stamps, uint64_t n)
{
    for (uint64_t x = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; x < n; x += (uint64_t)gridDim.x * blockDim.x)
        lat[x] = pack_word(ids[x], stamps ? (uint32_t)stamps[x] : word_stamp(lat[x]));
}

unsigned grid_for(uint64_t n, unsigned threads)
{
    uint64_t g = (n + threads - 1) / threads;
    if (g > 152ull * 64) g = 152ull * 64;
    return (unsigned)(g == 0 ? 1 : g);
}

template <int DIM, bool PERIM, bool ACT, bool EXTRA, bool CUBED>
cudaError_t launch_round_t(RoundArgs a, const RoundBufs &b, const RoundPos &p, cudaStream_t st)
{
    const auto bricks = [](uint32_t n, uint32_t log2) { return (n + (1u << log2) - 1) >> log2; };
    const uint32_t kx = bricks(a.nax, a.brick_lx), ky = bricks(a.nay, a.brick_ly),
                   kz = DIM == 3 ? bricks(a.naz, a.brick_lz) : 1;
    dim3 blocks(kx, ky, kz);
    if (ky > 65535u || kz > 65535u) {
        a.nbr_x = kx;
        a.nbr_y = ky;
        blocks = dim3(kx * ky * kz);
    }
    const unsigned threads = 1u << (a.brick_lx + a.brick_ly + (DIM == 3 ? a.brick_lz : 0));
    if (!a.pdl) {
        round_kernel<DIM, PERIM, ACT, EXTRA, CUBED><<<blocks, threads, 0, st>>>(a, b, p);
        return cudaGetLastError();
    }
    // programmatic dependent launch: the CTAs of this round may start while the
    // previous kernel of the stream drains (it allows it once all its CTAs have
    // started); they wait for its completion before they touch the lattice
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = blocks;
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = 0;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, round_kernel<DIM, PERIM, ACT, EXTRA, CUBED>, a, b, p);
}

template <int DIM, bool PERIM, bool ACT>
cudaError_t launch_round_t(const RoundArgs &a, const RoundBufs &b, const RoundPos &p, cudaStream_t st)
{
    const bool extra = b.Sc || a.chem || a.pers_dir;
    if (DIM == 3 && a.cubed)
        return extra ? launch_round_t<DIM, PERIM, ACT, true, DIM == 3>(a, b, p, st)
                     : launch_round_t<DIM, PERIM, ACT, false, DIM == 3>(a, b, p, st);
    return extra ? launch_round_t<DIM, PERIM, ACT, true, false>(a, b, p, st)
                 : launch_round_t<DIM, PERIM, ACT, false, false>(a, b, p, st);
}

}  // namespace

cudaError_t launch_round(int dim, bool perim, bool act, const RoundArgs &a, const RoundBufs &b, const RoundPos &p,
                         cudaStream_t st)
{
    if (dim == 2) {
        if (act) return perim ? launch_round_t<2, true, true>(a, b, p, st) : launch_round_t<2, false, true>(a, b, p, st);
        return perim ? launch_round_t<2, true, false>(a, b, p, st) : launch_round_t<2, false, false>(a, b, p, st);
    }
    if (act) return perim ? launch_round_t<3, true, true>(a, b, p, st) : launch_round_t<3, false, true>(a, b, p, st);
    return perim ? launch_round_t<3, true, false>(a, b, p, st) : launch_round_t<3, false, false>(a, b, p, st);
}

__global__ void batch_clamp_kernel(const BatchLattice *lats, const int2 *items)
{
    batch_clamp_item(lats, items[blockIdx.x]);
}

__global__ void batch_colours_kernel(const BatchLattice *lats)
{
    batch_colours_member(lats[blockIdx.x]);
}

// End of one batch MCS: every member moves to its next MCS.
__global__ void batch_advance_kernel(BatchLattice *lats, uint32_t n)
{
    for (uint32_t l = blockIdx.x * blockDim.x + threadIdx.x; l < n; l += gridDim.x * blockDim.x) {
        lats[l].t_start += 1;
        lats[l].g_start += lats[l].R;
    }
}

cudaError_t launch_batch_clamp(const BatchLattice *lats, const int2 *items, uint32_t n_items, cudaStream_t st)
{
    if (n_items == 0) return cudaSuccess;
    batch_clamp_kernel<<<n_items, 256, 0, st>>>(lats, items);
    return cudaGetLastError();
}

cudaError_t launch_batch_colours(const BatchLattice *lats, uint32_t n, cudaStream_t st)
{
    if (n == 0) return cudaSuccess;
    batch_colours_kernel<<<n, 64, 0, st>>>(lats);
    return cudaGetLastError();
}

cudaError_t launch_batch_advance(BatchLattice *lats, uint32_t n, cudaStream_t st)
{
    batch_advance_kernel<<<(n + 255) / 256, 256, 0, st>>>(lats, n);
    return cudaGetLastError();
}

template <int DIM, bool PERIM, bool ACT, bool EXTRA>
cudaError_t launch_batch_loop_t(const BatchLoopArgs &p, uint32_t threads, cudaStream_t st, uint32_t *grid_out)
{
    auto kern = batch_loop_kernel<DIM, PERIM, ACT, EXTRA>;
    int dev = 0, sms = 0, per_sm = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, (int)threads, 0);
    if (e != cudaSuccess) return e;
    uint64_t grid = (uint64_t)sms * (uint64_t)(per_sm > 0 ? per_sm : 1);
    if (grid > p.max_items) grid = p.max_items;
    if (grid < 2 && p.test_absent) grid = 2;  // someone must wait for the absent CTA
    if (grid < 1) grid = 1;
    *grid_out = (uint32_t)grid;
    BatchLattice *lats = p.lats;
    uint32_t n_lats = p.n_lats, r_max = p.r_max, n_clamp = p.n_clamp, n_mcs = p.n_mcs;
    const int4 *items = p.items;
    const int2 *clamp = p.clamp;
    const uint32_t *upto = p.upto_q;
    unsigned long long *bar = p.bar;
    unsigned *next = p.next;
    long long polls = p.max_polls;
    int *err = p.err;
    int absent = p.test_absent;
    void *args[] = {&lats, &n_lats, &items, &upto, &r_max, &clamp, &n_clamp, &n_mcs, &bar, &next, &polls, &err,
                    &absent};
    return cudaLaunchCooperativeKernel((const void *)kern, dim3((unsigned)grid), dim3(threads), args, 0, st);
}

cudaError_t launch_batch_loop(int dim, bool perim, bool act, bool motile, const BatchLoopArgs &p, uint32_t threads,
                              cudaStream_t st, uint32_t *grid_out)
{
#define CPM_LOOP(D, PE, AC)                                                                                    \
    (motile ? launch_batch_loop_t<D, PE, AC, true>(p, threads, st, grid_out)                                   \
            : launch_batch_loop_t<D, PE, AC, false>(p, threads, st, grid_out))
    if (dim == 2) {
        if (act) return perim ? CPM_LOOP(2, true, true) : CPM_LOOP(2, false, true);
        return perim ? CPM_LOOP(2, true, false) : CPM_LOOP(2, false, false);
    }
    if (act) return perim ? CPM_LOOP(3, true, true) : CPM_LOOP(3, false, true);
    return perim ? CPM_LOOP(3, true, false) : CPM_LOOP(3, false, false);
#undef CPM_LOOP
}

template <int DIM, bool PERIM, bool ACT>
cudaError_t batch_round_t(bool extra, const BatchLattice *lats, const int4 *items, uint32_t n_items, uint32_t q,
                          uint32_t threads, bool after_round, cudaStream_t st)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(n_items);
    cfg.blockDim = dim3(threads);
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = after_round ? 1 : 0;
    return extra ? cudaLaunchKernelEx(&cfg, batch_round_kernel<DIM, PERIM, ACT, true>, lats, items, q)
                 : cudaLaunchKernelEx(&cfg, batch_round_kernel<DIM, PERIM, ACT, false>, lats, items, q);
}

cudaError_t launch_batch_round(int dim, bool perim, bool act, bool extra, const BatchLattice *lats,
                               const int4 *items, uint32_t n_items, uint32_t q, uint32_t threads, bool after_round,
                               cudaStream_t st)
{
    if (n_items == 0) return cudaSuccess;
    if (dim == 2) {
        if (act) return perim ? batch_round_t<2, true, true>(extra, lats, items, n_items, q, threads, after_round, st)
                              : batch_round_t<2, false, true>(extra, lats, items, n_items, q, threads, after_round, st);
        return perim ? batch_round_t<2, true, false>(extra, lats, items, n_items, q, threads, after_round, st)
                     : batch_round_t<2, false, false>(extra, lats, items, n_items, q, threads, after_round, st);
    }
    if (act) return perim ? batch_round_t<3, true, true>(extra, lats, items, n_items, q, threads, after_round, st)
                          : batch_round_t<3, false, true>(extra, lats, items, n_items, q, threads, after_round, st);
    return perim ? batch_round_t<3, true, false>(extra, lats, items, n_items, q, threads, after_round, st)
                 : batch_round_t<3, false, false>(extra, lats, items, n_items, q, threads, after_round, st);
}

cudaError_t launch_recount(int dim, const int32_t *lat, const uint8_t *, int32_t *V, int32_t *A, uint32_t nx,
                           uint32_t ny, uint32_t nz, cudaStream_t st)
{
    const uint64_t n = (uint64_t)nx * ny * nz;
    if (dim == 2)
        recount_kernel<2><<<grid_for(n, 256), 256, 0, st>>>(lat, V, A, nx, ny, nz, n);
    else
        recount_kernel<3><<<grid_for(n, 256), 256, 0, st>>>(lat, V, A, nx, ny, nz, n);
    return cudaGetLastError();
}

cudaError_t launch_compare(const int32_t *V, const int32_t *A, const int32_t *V2, const int32_t *A2, int32_t n,
                           unsigned long long *n_bad, cudaStream_t st)
{
    compare_kernel<<<grid_for((uint64_t)n, 256), 256, 0, st>>>(V, A, V2, A2, n, n_bad);
    return cudaGetLastError();
}

cudaError_t launch_clamp_stamps(int32_t *lat, uint64_t n, uint32_t t, cudaStream_t st)
{
    clamp_kernel<<<grid_for(n, 256), 256, 0, st>>>(lat, n, t);
    return cudaGetLastError();
}

// Rows to cubes (the layout of cubed_off) or back, 16 bytes a thread.  A warp has a quarter of a cube, a CTA those of
// eight cubes next to each other along x, so that both sides are read and written in whole lines.
__global__ void __launch_bounds__(256) cube_kernel(int4 *cubes, int4 *rows, uint32_t nx, uint32_t ny, uint32_t nz, int to_rows)
{
    const uint32_t kx = nx / 8, groups = (kx + 7) / 8, ky = ny / 8;
    const uint32_t quarter = blockIdx.x & 3u;
    const uint32_t x8 = (blockIdx.x >> 2) % groups * 8 + (threadIdx.x >> 5), y8 = (blockIdx.x >> 2) / groups % ky,
                   z8 = (blockIdx.x >> 2) / groups / ky;
    if (x8 >= kx) return;
    const uint32_t w = quarter * 32 + (threadIdx.x & 31u);  // of the cube's 128 pieces
    const uint32_t x = x8 * 8 + (w >> 2 & 1u) * 4, y = y8 * 8 + (w & 1u) + (w >> 3 & 3u) * 2,
                   z = z8 * 8 + (w >> 1 & 1u) + (w >> 5) * 2;
    const uint64_t cube = (x8 + (uint64_t)kx * (y8 + (uint64_t)ky * z8)) * 128 + w;
    const uint64_t row = (x + (uint64_t)nx * (y + (uint64_t)ny * z)) / 4;
    if (to_rows) __stcs(rows + row, __ldcs(cubes + cube));
    else __stcs(cubes + cube, __ldcs(rows + row));
}

cudaError_t launch_cubes(int32_t *cubes, int32_t *rows, uint32_t nx, uint32_t ny, uint32_t nz, bool to_rows, cudaStream_t st)
{
    const uint64_t blocks = (uint64_t)((nx / 8 + 7) / 8) * (ny / 8) * (nz / 8) * 4;
    cube_kernel<<<(unsigned)blocks, 256, 0, st>>>(reinterpret_cast<int4 *>(cubes), reinterpret_cast<int4 *>(rows), nx, ny,
                                                  nz, to_rows ? 1 : 0);
    return cudaGetLastError();
}

cudaError_t launch_act_values(const int32_t *lat, const uint8_t *cell_type, const TypeParams &tp, uint64_t n,
                              uint32_t t_last, uint8_t *out, cudaStream_t st)
{
    act_values_kernel<<<grid_for(n, 256), 256, 0, st>>>(lat, cell_type, tp, n, t_last, out);
    return cudaGetLastError();
}

cudaError_t launch_unpack_ids(const int32_t *lat, int32_t *ids, uint64_t n, cudaStream_t st)
{
    if (n == 0) return cudaSuccess;
    unpack_ids_kernel<<<grid_for(n, 256), 256, 0, st>>>(lat, ids, n);
    return cudaGetLastError();
}

cudaError_t launch_pack_ids(int32_t *lat, const int32_t *ids, const uint8_t *stamps, uint64_t n, cudaStream_t st)
{
    if (n == 0) return cudaSuccess;
    pack_ids_kernel<<<grid_for(n, 256), 256, 0, st>>>(lat, ids, stamps, n);
    return cudaGetLastError();
}

}  // namespace cpmgb
