// Observations of a batch of lattices and the summary statistics made of
// them.  Observations: per cell its
// anchor (first site in raster order), volume, integer sums of the
// minimal-image offsets of its sites from the anchor (a centroid in one
// periodic image, Methods, "Composite variable tracking", Eq. 10), their
// second moments (cell shape) and its interface count (Eq. 3); per lattice the cell-medium neighbour pairs and
// the accepted copies so far.
//
// A thread walks along the slowest axis and keeps the sums of the cell it is in.
#include <cuda_runtime.h>

#include <cstdint>

#include "cpm_internal.h"

namespace cpmgb {
namespace {

constexpr int kObsThreads = 256;
constexpr double kArrestSpeed = 0.05;  // sites / MCS over a 50-MCS sub-track

__device__ __forceinline__ int min_image(int d, int n)
{
    // d in (-n, n); result in [-n/2, n - n/2)
    d += n / 2;
    if (d >= n) d -= n;
    if (d < 0) d += n;
    return d - n / 2;
}

__global__ void observe_init_kernel(const ObserveItem *items, int64_t *cells, int64_t *member)
{
    const ObserveItem it = items[blockIdx.x];
    for (int64_t r = threadIdx.x; r <= it.n_cells; r += blockDim.x) {
        int64_t *row = cells + (it.row0 + r) * kObsFields;
        row[0] = -1;  // all ones: the identity of the unsigned minimum
        for (int f = 1; f < kObsFields; ++f) row[f] = 0;
    }
    if (threadIdx.x == 0) {
        member[2 * blockIdx.x] = 0;
        member[2 * blockIdx.x + 1] = (int64_t)*it.accepts;
    }
}

// A walk: the sites (x, y) of a chunk of kWalk planes in 3D, x of a chunk of kWalk rows in 2D.  Threads
// next to each other walk next to each other along x.
constexpr uint32_t kWalk = 16;
struct Walk {
    uint32_t site, step, lo, hi;  // first site, distance to the next, extent [lo, hi) along the walked axis
    uint32_t x, y;                // the fixed coordinates (y: 3D only)
};
template <int DIM>
__device__ __forceinline__ uint32_t walk_count(const ObserveItem &it)
{
    return DIM == 3 ? it.nx * it.ny * ((it.nz + kWalk - 1) / kWalk) : it.nx * ((it.ny + kWalk - 1) / kWalk);
}
template <int DIM>
__device__ __forceinline__ Walk walk_of(const ObserveItem &it, uint32_t w)
{
    Walk r;
    r.x = w % it.nx;
    r.y = DIM == 3 ? w / it.nx % it.ny : 0;
    const uint32_t chunk = w / (DIM == 3 ? it.nx * it.ny : it.nx), n = DIM == 3 ? it.nz : it.ny;
    r.step = DIM == 3 ? it.nx * it.ny : it.nx;
    r.lo = chunk * kWalk;
    r.hi = r.lo + kWalk < n ? r.lo + kWalk : n;
    r.site = r.x + it.nx * r.y + r.step * r.lo;
    return r;
}
__device__ __forceinline__ int observed_id(const ObserveItem &it, uint32_t site)
{
    const int id = cell_id(it.lat[site]);
    return id > it.n_cells ? 0 : id;  // never above in a validated lattice; keeps the writes in bounds
}

// Along a walk the first site of a run of one cell has its lowest index.
template <int DIM>
__global__ void __launch_bounds__(kObsThreads) observe_anchor_kernel(const ObserveItem *items, int64_t *cells)
{
    const ObserveItem it = items[blockIdx.y];
    const uint32_t n = walk_count<DIM>(it);
    for (uint32_t w = blockIdx.x * blockDim.x + threadIdx.x; w < n; w += gridDim.x * blockDim.x) {
        const Walk k = walk_of<DIM>(it, w);
        int last = 0;
        uint32_t site = k.site;
        for (uint32_t z = k.lo; z < k.hi; ++z, site += k.step) {
            const int id = observed_id(it, site);
            if (id > 0 && id != last) {
                unsigned long long *a = reinterpret_cast<unsigned long long *>(cells + (it.row0 + id) * kObsFields);
                if (*reinterpret_cast<volatile unsigned long long *>(a) > site) atomicMin(a, (unsigned long long)site);
            }
            last = id;
        }
    }
}

// a / n for a < 2^31 by a multiplication: 2^(31 + l) / n rounded up, 2^l >= n, errs by less than 2^l / n of what
// would change the quotient (Granlund & Montgomery 1994)
struct Inverse {
    uint32_t mul, shift;
};
__device__ __forceinline__ Inverse inverse_of(uint32_t n)
{
    const uint32_t l = 32 - __clz(n - 1);
    return {(uint32_t)((1ull << (31 + l)) / n + 1), 31 + l};
}
__device__ __forceinline__ uint32_t quotient_of(uint32_t a, Inverse i)
{
    return (uint32_t)(((uint64_t)a * i.mul) >> i.shift);
}

// The sums of every cell.  A thread keeps the sums of the run at hand (sites of one cell next to each other
// along its walk) in registers: with the walk's coordinates fixed, a site costs the sums of its offset along the
// walk and the comparisons with its neighbours, of which each step loads only the plane (3D: nine words) or row
// (three) that comes into the window and counts the run's cell in it once.  In 3D the runs that have ended wait
// until a lane ends its second; then those of the warp are reduced cell by cell and added, a lane per field, to
// the CTA's sums in shared memory, which go to the cells after each set of walks.  Bound by instructions (127 a
// step of a warp, half of the slots used).  Sweep of 64 uneven lattices, the 32 in 3D (70 M sites): 413 us; with
// every run added to its cell at once, and the whole window compared at each step, 564.  Before walks, with a
// site per thread and twelve group reductions per site and group: 1.05 ms for the sweep's observation, 0.70 with
// walks; 1,024 runs of 64^2 sites 148 and 62 us.
constexpr int kObsSlots = 128;      // cells whose sums a CTA holds
constexpr int kSharedExtent = 1024; // the 32-bit sums of 4,096 sites hold offsets of lattices up to this extent
constexpr int kFarOffset = 11585;   // a run's 32-bit sum holds the squares of kWalk offsets up to this one
// FAR: some lattice has larger offsets along the walk (a variant of its own: the test of every offset costs 4%)
template <int DIM, bool FAR>
__global__ void __launch_bounds__(kObsThreads, DIM == 3 ? 3 : 4)
    observe_sums_kernel(const ObserveItem *items, int64_t *cells, int64_t *member)
{
    constexpr int P = DIM == 3 ? 9 : 3;  // sites of a window's plane
    constexpr int F = kObsFields - 1;    // sums of a cell, fields 1 ..
    __shared__ int keys[kObsSlots], sums[kObsSlots][F];
    const ObserveItem it = items[blockIdx.y];
    const int nx = (int)it.nx, ny = (int)it.ny, nz = (int)it.nz, nw = DIM == 3 ? nz : ny;
    const bool shared = DIM == 3 && nx <= kSharedExtent && ny <= kSharedExtent && nz <= kSharedExtent;
    const uint32_t n = walk_count<DIM>(it);
    const Inverse inv_x = inverse_of(it.nx), inv_y = inverse_of(it.ny);
    const int lane = threadIdx.x & 31;
    for (int q = threadIdx.x; q < kObsSlots; q += kObsThreads) keys[q] = 0;
    for (int q = threadIdx.x; q < kObsSlots * F; q += kObsThreads) (&sums[0][0])[q] = 0;
    __syncthreads();
    int medium = 0;
    for (uint32_t w0 = blockIdx.x * blockDim.x; w0 < n; w0 += gridDim.x * blockDim.x) {
        const bool walks = w0 + threadIdx.x < n;
        const Walk k = walk_of<DIM>(it, walks ? w0 + threadIdx.x : w0);
        // columns of the window: site numbers within a plane
        uint32_t col[P];
        {
            const uint32_t xs[3] = {k.x == 0 ? it.nx - 1 : k.x - 1, k.x, k.x + 1 == it.nx ? 0 : k.x + 1};
            const uint32_t ys[3] = {k.y == 0 ? it.ny - 1 : k.y - 1, k.y, k.y + 1 == it.ny ? 0 : k.y + 1};
#pragma unroll
            for (int c = 0; c < P; ++c) col[c] = xs[c % 3] + (DIM == 3 ? it.nx * ys[c / 3] : 0);
        }
        int prev[P], cur[P], next[P], zero_prev = 0, zero_cur = 0;
        const auto plane = [&](uint32_t z, int (&v)[P]) {
            int zeros = 0;
#pragma unroll
            for (int c = 0; c < P; ++c) {
                v[c] = cell_id(it.lat[col[c] + k.step * z]);
                zeros += v[c] == 0 ? 1 : 0;
            }
            return zeros;
        };
        zero_prev = plane(k.lo == 0 ? (uint32_t)nw - 1 : k.lo - 1, prev);
        zero_cur = plane(k.lo, cur);
        // a run: cell, offsets of the walk from its anchor, sums over its sites
        struct Run {
            int id, ox, oy, cnt, sw, sww, iface;
        };
        Run run{}, ended{};  // at hand, and one that has ended (3D)
        int aw = 0;          // anchor's coordinate along the walk
        const auto add_run = [&](const Run &r, int64_t sww) {
            unsigned long long *row = reinterpret_cast<unsigned long long *>(cells + (it.row0 + r.id) * kObsFields);
            const auto add = [&](int f, int64_t v) { atomicAdd(row + f, (unsigned long long)v); };
            const int64_t c = r.cnt;
            add(1, c);
            add(2, c * r.ox);
            add(5, r.iface);
            add(6, c * r.ox * r.ox);
            if (DIM == 3) {
                add(3, c * r.oy);
                add(4, r.sw);
                add(7, c * r.oy * r.oy);
                add(8, sww);
                add(9, c * r.ox * r.oy);
                add(10, (int64_t)r.sw * r.ox);
                add(11, (int64_t)r.sw * r.oy);
            } else {
                add(3, r.sw);
                add(7, sww);
                add(9, (int64_t)r.sw * r.ox);
            }
        };
        // 3D: the ended runs of a warp, cell by cell; lane f - 1 adds field f
        const auto flush = [&]() {
            unsigned open = __ballot_sync(0xffffffffu, ended.id > 0);
            while (open) {
                const int cell = __shfl_sync(0xffffffffu, ended.id, __ffs(open) - 1);
                const bool mine = ended.id == cell;
                open &= ~__ballot_sync(0xffffffffu, mine);
                const Run r = ended;
                int sum = 0;
                const auto add = [&](int f, int v) {
                    const int total = __reduce_add_sync(0xffffffffu, mine ? v : 0);
                    if (lane == f - 1) sum = total;
                };
                add(1, r.cnt);
                add(2, r.cnt * r.ox);
                add(3, r.cnt * r.oy);
                add(4, r.sw);
                add(5, r.iface);
                add(6, r.cnt * r.ox * r.ox);
                add(7, r.cnt * r.oy * r.oy);
                add(8, r.sww);
                add(9, r.cnt * r.ox * r.oy);
                add(10, r.sw * r.ox);
                add(11, r.sw * r.oy);
                int slot = -1;
                if (lane == 0) {
                    for (int p = 0, q = cell % kObsSlots; p < kObsSlots; ++p, q = (q + 1) % kObsSlots) {
                        const int held = atomicCAS(keys + q, 0, cell);
                        if (held == 0 || held == cell) {
                            slot = q;
                            break;
                        }
                    }
                }
                slot = __shfl_sync(0xffffffffu, slot, 0);
                if (lane < F && sum != 0) {
                    if (slot >= 0)
                        atomicAdd(&sums[slot][lane], sum);
                    else
                        atomicAdd(reinterpret_cast<unsigned long long *>(cells + (it.row0 + cell) * kObsFields) + lane + 1,
                                  (unsigned long long)(int64_t)sum);
                }
            }
            ended.id = 0;
        };
        const auto end_run = [&](bool ends) {
            if (!shared) {
                if (ends) add_run(run, run.sww);
                return;
            }
            if (__any_sync(0xffffffffu, ends && ended.id > 0)) flush();
            if (ends) ended = run;
        };
        const auto equal = [&](const int (&v)[P]) {
            int e = 0;
#pragma unroll
            for (int q = 0; q < P; ++q) e += v[q] == run.id ? 1 : 0;
            return e;
        };
        int same_prev = 0, same_cur = 0;  // sites of the run's cell in the planes
        for (uint32_t z = k.lo; z < k.lo + kWalk; ++z) {
            const bool here = walks && z < k.hi;
            int c = here ? cur[P / 2] : 0;
            if (c < 0 || c > it.n_cells) c = 0;
            const int zero_next = here ? plane(z + 1 == (uint32_t)nw ? 0 : z + 1, next) : 0;
            end_run(run.id > 0 && c != run.id);
            if (c != run.id) {
                run = Run{};
                run.id = c;
                if (c > 0) {
                    const uint32_t a = (uint32_t)cells[(it.row0 + c) * kObsFields], ya = quotient_of(a, inv_x), xa = a - ya * it.nx;
                    run.ox = min_image((int)k.x - (int)xa, nx);
                    if (DIM == 3) {
                        const uint32_t za = quotient_of(ya, inv_y);
                        run.oy = min_image((int)k.y - (int)(ya - za * it.ny), ny);
                        aw = (int)za;
                    } else {
                        aw = (int)ya;
                    }
                    same_prev = equal(prev);
                    same_cur = equal(cur);
                }
            }
            if (run.id > 0) {
                const int same_next = equal(next);
                const int iface = 3 * P - (same_prev + same_cur + same_next);
                medium += zero_prev + zero_cur + zero_next;
                const int ow = min_image((int)z - aw, nw);
                if (FAR && (ow > kFarOffset || ow < -kFarOffset)) {
                    // a run of its own, its square in 64 bits
                    add_run(Run{run.id, run.ox, run.oy, 1, ow, 0, iface}, (int64_t)ow * ow);
                } else {
                    ++run.cnt;
                    run.iface += iface;
                    run.sw += ow;
                    run.sww += ow * ow;
                }
                same_prev = same_cur;
                same_cur = same_next;
            }
#pragma unroll
            for (int q = 0; q < P; ++q) {
                prev[q] = cur[q];
                cur[q] = next[q];
            }
            zero_prev = zero_cur;
            zero_cur = zero_next;
        }
        end_run(run.id > 0);
        if (!shared) continue;
        flush();
        __syncthreads();
        for (int q = threadIdx.x; q < kObsSlots * F; q += kObsThreads) {
            const int v = sums[q / F][q % F];
            if (v == 0) continue;
            atomicAdd(reinterpret_cast<unsigned long long *>(cells + (it.row0 + keys[q / F]) * kObsFields + 1 + q % F),
                      (unsigned long long)(int64_t)v);
            sums[q / F][q % F] = 0;
        }
        __syncthreads();
        for (int q = threadIdx.x; q < kObsSlots; q += kObsThreads) keys[q] = 0;
        __syncthreads();
    }
    medium = __reduce_add_sync(0xffffffffu, medium);
    if (lane == 0 && medium)
        atomicAdd(reinterpret_cast<unsigned long long *>(member + 2 * blockIdx.y), (unsigned long long)medium);
}

constexpr int kSumThreads = 128, kSumWarps = kSumThreads / 32;
constexpr int kMaxLag = 20;  // step-direction autocorrelation lags (x every MCS)
constexpr size_t kSumUnitBytes = 48 * 1024;  // step directions held at a time (at least one cell's)
// dynamic shared memory of a summary of the most snapshots
constexpr size_t kSumMaxSmem = sizeof(double) * (5 + 3 * kSumWarps) * kSummaryMaxSnap + kSumUnitBytes;
static_assert(sizeof(double) * 2 * kSummaryMaxSnap <= kSumUnitBytes && sizeof(double) * 2 * kSumWarps * kMaxLag <= kSumUnitBytes,
              "a cell's directions and the lags' totals fit");
// scalar accumulators of one lattice, a copy per warp
enum {
    A_MSD = 0,       // 3 sums, then 3 counts
    A_SP = 6,        // speed sum, sum of squares, count
    A_ST = 9,        // straightness sum, count
    A_DAC = 11,      // 50-MCS direction cosine sum, count
    A_SLOW = 13,     // slow 50-MCS sub-tracks, count
    A_EL = 15,       // elongation sum, count
    A_AC = 17,       // sum and count of the direction cosines of the lag at hand
    A_N = 19
};

__device__ __forceinline__ double warp_sum(double v)
{
#pragma unroll
    for (int d = 16; d > 0; d /= 2) v += __shfl_xor_sync(0xffffffffu, v, d);
    return v;
}

// a / b with inv = 1 / b at hand: the product corrected by its residual (within an ulp of the quotient,
// three operations instead of a division's dozen)
__device__ __forceinline__ double quotient(double a, double b, double inv)
{
    const double q = a * inv;
    return fma(fma(-q, b, a), inv, q);
}

// One CTA per lattice, a warp per cell, its lanes over the snapshots.  Per cell: the centroid at
// every snapshot (anchor + offset sums / volume), unwrapped across snapshots by minimal-image
// steps; a cell absent at any snapshot has no track.  Per-snapshot volume and interface moments are
// sums of integers; the track statistics are summed per lane, then over lanes and warps in a fixed
// order.
//
// Bound by the FP64 unit (about two operations per SM and clock): what counts is the number of
// divisions and square roots.  A step's direction is formed once, not once per lag and partner, and
// the autocorrelation, which ends at its first value <= 0, is not taken beyond it where the CTA
// holds the directions of all its cells.  512 runs of 16 cells, 81 snapshots: 4.57 ms with a thread
// per cell and the directions formed per lag, 0.62 ms so.
__global__ void __launch_bounds__(kSumThreads) summarize_kernel(const ObserveItem *items, const int64_t *cells,
                                                                int64_t rows, const int64_t *member, int n_items,
                                                                int S1, int every, int cap, double *out)
{
    extern __shared__ double sum_smem[];
    __shared__ double part[kSumWarps][A_N];
    __shared__ double pers_s;
    __shared__ int open_s;
    const int run = blockIdx.x, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const ObserveItem it = items[run];
    // per snapshot: number of cells, V, V^2, A, A^2 over them
    unsigned long long *snap = reinterpret_cast<unsigned long long *>(sum_smem);
    // per warp: the track of its cell and the lengths of its 50-MCS displacements
    double *X = sum_smem + 5 * S1 + warp * 3 * S1, *Y = X + S1, *F = Y + S1;
    // per cell of the chunk: step directions ((0, 0) for a step of length 0 or a cell without a track)
    double *U = sum_smem + (5 + 3 * kSumWarps) * S1;
    for (int i = threadIdx.x; i < 5 * S1; i += blockDim.x) snap[i] = 0;
    if (threadIdx.x == 0) {
        pers_s = 0.5 * every;
        open_s = 1;
    }
    __syncthreads();
    const double nx = (double)it.nx, ny = (double)it.ny;
    const int lags[3] = {10, 50, 200};
    const int k50 = 50 % every == 0 ? 50 / every : 0;
    const int n_ac = S1 - 1 < kMaxLag + 1 ? S1 - 1 : kMaxLag + 1;  // lags 1 .. n_ac - 1
    const bool one_chunk = it.n_cells <= cap;
    double acc[A_N];
#pragma unroll
    for (int k = 0; k < A_N; ++k) acc[k] = 0.0;
    double ac_sum = 0.0, ac_cnt = 0.0;   // of lag 1 + lane, over all chunks but where one holds all cells
    for (int c0 = 1; c0 <= it.n_cells; c0 += cap) {
        const int nc = it.n_cells - c0 + 1 < cap ? it.n_cells - c0 + 1 : cap;
        for (int c = warp; c < nc; c += kSumWarps) {
            const int64_t row = it.row0 + c0 + c;
            double *UX = U + (size_t)c * 2 * S1, *UY = UX + S1;
            bool present = true;
            for (int s = lane; s < S1; s += 32) {
                const int64_t *r = cells + ((int64_t)s * rows + row) * kObsFields;
                const int64_t v = r[1];
                if (v <= 0) {
                    present = false;
                    continue;
                }
                atomicAdd(snap + s, 1ull);
                atomicAdd(snap + S1 + s, (unsigned long long)v);
                atomicAdd(snap + 2 * S1 + s, (unsigned long long)(v * v));
                atomicAdd(snap + 3 * S1 + s, (unsigned long long)r[5]);
                atomicAdd(snap + 4 * S1 + s, (unsigned long long)(r[5] * r[5]));
                const double V = (double)v, inv = 1.0 / V;
                const double mx = quotient((double)r[2], V, inv), my = quotient((double)r[3], V, inv);
                const double cxx = quotient((double)r[6], V, inv) - mx * mx;
                const double cyy = quotient((double)r[7], V, inv) - my * my;
                const double cxy = quotient((double)r[9], V, inv) - mx * my;
                const double t2 = cxx + cyy, det = cxx * cyy - cxy * cxy;
                const double disc = sqrt(fmax(t2 * t2 / 4.0 - det, 0.0));
                const double l1 = t2 / 2.0 + disc, l2 = t2 / 2.0 - disc;
                if (l2 > 1e-9) {
                    acc[A_EL] += sqrt(l1 / l2);
                    acc[A_EL + 1] += 1.0;
                }
                const uint32_t anchor = (uint32_t)r[0];  // below 2^31
                X[s] = (double)(anchor % it.nx) + mx;
                Y[s] = (double)(anchor / it.nx) + my;
            }
            present = __all_sync(0xffffffffu, present);
            __syncwarp();
            if (!present) {
                for (int s = lane; s < S1; s += 32) UX[s] = UY[s] = 0.0;
                __syncwarp();
                continue;
            }
            // minimal-image steps, then the track as their running sum
            for (int s = lane; s + 1 < S1; s += 32) {
                double dx = X[s + 1] - X[s], dy = Y[s + 1] - Y[s];
                if (fabs(dx) > 0.499 * nx) dx -= nx * rint(dx / nx);
                if (fabs(dy) > 0.499 * ny) dy -= ny * rint(dy / ny);
                UX[s] = dx;
                UY[s] = dy;
            }
            __syncwarp();
            if (lane < 2) {
                double *T = lane == 0 ? X : Y;
                const double *D = lane == 0 ? UX : UY;
                double p = 0.0;
                T[0] = 0.0;
                for (int s = 0; s + 1 < S1; ++s) {
                    p += D[s];
                    T[s + 1] = p;
                }
            }
            __syncwarp();
#pragma unroll
            for (int j = 0; j < 3; ++j) {
                const int k = lags[j] % every ? 0 : lags[j] / every;
                if (k <= 0 || k >= S1) continue;
                for (int s = lane; s + k < S1; s += 32) {
                    const double dx = X[s + k] - X[s], dy = Y[s + k] - Y[s];
                    acc[A_MSD + j] += dx * dx + dy * dy;
                }
                if (lane == 0) acc[A_MSD + 3 + j] += (double)(S1 - k);
            }
            double path = 0.0;
            for (int s = lane; s < S1; s += 32) {
                double ux = 0.0, uy = 0.0;
                if (s + 1 < S1) {
                    const double dx = X[s + 1] - X[s], dy = Y[s + 1] - Y[s];
                    const double sq = dx * dx + dy * dy, nrm = sqrt(sq);
                    path += nrm;
                    acc[A_SP + 1] += sq;
                    if (nrm > 0.0) {
                        const double inv = 1.0 / nrm;
                        ux = quotient(dx, nrm, inv);
                        uy = quotient(dy, nrm, inv);
                    }
                }
                UX[s] = ux;
                UY[s] = uy;
            }
            path = warp_sum(path);
            if (lane == 0 && S1 > 1) {
                acc[A_SP] += path;
                acc[A_SP + 2] += (double)(S1 - 1);
                if (path > 0.0) {
                    const double ex = X[S1 - 1] - X[0], ey = Y[S1 - 1] - Y[0];
                    acc[A_ST] += sqrt(ex * ex + ey * ey) / path;
                    acc[A_ST + 1] += 1.0;
                }
            }
            if (k50 > 0 && 2 * k50 < S1) {
                for (int s = lane; s + k50 < S1; s += 32) {
                    const double ax = X[s + k50] - X[s], ay = Y[s + k50] - Y[s];
                    const double na = sqrt(ax * ax + ay * ay);
                    F[s] = na;
                    acc[A_SLOW] += na / 50.0 < kArrestSpeed ? 1.0 : 0.0;
                }
                if (lane == 0) acc[A_SLOW + 1] += (double)(S1 - k50);
                __syncwarp();
                for (int s = lane; s + 2 * k50 < S1; s += 32) {
                    const double ax = X[s + k50] - X[s], ay = Y[s + k50] - Y[s];
                    const double bx = X[s + 2 * k50] - X[s + k50], by = Y[s + 2 * k50] - Y[s + k50];
                    const double na = F[s], nb = F[s + k50];
                    if (na > 0.0 && nb > 0.0) {
                        acc[A_DAC] += (ax * bx + ay * by) / (na * nb);
                        acc[A_DAC + 1] += 1.0;
                    }
                }
            }
            __syncwarp();
        }
        __syncthreads();
        // direction cosines of the chunk, lag by lag
        for (int k = 1; k < n_ac; ++k) {
            double sum = 0.0;
            int cnt = 0;
            for (int c = warp; c < nc; c += kSumWarps) {
                const double *UX = U + (size_t)c * 2 * S1, *UY = UX + S1;
                for (int s = lane; s + k + 1 < S1; s += 32) {
                    const double ax = UX[s], ay = UY[s], bx = UX[s + k], by = UY[s + k];
                    sum = fma(ax, bx, fma(ay, by, sum));
                    // a direction is (0, 0) only where there is none (no step)
                    cnt += (ax != 0.0 || ay != 0.0) && (bx != 0.0 || by != 0.0) ? 1 : 0;
                }
            }
            sum = warp_sum(sum);
            cnt = __reduce_add_sync(0xffffffffu, cnt);
            if (one_chunk) {
                if (lane == 0) {
                    part[warp][A_AC] = sum;
                    part[warp][A_AC + 1] = (double)cnt;
                }
                __syncthreads();
                if (threadIdx.x == 0) {
                    double cs = 0.0, cc = 0.0;
                    for (int w = 0; w < kSumWarps; ++w) {
                        cs += part[w][A_AC];
                        cc += part[w][A_AC + 1];
                    }
                    const double ck = cc > 0.0 ? cs / cc : 0.0;
                    if (ck > 0.0) pers_s += ck * every; else open_s = 0;
                }
                __syncthreads();
                if (!open_s) break;
            } else if (lane == k - 1) {
                ac_sum += sum;
                ac_cnt += (double)cnt;
            }
        }
        __syncthreads();
    }
    if (!one_chunk) {
        // the lags' totals over the warps, through the chunk's storage (at least 2 S1 doubles; 2 x 4 x 20 used)
        double *tot = U;
        if (lane < kMaxLag) {
            tot[(warp * kMaxLag + lane) * 2] = ac_sum;
            tot[(warp * kMaxLag + lane) * 2 + 1] = ac_cnt;
        }
        __syncthreads();
        if (threadIdx.x == 0) {
            for (int k = 1; k < n_ac; ++k) {
                double cs = 0.0, cc = 0.0;
                for (int w = 0; w < kSumWarps; ++w) {
                    cs += tot[(w * kMaxLag + k - 1) * 2];
                    cc += tot[(w * kMaxLag + k - 1) * 2 + 1];
                }
                const double ck = cc > 0.0 ? cs / cc : 0.0;
                if (!(ck > 0.0)) break;
                pers_s += ck * every;
            }
        }
    }
#pragma unroll
    for (int k = 0; k < A_AC; ++k) {
        const double v = warp_sum(acc[k]);
        if (lane == 0) part[warp][k] = v;
    }
    __syncthreads();
    if (warp != 0) return;
    // per-snapshot figures, lanes over the snapshots
    double tv = 0.0, ta = 0.0, tn = 0.0, vv = 0.0, av = 0.0, nv = 0.0, cf = 0.0, cfn = 0.0;
    for (int s = lane; s < S1; s += 32) {
        const double n = (double)snap[s], sV = (double)snap[S1 + s], sA = (double)snap[3 * S1 + s];
        tv += sV;
        ta += sA;
        tn += n;
        if (n > 0.0) {
            const double mv = sV / n, ma = sA / n;
            vv += fmax((double)snap[2 * S1 + s] / n - mv * mv, 0.0);
            av += fmax((double)snap[4 * S1 + s] / n - ma * ma, 0.0);
            nv += 1.0;
        }
        const double cm = (double)member[2 * ((int64_t)s * n_items + run)];
        const double cc = (sA - cm) / 2.0, tot = cc + cm;
        if (tot > 0.0) {
            cf += cc / tot;
            cfn += 1.0;
        }
    }
    tv = warp_sum(tv);
    ta = warp_sum(ta);
    tn = warp_sum(tn);
    vv = warp_sum(vv);
    av = warp_sum(av);
    nv = warp_sum(nv);
    cf = warp_sum(cf);
    cfn = warp_sum(cfn);
    if (lane != 0) return;
    double t[A_AC];
#pragma unroll
    for (int k = 0; k < A_AC; ++k) {
        t[k] = 0.0;
        for (int w = 0; w < kSumWarps; ++w) t[k] += part[w][k];
    }
    const double qnan = __longlong_as_double(0x7ff8000000000000ll);
    double *o = out + (int64_t)run * kSummaryStats;
    for (int k = 0; k < kSummaryStats; ++k) o[k] = qnan;
    // a statistic scaled by a target of 0 (no volume or perimeter constraint) is undefined: NaN
    if (tn > 0.0) {
        if (it.v_ref != 0.0) o[0] = tv / tn / it.v_ref;
        if (it.a_ref != 0.0) o[2] = ta / tn / it.a_ref;
    }
    if (nv > 0.0) {
        if (it.v_ref != 0.0) o[1] = sqrt(vv / nv) / it.v_ref;
        if (it.a_ref != 0.0) o[3] = sqrt(av / nv) / it.a_ref;
    }
    for (int j = 0; j < 3; ++j)
        if (t[A_MSD + 3 + j] > 0.0) o[4 + j] = t[A_MSD + j] / t[A_MSD + 3 + j];
    if (t[A_SP + 2] > 0.0) {
        const double m = t[A_SP] / every / t[A_SP + 2];
        o[7] = m;
        o[8] = sqrt(fmax(t[A_SP + 1] / ((double)every * every) / t[A_SP + 2] - m * m, 0.0));
    }
    if (t[A_DAC + 1] > 0.0) o[9] = t[A_DAC] / t[A_DAC + 1];
    if (S1 > 1) o[10] = pers_s;
    if (t[A_SLOW + 1] > 0.0) o[11] = t[A_SLOW] / t[A_SLOW + 1];
    if (S1 > 1) {
        const int64_t m0 = member[2 * (int64_t)run + 1];
        const int64_t m1 = member[2 * ((int64_t)(S1 - 1) * n_items + run) + 1];
        const double sites = (double)it.nx * it.ny * it.nz;
        o[12] = (double)(m1 - m0) / ((double)(S1 - 1) * every * sites);
    }
    if (cfn > 0.0) o[13] = cf / cfn;
    if (t[A_ST + 1] > 0.0) o[14] = t[A_ST] / t[A_ST + 1];
    if (t[A_EL + 1] > 0.0) o[15] = t[A_EL] / t[A_EL + 1];
}

// Persistence update (Eq. 6, Eq. 7) for every cell, one thread per cell,
// from this MCS's observation rows: record the centroid (anchor + offset
// sums / volume, NaN for an absent cell) in history slot t % H, then blend
// the unit displacement over dt MCS into p_hat.  Every operation is a single
// rounded double operation in the order the replay uses (no contraction).
__global__ void pers_update_kernel(const int64_t *cells, int32_t n_cells, uint32_t nx, uint32_t ny, uint32_t nz,
                                   const uint8_t *cell_type, const PersParams pp, double *hist, int32_t H,
                                   int64_t t, int64_t t0, double *dir)
{
    const int64_t c = 1 + (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (c > n_cells) return;
    const int64_t nc = (int64_t)n_cells + 1;
    const int64_t *r = cells + c * kObsFields;
    double *Xn = hist + 3 * (nc * (t % H) + c);
    const double qnan = __longlong_as_double(0x7ff8000000000000ll);
    if (r[1] <= 0) {
        Xn[0] = Xn[1] = Xn[2] = qnan;
        return;
    }
    const int64_t an = r[0], plane = (int64_t)nx * ny;
    const double V = (double)r[1];
    const double ac[3] = {(double)(an % nx), (double)((an / nx) % ny), (double)(an / plane)};
    for (int d = 0; d < 3; ++d) Xn[d] = __dadd_rn(ac[d], __ddiv_rn((double)r[2 + d], V));
    const int tp = cell_type[c];
    const int dt = pp.dt[tp];
    if (pp.lambda[tp] == 0 || dt < 1 || t - dt < t0) return;
    const double *Xo = hist + 3 * (nc * ((t - dt) % H) + c);
    if (isnan(Xo[0])) return;
    const double L[3] = {(double)nx, (double)ny, (double)nz};
    double D[3];
    for (int d = 0; d < 3; ++d) {
        const double v = __dsub_rn(Xn[d], Xo[d]);
        D[d] = __dsub_rn(v, __dmul_rn(L[d], rint(__ddiv_rn(v, L[d]))));
    }
    double n2 = __dmul_rn(D[0], D[0]);
    n2 = __dadd_rn(n2, __dmul_rn(D[1], D[1]));
    n2 = __dadd_rn(n2, __dmul_rn(D[2], D[2]));
    if (n2 == 0.0) return;
    const double n = __dsqrt_rn(n2), mu = pp.mu[tp], am = __dsub_rn(1.0, mu);
    double *ph = dir + 3 * c, q[3];
    for (int d = 0; d < 3; ++d) {
        const double u = __ddiv_rn(D[d], n);
        q[d] = __dadd_rn(__dmul_rn(am, u), __dmul_rn(mu, ph[d]));
    }
    double m2 = __dmul_rn(q[0], q[0]);
    m2 = __dadd_rn(m2, __dmul_rn(q[1], q[1]));
    m2 = __dadd_rn(m2, __dmul_rn(q[2], q[2]));
    if (m2 == 0.0) {
        ph[0] = ph[1] = ph[2] = 0.0;
        return;
    }
    const double m = __dsqrt_rn(m2);
    for (int d = 0; d < 3; ++d) ph[d] = __ddiv_rn(q[d], m);
}

}  // namespace

cudaError_t launch_pers_update(const int64_t *cells, int32_t n_cells, uint32_t nx, uint32_t ny, uint32_t nz,
                               const uint8_t *cell_type, const PersParams &pp, double *hist, int32_t H, int64_t t,
                               int64_t t0, double *dir, cudaStream_t st)
{
    if (n_cells < 1) return cudaSuccess;
    pers_update_kernel<<<(n_cells + 127) / 128, 128, 0, st>>>(cells, n_cells, nx, ny, nz, cell_type, pp, hist, H, t,
                                                              t0, dir);
    return cudaPeekAtLastError();
}

cudaError_t launch_summarize(const ObserveItem *d_items, uint32_t n_items, int32_t max_cells, const int64_t *cells,
                             int64_t rows, const int64_t *member, int32_t n_snap, int32_t every, double *out,
                             cudaStream_t st)
{
    if (n_items == 0) return cudaSuccess;
    if (n_snap < 1 || n_snap > kSummaryMaxSnap || every < 1) return cudaErrorInvalidValue;
    // cells whose step directions are held at a time, and room for the lags' totals of several chunks
    const size_t per_cell = sizeof(double) * 2 * (size_t)n_snap;
    size_t cap = kSumUnitBytes / per_cell;
    cap = cap < 1 ? 1 : (cap > (size_t)max_cells ? (max_cells > 0 ? (size_t)max_cells : 1) : cap);
    size_t units = cap * per_cell;
    if (units < sizeof(double) * 2 * kSumWarps * kMaxLag) units = sizeof(double) * 2 * kSumWarps * kMaxLag;
    const size_t smem = sizeof(double) * (5 + 3 * kSumWarps) * (size_t)n_snap + units;
    // the limit belongs to the kernel, not to the launch: every thread sets the same
    const cudaError_t e = cudaFuncSetAttribute(summarize_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSumMaxSmem);
    if (e != cudaSuccess) return e;
    summarize_kernel<<<n_items, kSumThreads, smem, st>>>(d_items, cells, rows, member, (int)n_items, n_snap, every,
                                                         (int)cap, out);
    return cudaPeekAtLastError();
}

cudaError_t launch_observe(int dim, const ObserveItem *d_items, uint32_t n_items, int64_t max_sites, uint32_t longest,
                           int64_t *cells, int64_t *member, cudaStream_t st)
{
    if (n_items == 0) return cudaSuccess;
    if (n_items > 65535u) return cudaErrorInvalidValue;
    observe_init_kernel<<<n_items, 256, 0, st>>>(d_items, cells, member);
    // a walk per thread, for the largest member; a few CTAs per SM in all
    int64_t bx = (max_sites / kWalk + kObsThreads - 1) / kObsThreads + 1;
    const int64_t most = 152 * 16 / (int64_t)n_items + 16;
    if (bx > most) bx = most;
    const dim3 grid((unsigned)bx, n_items);
    const bool far = longest / 2 > (uint32_t)kFarOffset;
    if (dim == 3) {
        observe_anchor_kernel<3><<<grid, kObsThreads, 0, st>>>(d_items, cells);
        if (far) observe_sums_kernel<3, true><<<grid, kObsThreads, 0, st>>>(d_items, cells, member);
        else observe_sums_kernel<3, false><<<grid, kObsThreads, 0, st>>>(d_items, cells, member);
    } else {
        observe_anchor_kernel<2><<<grid, kObsThreads, 0, st>>>(d_items, cells);
        if (far) observe_sums_kernel<2, true><<<grid, kObsThreads, 0, st>>>(d_items, cells, member);
        else observe_sums_kernel<2, false><<<grid, kObsThreads, 0, st>>>(d_items, cells, member);
    }
    return cudaPeekAtLastError();
}

}  // namespace cpmgb
