// Spans of rounds of small 3D lattices (cpm_span.cuh); one dimension per translation unit.
#include "cpm_span.cuh"

namespace cpmgb {

uint32_t span_cluster_3d(bool perim, bool act, bool extra) { return span_cluster_d<3>(perim, act, extra); }

cudaError_t launch_span_3d(bool perim, bool act, const RoundArgs &a, const LatticeBufs &l, const SpanPos &p,
                           cudaStream_t st)
{
    return launch_span_d<3>(perim, act, a, l, p, st);
}

cudaError_t launch_batch_span_3d(bool perim, bool act, bool motile, BatchLattice *lats, uint32_t n, uint32_t n_mcs,
                                 uint32_t threads, uint32_t smem, cudaStream_t st)
{
    return launch_batch_span_d<3>(perim, act, motile, lats, n, n_mcs, threads, smem, st);
}

}  // namespace cpmgb
