// Projection, SH colour and scene-adaptive shrinking (§3.1, §3.3) on sm_103a.
//
// project_kernel (project_impl.cuh): one thread per selected Gaussian computes the splat record
// (centre, conic, log-domain skip threshold, opacity, depth, colour, footprint
// radius) and its footprint record (tile rectangle, pair count, depth bits);
// then each warp enumerates its Gaussians' Gaussian-tile pairs and counts them
// into their tiles, from which the tile ranges of the sorted pair list follow
// (pairs.cu); the pairs of a Gaussian with more than kWarpWidePairs of them
// are counted by all the warp's lanes at once.
#include "project_impl.cuh"

namespace fgs {

template <int kDeg>
__global__ void __launch_bounds__(kProjectThreads, kProjectBlocks) project_kernel(
    DevTree t, const __grid_constant__ DevCamera cam, const uint32_t* __restrict__ sel, float* __restrict__ splat,
    uint4* __restrict__ foot, uint32_t* __restrict__ tile_cnt, FrameState* st)
{
    __shared__ proj::Rows<kDeg> S;
    grid_dep_wait();
    proj::project_walk<kDeg>(t, sel, S, splat, foot, tile_cnt, st,
                             [&](uint32_t e, uint32_t& n, uint32_t& tiles_x, uint32_t& tbase) -> const DevCamera& {
                                 n = e;
                                 tiles_x = (uint32_t)cam.tiles_x;
                                 tbase = 0u;
                                 return cam;
                             });
}

void launch_project(const DevTree& t, const DevCamera& cam, const uint32_t* sel, float* splat,
                    uint4* foot, uint32_t* tile_cnt, FrameState* st, int sms, cudaStream_t s)
{
    const int blocks = sms * kProjectBlocks;
    switch (t.sh_degree) {
    case 0: launch_pdl(project_kernel<0>, blocks, kProjectThreads, 0, s, t, cam, sel, splat, foot, tile_cnt, st); break;
    case 1: launch_pdl(project_kernel<1>, blocks, kProjectThreads, 0, s, t, cam, sel, splat, foot, tile_cnt, st); break;
    case 2: launch_pdl(project_kernel<2>, blocks, kProjectThreads, 0, s, t, cam, sel, splat, foot, tile_cnt, st); break;
    default: launch_pdl(project_kernel<3>, blocks, kProjectThreads, 0, s, t, cam, sel, splat, foot, tile_cnt, st); break;
    }
}

}  // namespace fgs
