// Per-tile front-to-back alpha blending (Eq. 2) and the KPC / GTC pre-render
// pass of the scene-adaptive shrinking (Eq. 5-7), sm_103a.
//
// The forward: one CTA of four warps per image tile, two for a tile that holds much of
// the frame's pairs; the tile's slice of the sorted value list is staged 128 Gaussians
// at a time and each warp walks it for its own blocks of pixels (blend_walk in
// blend_impl.cuh).
//
// The KPC pass: the same walk of whole tiles without an image, with the applied
// alpha * T summed for every pair (blend_walk_kpc).
//
// Blend decisions are exact: power, the log-domain skip test, alpha, the
// opacity clamp and the transmittance update use explicitly rounded binary32
// operations and a deterministic exp, so which Gaussians a pixel applies, and
// where it stops, do not depend on the compiler.  The culling only drops
// Gaussians that every pixel of the block would skip.  Colour accumulation may
// use FMA (it decides nothing).
#include "blend_impl.cuh"

namespace fgs {

template <bool kCount, bool kKeep>
__global__ void __launch_bounds__(blendk::kWalkChunk) blend_kernel(
    DevCamera cam, const uint2* __restrict__ ranges, const uint32_t* __restrict__ heavy,
    const uint32_t* __restrict__ vals, const float* __restrict__ splat, float* __restrict__ rgb,
    float* __restrict__ Tout, uint2* __restrict__ keep, FrameState* st)
{
    __shared__ __align__(128) blendk::WalkSmem<kKeep> S;
    grid_dep_wait();
    blendk::walk_grid(
        blockIdx.x, gridDim.x, (uint32_t)(cam.tiles_x * cam.tiles_y), ranges, heavy, st,
        [&](uint32_t tile, uint2 rg) {
            blendk::blend_walk<8, kCount, kKeep>(cam, tile, 0u, rg, S, vals, splat, rgb, Tout, keep, st);
        },
        [&](uint32_t tile, uint32_t part, uint2 rg) {
            blendk::blend_walk<16, kCount, kKeep>(cam, tile, part, rg, S, vals, splat, rgb, Tout, keep, st);
        });
}

__global__ void __launch_bounds__(blendk::kWalkChunk) blend_kpc_kernel(
    DevCamera cam, const uint2* __restrict__ ranges, const uint32_t* __restrict__ vals,
    const float* __restrict__ splat, float* __restrict__ kpc_out, float* __restrict__ G_out, FrameState* st)
{
    __shared__ __align__(128) blendk::KpcSmem S;
    grid_dep_wait();
    blendk::blend_walk_kpc(cam, blockIdx.x, ranges[blockIdx.x], S, vals, splat, kpc_out, G_out, st);
}

void launch_blend(const DevCamera& cam, const uint2* ranges, const uint32_t* heavy, const uint32_t* vals,
                  const float* splat, float* rgb, float* T, uint2* keep, FrameState* st, bool count,
                  cudaStream_t s)
{
    const int n_tiles = cam.tiles_x * cam.tiles_y;
    const int grid = n_tiles + 2 * split_slots(n_tiles);
    constexpr int threads = blendk::kWalkChunk;
    if (count)
        launch_pdl(blend_kernel<true, false>, grid, threads, 0, s, cam, ranges, heavy, vals, splat, rgb, T, keep, st);
    else if (keep)
        launch_pdl(blend_kernel<false, true>, grid, threads, 0, s, cam, ranges, heavy, vals, splat, rgb, T, keep, st);
    else
        launch_pdl(blend_kernel<false, false>, grid, threads, 0, s, cam, ranges, heavy, vals, splat, rgb, T, keep, st);
}

void launch_blend_kpc(const DevCamera& cam, const uint2* ranges, const uint32_t* vals,
                      const float* splat, float* kpc, float* G, FrameState* st, cudaStream_t s)
{
    const int n_tiles = cam.tiles_x * cam.tiles_y;
    launch_pdl(blend_kpc_kernel, n_tiles, blendk::kWalkChunk, 0, s, cam, ranges, vals, splat, kpc, G, st);
}

__global__ void eval_exp_kernel(const float* __restrict__ x, float* __restrict__ y, uint64_t n)
{
    const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
    for (uint64_t i = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; i < n; i += stride)
        y[i] = exp_cw(x[i]);
}

void launch_eval_exp(const float* x, float* y, uint64_t n, cudaStream_t s)
{
    uint64_t blocks = (n + 255) / 256;
    if (blocks > 4096) blocks = 4096;
    eval_exp_kernel<<<(unsigned)blocks, 256, 0, s>>>(x, y, n);
}

}  // namespace fgs
