// Batched multi-view form of the render path (many views of uneven resolution
// per call, sm_103a).
//
// All views go through one sequence of kernels instead of one sequence per view:
//  * bpred_kernel    R&L (§3.2) for every view: each node's centre and covariance
//                    are read once and tested against the views that may see it;
//  * banc_kernel     Ancestor filter per view: a node's ancestor path AP is read
//                    once for all views in which the node passed R&L;
//  * compaction      the per-view selection bits are one concatenated bit array
//                    [V][words]; the render path's counted compaction turns it into
//                    global entries v * n_pad + node (ascending: view, then node);
//  * bproject        projection and shrink of every entry with its view's camera;
//                    pairs are counted into global tile ids (the view's first
//                    tile + the tile), so the render path's tile scan, key
//                    scatter and per-tile sort order every view at once;
//  * bblend over all views' tiles; a CTA finds its view by binary search over
//    the views' first tiles and blends with that camera.
// Per view, selection, pairs, their order and every pixel are those of the
// single-view path with the same camera and tile shape.
#include "blend_impl.cuh"
#include "pairs_impl.cuh"
#include "project_impl.cuh"

#include <cstring>

namespace fgs {

// The cameras by value: the launch takes its copy, so the host may set the next call's at
// once and no staging buffer has to outlive a copy in flight.  (64 cameras are 9.5 KB of
// parameters; most batches need the smaller form.)
template <int N>
struct CameraPack {
    DevCamera c[N];
};

template <int N>
__global__ void __launch_bounds__(128) bcameras_kernel(const __grid_constant__ CameraPack<N> pack, int V,
                                                       DevCamera* __restrict__ dst)
{
    grid_dep_wait();
    for (int i = threadIdx.x; i < V * (int)(sizeof(DevCamera) / 4); i += blockDim.x)
        reinterpret_cast<uint32_t*>(dst)[i] = reinterpret_cast<const uint32_t*>(pack.c)[i];
}

template <int N>
static void launch_cameras(const DevCamera* cams, int V, DevCamera* dst, cudaStream_t s)
{
    CameraPack<N> pack;
    memcpy(pack.c, cams, sizeof(DevCamera) * V);
    launch_pdl(bcameras_kernel<N>, 1, 128, 0, s, pack, V, dst);
}

// R&L for V views: a warp takes chunks of 128 nodes g, g + W, g + 2W, ... (W warps), 32
// at a time: lane l tests the box of the l-th against every view's frustum planes (in
// shared memory, as the cameras); a chunk outside a view's frustum has no node with P
// there and its P bits are written as 0; the others are read by the whole warp, 4 nodes
// a lane, once for the views that need them, and evaluated for those.  The batch's
// counters are zeroed here first.  Bound: the box tests' issue and the in-frustum chunks'
// loads; a box tested by one lane a view, a chunk at a time, left most lanes idle and
// a round trip a chunk (8 views of 12.5M nodes: 111 us, now 70).
__global__ void __launch_bounds__(256, 3) bpred_kernel(DevTree t, const DevCamera* __restrict__ cams,
                                                    int V, uint32_t* __restrict__ pbits, FrameBegin begin)
{
    __shared__ DevCamera s_cam[kMaxBatchViews];
    __shared__ FrustumPlanes s_planes[kMaxBatchViews];
    grid_dep_wait();
    frame_begin(begin, (int)(blockIdx.x * blockDim.x + threadIdx.x), (int)(gridDim.x * blockDim.x));
    for (int i = threadIdx.x; i < V * (int)(sizeof(DevCamera) / 4); i += blockDim.x)
        reinterpret_cast<uint32_t*>(s_cam)[i] = reinterpret_cast<const uint32_t*>(cams)[i];
    __syncthreads();
    if ((int)threadIdx.x < V) frustum_planes(s_cam[threadIdx.x], s_planes[threadIdx.x]);
    __syncthreads();
    static_assert(kMaxBatchViews <= 64, "a view a bit of a 64-bit mask");
    const uint32_t n_words = t.n_pad >> 5, n_box = t.n_pad >> 7;
    const uint32_t lane = threadIdx.x & 31;
    const uint32_t n_warps = (gridDim.x * blockDim.x) >> 5;
    for (uint32_t cb = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; cb < n_box; cb += 32u * n_warps) {
        const uint32_t cl = cb + lane * n_warps;
        unsigned long long views = 0ull;                  // that may hold a centre of this lane's chunk
        if (cl < n_box) {
            const float4 lo = __ldg(t.cbox + 2 * cl), hi = __ldg(t.cbox + 2 * cl + 1);
            for (int v = 0; v < V; ++v) {
                if (chunk_outside(s_planes[v], lo, hi))
                    reinterpret_cast<uint4*>(pbits + (size_t)v * n_words)[cl] = make_uint4(0u, 0u, 0u, 0u);
                else
                    views |= 1ull << v;
            }
        }
        uint32_t todo = __ballot_sync(0xffffffffu, views != 0ull);
        while (todo) {
            const uint32_t j = (uint32_t)__ffs(todo) - 1u;
            todo &= todo - 1u;
            if (todo) {
                const uint32_t cn = cb + ((uint32_t)__ffs(todo) - 1u) * n_warps;
                const float* nx = t.mu + ((size_t)cn << 7) + (lane << 2);
                asm volatile("prefetch.global.L2 [%0];" ::"l"(nx));
                asm volatile("prefetch.global.L2 [%0];" ::"l"(nx + t.n_pad));
                asm volatile("prefetch.global.L2 [%0];" ::"l"(nx + 2 * (size_t)t.n_pad));
            }
            unsigned long long vm = ((unsigned long long)__shfl_sync(0xffffffffu, (uint32_t)(views >> 32), j) << 32) |
                                    __shfl_sync(0xffffffffu, (uint32_t)views, j);
            const uint32_t i = ((cb + j * n_warps) << 5) + lane;   // this lane's 4 nodes
            const uint32_t n0 = i << 2;
            const float4 mx = __ldg(reinterpret_cast<const float4*>(t.mu) + i);
            const float4 my = __ldg(reinterpret_cast<const float4*>(t.mu + t.n_pad) + i);
            const float4 mz = __ldg(reinterpret_cast<const float4*>(t.mu + 2 * (size_t)t.n_pad) + i);
            const uint32_t leaf = (__ldg(t.leaf_bits + (i >> 3)) >> ((i & 7) << 2)) & 0xFu;
            const float xs[4] = {mx.x, mx.y, mx.z, mx.w};
            const float ys[4] = {my.x, my.y, my.z, my.w};
            const float zs[4] = {mz.x, mz.y, mz.z, mz.w};
            float4 cv[6];
            bool have_cov = false;
            while (vm) {
                const int v = __ffsll((long long)vm) - 1;
                vm &= vm - 1ull;
                const DevCamera& cam = s_cam[v];
                float vz[4], txtz[4], tytz[4];
                uint32_t inf = 0;
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    float vx, vy;
                    camera_space(cam, xs[k], ys[k], zs[k], vx, vy, vz[k]);
                    txtz[k] = tytz[k] = 0.0f;
                    const bool in = (n0 + k < t.n) && frustum_test(cam, vx, vy, vz[k], txtz[k], tytz[k]);
                    inf |= (uint32_t)in << k;
                }
                uint32_t pnib = inf & leaf;
                const uint32_t need = inf & ~leaf;
                if (need) {
                    if (!have_cov) {
#pragma unroll
                        for (int q = 0; q < 6; ++q)
                            cv[q] = __ldg(reinterpret_cast<const float4*>(t.cov + q * (size_t)t.n_pad) + i);
                        have_cov = true;
                    }
#pragma unroll
                    for (int k = 0; k < 4; ++k) {
                        if (!((need >> k) & 1u)) continue;
                        float s6[6];
#pragma unroll
                        for (int q = 0; q < 6; ++q)
                            s6[q] = k == 0 ? cv[q].x : k == 1 ? cv[q].y : k == 2 ? cv[q].z : cv[q].w;
                        float a, b, cc, lam;
                        ewa_cov2d(cam, vz[k], txtz[k], tytz[k], s6, a, b, cc, lam);
                        if (fm(3.0f, fsq(lam)) <= cam.tau_R) pnib |= 1u << k;
                    }
                }
                uint32_t w = pnib << ((lane & 7) << 2);
                w |= __shfl_xor_sync(0xffffffffu, w, 1);
                w |= __shfl_xor_sync(0xffffffffu, w, 2);
                w |= __shfl_xor_sync(0xffffffffu, w, 4);
                if ((lane & 7) == 0) pbits[(size_t)v * n_words + (i >> 3)] = w;
            }
        }
    }
}

// Ancestor filter for V views, a warp 4 words of 32 nodes at a time: lane l reads word
// l % 4 of views l / 4, l / 4 + 8, ..., so the words without a P bit in any view (most)
// cost a few loads and stores for all 4 together.  For the others the path of each node
// is read once for all views (and the next such word's paths are prefetched), and the
// ancestors' bits of two views that have a P bit in the word in one batch of independent
// loads.  The survivors of every compaction tile are counted.  Bound: latency of the
// paths' and bits' loads (8 views of 12.5M nodes: 133 us; 238 with a word at a time over
// every view, an ancestor's bit looked up before the next).
__global__ void __launch_bounds__(256, 5) banc_kernel(DevTree t, int V, const uint32_t* __restrict__ pbits,
                                                      uint32_t* __restrict__ selbits, uint32_t* __restrict__ sel_cnt)
{
    grid_dep_wait();
    const uint32_t lane = threadIdx.x & 31;
    const uint32_t n_words = t.n_pad >> 5;                // a multiple of 128
    const uint32_t n_warps = (gridDim.x * blockDim.x) >> 5;
    for (uint32_t w0 = 4u * ((blockIdx.x * blockDim.x + threadIdx.x) >> 5); w0 < n_words; w0 += 4u * n_warps) {
        const uint32_t wl = w0 + (lane & 3u);
        uint32_t any = 0u;
        for (int v = (int)(lane >> 2); v < V; v += 8) any |= __ldg(pbits + (size_t)v * n_words + wl);
        any = __ballot_sync(0xffffffffu, any != 0u);
        any |= any >> 16;
        any |= any >> 8;
        uint32_t act = (any | any >> 4) & 0xFu;
        if (!((act >> (lane & 3u)) & 1u))
            for (int v = (int)(lane >> 2); v < V; v += 8) selbits[(size_t)v * n_words + wl] = 0u;
        while (act) {
            const uint32_t k = (uint32_t)__ffs(act) - 1u;
            act &= act - 1u;
            const uint32_t w = w0 + k;
            const uint32_t n = (w << 5) + lane;
            if (act && lane < t.depth)                    // the next word's paths
                asm volatile("prefetch.global.L2 [%0];" ::"l"(t.ap + (size_t)lane * t.n_pad +
                                                              ((size_t)(w0 + (uint32_t)__ffs(act) - 1u) << 5)));
            for (int vb = 0; vb < V; vb += 32) {          // 32 views at a time, lane l reads the word of view vb + l
                const uint32_t pw = vb + (int)lane < V ? __ldg(pbits + (size_t)(vb + lane) * n_words + w) : 0u;
                uint32_t vm = __ballot_sync(0xffffffffu, pw != 0u);
                if (vb + (int)lane < V && !pw) selbits[(size_t)(vb + lane) * n_words + w] = 0u;
                if (!vm) continue;
                uint32_t nodes = pw;                      // with a P bit in any of these views
#pragma unroll
                for (int o = 16; o; o >>= 1) nodes |= __shfl_xor_sync(0xffffffffu, nodes, o);
                const bool mine = (nodes >> lane) & 1u;
                uint32_t a[16];
#pragma unroll
                for (int q = 0; q < 16; ++q)
                    a[q] = mine && (uint32_t)q < t.depth ? __ldg(t.ap + (size_t)q * t.n_pad + n) : kApPad;
                while (vm) {                              // two views at a time
                    const uint32_t v0 = (uint32_t)__ffs(vm) - 1u;
                    vm &= vm - 1u;
                    const uint32_t v1 = vm ? (uint32_t)__ffs(vm) - 1u : v0;
                    vm &= vm - 1u;
                    const uint32_t* p0 = pbits + (size_t)(vb + v0) * n_words;
                    const uint32_t* p1 = pbits + (size_t)(vb + v1) * n_words;
                    bool k0 = (__shfl_sync(0xffffffffu, pw, v0) >> lane) & 1u;
                    bool k1 = (__shfl_sync(0xffffffffu, pw, v1) >> lane) & 1u;
                    uint32_t h0 = 0u, h1 = 0u;
#pragma unroll
                    for (int h = 0; h < 16; h += 8) {
                        if (h && t.depth <= 8u) break;
#pragma unroll
                        for (int q = h; q < h + 8; ++q)
                            if (a[q] != kApPad) {
                                if (k0) h0 |= __ldg(p0 + (a[q] >> 5)) >> (a[q] & 31);
                                if (k1) h1 |= __ldg(p1 + (a[q] >> 5)) >> (a[q] & 31);
                            }
                    }
                    k0 = k0 && !(h0 & 1u);
                    k1 = k1 && !(h1 & 1u);
                    // levels above the 16th (a tree so deep): one at a time
                    for (uint32_t q = 16; (k0 || k1) && q < t.depth; ++q) {
                        const uint32_t an = __ldg(t.ap + (size_t)q * t.n_pad + n);
                        if (an == kApPad) break;
                        if (__ldg(p0 + (an >> 5)) >> (an & 31) & 1u) k0 = false;
                        if (__ldg(p1 + (an >> 5)) >> (an & 31) & 1u) k1 = false;
                    }
                    const uint32_t b0 = __ballot_sync(0xffffffffu, k0), b1 = __ballot_sync(0xffffffffu, k1);
                    if (lane < 2u && (lane == 0u || v1 != v0)) {
                        const uint32_t b = lane ? b1 : b0;
                        const size_t at = (size_t)(vb + (lane ? v1 : v0)) * n_words + w;
                        selbits[at] = b;
                        if (b) atomicAdd(sel_cnt + at / kBatchSelTileWords, (uint32_t)__popc(b));
                    }
                }
            }
        }
    }
}

// Projection of every selected entry (entry = view * n_pad + node), with the
// pairs counted into global tile ids.
template <int kDeg>
__global__ void __launch_bounds__(kProjectThreads, kProjectBlocks) bproject_kernel(
    DevTree t, const DevCamera* __restrict__ cams, int V, const uint32_t* __restrict__ tile_base,
    const uint32_t* __restrict__ sel, float* __restrict__ splat, uint4* __restrict__ foot,
    uint32_t* __restrict__ tile_cnt, FrameState* st)
{
    __shared__ proj::Rows<kDeg> S;
    __shared__ DevCamera s_cam[kMaxBatchViews];
    __shared__ uint32_t s_base[kMaxBatchViews];
    grid_dep_wait();
    for (int i = threadIdx.x; i < V * (int)(sizeof(DevCamera) / 4); i += blockDim.x)
        reinterpret_cast<uint32_t*>(s_cam)[i] = reinterpret_cast<const uint32_t*>(cams)[i];
    for (int i = threadIdx.x; i < V; i += blockDim.x) s_base[i] = tile_base[i];
    __syncthreads();
    proj::project_walk<kDeg>(t, sel, S, splat, foot, tile_cnt, st,
                             [&](uint32_t e, uint32_t& n, uint32_t& tiles_x, uint32_t& tbase) -> const DevCamera& {
                                 const uint32_t v = e / t.n_pad;
                                 n = e - v * t.n_pad;
                                 tiles_x = (uint32_t)s_cam[v].tiles_x;
                                 tbase = s_base[v];
                                 return s_cam[v];
                             });
}

// Blend every tile of every view; the tile's view is found by binary search.
__global__ void __launch_bounds__(blendk::kWalkChunk) bblend_kernel(
    const DevCamera* __restrict__ cams, int V, uint32_t total_tiles, const uint32_t* __restrict__ tile_base,
    const unsigned long long* __restrict__ img_off, const uint2* __restrict__ ranges,
    const uint32_t* __restrict__ heavy, const uint32_t* __restrict__ vals, const float* __restrict__ splat,
    float* __restrict__ rgb, float* __restrict__ Tout, FrameState* st)
{
    __shared__ __align__(128) blendk::WalkSmem<false> S;
    __shared__ DevCamera s_cam;
    grid_dep_wait();
    // the tile's view: its camera to s_cam; first tile and image offset
    auto locate = [&](uint32_t gtile, uint32_t& base) {
        int lo = 0, hi = V;                            // largest v with tile_base[v] <= gtile
        while (hi - lo > 1) {
            const int mid = (lo + hi) >> 1;
            if (__ldg(tile_base + mid) <= gtile) lo = mid;
            else hi = mid;
        }
        for (int i = threadIdx.x; i < (int)(sizeof(DevCamera) / 4); i += blockDim.x)
            reinterpret_cast<uint32_t*>(&s_cam)[i] = reinterpret_cast<const uint32_t*>(cams + lo)[i];
        __syncthreads();
        base = __ldg(tile_base + lo);
        return __ldg(img_off + lo);
    };
    blendk::walk_grid(
        blockIdx.x, gridDim.x, total_tiles, ranges, heavy, st,
        [&](uint32_t gtile, uint2 rg) {
            uint32_t base;
            const unsigned long long o = locate(gtile, base);
            blendk::blend_walk<8, false, false>(s_cam, gtile - base, 0u, rg, S, vals, splat, rgb + 3 * o,
                                                Tout ? Tout + o : nullptr, nullptr, st);
        },
        [&](uint32_t gtile, uint32_t part, uint2 rg) {
            uint32_t base;
            const unsigned long long o = locate(gtile, base);
            blendk::blend_walk<16, false, false>(s_cam, gtile - base, part, rg, S, vals, splat, rgb + 3 * o,
                                                 Tout ? Tout + o : nullptr, nullptr, st);
        });
}

// ---------------------------------------------------------------------------
// launchers
// ---------------------------------------------------------------------------
void launch_batch_cameras(const DevCamera* cams, int V, DevCamera* dst, cudaStream_t s)
{
    if (V <= 16) launch_cameras<16>(cams, V, dst, s);
    else launch_cameras<kMaxBatchViews>(cams, V, dst, s);
}

void launch_batch_front(const DevTree& t, const DevCamera* cams, int V, uint32_t total_tiles,
                        const uint32_t* tile_base, uint32_t* pbits, uint32_t* selbits, uint32_t* sel,
                        uint32_t sel_cap, float* splat, uint4* foot, uint32_t* tile_cnt, uint32_t* large, uint32_t* heavy,
                        unsigned long long* items, unsigned long long* keys, uint32_t* vals,
                        unsigned long long cap, uint32_t* sel_cnt, unsigned long long* lb_scan,
                        uint2* ranges, FrameState* st, int sms, cudaStream_t s)
{
    const uint32_t n_words = t.n_pad >> 5;
    const uint32_t all_words = (uint32_t)((size_t)n_words * V);
    const FrameBegin begin{st, tile_cnt, (int)total_tiles, sel_cnt, (int)batch_sel_tiles(all_words)};
    int occ = 0;
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, bpred_kernel, 256, 0);
    launch_pdl(bpred_kernel, sms * (occ > 0 ? occ : 1), 256, 0, s, t, cams, V, pbits, begin);
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, banc_kernel, 256, 0);
    launch_pdl(banc_kernel, sms * (occ > 0 ? occ : 1), 256, 0, s, t, V, pbits, selbits, sel_cnt);
    launch_compact_counted_batch(selbits, all_words, sel, sel_cap, sel_cnt, st, s);
    const auto bproject = t.sh_degree == 0   ? bproject_kernel<0>
                          : t.sh_degree == 1 ? bproject_kernel<1>
                          : t.sh_degree == 2 ? bproject_kernel<2>
                                             : bproject_kernel<3>;
    launch_pdl(bproject, sms * kProjectBlocks, kProjectThreads, 0, s, t, cams, V, tile_base, sel, splat, foot,
               tile_cnt, st);
    launch_tile_scan(tile_cnt, ranges, total_tiles, large, cap, lb_scan, st, sms * occ_tile_scan(), s);
    launch_scatter_batch(cams, tile_base, t.n_pad, sel, foot, tile_cnt, items, cap, st, sms * occ_scatter(), s);
    launch_segsort(ranges, total_tiles, large, items, keys, vals, heavy, st, sms * occ_segsort(), s);
}

void launch_batch_blend(const DevCamera* cams, int V, uint32_t total_tiles, const uint32_t* tile_base,
                        const unsigned long long* img_off, const uint2* ranges, const uint32_t* heavy,
                        const uint32_t* vals, const float* splat, float* rgb, float* T, FrameState* st,
                        cudaStream_t s)
{
    const uint32_t grid = total_tiles + 2u * (uint32_t)split_slots((int)total_tiles);
    launch_pdl(bblend_kernel, grid, blendk::kWalkChunk, 0, s, cams, V, total_tiles, tile_base, img_off, ranges, heavy,
               vals, splat, rgb, T, st);
}

}  // namespace fgs
