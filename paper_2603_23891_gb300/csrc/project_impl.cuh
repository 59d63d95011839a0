// Per-Gaussian projection shared by the single-view and the batched kernels:
// EWA projection, footprint (3 sigma or shrunk to tau, §3.3), tile rectangle,
// pair count and SH colour.  Decision quantities use the explicitly rounded
// binary32 helpers of fgs_internal.cuh.
#pragma once

#include "pairs_impl.cuh"

namespace fgs {
namespace proj {


// Real spherical harmonics (Condon-Shortley phase), Cartesian form, normalisation
// constants from their closed forms: l=0 1/(2 sqrt(pi)); l=1 sqrt(3/(4 pi));
// l=2 sqrt(15/pi)/2, sqrt(5/pi)/4, sqrt(15/pi)/4; l=3 sqrt(35/(2 pi))/4,
// sqrt(105/pi)/2, sqrt(21/(2 pi))/4, sqrt(7/pi)/4, sqrt(105/pi)/4.
constexpr float kY00 = 0.28209479177387814f;
constexpr float kY1 = 0.48860251190291992f;
constexpr float kY2a = 1.0925484305920792f;
constexpr float kY2b = 0.31539156525252005f;
constexpr float kY2c = 0.54627421529603959f;
constexpr float kY3a = 0.59004358992664352f;
constexpr float kY3b = 2.8906114426405538f;
constexpr float kY3c = 0.45704579946446572f;
constexpr float kY3d = 0.37317633259011540f;
constexpr float kY3e = 1.4453057213202769f;

// Colour = sum_k Y_k(d) c[k][ch] + 0.5, clamped at 0, the coefficients read 16 bytes at a
// time from a staged row (K*3 floats padded to a multiple of 4) and accumulated on the
// fly; element e of the row is (k, ch) = (e / 3, e % 3).
template <int kDeg>
__device__ __forceinline__ void sh_colour(const float4* row, float x, float y, float z, float rgb[3])
{
    float Y[16];
#pragma unroll
    for (int k = 0; k < 16; ++k) Y[k] = 0.0f;
    Y[0] = kY00;
    if (kDeg >= 1) {
        Y[1] = -kY1 * y;
        Y[2] = kY1 * z;
        Y[3] = -kY1 * x;
    }
    if (kDeg >= 2) {
        const float xx = x * x, yy = y * y, zz = z * z;
        Y[4] = kY2a * x * y;
        Y[5] = -kY2a * y * z;
        Y[6] = kY2b * (2.0f * zz - xx - yy);
        Y[7] = -kY2a * x * z;
        Y[8] = kY2c * (xx - yy);
        if (kDeg >= 3) {
            Y[9] = -kY3a * y * (3.0f * xx - yy);
            Y[10] = kY3b * x * y * z;
            Y[11] = -kY3c * y * (4.0f * zz - xx - yy);
            Y[12] = kY3d * z * (2.0f * zz - 3.0f * xx - 3.0f * yy);
            Y[13] = -kY3c * x * (4.0f * zz - xx - yy);
            Y[14] = kY3e * z * (xx - yy);
            Y[15] = -kY3a * x * (xx - 3.0f * yy);
        }
    }
    constexpr int kNq = ((kDeg + 1) * (kDeg + 1) * 3 + 3) / 4;
    float acc[3] = {0.5f, 0.5f, 0.5f};
#pragma unroll
    for (int q = 0; q < kNq; ++q) {
        const float4 f = row[q];
        const float e[4] = {f.x, f.y, f.z, f.w};
#pragma unroll
        for (int r = 0; r < 4; ++r) {
            const int el = 4 * q + r;          // compile-time after unrolling
            if (el < 48) acc[el % 3] = fmaf(Y[el / 3], e[r], acc[el % 3]);
        }
    }
    rgb[0] = fmaxf(acc[0], 0.0f);
    rgb[1] = fmaxf(acc[1], 0.0f);
    rgb[2] = fmaxf(acc[2], 0.0f);
}

__device__ __forceinline__ float clampf(float v, float lo, float hi)
{
    v = v < lo ? lo : v;
    return v > hi ? hi : v;
}


// A node's attributes for the projection (DevTree::attr).
struct NodeAttr {
    float4 q0, q1, q2;
};

__device__ __forceinline__ NodeAttr load_attr(const DevTree& t, uint32_t n)
{
    const float4* a = t.attr + 3 * (size_t)n;
    return {__ldg(a), __ldg(a + 1), __ldg(a + 2)};
}

// Project a node with camera cam: the first two thirds of its splat record, its radius,
// and the footprint record {x0 | x1 << 16, y0 | y1 << 16, pair count, depth bits}.
__device__ __forceinline__ uint4 project_one(const DevCamera& cam, const NodeAttr& at, float4& rec0, float4& rec1,
                                             float& radius)
{
    const float4 q0 = at.q0, q1 = at.q1, q2 = at.q2;
    const float ftx = (float)cam.tiles_x, fty = (float)cam.tiles_y;
    uint32_t cnt = 0;
    // ---- decision-exact binary32: frustum, EWA covariance, footprint
    const float mx = q0.x, my = q0.y, mz = q0.z;
    const float s6[6] = {q1.x, q1.y, q1.z, q1.w, q2.x, q2.y};
    const float a0 = q0.w;
    const float ln_a0 = q2.z;
    float vx, vy, vz, txtz = 0.0f, tytz = 0.0f;
    camera_space(cam, mx, my, mz, vx, vy, vz);
    const bool inf = frustum_test(cam, vx, vy, vz, txtz, tytz);
    float a = 0.0f, b = 0.0f, c = 0.0f, lam = 0.0f;
    if (inf) ewa_cov2d(cam, vz, txtz, tytz, s6, a, b, c, lam);
    // x / z and y / z: the frustum test's quotients when it formed them (depth above 0.2)
    const float u = fa(fm(cam.fx, vz > 0.2f ? txtz : fd(vx, vz)), cam.cx);
    const float v = fa(fm(cam.fy, vz > 0.2f ? tytz : fd(vy, vz)), cam.cy);
    const float det = fs(fm(a, c), fm(b, b));
    const float lthr = fs(-5.5412635451584258f, ln_a0);   // -ln 255 - ln alpha0
    float A = 0.0f, B = 0.0f, C = 0.0f;
    radius = 0.0f;
    int32_t x0 = 0, x1 = 0, y0 = 0, y1 = 0;
    if (inf && det > 0.0f) {
        A = fd(c, det);
        B = fd(-b, det);
        C = fd(a, det);
        // 3-sigma radius, or the radius where alpha0 e^{-r^2/(2 lambda)} = tau,
        // capped at 3 sigma; alpha0 <= tau emits nothing (§3.3)
        float r = fm(3.0f, fsq(lam));
        bool drop = false;
        if (cam.shrink) {
            const float g = fm(2.0f, fs(ln_a0, cam.ln_tau));
            if (!(g > 0.0f)) drop = true;
            else if (g < 9.0f) r = fsq(fm(lam, g));
        }
        if (!drop) {
            radius = r;
            // tiles are powers of two wide and high, so x / w is x * (1 / w) bit for bit
            // (both the correctly rounded x * 2^-k)
            const float iw = __uint_as_float((uint32_t)(127 - cam.tile_shift_x) << 23);
            const float ih = __uint_as_float((uint32_t)(127 - cam.tile_shift_y) << 23);
            const float fx0 = clampf(floorf(fm(fs(u, r), iw)), 0.0f, ftx);
            const float fx1 = clampf(fa(floorf(fm(fa(u, r), iw)), 1.0f), 0.0f, ftx);
            const float fy0 = clampf(floorf(fm(fs(v, r), ih)), 0.0f, fty);
            const float fy1 = clampf(fa(floorf(fm(fa(v, r), ih)), 1.0f), 0.0f, fty);
            x0 = (int32_t)fx0; x1 = (int32_t)fx1; y0 = (int32_t)fy0; y1 = (int32_t)fy1;
            if (x1 > x0 && y1 > y0) cnt = (uint32_t)((x1 - x0) * (y1 - y0));
        }
    }
    rec0 = make_float4(u, v, A, B);
    rec1 = make_float4(C, lthr, a0, vz);
    return make_uint4((uint32_t)x0 | ((uint32_t)x1 << 16), (uint32_t)y0 | ((uint32_t)y1 << 16), cnt,
                      __float_as_uint(vz));
}

constexpr int kWarps = kProjectThreads / 32;

// Row stride in shared memory, in 16-byte units: odd, so that the 8 lanes of a
// quarter-warp, each reading its own row, hit different banks.
template <int kDeg>
struct Rows {
    static constexpr int kQ = ((kDeg + 1) * (kDeg + 1) * 3 + 3) / 4;
    static constexpr int kStride = kQ | 1;
    float4 v[kWarps][32 * kStride];
};

// The projection of the selected entries sel[m], m < M: splat record, footprint record,
// pairs counted into their tiles.  A warp takes 32 consecutive entries, one a lane.
// view(e, n, tiles_x, first tile) gives entry e's node and camera.
//
// Bound: latency of two dependent gathers (attributes, then the SH rows of those that
// emit pairs: no pixel reads the colour of the others, about 40% of a selection under
// shrinking, so their rows are not fetched).  So the rows are copied to shared memory
// asynchronously, whole rows by consecutive lanes (a lane's own 16-byte loads touch half
// of each sector and wait where they are used), while the warp counts its pairs and the
// next 32 entries' attributes are on their way.  537K Gaussians of degree 3 (450K emitting,
// 1.13M pairs): 44 -> 37 us, 157 MB; 8 views, 7.5M entries: 258 -> 252 us, 1.45 GB of DRAM.
template <int kDeg, class View>
__device__ __forceinline__ void project_walk(const DevTree& t, const uint32_t* __restrict__ sel, Rows<kDeg>& S,
                                             float* __restrict__ splat, uint4* __restrict__ foot,
                                             uint32_t* __restrict__ tile_cnt, FrameState* st, View view)
{
    constexpr int kQ = Rows<kDeg>::kQ, kStride = Rows<kDeg>::kStride;
    const uint32_t lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const uint32_t M = st->M, step = gridDim.x * kProjectThreads;
    float4* rows = S.v[warp];
    uint32_t base = blockIdx.x * kProjectThreads + warp * 32u;
    if (base >= M) return;
    uint32_t emitting = 0;
    uint32_t e = __ldg(sel + min(base + lane, M - 1u)), n, tiles_x, tbase;
    const DevCamera* cam = &view(e, n, tiles_x, tbase);
    NodeAttr at = load_attr(t, n);
    uint32_t e_next = base + step < M ? __ldg(sel + min(base + step + lane, M - 1u)) : e;
    while (true) {
        const uint32_t m = base + lane;
        float4 rec0, rec1;
        float radius;
        uint4 f = project_one(*cam, at, rec0, rec1, radius);
        if (m >= M) f.z = 0u;
        const uint32_t emit = __ballot_sync(0xffffffffu, f.z > 0u);
        emitting += (uint32_t)__popc(emit);
        // the SH rows of the emitting lanes (in a small view of a large scene often none): 16
        // bytes a lane and step, row by row
        if (emit) {
#pragma unroll
            for (int i = 0; i < kQ; ++i) {
                const uint32_t idx = (uint32_t)i * 32u + lane, r = idx / kQ, k = idx - r * kQ;
                const uint32_t nr = __shfl_sync(0xffffffffu, n, r);
                if ((emit >> r) & 1u)
                    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(
                                     (uint32_t)__cvta_generic_to_shared(rows + r * kStride + k)),
                                 "l"(t.sh + (size_t)nr * t.sh_stride + 4 * k)
                                 : "memory");
            }
        }
        // direction to the colour; then the next entries' attributes
        float dx = at.q0.x - cam->campos[0], dy = at.q0.y - cam->campos[1], dz = at.q0.z - cam->campos[2];
        const uint32_t cur_tx = tiles_x, cur_tb = tbase;
        const bool more = base + step < M;
        if (more) {
            cam = &view(e_next, n, tiles_x, tbase);
            at = load_attr(t, n);
            if (base + 2u * step < M) e_next = __ldg(sel + min(base + 2u * step + lane, M - 1u));
        }
        float4* out = reinterpret_cast<float4*>(splat + (size_t)m * kSplatStride);
        if (m < M) {
            foot[m] = f;
            out[0] = rec0;
            out[1] = rec1;
        }
        warp_count_pairs(f.z, f.x, f.y, cur_tx, cur_tb, tile_cnt);
        asm volatile("cp.async.wait_all;" ::: "memory");
        __syncwarp();
        // ---- colour (FMA allowed: decides nothing)
        float rgb[3] = {0.0f, 0.0f, 0.0f};
        if (f.z) {
            const float il = rsqrtf(dx * dx + dy * dy + dz * dz);
            dx *= il; dy *= il; dz *= il;
            sh_colour<kDeg>(rows + lane * kStride, dx, dy, dz, rgb);
        }
        if (m < M) out[2] = make_float4(rgb[0], rgb[1], rgb[2], radius);
        if (!more) break;
        base += step;
        __syncwarp();                              // the rows are read before they are overwritten
    }
    if (lane == 0 && emitting) atomicAdd(&st->n_emitting, emitting);
}

}  // namespace proj
}  // namespace fgs
