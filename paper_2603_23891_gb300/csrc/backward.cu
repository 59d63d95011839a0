// Differentiable form of the render path: parameter preparation, and the
// hand-written backward of blending (Eq. 2), EWA projection and SH colour.
//
// Selection, tile rectangles and every skip / stop decision of blending are
// held fixed (a discrete cut), as in 3DGS training.  Per-Gaussian parameters:
// mean mu, log-scale s, quaternion q (any norm), opacity logit l, SH
// coefficients; Sigma = R(q/|q|) diag(e^{2s}) R^T, alpha0 = sigmoid(l).
//
// blend_bwd_kernel starts from each pixel's final transmittance and stop position (the
// 8 bytes per pixel that a FGS_RENDER_KEEP forward kept, or that the forward's walk,
// run once more without an image, leaves) and walks the tile back to front,
// recovering T before each Gaussian as T / (1 - alpha); chunks past the last stop of
// the tile are never loaded.  The gradients with respect to the splat record (u, v,
// conic A B C, alpha0, colour) of a Gaussian are summed over a 4x4 block of pixels by one lane
// and added per Gaussian; project_bwd_kernel then applies the chain rule to the
// parameters.
#include "blend_impl.cuh"

#include "project_impl.cuh"

namespace fgs {

constexpr int kGS = 12;   // floats per splat gradient: u v A B C a0 r g b (3 spare)

// ---------------------------------------------------------------------------
// parameters -> binary32 attributes, in one fixed operation order (no fused
// operations), so that the selection and blending decisions taken on them are
// reproducible bit for bit by any IEEE binary32 implementation of that order
// ---------------------------------------------------------------------------

// ln x for positive normal x: x = 2^e m, m in [sqrt(1/2), sqrt(2)] from the
// exponent bits; ln m = 2 atanh(s), s = (m - 1) / (m + 1), by the odd series
// 2 s (1 + s^2/3 + s^4/5 + s^6/7 + s^8/9) (|s| < 0.172, truncation below 1e-9
// relative; Abramowitz & Stegun 4.1.27); plus e ln 2.
__device__ __forceinline__ float ln_cw(float x)
{
    const uint32_t b = __float_as_uint(x);
    int e = (int)((b >> 23) & 0xffu) - 127;
    float m = __uint_as_float((b & 0x7fffffu) | 0x3f800000u);
    if (m > 1.41421356f) {
        m = fm(m, 0.5f);
        e += 1;
    }
    const float s = fd(fs(m, 1.0f), fa(m, 1.0f));
    const float s2 = fm(s, s);
    float p = 0.111111111f;
    p = fa(fm(p, s2), 0.142857143f);
    p = fa(fm(p, s2), 0.2f);
    p = fa(fm(p, s2), 0.333333333f);
    p = fa(fm(p, s2), 1.0f);
    return fa(fm((float)e, 0.693147182f), fm(fm(2.0f, s), p));
}

struct ParamPtrs {
    const float* mu;          // [3][n]
    const float* log_scale;   // [3][n]
    const float* quat;        // [4][n] (w, x, y, z), any non-zero norm
    const float* logit;       // [n]
    const float* sh;          // [n][K][3]
    uint32_t n;
};

constexpr float kLogitMax = 80.0f;

// Sigma = R(q/|q|) diag(e^{2 s}) R(q/|q|)^T (6 upper-triangle entries, order
// xx xy xz yy yz zz) and the pieces the backward needs.
__device__ __forceinline__ void sigma_from(const ParamPtrs& p, uint32_t n, float cov[6], float R[9],
                                           float s2[3], float qh[4], float& qn)
{
    const size_t N = p.n;
    const float w = p.quat[n], x = p.quat[N + n], y = p.quat[2 * N + n], z = p.quat[3 * N + n];
    qn = fsq(fa(fa(fa(fm(w, w), fm(x, x)), fm(y, y)), fm(z, z)));
    const float qw = fd(w, qn), qx = fd(x, qn), qy = fd(y, qn), qz = fd(z, qn);
    qh[0] = qw; qh[1] = qx; qh[2] = qy; qh[3] = qz;
    R[0] = fs(1.0f, fm(2.0f, fa(fm(qy, qy), fm(qz, qz))));
    R[1] = fm(2.0f, fs(fm(qx, qy), fm(qw, qz)));
    R[2] = fm(2.0f, fa(fm(qx, qz), fm(qw, qy)));
    R[3] = fm(2.0f, fa(fm(qx, qy), fm(qw, qz)));
    R[4] = fs(1.0f, fm(2.0f, fa(fm(qx, qx), fm(qz, qz))));
    R[5] = fm(2.0f, fs(fm(qy, qz), fm(qw, qx)));
    R[6] = fm(2.0f, fs(fm(qx, qz), fm(qw, qy)));
    R[7] = fm(2.0f, fa(fm(qy, qz), fm(qw, qx)));
    R[8] = fs(1.0f, fm(2.0f, fa(fm(qx, qx), fm(qy, qy))));
#pragma unroll
    for (int k = 0; k < 3; ++k) s2[k] = exp_cw(fm(2.0f, p.log_scale[k * N + n]));
    constexpr int ij[6][2] = {{0, 0}, {0, 1}, {0, 2}, {1, 1}, {1, 2}, {2, 2}};
#pragma unroll
    for (int e = 0; e < 6; ++e) {
        const int i = ij[e][0], j = ij[e][1];
        cov[e] = fa(fa(fm(fm(R[3 * i], s2[0]), R[3 * j]), fm(fm(R[3 * i + 1], s2[1]), R[3 * j + 1])),
                    fm(fm(R[3 * i + 2], s2[2]), R[3 * j + 2]));
    }
}

__device__ __forceinline__ float clamp_logit(float l)
{
    return l < -kLogitMax ? -kLogitMax : (l > kLogitMax ? kLogitMax : l);
}

// Parameters -> the tree attributes the frame kernels read: mu, Sigma,
// alpha0 = sigmoid(l), ln alpha0 = -ln(1 + e^{-l}) (l clamped to [-80, 80]), the boxes of
// 128 centres, SH.  Three passes over different data in one launch: the SH rows
// (coefficients [n][K3] -> rows of sh_stride floats; vec: sh_stride == K3 and the source
// 16-byte aligned, so one flat copy by 16-byte loads, four in flight a thread), the
// boxes (a warp a chunk, from the parameters), the attributes (a thread a node).
// Bound: HBM, 4 (11 + K3) bytes read and 4 (21 + sh_stride) written a node.  1.25M nodes
// of degree 3: 135 us as three launches with 4-byte SH copies.
template <int kDeg>
__global__ void __launch_bounds__(256) prep_kernel(DevTree t, ParamPtrs p, bool vec)
{
    grid_dep_wait();
    const uint32_t tid = blockIdx.x * blockDim.x + threadIdx.x, nt = gridDim.x * blockDim.x;
    constexpr uint64_t K3 = (kDeg + 1) * (kDeg + 1) * 3;
    float* sh = const_cast<float*>(t.sh);
    if (K3 % 4 == 0 && vec) {
        const uint64_t total = (uint64_t)t.n * K3 / 4;
        const float4* src = reinterpret_cast<const float4*>(p.sh);
        float4* dst = reinterpret_cast<float4*>(sh);
        uint64_t i = tid;
        for (; i + 3ull * nt < total; i += 4ull * nt) {
            float4 v[4];
#pragma unroll
            for (int k = 0; k < 4; ++k) v[k] = __ldcs(src + i + (uint64_t)k * nt);
#pragma unroll
            for (int k = 0; k < 4; ++k) dst[i + (uint64_t)k * nt] = v[k];
        }
        for (; i < total; i += nt) dst[i] = __ldcs(src + i);
    } else {
        const uint64_t total = (uint64_t)t.n * K3;
        for (uint64_t i = tid; i < total; i += nt) {
            const uint64_t n = i / K3;                              // a multiply: K3 is a constant
            sh[n * t.sh_stride + (i - n * K3)] = __ldg(p.sh + i);
        }
    }
    chunk_boxes(p.mu, p.n, p.n, t.n_pad >> 7, const_cast<float4*>(t.cbox), tid, nt);
    float* mu = const_cast<float*>(t.mu);
    float* cov = const_cast<float*>(t.cov);
    const size_t np = t.n_pad, N = p.n;
    for (uint32_t n = tid; n < p.n; n += nt) {
#pragma unroll
        for (int k = 0; k < 3; ++k) mu[k * np + n] = p.mu[k * N + n];
        float c6[6], R[9], s2[3], qh[4], qn;
        sigma_from(p, n, c6, R, s2, qh, qn);
#pragma unroll
        for (int k = 0; k < 6; ++k) cov[k * np + n] = c6[k];
        const float den = fa(1.0f, exp_cw(-clamp_logit(p.logit[n])));
        const float a0 = fd(1.0f, den), la0 = -ln_cw(den);
        float4* attr = const_cast<float4*>(t.attr) + 3 * (size_t)n;
        attr[0] = make_float4(p.mu[n], p.mu[N + n], p.mu[2 * N + n], a0);
        attr[1] = make_float4(c6[0], c6[1], c6[2], c6[3]);
        attr[2] = make_float4(c6[4], c6[5], la0, 0.0f);
    }
}

// ---------------------------------------------------------------------------
// blend backward
// ---------------------------------------------------------------------------
// Shared memory of the back-to-front gradient walk.
struct BwdWarp {                                                  // one warp's: 32 entries at a time
    float n[32][blendk::kParkStride];                             // -power at a block's 16 pixels
    float w[32][blendk::kParkStride];                             // alpha T, 0 where the entry is not applied
    float g[32][blendk::kParkStride];                             // dL/dpower, 0 likewise
    float4 col[32];                                               // alpha0, r, g, b
    uint8_t list[4][blendk::kWalkChunk];                          // per block: the chunk's records it may meet
};
struct BwdSmem {
    float4 r0[blendk::kWalkChunk];                                // u, v, A, B
    float4 r1[blendk::kWalkChunk];                                // C, lthr, alpha0, depth
    float4 r2[blendk::kWalkChunk];                                // r, g, b, radius
    uint16_t mask[blendk::kWalkChunk];
    float dC[3][256];                                             // dL/dC by block, in the parked order
    uint32_t last[blendk::kWalkWarps];
    BwdWarp w[blendk::kWalkWarps];
};

// Gradient walk of a tile (kLanes = 8) or its half `part` (kLanes = 16), laid out as the
// forward's walk (blend_walk): lanes, blocks, chunks, lists and the test are the same,
// the chunks and the lists' groups of kLanes entries taken from the last to the first.
// keep holds each pixel's {final T, stop}; a pixel takes part in the list entries
// before its stop.  Per group of entries:
//  * test: a lane an entry, as in the forward;
//  * apply: a lane its own pixels' hits, back to front: T before the entry is
//    T / (1 - alpha), D = dL/dC . (colour behind) follows, and w = alpha T and
//    dL/dpower are parked for (entry, pixel);
//  * gather: a lane an entry again: the sums over the block's 16 pixels of w dL/dC and
//    of dL/dpower times 1, dx, dy, dx^2, dx dy, dy^2, two pixels to an instruction, from
//    which the splat's nine gradients follow, added with three reductions (two of four
//    floats).  (With a lane a pixel throughout, every list entry cost 9 products, 11
//    shuffles and 9 reductions for 32 pixels, hit or not: about 130 instructions.)
// Bound: instruction issue.
template <int kLanes>
__device__ __forceinline__ void blend_bwd_walk(const DevCamera& cam, uint32_t tile, uint32_t part, uint2 rg,
                                               BwdSmem& S, const uint32_t* __restrict__ vals,
                                               const float* __restrict__ splat, const uint2* __restrict__ keep,
                                               const float* __restrict__ dL_drgb, float* __restrict__ gsplat,
                                               const FrameState* st)
{
    using namespace blendk;
    constexpr bool kTwo = kLanes == 8;                             // pixels a lane
    constexpr uint32_t kC = kWalkChunk, kBlocks = 32 / kLanes;
    constexpr uint32_t kPx0 = kTwo ? 0xAAAAu : 0xFFFFu, kPx1 = kTwo ? 0x5555u : 0u;      // mask bits a pixel
    const uint32_t tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const uint32_t b = lane / kLanes, i = lane % kLanes;
    const uint32_t M = st->M;
    BwdWarp& W = S.w[warp];
    const int32_t tx0 = (int32_t)(tile % (uint32_t)cam.tiles_x) * cam.tile_w;
    const int32_t ty0 = (int32_t)(tile / (uint32_t)cam.tiles_x) * cam.tile_h;
    const uint32_t fb = kTwo ? 4u * warp : 8u * part + 2u * warp;
    int32_t ox, oy;
    uint32_t bsh;
    walk_origin(cam, fb >> 2, ox, oy, bsh);
    const uint32_t bb = (fb & 3u) + b;
    const int32_t bx0 = tx0 + ox + (int32_t)((bb & ((1u << bsh) - 1u)) << 2);
    const int32_t by0 = ty0 + oy + (int32_t)((bb >> bsh) << 2);
    const uint32_t pp = kTwo ? i : i >> 1;
    const int32_t x = bx0 + (int32_t)(pp & 3u);
    const int32_t y = by0 + (int32_t)(pp >> 2 << 1) + (kTwo ? 0 : 1 - (int32_t)(i & 1u));
    const uint32_t park = kTwo ? 2u * i : i ^ 1u;                  // the first pixel's place in the parked order

    // the pixels' forward outcome: final T, stop position; dL/dC
    f32x2 T, dC0, dC1, dC2;
    uint32_t lim[2] = {rg.x, rg.x};
    {
        float t[2] = {1.0f, 1.0f}, d[3][2] = {};
        const size_t hw = (size_t)cam.width * cam.height;
#pragma unroll
        for (int k = 0; k < (kTwo ? 2 : 1); ++k) {
            if (x < cam.width && y + k < cam.height) {
                const size_t pix = (size_t)(y + k) * cam.width + x;
                const uint2 kp = __ldg(keep + pix);
                t[k] = __uint_as_float(kp.x);
                lim[k] = kp.y;
#pragma unroll
                for (int c = 0; c < 3; ++c) d[c][k] = __ldg(dL_drgb + c * hw + pix);
            }
#pragma unroll
            for (int c = 0; c < 3; ++c) S.dC[c][32u * kBlocks / 2u * warp + 16u * b + park + k] = d[c][k];
        }
        T = pack2(t[0], t[1]);
        dC0 = pack2(d[0][0], d[0][1]);
        dC1 = pack2(d[1][0], d[1][1]);
        dC2 = pack2(d[2][0], d[2][1]);
    }
    // dL/dC . colour behind
    f32x2 D = mul2(mul2(dC0, dup2(cam.bg[0])), T);
    D = fma2(mul2(dC1, dup2(cam.bg[1])), T, D);
    D = fma2(mul2(dC2, dup2(cam.bg[2])), T, D);

    // the blocks' last stops, and the walk's
    uint32_t blim = max(lim[0], lim[1]);
#pragma unroll
    for (int o = kLanes / 2; o > 0; o >>= 1) blim = max(blim, __shfl_xor_sync(kFull, blim, o));
    uint32_t bl[kBlocks];
#pragma unroll
    for (uint32_t k = 0; k < kBlocks; ++k) bl[k] = __shfl_sync(kFull, blim, k * kLanes);
    uint32_t e = bl[0];
#pragma unroll
    for (uint32_t k = 1; k < kBlocks; ++k) e = max(e, bl[k]);
    if (lane == 0) S.last[warp] = e;
    __syncthreads();
#pragma unroll
    for (int k = 0; k < kWalkWarps; ++k) e = max(e, S.last[k]);
    e = min(e, rg.y);                    // no pixel of the tile (half) reaches past e
    if (e <= rg.x) return;

    f32x2 npx[4], npy[2];                                          // minus the block's pixel centres
#pragma unroll
    for (int k = 0; k < 4; ++k) npx[k] = dup2(-fa((float)(bx0 + k), 0.5f));
#pragma unroll
    for (int k = 0; k < 2; ++k)
        npy[k] = pack2(-fa((float)(by0 + 2 * k), 0.5f), -fa((float)(by0 + 2 * k + 1), 0.5f));

    const uint32_t n_chunks = (e - rg.x + kC - 1u) / kC;
    uint32_t m = 0u;
    {
        const uint32_t at = rg.x + (n_chunks - 1u) * kC + tid;
        if (at < e) m = __ldg(vals + at);
    }
    for (uint32_t c = n_chunks; c-- > 0u;) {
        const uint32_t s0 = rg.x + c * kC;
        const uint32_t cnt = e - s0 < kC ? e - s0 : kC;
        // ---- stage
        if (tid < cnt) {
            if (m >= M) m = 0;      // only after a failed sort (status already latched)
            const float4* g = reinterpret_cast<const float4*>(splat + (size_t)m * kSplatStride);
            const float4 g0 = __ldg(g), g1 = __ldg(g + 1), g2 = __ldg(g + 2);
            S.r0[tid] = g0;
            S.r1[tid] = staged_r1(g1);
            S.r2[tid] = g2;
            S.mask[tid] = (uint16_t)walk_mask(cam, tx0, ty0, g0.x, g0.y, g0.z, g0.w, g1.x, g1.y);
        }
        if (c > 0u) m = __ldg(vals + s0 - kC + tid);
        __syncthreads();
        // ---- list: the block's records before its last stop; how many before each pixel's own
        uint32_t len[kBlocks] = {}, own[2] = {0u, 0u};
        const uint32_t lt = (1u << lane) - 1u;
        for (uint32_t j0 = 0; j0 < cnt; j0 += 32) {
            const uint32_t j = j0 + lane;
            const uint32_t bm = j < cnt ? (uint32_t)S.mask[j] >> fb : 0u;
            uint32_t mine = 0u;
#pragma unroll
            for (uint32_t k = 0; k < kBlocks; ++k) {
                const bool in = (bm & (1u << k)) && s0 + j < bl[k];
                const uint32_t v = __ballot_sync(kFull, in);
                if (in) W.list[k][len[k] + __popc(v & lt)] = (uint8_t)j;
                len[k] += __popc(v);
                mine = b == k ? v : mine;
            }
#pragma unroll
            for (int k = 0; k < (kTwo ? 2 : 1); ++k) {
                const uint32_t r = lim[k] > s0 + j0 ? lim[k] - s0 - j0 : 0u;   // the pixel's records of these 32
                own[k] += __popc(mine & ~(r < 32u ? kFull << r : 0u));
            }
        }
        __syncwarp();
        uint32_t left = len[0];
#pragma unroll
        for (uint32_t k = 1; k < kBlocks; ++k) left = b == k ? len[k] : left;
        const uint32_t en = (uint32_t)kLanes - 1u - i;             // (the transposition leaves entry 0 on top)
        while (__any_sync(kFull, left != 0u)) {
            // ---- test: one entry a lane at its block's 16 pixels; entry 0 is the list's last
            const bool valid = en < left;
            const uint32_t rs = valid ? W.list[b][left - 1u - en] : 0u;
            const uint32_t sl = b * kLanes + en;
            uint32_t hits = 0u;
            {
                const float4 a = S.r0[rs], cc = S.r1[rs], q = S.r2[rs];
                W.col[sl] = make_float4(cc.z, q.x, q.y, q.z);
                f32x2 dx[4];
#pragma unroll
                for (int k = 0; k < 4; ++k) dx[k] = add2(dup2(a.x), npx[k]);
                const f32x2 hA = dup2(fm(0.5f, a.z)), B2 = dup2(a.w), hC = dup2(fm(0.5f, cc.x)), K = dup2(-cc.y);
#pragma unroll
                for (int rp = 1; rp >= 0; --rp) {
                    const f32x2 dy = add2(dup2(a.y), npy[rp]);
                    const f32x2 bdy = mul2(B2, dy), cdy = mul2(mul2(hC, dy), dy);
                    f32x2 n[4];
#pragma unroll
                    for (int k = 3; k >= 0; --k) {
                        n[k] = fma2(fma2(hA, dx[k], bdy), dx[k], cdy);
                        const float2 p = unpack2(mul2(n[k], fma2(n[k], dup2(-1.0f), K)));
                        hits = __funnelshift_l(__float_as_uint(p.x), hits, 1);
                        hits = __funnelshift_l(__float_as_uint(p.y), hits, 1);
                    }
                    float* pn = &W.n[sl][8 * rp];
                    *reinterpret_cast<ulonglong2*>(pn) = make_ulonglong2(n[0], n[1]);
                    *reinterpret_cast<ulonglong2*>(pn + 4) = make_ulonglong2(n[2], n[3]);
                }
                hits = valid ? ~hits & 0xFFFFu : 0u;
            }
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                *reinterpret_cast<float4*>(&W.w[sl][4 * k]) = make_float4(0.f, 0.f, 0.f, 0.f);
                *reinterpret_cast<float4*>(&W.g[sl][4 * k]) = make_float4(0.f, 0.f, 0.f, 0.f);
            }
            // the first left - own entries lie behind the pixel's stop
            const uint32_t d0 = left > own[0] ? left - own[0] : 0u, d1 = left > own[1] ? left - own[1] : 0u;
            uint32_t mask = transpose_bits<kLanes>(hits, i) &
                            ((kPx0 & shr0(0xFFFFu, (kTwo ? 2u : 1u) * d0)) | (kPx1 & shr0(0xFFFFu, 2u * d1)));
            mask <<= 16;
            __syncwarp();
            // ---- apply
            while (__any_sync(kFull, mask != 0u)) {
                uint32_t sh = clz_or_ones(mask);
                if (kTwo) sh &= ~1u;
                const uint32_t h = mask & shr0(kTwo ? 0xC0000000u : 0x80000000u, sh);
                const bool h0 = (h & (kPx0 << 16)) != 0u, h1 = (h & (kPx1 << 16)) != 0u;
                mask ^= h;
                const uint32_t at = b * kLanes + ((kTwo ? sh >> 1 : sh) & (kLanes - 1u));
                const float4 cv = W.col[at];
                auto alpha1 = [&](float n) {                       // before the clamp
                    uint32_t t;
                    const float p = exp_poly_neg(n, t);
                    return fm(cv.x, fm(p, __uint_as_float((t << 23) + (127u << 23))));
                };
                // dL/dC . colour; a pixel that does not apply the entry keeps D (0 times an
                // infinite colour would not be 0)
                f32x2 qd = fma2(dC2, dup2(cv.w), fma2(dC1, dup2(cv.z), mul2(dC0, dup2(cv.y))));
                if constexpr (kTwo) {
                    const float2 q = unpack2(qd);
                    qd = pack2(h0 ? q.x : 0.0f, h1 ? q.y : 0.0f);
                    const float2 n = *reinterpret_cast<const float2*>(&W.n[at][park]);
                    const float r0 = alpha1(n.x), r1 = alpha1(n.y);
                    const f32x2 al = pack2(h0 ? fminf(r0, 0.99f) : 0.0f, h1 ? fminf(r1, 0.99f) : 0.0f);
                    const float2 om = unpack2(fma2(al, dup2(-1.0f), dup2(1.0f)));
                    const f32x2 iom = pack2(rcp1(om.x), rcp1(om.y));
                    T = mul2(T, iom);                              // before the entry
                    const f32x2 w = mul2(al, T);
                    const float2 gp = unpack2(mul2(fma2(mul2(iom, D), dup2(-1.0f), mul2(T, qd)), al));
                    D = fma2(w, qd, D);
                    if (h) {
                        *reinterpret_cast<f32x2*>(&W.w[at][park]) = w;
                        // a clamped alpha does not move
                        *reinterpret_cast<float2*>(&W.g[at][park]) =
                            make_float2(h0 && r0 < 0.99f ? gp.x : 0.0f, h1 && r1 < 0.99f ? gp.y : 0.0f);
                    }
                } else {
                    const float r0 = alpha1(W.n[at][park]);
                    const float al = h0 ? fminf(r0, 0.99f) : 0.0f;
                    const float iom = rcp1(1.0f - al), q0 = unpack2(qd).x, d = unpack2(D).x;
                    const float t = unpack2(T).x * iom, w = al * t;
                    if (h0) {
                        W.w[at][park] = w;
                        W.g[at][park] = r0 < 0.99f ? (t * q0 - iom * d) * al : 0.0f;
                    }
                    T = pack2(t, 0.0f);
                    D = pack2(h0 ? fmaf(w, q0, d) : d, 0.0f);
                }
            }
            __syncwarp();
            // ---- gather: the entry's sums over the block's pixels
            if (hits) {
                f32x2 R = 0ull, G = 0ull, Bs = 0ull, S0 = 0ull, Sx = 0ull, Sy = 0ull, Sxx = 0ull, Sxy = 0ull, Syy = 0ull;
                const uint32_t dc = 32u * kBlocks / 2u * warp + 16u * b;
                const float4 a = S.r0[rs], cc = S.r1[rs];
                f32x2 dx[4];
#pragma unroll
                for (int k = 0; k < 4; ++k) dx[k] = add2(dup2(a.x), npx[k]);
#pragma unroll
                for (int rp = 0; rp < 2; ++rp) {
                    f32x2 sr = 0ull, rx = 0ull;
#pragma unroll
                    for (int k = 0; k < 4; k += 2) {
                        const int o = 8 * rp + 2 * k;
                        const ulonglong2 w = *reinterpret_cast<const ulonglong2*>(&W.w[sl][o]);
                        const ulonglong2 g = *reinterpret_cast<const ulonglong2*>(&W.g[sl][o]);
                        const ulonglong2 c0 = *reinterpret_cast<const ulonglong2*>(&S.dC[0][dc + o]);
                        const ulonglong2 c1 = *reinterpret_cast<const ulonglong2*>(&S.dC[1][dc + o]);
                        const ulonglong2 c2 = *reinterpret_cast<const ulonglong2*>(&S.dC[2][dc + o]);
                        R = fma2(w.y, c0.y, fma2(w.x, c0.x, R));
                        G = fma2(w.y, c1.y, fma2(w.x, c1.x, G));
                        Bs = fma2(w.y, c2.y, fma2(w.x, c2.x, Bs));
                        sr = add2(g.y, add2(g.x, sr));
                        const f32x2 x0 = mul2(g.x, dx[k]), x1 = mul2(g.y, dx[k + 1]);
                        rx = add2(x1, add2(x0, rx));
                        Sxx = fma2(x1, dx[k + 1], fma2(x0, dx[k], Sxx));
                    }
                    S0 = add2(S0, sr);
                    Sx = add2(Sx, rx);
                    const f32x2 dy = add2(dup2(a.y), npy[rp]), ry = mul2(sr, dy);
                    Sxy = fma2(rx, dy, Sxy);
                    Sy = add2(Sy, ry);
                    Syy = fma2(ry, dy, Syy);
                }
                auto total = [](f32x2 v) {
                    const float2 f = unpack2(v);
                    return f.x + f.y;
                };
                const float sx = total(Sx), sy = total(Sy);
                float* out = gsplat + (size_t)min(__ldg(vals + s0 + rs), M - 1u) * kGS;
                // d power / du = -(A dx + B dy), likewise for v; d alpha / d alpha0 = alpha / alpha0
                atomicAdd(reinterpret_cast<float4*>(out),
                          make_float4(-(a.z * sx + a.w * sy), -(cc.x * sy + a.w * sx), -0.5f * total(Sxx), -total(Sxy)));
                atomicAdd(reinterpret_cast<float4*>(out) + 1,
                          make_float4(-0.5f * total(Syy), total(S0) / cc.z, total(R), total(G)));
                atomicAdd(out + 8, total(Bs));
            }
            __syncwarp();
            left -= min(left, (uint32_t)kLanes);
        }
        __syncthreads();
    }
}

// Gradients to zero: p[0..3] of per_node[k] floats a node for all n nodes, sh ([n][k3])
// for the nodes without a bit in selbits (the others' rows are all written later).  vec:
// rows of sh are multiples of 16 bytes and aligned.
struct GradZero {
    float* p[4];
    uint32_t per_node[4];
    float* sh;
    uint32_t k3;
    bool vec;
    const uint32_t* selbits;
    uint32_t n;
    uint32_t blocks;
};

// Block `part` of n_parts' share of the zeros, past L2 (nothing reads them soon): 16-byte
// stores where the array allows.
__device__ __forceinline__ void zero_share(const GradZero& z, uint32_t part, uint32_t n_parts)
{
    const float4 zero4 = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
    for (int k = 0; k < 4; ++k) {
        const uint64_t total = (uint64_t)z.per_node[k] * z.n;
        const uint64_t lo = total * part / n_parts, hi = total * (part + 1ull) / n_parts;
        float* p = z.p[k];
        uint64_t a = lo + ((4ull - (((uint64_t)p / 4ull + lo) & 3ull)) & 3ull);      // the first 16-byte boundary
        if (a > hi) a = hi;
        const uint64_t b = a + ((hi - a) & ~3ull);
        for (uint64_t i = lo + threadIdx.x; i < a; i += blockDim.x) p[i] = 0.0f;
        for (uint64_t i = a + 4ull * threadIdx.x; i < b; i += 4ull * blockDim.x)
            __stcs(reinterpret_cast<float4*>(p + i), zero4);
        for (uint64_t i = b + threadIdx.x; i < hi; i += blockDim.x) p[i] = 0.0f;
    }
    // a warp 32 nodes (a word of selbits) at a time, 16 (or 4) bytes a lane and step
    const uint32_t lane = threadIdx.x & 31, n_words = (z.n + 31u) >> 5, n_warps = n_parts * (blockDim.x >> 5);
    const uint32_t unit = z.vec ? 4u : 1u, q = z.k3 / unit;
    const uint32_t inv = (65536u + q - 1u) / q;           // i / q = i * inv >> 16 for i < 32 q <= 1536 and these q
    for (uint32_t w = part * (blockDim.x >> 5) + (threadIdx.x >> 5); w < n_words; w += n_warps) {
        const uint32_t left = z.n - (w << 5);
        const uint32_t rows = ~__ldg(z.selbits + w) & (left < 32u ? (1u << left) - 1u : 0xFFFFFFFFu);
        if (!rows) continue;
        float* p = z.sh + ((size_t)w << 5) * z.k3;
        for (uint32_t i = lane; i < 32u * q; i += 32u)
            if ((rows >> (i * inv >> 16)) & 1u) {
                if (z.vec) __stcs(reinterpret_cast<float4*>(p) + i, zero4);
                else p[i] = 0.0f;
            }
    }
}

// keep holds each pixel's {final T, stop} (kept by a FGS_RENDER_KEEP forward, or
// recomputed by the forward's walk without an image just before).  zero: the gradients
// of nodes outside the selection, written by the first zero.blocks blocks beside the
// walk, where HBM idles (1.25M nodes of degree 3, 537K selected: 43 us of memsets and their
// launches before; a share of the zeros in every block delayed its walk, 252 us instead
// of 190; all rows by blocks of their own 224, the unselected nodes' alone 214).
__global__ void __launch_bounds__(blendk::kWalkChunk) blend_bwd_kernel(
    DevCamera cam, const uint2* __restrict__ ranges, const uint32_t* __restrict__ heavy,
    const uint32_t* __restrict__ vals, const float* __restrict__ splat, const uint2* __restrict__ keep,
    const float* __restrict__ dL_drgb, float* __restrict__ gsplat, GradZero zero, const FrameState* st)
{
    __shared__ __align__(128) BwdSmem S;
    grid_dep_wait();
    if (blockIdx.x < zero.blocks) {
        zero_share(zero, blockIdx.x, zero.blocks);
        return;
    }
    blendk::walk_grid(
        blockIdx.x - zero.blocks, gridDim.x - zero.blocks, (uint32_t)(cam.tiles_x * cam.tiles_y), ranges, heavy, st,
        [&](uint32_t tile, uint2 rg) {
            blend_bwd_walk<8>(cam, tile, 0u, rg, S, vals, splat, keep, dL_drgb, gsplat, st);
        },
        [&](uint32_t tile, uint32_t part, uint2 rg) {
            blend_bwd_walk<16>(cam, tile, part, rg, S, vals, splat, keep, dL_drgb, gsplat, st);
        });
}

// ---------------------------------------------------------------------------
// projection / SH backward (one thread per selected Gaussian)
// ---------------------------------------------------------------------------
namespace {

// Real SH basis (Cartesian form, degree kDeg <= 3) and its partial derivatives
// in (x, y, z), treating the three as independent.
template <int kDeg>
__device__ __forceinline__ void sh_basis_grad(float x, float y, float z, float Y[16], float dY[16][3])
{
    using namespace proj;
#pragma unroll
    for (int k = 0; k < 16; ++k) {
        Y[k] = 0.0f;
        dY[k][0] = dY[k][1] = dY[k][2] = 0.0f;
    }
    Y[0] = kY00;
    if (kDeg < 1) return;
    Y[1] = -kY1 * y; dY[1][1] = -kY1;
    Y[2] = kY1 * z;  dY[2][2] = kY1;
    Y[3] = -kY1 * x; dY[3][0] = -kY1;
    if (kDeg < 2) return;
    const float xx = x * x, yy = y * y, zz = z * z;
    Y[4] = kY2a * x * y;                 dY[4][0] = kY2a * y;           dY[4][1] = kY2a * x;
    Y[5] = -kY2a * y * z;                dY[5][1] = -kY2a * z;          dY[5][2] = -kY2a * y;
    Y[6] = kY2b * (2.0f * zz - xx - yy); dY[6][0] = -2.0f * kY2b * x;   dY[6][1] = -2.0f * kY2b * y;
    dY[6][2] = 4.0f * kY2b * z;
    Y[7] = -kY2a * x * z;                dY[7][0] = -kY2a * z;          dY[7][2] = -kY2a * x;
    Y[8] = kY2c * (xx - yy);             dY[8][0] = 2.0f * kY2c * x;    dY[8][1] = -2.0f * kY2c * y;
    if (kDeg < 3) return;
    Y[9] = -kY3a * y * (3.0f * xx - yy);
    dY[9][0] = -6.0f * kY3a * x * y;
    dY[9][1] = -kY3a * (3.0f * xx - 3.0f * yy);
    Y[10] = kY3b * x * y * z;
    dY[10][0] = kY3b * y * z;
    dY[10][1] = kY3b * x * z;
    dY[10][2] = kY3b * x * y;
    Y[11] = -kY3c * y * (4.0f * zz - xx - yy);
    dY[11][0] = 2.0f * kY3c * x * y;
    dY[11][1] = -kY3c * (4.0f * zz - xx - 3.0f * yy);
    dY[11][2] = -8.0f * kY3c * y * z;
    Y[12] = kY3d * z * (2.0f * zz - 3.0f * xx - 3.0f * yy);
    dY[12][0] = -6.0f * kY3d * x * z;
    dY[12][1] = -6.0f * kY3d * y * z;
    dY[12][2] = kY3d * (6.0f * zz - 3.0f * xx - 3.0f * yy);
    Y[13] = -kY3c * x * (4.0f * zz - xx - yy);
    dY[13][0] = -kY3c * (4.0f * zz - 3.0f * xx - yy);
    dY[13][1] = 2.0f * kY3c * x * y;
    dY[13][2] = -8.0f * kY3c * x * z;
    Y[14] = kY3e * z * (xx - yy);
    dY[14][0] = 2.0f * kY3e * x * z;
    dY[14][1] = -2.0f * kY3e * y * z;
    dY[14][2] = kY3e * (xx - yy);
    Y[15] = -kY3a * x * (xx - 3.0f * yy);
    dY[15][0] = -kY3a * (3.0f * xx - 3.0f * yy);
    dY[15][1] = 6.0f * kY3a * x * y;
}

}  // namespace

struct GradPtrs {
    float* mu;          // [3][n]
    float* log_scale;   // [3][n]
    float* quat;        // [4][n]
    float* logit;       // [n]
    float* sh;          // [n][K][3]
};

// Chain rule for selected Gaussian m (node sel[m]): splat gradient -> mean,
// log-scale, quaternion, logit, SH.  Each node appears once in the selection,
// so plain stores do, and loads and stores when accumulating (reductions in global memory
// flush subnormal numbers; two accumulating views of 375K nodes 408 us with them, 418 so,
// of degree 2 402 and 406, 437 with one old value in flight at a time).
//
// Each warp takes 32 consecutive selected Gaussians per iteration, one per
// lane.  Their SH rows (3 K floats each, contiguous per node) are staged in
// shared memory with coalesced asynchronous copies, and the SH gradient rows
// leave the same way, 16 bytes at a time where the rows are multiples of 16 bytes and
// the arrays aligned (vec; degrees 1 and 3), else 4.  A lane reads its row four floats
// at a time: the row stride is a multiple of 4 floats and odd in units of 4, so the 8
// lanes of a quarter-warp hit different banks.  Bound: the latency of the rows (8 blocks
// of 2 warps an SM, by shared memory and registers), so the next group's rows are copied
// and its other inputs prefetched while this one is computed (537K Gaussians of degree 3:
// 73 -> 54 us; accumulating 264K: 36 -> 33).
__device__ __forceinline__ void cp_async4(float* smem, const float* gmem)
{
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"((uint32_t)__cvta_generic_to_shared(smem)), "l"(gmem)
                 : "memory");
}
__device__ __forceinline__ void cp_async16(float* smem, const float* gmem)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((uint32_t)__cvta_generic_to_shared(smem)), "l"(gmem)
                 : "memory");
}

__device__ __forceinline__ void prefetch_l2(const float* p) { asm volatile("prefetch.global.L2 [%0];" ::"l"(p)); }

constexpr int kPbWarps = 2;   // warps per projection-backward block

template <int kDeg, bool kAccumulate>
__global__ void __launch_bounds__(kPbWarps * 32, 16 / kPbWarps) project_bwd_kernel(DevTree t, DevCamera cam, ParamPtrs p,
                                                          const uint32_t* __restrict__ sel,
                                                          const float* __restrict__ gsplat,
                                                          GradPtrs gr, bool vec, const FrameState* st)
{
    constexpr int K = (kDeg + 1) * (kDeg + 1);
    constexpr int K3 = 3 * K, Q = (K3 + 3) / 4, RS = 4 * (Q | 1);
    __shared__ __align__(16) float s_rows[kPbWarps][2][32 * RS];      // the next group's rows land during this one's work
    grid_dep_wait();
    const uint32_t M = st->M;
    const size_t N = p.n;
    const float* W = cam.R;
    const uint32_t lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const uint32_t step = gridDim.x * kPbWarps * 32;
    auto node = [&](uint32_t at) { return at < M ? sel[min(at + lane, M - 1u)] : 0u; };
    // the SH rows of the group at `at` (nodes nn, one a lane) with asynchronous copies, all
    // in flight at once
    auto stage = [&](uint32_t at, uint32_t nn, float* to) {
        if (at >= M) return;
        if (K3 % 4 == 0 && vec) {
#pragma unroll
            for (int i = 0; i < Q; ++i) {
                const uint32_t idx = (uint32_t)i * 32u + lane, r = idx / Q, k = 4u * (idx - r * Q);
                const uint32_t nr = __shfl_sync(0xffffffffu, nn, r);
                cp_async16(to + r * RS + k, p.sh + (size_t)nr * K3 + k);
            }
        } else {
            for (int i = 0; i < K3; ++i) {
                const uint32_t idx = (uint32_t)i * 32u + lane, r = idx / K3, k = idx - r * K3;
                const uint32_t nr = __shfl_sync(0xffffffffu, nn, r);
                cp_async4(to + r * RS + k, p.sh + (size_t)nr * K3 + k);
            }
        }
    };
    uint32_t base = (blockIdx.x * kPbWarps + warp) * 32;
    uint32_t n = node(base), n_next = node(base + step);
    stage(base, n, s_rows[warp][0]);
    asm volatile("cp.async.commit_group;" ::: "memory");
    for (uint32_t buf = 0; base < M; base += step, buf ^= 1u) {
        const uint32_t m = base + lane;
        const bool act = m < M;
        float* rows = s_rows[warp][buf];
        float* row = rows + lane * RS;
        stage(base + step, n_next, s_rows[warp][buf ^ 1u]);
        asm volatile("cp.async.commit_group;" ::: "memory");
        const uint32_t n_after = base + step < M ? node(base + 2u * step) : 0u;
        if (base + step < M) {                            // the next group's other inputs, to L2
#pragma unroll
            for (int k = 0; k < 3; ++k) {
                prefetch_l2(p.mu + k * N + n_next);
                prefetch_l2(p.log_scale + k * N + n_next);
            }
#pragma unroll
            for (int k = 0; k < 4; ++k) prefetch_l2(p.quat + k * N + n_next);
            prefetch_l2(p.logit + n_next);
            const size_t row = (size_t)(base + step) * kGS + lane * 32u;      // kGS lines of 32 floats
            if (lane < (uint32_t)kGS && row < (size_t)M * kGS) prefetch_l2(gsplat + row);
        }
        asm volatile("cp.async.wait_group 1;" ::: "memory");
        __syncwarp();
        const float* gs = gsplat + (size_t)(act ? m : base) * kGS;
        const float gu = gs[0], gv = gs[1], gA = gs[2], gB = gs[3], gC = gs[4], ga0 = gs[5];
        const float gcol[3] = {gs[6], gs[7], gs[8]};
        const float mu[3] = {p.mu[n], p.mu[N + n], p.mu[2 * N + n]};
        // camera space (the Gaussian passed the frustum test, so the tangent
        // clamp of the EWA Jacobian is inactive)
        const float x = W[0] * mu[0] + W[1] * mu[1] + W[2] * mu[2] + cam.t[0];
        const float y = W[3] * mu[0] + W[4] * mu[1] + W[5] * mu[2] + cam.t[1];
        const float z = W[6] * mu[0] + W[7] * mu[1] + W[8] * mu[2] + cam.t[2];
        const float iz = 1.0f / z, iz2 = iz * iz;
        float c6[6], Rq[9], s2[3], qh[4], qn;
        sigma_from(p, n, c6, Rq, s2, qh, qn);
        const float Sg[3][3] = {{c6[0], c6[1], c6[2]}, {c6[1], c6[3], c6[4]}, {c6[2], c6[4], c6[5]}};
        const float J[2][3] = {{cam.fx * iz, 0.0f, -cam.fx * x * iz2}, {0.0f, cam.fy * iz, -cam.fy * y * iz2}};
        float Mm[2][3], MS[2][3];
#pragma unroll
        for (int i = 0; i < 2; ++i)
#pragma unroll
            for (int j = 0; j < 3; ++j) Mm[i][j] = J[i][0] * W[j] + J[i][1] * W[3 + j] + J[i][2] * W[6 + j];
#pragma unroll
        for (int i = 0; i < 2; ++i)
#pragma unroll
            for (int j = 0; j < 3; ++j) MS[i][j] = Mm[i][0] * Sg[0][j] + Mm[i][1] * Sg[1][j] + Mm[i][2] * Sg[2][j];
        const float a = MS[0][0] * Mm[0][0] + MS[0][1] * Mm[0][1] + MS[0][2] * Mm[0][2] + 0.3f;
        const float b = MS[0][0] * Mm[1][0] + MS[0][1] * Mm[1][1] + MS[0][2] * Mm[1][2];
        const float c = MS[1][0] * Mm[1][0] + MS[1][1] * Mm[1][1] + MS[1][2] * Mm[1][2] + 0.3f;
        const float det = a * c - b * b, id2 = 1.0f / (det * det);
        // conic (A, B, C) = (c, -b, a) / det  ->  Sigma_2D entries (a, b, c)
        const float ga = (gA * (-c * c) + gB * (b * c) + gC * (-b * b)) * id2;
        const float gb = (gA * (2.0f * b * c) - gB * (det + 2.0f * b * b) + gC * (2.0f * a * b)) * id2;
        const float gc = (gA * (-b * b) + gB * (a * b) + gC * (-a * a)) * id2;
        const float G2[2][2] = {{ga, 0.5f * gb}, {0.5f * gb, gc}};
        // Sigma_2D = M Sigma M^T: dL/dSigma = M^T G2 M, dL/dM = 2 G2 M Sigma
        float GS[3][3], GM[2][3], GJ[2][3];
#pragma unroll
        for (int i = 0; i < 3; ++i)
#pragma unroll
            for (int j = 0; j < 3; ++j) {
                float v = 0.0f;
#pragma unroll
                for (int k = 0; k < 2; ++k)
#pragma unroll
                    for (int l = 0; l < 2; ++l) v += Mm[k][i] * G2[k][l] * Mm[l][j];
                GS[i][j] = v;
            }
#pragma unroll
        for (int i = 0; i < 2; ++i)
#pragma unroll
            for (int j = 0; j < 3; ++j) GM[i][j] = 2.0f * (G2[i][0] * MS[0][j] + G2[i][1] * MS[1][j]);
        // M = J W
#pragma unroll
        for (int i = 0; i < 2; ++i)
#pragma unroll
            for (int k = 0; k < 3; ++k)
                GJ[i][k] = GM[i][0] * W[3 * k] + GM[i][1] * W[3 * k + 1] + GM[i][2] * W[3 * k + 2];
        // (u, v) and J as functions of the camera-space centre
        const float gx = gu * cam.fx * iz - GJ[0][2] * cam.fx * iz2;
        const float gy = gv * cam.fy * iz - GJ[1][2] * cam.fy * iz2;
        const float gz = -(gu * cam.fx * x + gv * cam.fy * y) * iz2 - (GJ[0][0] * cam.fx + GJ[1][1] * cam.fy) * iz2 +
                         2.0f * (GJ[0][2] * cam.fx * x + GJ[1][2] * cam.fy * y) * iz2 * iz;
        float gmu[3];
#pragma unroll
        for (int j = 0; j < 3; ++j) gmu[j] = W[j] * gx + W[3 + j] * gy + W[6 + j] * gz;
        // Sigma = R diag(s2) R^T: dL/dR = 2 GS R diag(s2), dL/ds_k = 2 s2_k (R^T GS R)_kk
        float G[9], gls[3];
#pragma unroll
        for (int i = 0; i < 3; ++i)
#pragma unroll
            for (int k = 0; k < 3; ++k)
                G[3 * i + k] = 2.0f * (GS[i][0] * Rq[k] + GS[i][1] * Rq[3 + k] + GS[i][2] * Rq[6 + k]) * s2[k];
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            float v = 0.0f;
#pragma unroll
            for (int i = 0; i < 3; ++i)
#pragma unroll
                for (int j = 0; j < 3; ++j) v += Rq[3 * i + k] * GS[i][j] * Rq[3 * j + k];
            gls[k] = 2.0f * s2[k] * v;
        }
        // R(q/|q|): derivatives of the nine entries in the unit quaternion
        const float w_ = qh[0], x_ = qh[1], y_ = qh[2], z_ = qh[3];
        float gq[4];
        gq[0] = 2.0f * (-z_ * G[1] + y_ * G[2] + z_ * G[3] - x_ * G[5] - y_ * G[6] + x_ * G[7]);
        gq[1] = 2.0f * (y_ * G[1] + z_ * G[2] + y_ * G[3] - 2.0f * x_ * G[4] - w_ * G[5] + z_ * G[6] +
                        w_ * G[7] - 2.0f * x_ * G[8]);
        gq[2] = 2.0f * (-2.0f * y_ * G[0] + x_ * G[1] + w_ * G[2] + x_ * G[3] + z_ * G[5] - w_ * G[6] +
                        z_ * G[7] - 2.0f * y_ * G[8]);
        gq[3] = 2.0f * (-2.0f * z_ * G[0] - w_ * G[1] + x_ * G[2] + w_ * G[3] - 2.0f * z_ * G[4] + y_ * G[5] +
                        x_ * G[6] + y_ * G[7]);
        const float dotq = gq[0] * w_ + gq[1] * x_ + gq[2] * y_ + gq[3] * z_;
        // alpha0 = sigmoid(l)
        const float l = p.logit[n];
        const float a0 = 1.0f / (1.0f + __expf(-l));
        const float glogit = (l < -kLogitMax || l > kLogitMax) ? 0.0f : ga0 * a0 * (1.0f - a0);
        // colour = max(0, 1/2 + sum_k Y_k(d) c_k), d = (mu - campos) / |mu - campos|
        float d[3] = {mu[0] - cam.campos[0], mu[1] - cam.campos[1], mu[2] - cam.campos[2]};
        const float idl = rsqrtf(d[0] * d[0] + d[1] * d[1] + d[2] * d[2]);
#pragma unroll
        for (int k = 0; k < 3; ++k) d[k] *= idl;
        float Y[16], dY[16][3];
        sh_basis_grad<kDeg>(d[0], d[1], d[2], Y, dY);
        float gd[3] = {0.0f, 0.0f, 0.0f}, g3[3] = {0.5f, 0.5f, 0.5f};
        float4* row4 = reinterpret_cast<float4*>(row);
#pragma unroll
        for (int v = 0; v < Q; ++v) {
            const float4 f = row4[v];
            const float e[4] = {f.x, f.y, f.z, f.w};
#pragma unroll
            for (int r = 0; r < 4; ++r)
                if (4 * v + r < K3) g3[(4 * v + r) % 3] += Y[(4 * v + r) / 3] * e[r];
        }
#pragma unroll
        for (int ch = 0; ch < 3; ++ch) g3[ch] = g3[ch] > 0.0f ? gcol[ch] : 0.0f;
#pragma unroll
        for (int v = 0; v < Q; ++v) {
            const float4 f = row4[v];
            float e[4] = {f.x, f.y, f.z, f.w};
#pragma unroll
            for (int r = 0; r < 4; ++r)
                if (4 * v + r < K3) {
                    const int k = (4 * v + r) / 3, ch = (4 * v + r) % 3;      // compile-time after unrolling
                    const float cg = e[r] * g3[ch];
                    gd[0] += cg * dY[k][0];
                    gd[1] += cg * dY[k][1];
                    gd[2] += cg * dY[k][2];
                    e[r] = Y[k] * g3[ch];              // the row now holds the SH gradient
                }
            row4[v] = make_float4(e[0], e[1], e[2], e[3]);
        }
        __syncwarp();
        float old[11] = {};                               // what the other gradients are added to
        if (kAccumulate && act) {
#pragma unroll
            for (int k = 0; k < 3; ++k) {
                old[k] = gr.mu[k * N + n];
                old[3 + k] = gr.log_scale[k * N + n];
            }
#pragma unroll
            for (int k = 0; k < 4; ++k) old[6 + k] = gr.quat[k * N + n];
            old[10] = gr.logit[n];
        }
        // SH gradient rows out, coalesced; when adding, kB old values in flight a lane
        if (K3 % 4 == 0 && vec) {
            constexpr int kB = kAccumulate ? 4 : 1;
            auto at = [&](int i, uint32_t& r, uint32_t& k) {
                const uint32_t idx = (uint32_t)i * 32u + lane;
                r = idx / Q;
                k = 4u * (idx - r * Q);
                return reinterpret_cast<float4*>(gr.sh + (size_t)__shfl_sync(0xffffffffu, n, r) * K3 + k);
            };
#pragma unroll
            for (int i0 = 0; i0 < Q; i0 += kB) {
                uint32_t r, k;
                float4 held[kB];
                if (kAccumulate)
#pragma unroll
                    for (int j = 0; j < kB && i0 + j < Q; ++j) {
                        const float4* p = at(i0 + j, r, k);
                        if (base + r < M) held[j] = *p;
                    }
#pragma unroll
                for (int j = 0; j < kB && i0 + j < Q; ++j) {
                    float4* p = at(i0 + j, r, k);
                    float4 g = *reinterpret_cast<const float4*>(rows + r * RS + k);
                    if (kAccumulate) g = make_float4(held[j].x + g.x, held[j].y + g.y, held[j].z + g.z, held[j].w + g.w);
                    if (base + r < M) *p = g;
                }
            }
        } else {
            constexpr int kB = K3 % 9 == 0 ? 9 : K3 % 6 == 0 ? 6 : 3;
            auto at = [&](int i, uint32_t& r, uint32_t& k) {
                const uint32_t idx = (uint32_t)i * 32u + lane;
                r = idx / K3;
                k = idx - r * K3;
                return gr.sh + (size_t)__shfl_sync(0xffffffffu, n, r) * K3 + k;
            };
#pragma unroll 1
            for (int i0 = 0; i0 < K3; i0 += kB) {
                uint32_t r, k;
                float held[kB] = {};
                if (kAccumulate)
#pragma unroll
                    for (int j = 0; j < kB; ++j) {
                        const float* p = at(i0 + j, r, k);
                        if (base + r < M) held[j] = *p;
                    }
#pragma unroll
                for (int j = 0; j < kB; ++j) {
                    float* p = at(i0 + j, r, k);
                    const float g = rows[r * RS + k];
                    if (base + r < M) *p = kAccumulate ? held[j] + g : g;
                }
            }
        }
        __syncwarp();
        const uint32_t nn = n;
        n = n_next;
        n_next = n_after;
        if (!act) continue;
        const float dd = gd[0] * d[0] + gd[1] * d[1] + gd[2] * d[2];
#pragma unroll
        for (int k = 0; k < 3; ++k) gmu[k] += (gd[k] - d[k] * dd) * idl;
        float gqn[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) gqn[k] = (gq[k] - qh[k] * dotq) / qn;
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            gr.mu[k * N + nn] = kAccumulate ? old[k] + gmu[k] : gmu[k];
            gr.log_scale[k * N + nn] = kAccumulate ? old[3 + k] + gls[k] : gls[k];
        }
#pragma unroll
        for (int k = 0; k < 4; ++k) gr.quat[k * N + nn] = kAccumulate ? old[6 + k] + gqn[k] : gqn[k];
        gr.logit[nn] = kAccumulate ? old[10] + glogit : glogit;
    }
}

__global__ void __launch_bounds__(128) zero_rows_kernel(float4* __restrict__ gsplat, const FrameState* st)
{
    grid_dep_wait();
    const uint32_t n4 = st->M * (uint32_t)(kGS / 4);
    for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < n4; i += gridDim.x * blockDim.x)
        gsplat[i] = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
}

// ---------------------------------------------------------------------------
// launchers
// ---------------------------------------------------------------------------
void launch_prep_params(const DevTree& t, const float* mu, const float* log_scale, const float* quat,
                        const float* logit, const float* sh, int blocks, cudaStream_t s)
{
    const ParamPtrs p{mu, log_scale, quat, logit, sh, t.n};
    const uint32_t K3 = (t.sh_degree + 1) * (t.sh_degree + 1) * 3;
    const bool vec = t.sh_stride == K3 && ((uintptr_t)sh & 15u) == 0;
    switch (t.sh_degree) {
    case 0: launch_pdl(prep_kernel<0>, blocks, 256, 0, s, t, p, vec); break;
    case 1: launch_pdl(prep_kernel<1>, blocks, 256, 0, s, t, p, vec); break;
    case 2: launch_pdl(prep_kernel<2>, blocks, 256, 0, s, t, p, vec); break;
    default: launch_pdl(prep_kernel<3>, blocks, 256, 0, s, t, p, vec); break;
    }
}

template <int kDeg>
static void launch_project_bwd(const DevTree& t, const DevCamera& cam, const ParamPtrs& p,
                               const uint32_t* sel, const float* gsplat, const GradPtrs& gr,
                               bool accumulate, int blocks, const FrameState* st, cudaStream_t s)
{
    constexpr int K3 = 3 * (kDeg + 1) * (kDeg + 1);
    const bool vec = K3 % 4 == 0 && (((uintptr_t)p.sh | (uintptr_t)gr.sh) & 15u) == 0;
    if (accumulate)
        launch_pdl(project_bwd_kernel<kDeg, true>, blocks, kPbWarps * 32, 0, s, t, cam, p, sel, gsplat, gr, vec, st);
    else
        launch_pdl(project_bwd_kernel<kDeg, false>, blocks, kPbWarps * 32, 0, s, t, cam, p, sel, gsplat, gr, vec, st);
}

void launch_backward(const DevTree& t, const DevCamera& cam, const uint2* ranges, const uint32_t* heavy,
                     const uint32_t* vals,
                     const float* splat, uint2* keep, bool kept, const uint32_t* sel, const uint32_t* selbits,
                     const float* dL_drgb, float* gsplat, const float* const params[5], float* const grads[5], bool accumulate,
                     int sms, FrameState* st, cudaStream_t s)
{
    // gsplat rows of the selected Gaussians start at zero: the blend backward adds into them
    launch_pdl(zero_rows_kernel, sms * 8, 128, 0, s, reinterpret_cast<float4*>(gsplat), st);
    if (!kept) launch_blend(cam, ranges, heavy, vals, splat, nullptr, nullptr, keep, st, false, s);
    const ParamPtrs p{params[0], params[1], params[2], params[3], params[4], t.n};
    const GradPtrs gr{grads[0], grads[1], grads[2], grads[3], grads[4]};
    // nodes outside the selection get zero gradient
    const uint32_t K3 = (t.sh_degree + 1) * (t.sh_degree + 1) * 3;
    const GradZero zero{{gr.mu, gr.log_scale, gr.quat, gr.logit}, {3, 3, 4, 1}, gr.sh, K3,
                        K3 % 4 == 0 && ((uintptr_t)gr.sh & 15u) == 0, selbits, t.n, accumulate ? 0u : (uint32_t)sms};
    const int n_tiles = cam.tiles_x * cam.tiles_y;
    launch_pdl(blend_bwd_kernel, n_tiles + 2 * split_slots(n_tiles) + (int)zero.blocks, blendk::kWalkChunk, 0, s, cam,
               ranges, heavy, vals, splat, keep, dL_drgb, gsplat, zero, st);
    const int blocks = sms * (16 / kPbWarps);
    switch (t.sh_degree) {
    case 0: launch_project_bwd<0>(t, cam, p, sel, gsplat, gr, accumulate, blocks, st, s); break;
    case 1: launch_project_bwd<1>(t, cam, p, sel, gsplat, gr, accumulate, blocks, st, s); break;
    case 2: launch_project_bwd<2>(t, cam, p, sel, gsplat, gr, accumulate, blocks, st, s); break;
    default: launch_project_bwd<3>(t, cam, p, sel, gsplat, gr, accumulate, blocks, st, s); break;
    }
}

}  // namespace fgs
