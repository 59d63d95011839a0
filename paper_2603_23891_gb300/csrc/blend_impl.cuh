// Per-tile blending machinery shared by the single-view and the batched blend
// kernels (see blend.cu for the design).
#pragma once

#include "fgs_internal.cuh"

#include <type_traits>

namespace fgs {
namespace blendk {

// ---------------------------------------------------------------------------
// The forward's walk
// ---------------------------------------------------------------------------
// One CTA of four warps walks a tile (kLanes = 8) or half of one (kLanes = 16).  A
// tile is 16 blocks of 4x4 pixels; a warp has 32 / kLanes blocks, kLanes lanes each:
// four blocks with two pixels a lane, or two blocks with one.
//  * Stage: 128 records at a time, one a thread, into shared memory; the thread boxes
//    its record against the tile's blocks (walk_mask).
//  * List: each warp gives every block of its own an ordered list of the records it
//    may meet.
//  * Test, kLanes entries of each block at a time: a lane takes ONE ENTRY and computes
//    its power at the block's 16 pixels, two pixels to an instruction (binary32
//    pairs): the products with dy, and dx itself, are shared by a row and a column, so
//    a pixel costs two fused multiply-adds, and the two skip tests one more and a
//    product, whose sign is the answer.  The powers are parked in shared memory and
//    the lanes' 16-bit answers transposed, so that a lane then holds the answers of
//    all the entries for ITS PIXELS.  (With a lane a pixel from the start every entry
//    was read by every lane and its offsets and products formed again in each: 16
//    instructions for 32 evaluations; here about 150 for 512.)
//  * Apply: each lane takes its own pixels' next two entries, front to back.  Entries
//    wait in a window of two groups, so a lane with few hits in one group goes on with
//    the next while the others finish (idle lanes on the blob workload: 51% of the
//    turns with one group, 38% with two, 37% with four).
// Bound: instruction issue.  Two pixels a lane takes the fewest instructions; one pixel
// a lane takes a fifth more, but half the turns for each warp, and twice the warps:
// it is taken for the tiles whose walk would outlast the rest of the frame
// (split_pairs).
typedef unsigned long long f32x2;

__device__ __forceinline__ f32x2 pack2(float a, float b)
{
    f32x2 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
    return r;
}
__device__ __forceinline__ f32x2 dup2(float a) { return pack2(a, a); }
__device__ __forceinline__ float2 unpack2(f32x2 v)
{
    float2 r;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(v));
    return r;
}
// Each half rounded to nearest even on its own, as the scalar operations are.
__device__ __forceinline__ f32x2 fma2(f32x2 a, f32x2 b, f32x2 c)
{
    f32x2 r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}
__device__ __forceinline__ f32x2 add2(f32x2 a, f32x2 b)
{
    f32x2 r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ f32x2 mul2(f32x2 a, f32x2 b)
{
    f32x2 r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}

// A record's {C, lthr, alpha0, depth} as it is staged: no power below -87 passes the skip
// test, where exp is 0 and the entry would change nothing (exp_poly_neg's range).
__device__ __forceinline__ float4 staged_r1(float4 r)
{
    r.y = fmaxf(r.y, -87.0f);
    return r;
}

// Leading zeros; all ones for 0.
__device__ __forceinline__ uint32_t clz_or_ones(uint32_t v)
{
    uint32_t r;
    asm("bfind.shiftamt.u32 %0, %1;" : "=r"(r) : "r"(v));
    return r;
}
// A shift by 32 or more gives 0.
__device__ __forceinline__ uint32_t shr0(uint32_t v, uint32_t n)
{
    uint32_t r;
    asm("shr.u32 %0, %1, %2;" : "=r"(r) : "r"(v), "r"(n));
    return r;
}

// exp_hit's polynomial at -n (n = -power: the same operations on the negated argument;
// r and the odd coefficients change sign, every rounding is the same); t0's low bits
// are k, 2^k is still to be applied.  Scalar: the constants are immediates (a packed
// operation would read each pair from constant memory first, as many instructions).
__device__ __forceinline__ float exp_poly_neg(float n, uint32_t& t0)
{
    const float t = ff(n, -1.44269504088896341f, 12582912.0f);
    const float kf = fs(t, 12582912.0f);
    float r = ff(kf, 0.693359375f, n);
    r = ff(kf, -2.12194440e-4f, r);
    float p = ff(-1.98412698412698413e-4f, r, 1.38888888888888889e-3f);
    p = ff(p, r, -8.33333333333333333e-3f);
    p = ff(p, r, 4.16666666666666667e-2f);
    p = ff(p, r, -1.66666666666666667e-1f);
    p = ff(p, r, 0.5f);
    p = ff(p, r, -1.0f);
    p = ff(p, r, 1.0f);
    t0 = __float_as_uint(t);
    return p;
}

constexpr int kWalkWarps = 4;       // warps of a CTA
constexpr int kWalkChunk = 32 * kWalkWarps;   // pairs staged at a time, one a thread
constexpr int kParkStride = 20;     // floats of a parked entry (16, padded: conflict-free stores)
constexpr uint32_t kFull = 0xffffffffu;

// One warp's.  Window slots: 2 kLanes of each of its 32 / kLanes blocks.
template <bool kKeep>
struct WalkWarp {
    float pw[64][kParkStride];                    // -power at a block's 16 pixels
    float4 col[64][2];                            // alpha0, r, g, b twice each
    uint32_t pos[kKeep ? 64 : 1];                 // pair index
    uint8_t list[4][kWalkChunk];                  // per block: the chunk's records it may meet
};

template <bool kKeep>
struct WalkSmem {
    float4 r0[kWalkChunk];                        // u, v, A, B
    float4 r1[kWalkChunk];                        // C, lthr, alpha0, depth
    float4 r2[kWalkChunk];                        // r, g, b, radius
    uint16_t mask[kWalkChunk];                    // walk_mask
    WalkWarp<kKeep> w[kWalkWarps];
};

// A tile's blocks in fours: origin in the tile of the w-th four, 2x2 blocks (64x4
// tiles: 4x1), 2^bsh blocks across.
__device__ __forceinline__ void walk_origin(const DevCamera& cam, uint32_t w, int32_t& ox, int32_t& oy,
                                            uint32_t& bsh)
{
    bsh = cam.tile_shift_x == 6 ? 2u : 1u;
    const uint32_t wsh = (uint32_t)cam.tile_shift_x - 2u - bsh;    // log2(fours across)
    ox = (int32_t)((w & ((1u << wsh) - 1u)) << (bsh + 2u));
    oy = (int32_t)((w >> wsh) << (4u - bsh));
}

// Which blocks of the tile may hold a pixel whose binary32 power reaches the
// Gaussian's skip threshold lthr; bit 4 w + b: block b of the w-th four (walk_origin's
// layout).  Exactly, power >= lthr is the ellipse d^T Q d <= s with Q = [[A, B], [B, C]]
// and s = -2 lthr, whose bounding box has half-widths sqrt(s C / det Q) and
// sqrt(s A / det Q).  Margins, for cond(Q) < 1e4 (cond(Q) <= tr^2 / det; beyond that, or
// for a singular Q, every block keeps the Gaussian):
//  * the binary32 power (offsets rounded, three products, two fused
//    multiply-adds) is within 11 * 2^-24 * cond(Q) < 0.7% of the exact form at
//    the exact offsets, so a pixel passing the test lies in the ellipse of
//    s' = 1.05 s + 1e-4;
//  * det Q computed in binary32 loses at most 2^-24 cond(Q) / 2 < 3e-4
//    relative, and the approximate quotient and roots 1e-6, so the computed
//    half-widths are within 2e-4 relative of the exact ones for s' (the 5% in s leaves
//    2% of the half-width spare);
//  * the box is further widened by 0.1% and 0.01 px for the roundings of
//    u - tx0, v - ty0 and of the bounds below.
// A block left out of the mask would have skipped the Gaussian at every one of
// its pixels.  Block column c spans pixel centres tx0 + 4 c + [0.5, 3.5], row r
// ty0 + 4 r + [0.5, 3.5]; the mask is the block of columns x rows the box meets.
__device__ __forceinline__ uint32_t walk_mask(const DevCamera& cam, int32_t tx0, int32_t ty0, float u, float v,
                                              float A, float B, float C, float lthr)
{
    if (!(lthr <= 0.0f)) return 0u;
    const float det = A * C - B * B;
    const float tr = A + C;
    if (!(det > 0.0f) || tr * tr > 1e4f * det) return 0xFFFFu;
    const float sd = __fdividef(fmaf(-2.1f, lthr, 1e-4f), det);
    float ex, ey;
    asm("sqrt.approx.f32 %0, %1;" : "=f"(ex) : "f"(sd * C));
    asm("sqrt.approx.f32 %0, %1;" : "=f"(ey) : "f"(sd * A));
    ex = fmaf(ex, 1.001f, 0.01f);
    ey = fmaf(ey, 1.001f, 0.01f);
    const int32_t sh = cam.tile_shift_x - 2;                 // log2(block columns)
    const int32_t ncol = 1 << sh, nrow = 16 >> sh;
    const float ux = u - (float)tx0, vy = v - (float)ty0;
    const int32_t c_lo = max(0, (int32_t)ceilf((ux - ex - 3.5f) * 0.25f));
    const int32_t c_hi = min(ncol - 1, (int32_t)floorf((ux + ex - 0.5f) * 0.25f));
    const int32_t r_lo = max(0, (int32_t)ceilf((vy - ey - 3.5f) * 0.25f));
    const int32_t r_hi = min(nrow - 1, (int32_t)floorf((vy + ey - 0.5f) * 0.25f));
    if (c_lo > c_hi || r_lo > r_hi) return 0u;
    uint32_t cols = ((2u << c_hi) - 1u) & ~((1u << c_lo) - 1u);
    if (sh == 4) return cols;                                // 64x4 tiles: four columns a four
    cols = (cols | cols << 4) & 0x0F0Fu;                     // two columns a four: every pair to its nibble
    cols = (cols | cols << 2) & 0x3333u;
    uint32_t m = 0;
    for (int32_t r = r_lo; r <= r_hi; ++r) m |= cols << (((r >> 1) << (sh + 1)) + ((r & 1) << 1));
    return m;
}

// 16-bit rows of 16 / kLanes-bit elements, kLanes lanes by kLanes: lane l of a group
// ends with element k = lane k's element l.
template <int kLanes>
__device__ __forceinline__ uint32_t transpose_bits(uint32_t x, uint32_t i)
{
    uint32_t t = __shfl_xor_sync(kFull, x, kLanes / 2);
    x = __byte_perm(x, t, (i & (kLanes / 2)) ? 0x4415u : 0x4440u) & 0xFFFFu;
    t = __shfl_xor_sync(kFull, x, kLanes / 4);
    const uint32_t m4 = (i & (kLanes / 4)) ? 0xF0F0u : 0x0F0Fu;
    x = (x & m4) | (__funnelshift_l(t, t, (i & (kLanes / 4)) ? 28u : 4u) & (0xFFFFu ^ m4));
    t = __shfl_xor_sync(kFull, x, kLanes / 8);
    const uint32_t m2 = (i & (kLanes / 8)) ? 0xCCCCu : 0x3333u;
    x = (x & m2) | (__funnelshift_l(t, t, (i & (kLanes / 8)) ? 30u : 2u) & (0xFFFFu ^ m2));
    if (kLanes == 16) {
        t = __shfl_xor_sync(kFull, x, 1);
        const uint32_t m1 = (i & 1u) ? 0xAAAAu : 0x5555u;
        x = (x & m1) | (__funnelshift_l(t, t, (i & 1u) ? 31u : 1u) & (0xFFFFu ^ m1));
    }
    return x;
}

// Blend one image tile (kLanes = 8) or its half `part` (kLanes = 16).  `tile` is the
// tile in the camera's grid, rg its range of the sorted pairs.  rgb / Tout are the
// camera's own image planes, either may be null.  With kKeep, keep_out receives per
// pixel {final T bits, stop position}: the sorted-pair index of the Gaussian the pixel
// stopped at, or the tile's end if it did not stop; the differentiable form's
// backward walks each pixel from there.  kCount adds the work counters of FrameState
// (steps of 32 pixel evaluations, evaluations, alpha applications, steps with one).
template <int kLanes, bool kCount, bool kKeep>
__device__ __forceinline__ void blend_walk(const DevCamera& cam, uint32_t tile, uint32_t part, uint2 rg,
                                           WalkSmem<kKeep>& S, const uint32_t* __restrict__ vals,
                                           const float* __restrict__ splat, float* __restrict__ rgb,
                                           float* __restrict__ Tout, uint2* __restrict__ keep_out, FrameState* st)
{
    static_assert(kLanes == 8 || kLanes == 16, "lanes a block");
    constexpr bool kTwo = kLanes == 8;                             // pixels a lane
    constexpr uint32_t kC = kWalkChunk, kBlocks = 32 / kLanes, kSlots = 2 * kLanes;
    constexpr uint32_t kPx0 = kTwo ? 0xAAAAAAAAu : kFull, kPx1 = kTwo ? 0x55555555u : 0u;   // window bits a pixel
    const uint32_t tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const uint32_t b = lane / kLanes, i = lane % kLanes;
    const uint32_t M = st->M;
    const uint32_t e = rg.y;
    WalkWarp<kKeep>& W = S.w[warp];
    uint32_t m = rg.x + tid < e ? __ldg(vals + rg.x + tid) : 0u;
    const int32_t tx0 = (int32_t)(tile % (uint32_t)cam.tiles_x) * cam.tile_w;
    const int32_t ty0 = (int32_t)(tile / (uint32_t)cam.tiles_x) * cam.tile_h;
    // the warp's first block among the tile's 16, in fours
    const uint32_t fb = kTwo ? 4u * warp : 8u * part + 2u * warp;
    int32_t ox, oy;
    uint32_t bsh;
    walk_origin(cam, fb >> 2, ox, oy, bsh);
    const uint32_t bb = (fb & 3u) + b;
    const int32_t bx0 = tx0 + ox + (int32_t)((bb & ((1u << bsh) - 1u)) << 2);
    const int32_t by0 = ty0 + oy + (int32_t)((bb >> bsh) << 2);
    // this lane's pixels: (x, y) and (x, y + 1), or one of the two
    const uint32_t pp = kTwo ? i : i >> 1;
    const int32_t x = bx0 + (int32_t)(pp & 3u);
    const int32_t y = by0 + (int32_t)(pp >> 2 << 1) + (kTwo ? 0 : 1 - (int32_t)(i & 1u));
    uint32_t live = x < cam.width ? (y < cam.height ? kPx0 : 0u) | (y + 1 < cam.height ? kPx1 : 0u) : 0u;
    f32x2 T = dup2(1.0f), Cr = 0ull, Cg = 0ull, Cb = 0ull;         // kTwo: a pixel each half, else the low half

    f32x2 npx[4], npy[2];                                          // minus the block's pixel centres
#pragma unroll
    for (int k = 0; k < 4; ++k) npx[k] = dup2(-fa((float)(bx0 + k), 0.5f));
#pragma unroll
    for (int k = 0; k < 2; ++k)
        npy[k] = pack2(-fa((float)(by0 + 2 * k), 0.5f), -fa((float)(by0 + 2 * k + 1), 0.5f));
    // every window slot's colour finite from the start
#pragma unroll
    for (int k = 0; k < 4; ++k)
        reinterpret_cast<float4*>(&W.col[0][0])[32 * k + (int)lane] = make_float4(0.f, 0.f, 0.f, 0.f);

    uint32_t mask = 0u;          // window: 16 bits a group of kLanes entries, the older in the upper half
    uint32_t par = 0u;           // the older group's half of the window slots: 0 or kLanes
    // a colour or a coefficient is not finite (or huge), or an applied alpha may not be normal
    // (an opacity that its logarithm, and so the threshold, does not describe)
    bool careful = false;
    uint32_t c_steps = 0, c_evals = 0, c_hits = 0, c_active = 0, c_proc = 0, c_old = 0, c_new = 0;

    // the lane's next entry out of the window: its slot, and which pixels it applies to
    auto take = [&](uint32_t& sl, bool& h0, bool& h1) {
        uint32_t sh = clz_or_ones(mask);
        if (kTwo) sh &= ~1u;
        const uint32_t h = mask & shr0(kTwo ? 0xC0000000u : 0x80000000u, sh);
        h0 = (h & kPx0) != 0u;
        h1 = (h & kPx1) != 0u;
        if (kCount) {
            c_hits += (uint32_t)h0 + (uint32_t)h1;
            c_proc |= h;
        }
        mask ^= h;
        sl = b * kSlots + (((kTwo ? sh >> 1 : sh) ^ par) & (kSlots - 1u));
    };
    // the later entries of the window need no evaluation by a pixel stopping at slot sl
    auto uncount = [&](uint32_t sl) {
        const uint32_t p = (sl & (kSlots - 1u)) ^ par;
        return p < (uint32_t)kLanes ? c_old - p - 1u + c_new : c_new - (p - (uint32_t)kLanes) - 1u;
    };
    // two pixels: those that stop before this Gaussian keep T and add nothing (rare)
    auto stop2 = [&](uint32_t sl, f32x2& al, f32x2& Tn) {
        const float2 tn = unpack2(Tn), to = unpack2(T);
        const bool s0 = tn.x < 0.0001f, s1 = tn.y < 0.0001f;
        if (!(s0 || s1)) return;
        if (kKeep) {
            const uint32_t at = W.pos[sl];
            if (s0) keep_out[(size_t)y * cam.width + x] = make_uint2(__float_as_uint(to.x), at);
            if (s1) keep_out[(size_t)(y + 1) * cam.width + x] = make_uint2(__float_as_uint(to.y), at);
        }
        if (kCount) c_evals -= ((uint32_t)s0 + (uint32_t)s1) * uncount(sl);
        const float2 ao = unpack2(al);
        al = pack2(s0 ? 0.0f : ao.x, s1 ? 0.0f : ao.y);
        Tn = pack2(s0 ? to.x : tn.x, s1 ? to.y : tn.y);
        live &= (s0 ? kPx1 : kFull) & (s1 ? kPx0 : kFull);
        mask &= live;
    };
    // apply the window's entries, two a turn, until no lane has one left under `gate`;
    // `care`: colours and powers may be infinite or NaN (0 times one is not 0), alpha subnormal
    auto apply = [&](uint32_t gate, auto care) {
        constexpr bool kCare = decltype(care)::value;
        // alpha for parked power n, 0 where the entry is not applied
        auto alpha1 = [&](float n, float a0, bool h) {
            uint32_t t;
            const float p = exp_poly_neg(n, t);
            // alpha0 p 2^k: a normal alpha takes 2^k into its exponent
            const float al = kCare ? fm(a0, fm(p, __uint_as_float((t << 23) + (127u << 23))))
                                   : __uint_as_float((t << 23) + __float_as_uint(fm(a0, p)));
            return h ? fminf(al, 0.99f) : 0.0f;
        };
        auto add1 = [&](const float4& q0, const float4& q1, float w, float& r, float& g, float& bl) {
            if (kCare && w == 0.0f) return;
            r = fmaf(q0.z, w, r);
            g = fmaf(q1.x, w, g);
            bl = fmaf(q1.z, w, bl);
        };
        while (__any_sync(kFull, (mask & gate) != 0u)) {
            uint32_t sa, sb;
            bool a0, a1, b0, b1;
            take(sa, a0, a1);
            take(sb, b0, b1);
            const float4 qa0 = W.col[sa][0], qa1 = W.col[sa][1];
            const float4 qb0 = W.col[sb][0], qb1 = W.col[sb][1];
            if constexpr (kTwo) {
                auto alpha2 = [&](uint32_t sl, float al0, bool h0, bool h1) {
                    const float2 n = *reinterpret_cast<const float2*>(&W.pw[sl][2 * i]);
                    return pack2(alpha1(n.x, al0, h0), alpha1(n.y, al0, h1));
                };
                auto add2c = [&](const float4& q0, const float4& q1, f32x2 w) {
                    if (!kCare) {
                        Cr = fma2(pack2(q0.z, q0.w), w, Cr);
                        Cg = fma2(pack2(q1.x, q1.y), w, Cg);
                        Cb = fma2(pack2(q1.z, q1.w), w, Cb);
                    } else {
                        const float2 wo = unpack2(w);
                        float2 r = unpack2(Cr), g = unpack2(Cg), bl = unpack2(Cb);
                        add1(q0, q1, wo.x, r.x, g.x, bl.x);
                        add1(q0, q1, wo.y, r.y, g.y, bl.y);
                        Cr = pack2(r.x, r.y);
                        Cg = pack2(g.x, g.y);
                        Cb = pack2(bl.x, bl.y);
                    }
                };
                f32x2 al = alpha2(sa, qa0.x, a0, a1), be = alpha2(sb, qb0.x, b0, b1);
                f32x2 Ta = mul2(T, fma2(al, dup2(-1.0f), dup2(1.0f)));
                f32x2 Tb = mul2(Ta, fma2(be, dup2(-1.0f), dup2(1.0f)));
                const float2 tb = unpack2(Tb);
                if (__any_sync(kFull, fminf(tb.x, tb.y) < 0.0001f)) {
                    const uint32_t was = live;
                    const f32x2 To = T;
                    stop2(sa, al, Ta);
                    // a pixel that stopped at the first does not see the second
                    const bool g0 = (was ^ live) & 2u, g1 = (was ^ live) & 1u;
                    const float2 bo = unpack2(be);
                    if (kCount) c_hits -= (uint32_t)(g0 && b0) + (uint32_t)(g1 && b1);
                    be = pack2(g0 ? 0.0f : bo.x, g1 ? 0.0f : bo.y);
                    Tb = mul2(Ta, fma2(be, dup2(-1.0f), dup2(1.0f)));
                    T = Ta;
                    stop2(sb, be, Tb);
                    T = To;
                }
                add2c(qa0, qa1, mul2(al, T));
                add2c(qb0, qb1, mul2(be, Ta));
                T = Tb;
            } else {
                const float t0 = unpack2(T).x;
                float al = alpha1(W.pw[sa][i ^ 1u], qa0.x, a0), be = alpha1(W.pw[sb][i ^ 1u], qb0.x, b0);
                float ta = fm(t0, fs(1.0f, al)), tb = fm(ta, fs(1.0f, be));
                if (__any_sync(kFull, tb < 0.0001f)) {
                    if (tb < 0.0001f) {                            // stops before one of the two
                        const bool first = ta < 0.0001f;
                        const uint32_t sl = first ? sa : sb;
                        if (kCount) {
                            c_evals -= uncount(sl);
                            c_hits -= (uint32_t)(first && b0);
                        }
                        if (first) {
                            al = 0.0f;
                            ta = t0;
                        }
                        be = 0.0f;
                        tb = ta;
                        live = mask = 0u;
                        if (kKeep) keep_out[(size_t)y * cam.width + x] = make_uint2(__float_as_uint(ta), W.pos[sl]);
                    }
                }
                float r = unpack2(Cr).x, g = unpack2(Cg).x, bl = unpack2(Cb).x;
                add1(qa0, qa1, al * t0, r, g, bl);
                add1(qb0, qb1, be * ta, r, g, bl);
                Cr = pack2(r, 0.0f);
                Cg = pack2(g, 0.0f);
                Cb = pack2(bl, 0.0f);
                T = pack2(tb, 0.0f);
            }
        }
    };

    for (uint32_t s0 = rg.x; s0 < e; s0 += kC) {
        const uint32_t cnt = e - s0 < kC ? e - s0 : kC;
        // ---- stage: one record a thread, and the blocks it may meet
        bool odd = false;
        if (tid < cnt) {
            if (m >= M) m = 0;      // only after a failed sort (status already latched)
            const float4* g = reinterpret_cast<const float4*>(splat + (size_t)m * kSplatStride);
            const float4 g0 = __ldg(g), g1 = __ldg(g + 1), g2 = __ldg(g + 2);
            S.r0[tid] = g0;
            S.r1[tid] = staged_r1(g1);
            S.r2[tid] = g2;
            const uint32_t mask_tid = walk_mask(cam, tx0, ty0, g0.x, g0.y, g0.z, g0.w, g1.x, g1.y);
            S.mask[tid] = (uint16_t)mask_tid;
            odd = mask_tid && !(fabsf(g2.x) + fabsf(g2.y) + fabsf(g2.z) + fabsf(g0.x) + fabsf(g0.y) + fabsf(g0.z) +
                                        fabsf(g0.w) + fabsf(g1.x) <= 1.0e9f &&
                                g1.y >= -20.0f && g1.z >= 1.0e-20f);
        }
        const bool last = s0 + kC >= e;
        if (s0 + kC + tid < e) m = __ldg(vals + s0 + kC + tid);
        careful |= __syncthreads_or(odd) != 0;
        if (__any_sync(kFull, live != 0u)) {
            // ---- list
            uint32_t len[kBlocks] = {};
            const uint32_t lt = (1u << lane) - 1u;
            for (uint32_t j = lane; j < cnt + lane; j += 32) {
                const uint32_t bm = j < cnt ? (uint32_t)S.mask[j] >> fb : 0u;
#pragma unroll
                for (uint32_t k = 0; k < kBlocks; ++k) {
                    const uint32_t v = __ballot_sync(kFull, bm & (1u << k));
                    if (bm & (1u << k)) W.list[k][len[k] + __popc(v & lt)] = (uint8_t)j;
                    len[k] += __popc(v);
                }
            }
            __syncwarp();
            uint32_t left = len[0];
#pragma unroll
            for (uint32_t k = 1; k < kBlocks; ++k) left = b == k ? len[k] : left;
            const uint32_t en = (uint32_t)kLanes - 1u - i;         // (the transposition leaves entry 0 on top)
            const uint8_t* next = &W.list[b][en];
            for (;;) {
                const bool test = __any_sync(kFull, left != 0u);
                if (!test && !(last && __any_sync(kFull, mask != 0u))) break;
                if (test) {
                    // ---- test: one entry a lane at its block's 16 pixels
                    const bool valid = en < left;
                    const uint32_t rs = valid ? *next : 0u;
                    const float4 a = S.r0[rs];
                    const float4 c = S.r1[rs];
                    const float4 q = S.r2[rs];
                    const uint32_t sl = b * kSlots + ((par ^ (uint32_t)kLanes) | en);
                    if (valid) {
                        W.col[sl][0] = make_float4(c.z, c.z, q.x, q.x);
                        W.col[sl][1] = make_float4(q.y, q.y, q.z, q.z);
                        if (kKeep) W.pos[sl] = s0 + rs;
                    }
                    const f32x2 hA = dup2(fm(0.5f, a.z)), B2 = dup2(a.w), hC = dup2(fm(0.5f, c.x)), K = dup2(-c.y);
                    const f32x2 u2 = dup2(a.x), v2 = dup2(a.y);
                    f32x2 dx[4];
#pragma unroll
                    for (int k = 0; k < 4; ++k) dx[k] = add2(u2, npx[k]);
                    uint32_t miss = 0u;
#pragma unroll
                    for (int rp = 1; rp >= 0; --rp) {
                        const f32x2 dy = add2(v2, npy[rp]);
                        const f32x2 bdy = mul2(B2, dy), cdy = mul2(mul2(hC, dy), dy);
                        f32x2 n[4];
#pragma unroll
                        for (int k = 3; k >= 0; --k) {
                            n[k] = fma2(fma2(hA, dx[k], bdy), dx[k], cdy);         // -power, >= 0 where it counts
                            // 0 <= n <= K exactly if n (K - n) is not negative (n is never -0; NaN passes)
                            const float2 p = unpack2(mul2(n[k], fma2(n[k], dup2(-1.0f), K)));
                            miss = __funnelshift_l(__float_as_uint(p.x), miss, 1);
                            miss = __funnelshift_l(__float_as_uint(p.y), miss, 1);
                        }
                        float* pw = &W.pw[sl][8 * rp];
                        *reinterpret_cast<ulonglong2*>(pw) = make_ulonglong2(n[0], n[1]);
                        *reinterpret_cast<ulonglong2*>(pw + 4) = make_ulonglong2(n[2], n[3]);
                    }
                    mask |= transpose_bits<kLanes>(valid ? ~miss & 0xFFFFu : 0u, i) & live;
                    const uint32_t took = min(left, (uint32_t)kLanes);
                    if (kCount) {
                        c_steps += (kTwo ? 2u : 1u) * __reduce_max_sync(kFull, took);
                        c_evals += took * ((live >> 31) + (kTwo ? live & 1u : 0u));
                        c_new = took;
                    }
                    left -= took;
                    next += kLanes;
                    __syncwarp();
                }
                const uint32_t gate = test ? 0xFFFF0000u : kFull;
                if (careful) apply(gate, std::true_type{});
                else apply(gate, std::false_type{});
                __syncwarp();
                if (test) {
                    mask <<= 16;
                    par ^= (uint32_t)kLanes;
                }
                if (kCount) {
                    c_active += __popc(__reduce_or_sync(kFull, c_proc & gate));
                    c_proc = test ? c_proc << 16 : 0u;
                    c_old = c_new;
                    c_new = 0u;
                }
                if (__all_sync(kFull, live == 0u)) break;
            }
        }
        // the next chunk's records may replace this one's; all pixels stopped: no more chunks
        if (!last && __syncthreads_and(live == 0u)) break;
    }
    if (kCount) {
        c_evals = warp_sum_u32(c_evals);
        c_hits = warp_sum_u32(c_hits);
        if (lane == 0) {
            atomicAdd(&st->blend_entries, (unsigned long long)c_steps);
            atomicAdd(&st->blend_evals, (unsigned long long)c_evals);
            atomicAdd(&st->blend_hits, (unsigned long long)c_hits);
            atomicAdd(&st->blend_active, (unsigned long long)c_active);
        }
    }
    const float2 t = unpack2(T), r = unpack2(Cr), g = unpack2(Cg), bl = unpack2(Cb);
    const size_t hw = (size_t)cam.width * cam.height;
#pragma unroll
    for (int k = 0; k < (kTwo ? 2 : 1); ++k) {
        if (x >= cam.width || y + k >= cam.height) continue;
        const size_t pix = (size_t)(y + k) * cam.width + x;
        const float tk = k ? t.y : t.x;
        if (rgb) {
            rgb[pix] = fmaf(tk, cam.bg[0], k ? r.y : r.x);
            rgb[hw + pix] = fmaf(tk, cam.bg[1], k ? g.y : g.x);
            rgb[2 * hw + pix] = fmaf(tk, cam.bg[2], k ? bl.y : bl.x);
        }
        if (Tout) Tout[pix] = tk;
        // a live pixel did not stop
        if (kKeep && (live & (k ? kPx1 : kPx0))) keep_out[pix] = make_uint2(__float_as_uint(tk), e);
    }
}

// ---------------------------------------------------------------------------
// The KPC pre-render of a tile (Eq. 5-6)
// ---------------------------------------------------------------------------
struct KpcWarp {                                  // one warp's: 32 entries at a time
    float n[32][kParkStride];                     // -power at a block's 16 pixels
    float w[32][kParkStride];                     // alpha T, 0 where the entry is not applied
    float a0[32];
    uint8_t list[4][kWalkChunk];                  // per block: the chunk's records it may meet
};
struct KpcSmem {
    float4 r0[kWalkChunk];                        // u, v, A, B
    float4 r1[kWalkChunk];                        // C, lthr, alpha0, depth
    uint16_t mask[kWalkChunk];                    // walk_mask
    float part[16][kWalkChunk];                   // a record's sum over each block
    double red[kWalkWarps];
    KpcWarp w[kWalkWarps];
};

// blend_walk<8> without an image: after each group of 8 entries of each block a lane
// an entry sums the applied alpha T over its block's pixels, and after each chunk a
// thread a record adds up its blocks in their order.  Writes kpc_out of every pair of
// the tile and the tile's mean G_out[tile] (NaN for a tile without pairs).
__device__ __forceinline__ void blend_walk_kpc(const DevCamera& cam, uint32_t tile, uint2 rg, KpcSmem& S,
                                               const uint32_t* __restrict__ vals, const float* __restrict__ splat,
                                               float* __restrict__ kpc_out, float* __restrict__ G_out,
                                               const FrameState* st)
{
    constexpr uint32_t kC = kWalkChunk;
    const uint32_t tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const uint32_t b = lane >> 3, i = lane & 7u;
    const uint32_t M = st->M;
    const uint32_t e = rg.y;
    KpcWarp& W = S.w[warp];
    uint32_t m = rg.x + tid < e ? __ldg(vals + rg.x + tid) : 0u;
    const int32_t tx0 = (int32_t)(tile % (uint32_t)cam.tiles_x) * cam.tile_w;
    const int32_t ty0 = (int32_t)(tile / (uint32_t)cam.tiles_x) * cam.tile_h;
    int32_t ox, oy;
    uint32_t bsh;
    walk_origin(cam, warp, ox, oy, bsh);
    const int32_t bx0 = tx0 + ox + (int32_t)((b & ((1u << bsh) - 1u)) << 2);
    const int32_t by0 = ty0 + oy + (int32_t)((b >> bsh) << 2);
    const int32_t x = bx0 + (int32_t)(i & 3u), y = by0 + (int32_t)(i >> 2 << 1);
    uint32_t live = x < cam.width ? (y < cam.height ? 0xAAAAAAAAu : 0u) | (y + 1 < cam.height ? 0x55555555u : 0u) : 0u;
    f32x2 T = dup2(1.0f);
    f32x2 npx[4], npy[2];
#pragma unroll
    for (int k = 0; k < 4; ++k) npx[k] = dup2(-fa((float)(bx0 + k), 0.5f));
#pragma unroll
    for (int k = 0; k < 2; ++k)
        npy[k] = pack2(-fa((float)(by0 + 2 * k), 0.5f), -fa((float)(by0 + 2 * k + 1), 0.5f));
    double acc = 0.0;                             // this thread's share of the tile's sum (fixed order)

    for (uint32_t s0 = rg.x; s0 < e; s0 += kC) {
        const uint32_t cnt = e - s0 < kC ? e - s0 : kC;
        uint32_t my_mask = 0u;
        if (tid < cnt) {
            if (m >= M) m = 0;      // only after a failed sort (status already latched)
            const float4* g = reinterpret_cast<const float4*>(splat + (size_t)m * kSplatStride);
            const float4 g0 = __ldg(g), g1 = __ldg(g + 1);
            S.r0[tid] = g0;
            S.r1[tid] = staged_r1(g1);
            my_mask = walk_mask(cam, tx0, ty0, g0.x, g0.y, g0.z, g0.w, g1.x, g1.y);
            S.mask[tid] = (uint16_t)my_mask;
#pragma unroll
            for (int k = 0; k < 16; ++k) S.part[k][tid] = 0.0f;
        }
        if (s0 + kC + tid < e) m = __ldg(vals + s0 + kC + tid);
        __syncthreads();
        if (__any_sync(kFull, live != 0u)) {
            uint32_t len[4] = {};
            const uint32_t lt = (1u << lane) - 1u;
            for (uint32_t j = lane; j < cnt + lane; j += 32) {
                const uint32_t bm = j < cnt ? (uint32_t)S.mask[j] >> (4u * warp) : 0u;
#pragma unroll
                for (uint32_t k = 0; k < 4; ++k) {
                    const uint32_t v = __ballot_sync(kFull, bm & (1u << k));
                    if (bm & (1u << k)) W.list[k][len[k] + __popc(v & lt)] = (uint8_t)j;
                    len[k] += __popc(v);
                }
            }
            __syncwarp();
            uint32_t left = b == 0 ? len[0] : b == 1 ? len[1] : b == 2 ? len[2] : len[3];
            const uint32_t en = 7u - i, sl = b * 8u + en;
            const uint8_t* next = &W.list[b][en];
            while (__any_sync(kFull, left != 0u)) {
                // ---- test: one entry a lane at its block's 16 pixels
                const bool valid = en < left;
                const uint32_t rs = valid ? *next : 0u;
                const float4 a = S.r0[rs], c = S.r1[rs];
                W.a0[sl] = c.z;
                const f32x2 hA = dup2(fm(0.5f, a.z)), B2 = dup2(a.w), hC = dup2(fm(0.5f, c.x)), K = dup2(-c.y);
                f32x2 dx[4];
#pragma unroll
                for (int k = 0; k < 4; ++k) dx[k] = add2(dup2(a.x), npx[k]);
                uint32_t hits = 0u;
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
#pragma unroll
                for (int k = 0; k < 4; ++k)
                    *reinterpret_cast<float4*>(&W.w[sl][4 * k]) = make_float4(0.f, 0.f, 0.f, 0.f);
                uint32_t mask = (transpose_bits<8>(hits, i) & live) << 16;
                __syncwarp();
                // ---- apply
                while (__any_sync(kFull, mask != 0u)) {
                    const uint32_t sh = clz_or_ones(mask) & ~1u;
                    const uint32_t h = mask & shr0(0xC0000000u, sh);
                    const bool h0 = (h & 0xAAAAAAAAu) != 0u, h1 = (h & 0x55555555u) != 0u;
                    mask ^= h;
                    const uint32_t at = b * 8u + ((sh >> 1) & 7u);
                    const float a0 = W.a0[at];
                    const float2 n = *reinterpret_cast<const float2*>(&W.n[at][2 * i]);
                    auto alpha1 = [&](float nn, bool on) {
                        uint32_t t;
                        const float p = exp_poly_neg(nn, t);
                        const float al = fm(a0, fm(p, __uint_as_float((t << 23) + (127u << 23))));
                        return on ? fminf(al, 0.99f) : 0.0f;
                    };
                    const f32x2 al = pack2(alpha1(n.x, h0), alpha1(n.y, h1));
                    const f32x2 Tn = mul2(T, fma2(al, dup2(-1.0f), dup2(1.0f)));
                    float2 w = unpack2(mul2(al, T)), tn = unpack2(Tn);
                    if (fminf(tn.x, tn.y) < 0.0001f) {             // stops before this Gaussian
                        const float2 to = unpack2(T);
                        const bool q0 = tn.x < 0.0001f, q1 = tn.y < 0.0001f;
                        w = make_float2(q0 ? 0.0f : w.x, q1 ? 0.0f : w.y);
                        tn = make_float2(q0 ? to.x : tn.x, q1 ? to.y : tn.y);
                        live &= (q0 ? 0x55555555u : kFull) & (q1 ? 0xAAAAAAAAu : kFull);
                        mask &= live;
                    }
                    T = pack2(tn.x, tn.y);
                    if (h) *reinterpret_cast<float2*>(&W.w[at][2 * i]) = w;
                }
                __syncwarp();
                // ---- gather
                if (hits) {
                    f32x2 s2 = 0ull;
#pragma unroll
                    for (int k = 0; k < 4; ++k) {
                        const ulonglong2 v = *reinterpret_cast<const ulonglong2*>(&W.w[sl][4 * k]);
                        s2 = add2(v.y, add2(v.x, s2));
                    }
                    const float2 f = unpack2(s2);
                    S.part[4u * warp + b][rs] = f.x + f.y;
                }
                __syncwarp();
                left -= min(left, 8u);
                next += 8;
                if (__all_sync(kFull, live == 0u)) break;
            }
        }
        __syncthreads();
        if (tid < cnt) {
            float k = 0.0f;
#pragma unroll
            for (int h = 0; h < 16; ++h)
                if ((my_mask >> h) & 1u) k += S.part[h][tid];
            kpc_out[s0 + tid] = k;
            acc += (double)k;
        }
        __syncthreads();
    }
    // Eq. 6: G = mean KPC over the tile's pairs; fixed-order block reduction
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(kFull, acc, o);
    if (lane == 0) S.red[warp] = acc;
    __syncthreads();
    if (tid == 0) {
        const uint32_t n = e - rg.x;
        double sum = 0.0;
        for (int k = 0; k < kWalkWarps; ++k) sum += S.red[k];
        G_out[tile] = n > 0 ? (float)(sum / (double)n) : __int_as_float(0x7fc00000);
    }
}

// CTA bid's share of a grid of n_ctas: the halves of the split tiles (heavy[], listed by
// the sort) first, two CTAs for each of the split_slots there may be, then the n_tiles
// tiles, those that are not split.
template <class Whole, class Half>
__device__ __forceinline__ void walk_grid(uint32_t bid, uint32_t n_ctas, uint32_t n_tiles, const uint2* __restrict__ ranges,
                                          const uint32_t* __restrict__ heavy, const FrameState* st, Whole whole,
                                          Half half)
{
    const uint32_t n_half = n_ctas - n_tiles;
    if (bid < n_half) {
        if (bid >> 1 >= st->tickets[kTicketHeavy]) return;
        const uint32_t tile = heavy[bid >> 1];
        half(tile, bid & 1u, ranges[tile]);
    } else {
        const uint32_t tile = bid - n_half;
        const uint2 rg = ranges[tile];
        if (rg.y - rg.x > st->split) return;
        whole(tile, rg);
    }
}


}  // namespace blendk
}  // namespace fgs
