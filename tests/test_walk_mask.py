"""The blend walk's block mask (blend_impl.cuh, walk_mask and walk_origin), restated in numpy
binary32 for all four tile shapes, is conservative: every pixel whose binary32 power passes
both skip tests lies in a block of the mask.  The quotient and the square roots, which the
kernel takes approximately, are taken at the low end of their error bounds (two units in
the last place for __fdividef, 2^-23 relative for sqrt.approx), where the box is smallest;
the determinant in every contraction.  Without the margins the same masks lose pixels."""
import numpy as np
import pytest

from test_cull_margins import boundary_gaussians, dets, fma, power, random_gaussians

f32 = np.float32
SHAPES = [(16, 16), (32, 8), (8, 32), (64, 4)]


def block_of_bit(tw, bit):
    """Column and row of the 4x4 block of mask bit 4 w + b: walk_origin's w-th four, block b of it."""
    shift = tw.bit_length() - 1
    bsh = 2 if shift == 6 else 1
    wsh = shift - 2 - bsh
    w, b = bit >> 2, bit & 3
    x = ((w & ((1 << wsh) - 1)) << (bsh + 2)) + ((b & ((1 << bsh) - 1)) << 2)
    y = ((w >> wsh) << (4 - bsh)) + ((b >> bsh) << 2)
    return x >> 2, y >> 2


def walk_mask(u, v, A, B, C, lthr, tx0, ty0, tw, det, margins=True):
    sh = (tw.bit_length() - 1) - 2
    ncol, nrow = 1 << sh, 16 >> sh
    tr = A + C
    full = ~(det > 0) | (tr * tr > f32(1e4) * det)
    with np.errstate(all="ignore"):
        s = fma(np.full_like(lthr, f32(-2.1)), lthr, np.full_like(lthr, f32(1e-4))) if margins else f32(-2.0) * lthr
        sd = (s / det) * f32(1.0 - 2.0 ** -22)
        ex, ey = (np.sqrt(sd * x) * f32(1.0 - 2.0 ** -23) for x in (C, A))
        if margins:
            ex, ey = (fma(e, np.full_like(e, f32(1.001)), np.full_like(e, f32(0.01))) for e in (ex, ey))

        def span(c, e, n):
            lo = np.maximum(0, np.nan_to_num(np.ceil((c - e - f32(3.5)) * f32(0.25)), nan=0, posinf=1e9, neginf=-1e9))
            hi = np.minimum(n - 1, np.nan_to_num(np.floor((c + e - f32(0.5)) * f32(0.25)), nan=0, posinf=1e9, neginf=-1e9))
            return lo.astype(np.int64), hi.astype(np.int64)

        c_lo, c_hi = span(u - f32(tx0), ex, ncol)
        r_lo, r_hi = span(v - f32(ty0), ey, nrow)
    some = (c_lo <= c_hi) & (r_lo <= r_hi)
    cl, ch = np.where(some, c_lo, 0), np.where(some, c_hi, 0)
    cols = ((2 << ch) - 1) & ~((1 << cl) - 1)
    if sh == 4:
        m = cols
    else:
        cols = (cols | cols << 4) & 0x0F0F
        cols = (cols | cols << 2) & 0x3333
        m = np.zeros_like(cols)
        for r in range(nrow):
            m |= np.where((r >= r_lo) & (r <= r_hi), cols << (((r >> 1) << (sh + 1)) + ((r & 1) << 1)), 0)
    m = np.where(some, m, 0)
    return np.where(~(lthr <= 0), 0, np.where(full, 0xFFFF, m)) & 0xFFFF


@pytest.mark.parametrize("tile", SHAPES, ids=lambda s: f"{s[0]}x{s[1]}")
def test_every_bit_is_one_block(tile):
    tw, th = tile
    blocks = {block_of_bit(tw, bit) for bit in range(16)}
    assert blocks == {(c, r) for c in range(tw // 4) for r in range(th // 4)}


@pytest.mark.parametrize("tile", SHAPES, ids=lambda s: f"{s[0]}x{s[1]}")
def test_mask_keeps_every_block_with_a_passing_pixel(tile):
    tw, th = tile
    tx0, ty0 = 5 * tw, 3 * th
    ys, xs = np.mgrid[0:th, 0:tw]
    px, py = (xs.ravel() + tx0).astype(f32) + f32(0.5), (ys.ravel() + ty0).astype(f32) + f32(0.5)
    bit_at = {block_of_bit(tw, b): b for b in range(16)}
    bit = np.array([bit_at[(x // 4, y // 4)] for x, y in zip(xs.ravel(), ys.ravel())])
    rng = np.random.default_rng(tw)
    hits = kept = masks = lost_without = 0
    for it in range(6):
        g = boundary_gaussians(rng, 16000, tx0, ty0, tw, th, 4, 4) if it % 2 else random_gaussians(rng, 16000, tx0, ty0, tw)
        u, v, A, B, C, lthr = g
        p = power(u, v, A, B, C, px, py)
        hit = ~((p > 0) | (p < lthr[:, None]))
        hits += int(hit.sum())
        for det in dets(A, B, C):
            m = walk_mask(*g, tx0, ty0, tw, det)
            missed = hit & ((m[:, None] >> bit) & 1 == 0)
            assert not missed.any(), np.flatnonzero(missed.any(1))[:1]
            kept += int(sum(((m >> b) & 1).sum() for b in range(16)))
            masks += 16 * len(m)
        exact = walk_mask(*g, tx0, ty0, tw, dets(A, B, C)[0], margins=False)
        lost_without += int((hit & ((exact[:, None] >> bit) & 1 == 0)).sum())
    assert hits > 100000 and kept < 0.8 * masks and lost_without > 50
