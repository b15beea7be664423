"""CPU check of the assignment kernel's 32-bit distance form (DOT32) at its present tile of 64 columns: wherever the host's
bound 3 wc' vmax^2 + 6 ws' R^2 < 2^31 with R = 16 (63 + 3S) picks it, every partial sum in the kernel's order stays below
2^31 in magnitude, evaluated in exact integers at the extremes. The kernel stages K = wc' |c|^2 + ws' |x|^2 and the factors
-32 ws' x, -32 ws' y, -32 wc' c of plain pixel values, forms K + column term + row term once per candidate, adds the row
factor from row to row (once more after the last one), and for each row adds the three colour terms to it in turn. The parameter sets
that this tile admits and one of 128 columns would not are among them."""
from __future__ import annotations

import itertools

from test_seg_distance_bounds_cpu import weights

TILE_W, ROWS = 64, 5
TILE_ROWS = 4 * ROWS


def dot_bound(S, m, bd, tile):
    wcn, wsn = weights(S, m, bd)
    vmax, R = 16 * ((1 << bd) - 1), 16 * (tile - 1 + 3 * S)
    return wcn * 3 * vmax * vmax + wsn * 6 * R * R


def extreme_partial_sum(S, m, bd):
    wcn, wsn = weights(S, m, bd)
    vmax = (1 << bd) - 1
    # a mean lies in a cell next to the pixel's: at most 2 S - 1 pixels beyond the tile, and so does its position
    xs, ys = ([16 * -(2 * S), 16 * (n - 1 + 2 * S)] for n in (TILE_W, TILE_ROWS))
    worst = 0
    for xk, yk in itertools.product(xs, ys):
        for ck in itertools.product((0, 16 * vmax), repeat=3):
            K = wcn * sum(c * c for c in ck) + wsn * (xk * xk + yk * yk)
            fx, fy, fc = -32 * wsn * xk, -32 * wsn * yk, [-32 * wcn * c for c in ck]
            worst = max(worst, K, abs(fx), abs(fy), *(abs(f) for f in fc))
            for px in (0, TILE_W - 1):
                worst = max(worst, abs(K + px * fx))
                for py in (0, TILE_ROWS - 1, TILE_ROWS):  # the first row of a group to the step past the last one
                    t = K + px * fx + py * fy
                    for v in itertools.product((0, vmax), repeat=3):
                        worst = max(worst, *(abs(s) for s in itertools.accumulate((v[c] * fc[c] for c in range(3)), initial=t)))
    return worst


def test_partial_sums_fit_wherever_the_host_picks_the_form():
    only_here = n = 0
    for S, m, bd in itertools.product(range(1, 65), (0, 1, 2, 5, 10, 20, 40, 90, 255), (4, 6, 7, 8, 9, 10, 12)):
        if dot_bound(S, m, bd, TILE_W) >= 1 << 31:
            continue
        only = dot_bound(S, m, bd, 128) >= 1 << 31
        if not only and (S * m + bd) % 3:  # every set near the limit, a third of the others
            continue
        n, only_here = n + 1, only_here + only
        assert extreme_partial_sum(S, m, bd) < 1 << 31, (S, m, bd)
    assert n > 150 and only_here >= 20


def test_sets_that_the_narrower_tile_admits():
    for S, m, bd in ((6, 5, 6), (11, 10, 6), (18, 20, 6)):
        assert dot_bound(S, m, bd, TILE_W) < 1 << 31 <= dot_bound(S, m, bd, 128)
