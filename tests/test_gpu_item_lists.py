"""The gridding fold at the limits of its work-item lists, with rows that all
anchor in one tile, so that the list has the length it is named for (lists up
to 32 items are summed by the cell, longer ones in groups of 16 first).
Against the FP64 oracle; tolerances as in test_gpu_operator.py."""
import numpy as np
import pytest

import synth
from oracle import gridding as og

TOL = {"fp64": 1e-12, "fp32": 1e-5, "fp32_kahan": 1e-5}
CHUNK, DL = 16, 1e-3
LISTS = [1, 16, 31, 32, 33, 47, 48, 49, 64, 65]
# grids summed one cell a thread, then four (from some 790 cells a side: all of
# 2 x 448, and of 2 x 512 a square that starts at no multiple of four cells)
GRIDS = [(48, 16), (48, 32), (448, 16), (448, 32), (512, 16), (512, 32)]


def rel(a, b):
    return float(np.linalg.norm(a - b) / np.linalg.norm(b))


def tile_of(gu, gv, Ng, tile):
    """Tile indices of the rows' footprint anchors (cell k at index k + Ng / 2)."""
    a = [(np.floor(g - 3.5).astype(np.int64) + 1 + Ng // 2) % Ng // tile for g in (gv, gu)]
    return a[0] * (Ng // tile) + a[1]


def observation(N, tile, items):
    """u, v whose longest list has `items` work items of CHUNK rows (the last
    one five rows short): all its rows anchor in one tile near the origin, no
    other tile has more than one item; at 512 px the outermost footprint reaches
    cell 439."""
    rng = np.random.default_rng(items)
    Ng = 2 * N
    corner = (Ng // 2 // tile) * tile - Ng // 2   # grid cell of the tile's first anchor
    n = items * CHUNK - 5
    gu, gv = (corner + 2.5 + rng.uniform(0.01, tile - 0.01, n) for _ in range(2))
    u2, v2 = synth.random_uv(300, N, DL, rng, frac_of_grid=0.42)
    gu2, gv2 = u2 * Ng * DL, v2 * Ng * DL
    gu2[0], gv2[0] = 436.2 / 512 * N, 0.1
    t = tile_of(gu2, gv2, Ng, tile)
    keep, home = np.zeros(len(t), bool), tile_of(gu[:1], gv[:1], Ng, tile)[0]
    for k in np.unique(t[t != home]):
        keep[np.flatnonzero(t == k)[:CHUNK]] = True
    order = rng.permutation(n + int(keep.sum()))
    return (np.concatenate([a, b[keep]])[order] / (Ng * DL) for a, b in ((gu, gu2), (gv, gv2)))


@pytest.mark.parametrize("items", LISTS)
@pytest.mark.parametrize("N,tile", GRIDS)
def test_lists_have_the_stated_length(N, tile, items):
    u, v = observation(N, tile, items)
    A = og.GriddedOperator(u, v, N, DL)
    rows = np.bincount(tile_of(A.gu, A.gv, 2 * N, tile))
    lists = -(-rows // CHUNK)
    assert lists.max() == items and np.sort(lists)[-2] == 1
    if N == 512:   # the square of reached cells: four cells a thread, unaligned start
        reach = max(np.abs(c).max() for a in (A.c0u, A.c0v) for c in (a, a + 6))
        assert reach < N and (2 * reach + 1) ** 2 / 4 >= 152 * 1024 and (N - reach) % 4


@pytest.mark.gpu
@pytest.mark.parametrize("items", LISTS)
@pytest.mark.parametrize("N,tile", GRIDS)
@pytest.mark.parametrize("precision", ["fp64", "fp32", "fp32_kahan"])
def test_fold_of_long_lists(precision, N, tile, items):
    import torch
    import paper_2406_18356_gb300 as ms
    u, v = observation(N, tile, items)
    rng = np.random.default_rng(N + items)
    vis = rng.standard_normal(len(u)) + 1j * rng.standard_normal(len(u))
    plan = ms.Plan(u, v, N, DL, 9.0, 2.0, precision=precision, levels=2, tile=tile, chunk=CHUNK)
    d = torch.from_numpy(vis).to("cuda", plan.complex_dtype)
    got = plan.grid("ALL", d).cpu().numpy()
    assert rel(got, og.GriddedOperator(u, v, N, DL).dirty(vis)) <= TOL[precision]
    both = plan.grid_batch([(0, "ALL"), (0, "L")], [d, d])
    np.testing.assert_array_equal(both[0].cpu().numpy(), got)
    assert torch.equal(both[1], plan.grid("L", d))
    plan.close()


# (48: cuFFT sides use the whole grid)
@pytest.mark.gpu
@pytest.mark.parametrize("N,want", [(48, 48), (64, 58), (512, 439)])
def test_grid_extent(N, want):
    import paper_2406_18356_gb300 as ms
    u, v = observation(N, 16, 2)
    plan = ms.Plan(u, v, N, DL, 9.0, 2.0, levels=2)
    A = og.GriddedOperator(u, v, N, DL)
    if N != 48:
        assert want == max(np.abs(c).max() for a in (A.c0u, A.c0v) for c in (a, a + 6))
    assert plan.grid_extent() == want
    plan.close()
