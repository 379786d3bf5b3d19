"""The operator's own transforms over their range of sides and uv extents, the
kernel-weight tables, and degridding into buffers that are read as well,
against the FP64 oracle (tolerances as in test_gpu_operator.py)."""
import numpy as np
import pytest

import synth
from oracle import gridding as og

pytestmark = pytest.mark.gpu

TOL = {"fp64": 1e-12, "fp32": 1e-5, "fp32_kahan": 1e-5}


@pytest.fixture(scope="module")
def ms():
    import torch
    import paper_2406_18356_gb300 as pkg
    from paper_2406_18356_gb300 import _build
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    _build.build()
    pkg.load_library()
    return pkg


def rel(a, b):
    return float(np.linalg.norm(a - b) / np.linalg.norm(b))


# short: cells near the origin only; edge: footprints that wrap around the grid
@pytest.mark.parametrize("reach", [0.02, 0.3, 0.499])
@pytest.mark.parametrize("N", [16, 64, 512, 1024])
@pytest.mark.parametrize("precision", ["fp64", "fp32", "fp32_kahan"])
def test_both_directions(ms, N, reach, precision):
    import torch
    rng = np.random.default_rng(N)
    dl, n = 1e-3, 700
    u, v = synth.random_uv(n, N, dl, rng, frac_of_grid=reach)
    A = og.GriddedOperator(u, v, N, dl)
    plan = ms.Plan(u, v, N, dl, 0.2 * N, 2.0, precision=precision, levels=2)
    img = rng.standard_normal((N, N))
    vis = rng.standard_normal(n) + 1j * rng.standard_normal(n)
    got = plan.degrid("ALL", torch.from_numpy(img).to("cuda", plan.real_dtype)).cpu().numpy()
    assert rel(got, A.forward(img)) <= TOL[precision]
    got = plan.grid("ALL", torch.from_numpy(vis).to("cuda", plan.complex_dtype)).cpu().numpy()
    assert rel(got, A.dirty(vis)) <= TOL[precision]
    plan.close()


# beta within and above the range of the FP64 weight tables (the oracle's
# deapodization holds 1e-13 from the default, 16.1, on: its quadrature in t has
# the kernel's square-root ends, 1.6e-10 at beta = 8)
@pytest.mark.parametrize("beta", [16.1, 31.9, 33.0])
def test_kernel_shapes(ms, beta):
    import torch
    rng = np.random.default_rng(3)
    u, v = synth.random_uv(900, 32, 1e-3, rng)
    A = og.GriddedOperator(u, v, 32, 1e-3, beta=beta)
    plan = ms.Plan(u, v, 32, 1e-3, 6.0, 2.0, es_beta=beta, levels=2)
    img = rng.standard_normal((32, 32))
    vis = A.forward(img)
    got = plan.degrid("ALL", torch.from_numpy(img).cuda()).cpu().numpy()
    assert rel(got, vis) <= TOL["fp64"]
    got = plan.grid("ALL", torch.from_numpy(vis).cuda()).cpu().numpy()
    assert rel(got, A.dirty(vis)) <= TOL["fp64"]
    plan.close()


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
def test_degridding_into_its_observed_rows(ms, precision):
    """vis_out may be vis_obs, shifted over it, or shared by jobs that
    read it: every row is taken before any row it depends on is written."""
    import torch
    w = synth.tiny(npix=32, n_ant=12, n_dumps=10, seed=4)
    plan = ms.Plan(w.u[0], w.v[0], 32, w.pixel_size, w.ell_px, w.delta_px, precision=precision,
                   levels=2)
    rng = np.random.default_rng(0)
    img = torch.from_numpy(rng.standard_normal((32, 32))).to("cuda", plan.real_dtype)
    obs = torch.from_numpy(w.vis[0]).to("cuda", plan.complex_dtype)
    apart = {p: plan.degrid(p, img, obs, out=obs.clone()) for p in ("L", "H", "ALL")}
    same = obs.clone()
    plan.degrid("ALL", img, same, out=same)
    assert torch.equal(same, apart["ALL"])
    long = torch.cat([obs, obs[:7]])       # out starts 7 rows into obs
    plan.degrid("ALL", img, long[:-7], out=long[7:])
    assert torch.equal(long[7:], apart["ALL"])
    shared = obs.clone()
    plan.degrid_batch([(0, "L"), (0, "H")], [img, img], [shared, shared], outs=[shared, shared])
    rows = {p: torch.from_numpy(plan.partition_rows(p).astype(np.int64)).cuda() for p in "LH"}
    for p in "LH":   # rows of both partitions get the same value from either
        assert torch.equal(shared[rows[p]], apart[p][rows[p]])
    plan.close()


# work items of one tile around the fold's limits (lists up to 32 are summed
# by the cell, longer ones in groups of 16 first), the other tiles with few, on
# a grid summed one cell a thread and one summed four
@pytest.mark.parametrize("items", [1, 31, 32, 33, 48, 49, 70])
@pytest.mark.parametrize("N,tile", [(48, 16), (48, 32), (448, 16)])
@pytest.mark.parametrize("precision", ["fp64", "fp32", "fp32_kahan"])
def test_long_item_lists(ms, precision, N, tile, items):
    import torch
    rng = np.random.default_rng(items)
    dl, chunk = 1e-3, 16
    n = items * chunk - 5
    u = rng.uniform(2.0, tile - 3.0, n) / (2 * N * dl)   # inside the tile at the origin
    v = rng.uniform(2.0, tile - 3.0, n) / (2 * N * dl)
    u2, v2 = synth.random_uv(200, N, dl, rng)
    u, v = np.concatenate([u, u2]), np.concatenate([v, v2])
    vis = rng.standard_normal(len(u)) + 1j * rng.standard_normal(len(u))
    A = og.GriddedOperator(u, v, N, dl)
    plan = ms.Plan(u, v, N, dl, 9.0, 2.0, precision=precision, levels=2, tile=tile, chunk=chunk)
    d = torch.from_numpy(vis).to("cuda", plan.complex_dtype)
    got = plan.grid("ALL", d).cpu().numpy()
    assert rel(got, A.dirty(vis)) <= TOL[precision]
    both = plan.grid_batch([(0, "ALL"), (0, "L")], [d, d])
    np.testing.assert_array_equal(both[0].cpu().numpy(), got)
    assert torch.equal(both[1], plan.grid("L", d))
    plan.close()
