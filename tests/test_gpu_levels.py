"""Dictionary transforms and FISTA on image sides whose coarse levels are no
multiples of a tile or of a 16-byte vector, against the FP64 oracle (the tests
of the usual sides are in test_gpu_solver.py).  Coefficients and images are
sums of at most 2 x 4 x 16 products per level and direction, so FP64 holds
1e-12 and FP32 1e-5 relative L2 (the operators' bar)."""
import numpy as np
import pytest

import synth
from oracle.wavelets import Dictionary

pytestmark = pytest.mark.gpu


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


# 480 = 16 x 30 and 240 = 16 x 15: coarsest subbands of side 30 and 15, whose
# rows start on no 16-byte boundary; 176 = 16 x 11 and 96 = 16 x 6
@pytest.mark.parametrize("precision,tol", [("fp64", 1e-12), ("fp32", 1e-5)])
@pytest.mark.parametrize("N,J", [(480, 4), (240, 4), (176, 4), (96, 4), (112, 3)])
def test_transforms_on_odd_coarse_levels(ms, N, J, precision, tol):
    import torch
    w = synth.tiny(npix=32)
    plan = ms.Plan(w.u[0], w.v[0], N, w.pixel_size * 32 / N, 0.1 * N, 3.0, precision=precision,
                   levels=J)
    dt = torch.float64 if precision == "fp64" else torch.float32
    rng = np.random.default_rng(N)
    alpha, x = rng.standard_normal((8, N, N)), rng.standard_normal((N, N))
    W = Dictionary(N, 8, J)
    got = plan.dictionary_synthesis(torch.from_numpy(alpha).to("cuda", dt)).double().cpu().numpy()
    assert rel(got, W.synth(alpha)) <= tol
    got = plan.dictionary_analysis(torch.from_numpy(x).to("cuda", dt)).double().cpu().numpy()
    assert rel(got, W.analysis(x)) <= tol
    plan.close()


# level 1 of the synthesis, FP32: 4 output pairs a thread (1024 px: 1024
# tiles), 2 (fewer tiles), straight from the coefficient planes (one level),
# with fewer bases; FP64 beside it
@pytest.mark.parametrize("precision,tol", [("fp64", 1e-12), ("fp32", 1e-5)])
@pytest.mark.parametrize("N,J,M", [(1024, 2, 8), (320, 1, 8), (288, 2, 3), (256, 1, 1)])
def test_synthesis_sum_over_bases(ms, N, J, M, precision, tol):
    import torch
    w = synth.tiny(npix=32)
    plan = ms.Plan(w.u[0], w.v[0], N, w.pixel_size * 32 / N, 0.1 * N, 3.0, precision=precision,
                   levels=J, n_bases=M)
    dt = torch.float64 if precision == "fp64" else torch.float32
    alpha = np.random.default_rng(N).standard_normal((M, N, N))
    got = plan.dictionary_synthesis(torch.from_numpy(alpha).to("cuda", dt)).double().cpu().numpy()
    assert rel(got, Dictionary(N, M, J).synth(alpha)) <= tol
    plan.close()


@pytest.mark.parametrize("precision,tol", [("fp64", 1e-9), ("fp32", 2e-5)])
@pytest.mark.parametrize("N,J", [(176, 4), (480, 4), (96, 4)])
def test_fista_on_odd_coarse_levels(ms, N, J, precision, tol):
    """Three iterations of step one's problem (the prox fused into the level
    kernels), started from given coefficients."""
    import torch
    from oracle.gridding import GriddedOperator, partition
    from oracle.solver import Problem, fista, psf_spectrum
    w = synth.tiny(npix=32)
    dl = w.pixel_size * 32 / N
    ell, delta = 0.1 * N, 3.0
    plan = ms.Plan(w.u[0], w.v[0], N, dl, ell, delta, precision=precision, levels=J)
    dt = torch.float64 if precision == "fp64" else torch.float32
    rng = np.random.default_rng(N)
    res, start = rng.standard_normal((N, N)), rng.standard_normal((8, N, N))
    in_l, _ = partition(w.u[0], w.v[0], N, dl, ell, delta)
    A = GriddedOperator(w.u[0][in_l], w.v[0][in_l], N, dl)
    lam = 0.5
    prob = Problem("low", Dictionary(N, 8, J), psf_spectrum(A.psf()), res, lam)
    ref = fista(prob, 3, beta0=start)
    beta = torch.from_numpy(start).to("cuda", dt)
    model, st = plan.minor_cycle("low", torch.from_numpy(res).to("cuda", dt), lam, 3, beta=beta)
    assert st.iterations == 3
    assert rel(beta.double().cpu().numpy(), ref.beta) <= tol
    assert rel(model.double().cpu().numpy(), prob.W.synth(ref.beta)) <= tol
    plan.close()
