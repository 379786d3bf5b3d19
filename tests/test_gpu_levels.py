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
