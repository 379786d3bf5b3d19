"""The largest sides of the operator's and the linear operator's own
transforms, and batches of minor cycles that take the widest tiles."""
import numpy as np
import pytest

import synth
import test_gpu_batch_fista as batch
import test_gpu_linear_transforms as linear
from oracle import gridding as og

pytestmark = pytest.mark.gpu

TOL = {"fp64": 1e-12, "fp32": 1e-5, "fp32_kahan": 1e-5}   # as in test_gpu_operator.py


def rel(a, b):
    return float((a - b).norm() / b.norm())


class Reference:
    """A = G F Z D and its scaled adjoint by torch in FP64: the oracle's
    deapodization and footprints, the FFT of the whole padded grid."""

    def __init__(self, u, v, N, dl):
        import torch
        A = og.GriddedOperator(u, v, N, dl)
        cells, weights = [], []
        for j in range(7):
            for i in range(7):
                cv, cu = A.c0v + j, A.c0u + i
                cells.append((cv % A.ngrid) * A.ngrid + cu % A.ngrid)
                weights.append(og.es_kernel(A.gv - cv, 7, A.beta) *
                               og.es_kernel(A.gu - cu, 7, A.beta))
        self.N, self.Ng, self.rows = N, A.ngrid, len(u)
        self.cells = torch.from_numpy(np.stack(cells)).cuda()
        self.weights = torch.from_numpy(np.stack(weights)).cuda()
        psi = torch.from_numpy(A.psi).cuda()
        self.psi2 = psi[:, None] * psi[None]
        self.at = torch.from_numpy(A.pad_index).cuda()

    def forward(self, image):
        import torch
        grid = torch.zeros((self.Ng, self.Ng), dtype=torch.complex128, device="cuda")
        grid[self.at[:, None], self.at[None]] = (image / self.psi2).to(torch.complex128)
        return (torch.fft.fft2(grid).reshape(-1)[self.cells] * self.weights).sum(0)

    def dirty(self, vis):
        import torch
        grid = torch.zeros(self.Ng * self.Ng, dtype=torch.complex128, device="cuda")
        grid.index_add_(0, self.cells.reshape(-1), (vis[None] * self.weights).reshape(-1))
        image = torch.fft.ifft2(grid.reshape(self.Ng, self.Ng)) * float(self.Ng) ** 2
        return image[self.at[:, None], self.at[None]].real / self.psi2 / self.rows


# (64: the reference against the sides that the oracle covers)
@pytest.mark.parametrize("N", [64, 2048, 4096])
@pytest.mark.parametrize("reach", [0.3, 0.499])
def test_operator(N, reach):
    import torch
    import paper_2406_18356_gb300 as ms
    rng = np.random.default_rng(N)
    dl, n = 1e-3, 700
    u, v = synth.random_uv(n, N, dl, rng, frac_of_grid=reach)
    ref = Reference(u, v, N, dl)
    img = torch.from_numpy(rng.standard_normal((N, N))).cuda()
    vis = torch.from_numpy(rng.standard_normal(n) + 1j * rng.standard_normal(n)).cuda()
    forward, dirty = ref.forward(img), ref.dirty(vis)
    if N == 64:
        A = og.GriddedOperator(u, v, N, dl)
        assert rel(forward, torch.from_numpy(A.forward(img.cpu().numpy())).cuda()) <= 1e-12
        assert rel(dirty, torch.from_numpy(A.dirty(vis.cpu().numpy())).cuda()) <= 1e-12
    for precision, tol in TOL.items():
        plan = ms.Plan(u, v, N, dl, 0.2 * N, 2.0, precision=precision, levels=1, n_bases=1)
        assert rel(plan.degrid("ALL", img.to(plan.real_dtype)), forward) <= tol, precision
        assert rel(plan.grid("ALL", vis.to(plan.complex_dtype)), dirty) <= tol, precision
        plan.close()


# L = 8192 in FP64 (3072: L = 4/3 of 2N) and in FP32 below 8/5 of 2N (2624; 2560
# goes to cuFFT), 8/5 at L = 4096
@pytest.mark.parametrize("precision,sides", [("fp64", (1536, 2048, 3072, 4096)),
                                             ("fp32", (1280, 2560, 2624))])
def test_linear_operator(precision, sides):
    linear.test_first_iteration_is_the_convolved_residual(precision, sides)


@pytest.mark.parametrize("precision,tol", [("fp64", 1e-11), ("fp32", 2e-5)])
@pytest.mark.parametrize("npix,channels", [(512, 3), (1024, 1)])
def test_minor_cycle_batch(npix, channels, precision, tol):
    """9 jobs of 512 px, 3 of 1024: as test_gpu_batch_fista.py."""
    import paper_2406_18356_gb300 as ms
    w = synth.multi_channel(npix=npix, nchan=channels, n_ant=16, n_dumps=16, span_h=4.0,
                            flag_max=0.3, with_vis=True, seed=3)
    plan = batch._plan(ms, w, precision)
    jobs = batch._jobs(plan, w, channels)
    models, stats = plan.minor_cycle_batch(jobs, 12)
    for j, m, st in zip(jobs, models, stats):
        want, rst = batch._per_job(plan, j, 12)
        assert st.iterations == rst.iterations == 12
        np.testing.assert_allclose(st.trace, rst.trace, rtol=tol)
        assert rel(m.double(), want.double()) <= tol, (j["step"], j["chan"])
    plan.close()
