"""The linear PSF operator at the sizes of its transform rule (own kernels of
length 2N or the next power of two, cuFFT on the 2N x 2N field otherwise)."""
import pytest

import synth

pytestmark = pytest.mark.gpu


# L = 2N, L > 2N by up to 8/5 (FP32) or 4/3 (FP64), and sides that keep cuFFT
# (FP32: 144, 272; FP64 also 80)
@pytest.mark.parametrize("precision,sides", [
    ("fp32", (16, 32, 48, 80, 96, 112, 128, 144, 192, 256, 272, 448, 512, 1024, 2048, 4096)),
    ("fp64", (16, 48, 64, 80, 128, 192, 256, 448, 512, 1024)),
    ("fp32_kahan", (32, 96, 256)),
])
def test_first_iteration_is_the_convolved_residual(precision, sides):
    """From zero, one iteration without threshold gives W beta_1 = (2 M /
    theta) H i~; H i~ by torch in FP64 from the PSF of a 2N plan.  FP32: the
    gridded PSF and two transforms of up to 13 stages, 1e-6 each, on a result
    within an order of magnitude of its input."""
    import torch
    import paper_2406_18356_gb300 as ms
    tol = 1e-10 if precision == "fp64" else 2e-5
    for N in sides:
        w = synth.tiny(npix=N, n_ant=12, n_dumps=8, seed=N)
        kw = dict(levels=1, n_bases=2)
        plan = ms.Plan(w.u[0], w.v[0], N, w.pixel_size, w.ell_px, w.delta_px,
                       precision=precision, convolution="linear", **kw)
        wide = ms.Plan(w.u[0], w.v[0], 2 * N, w.pixel_size, 2 * w.ell_px, 2 * w.delta_px,
                       precision="fp64", **kw)
        vis = torch.from_numpy(w.vis[0]).cuda().to(plan.complex_dtype)
        res = plan.grid("ALL", vis)
        spec = torch.fft.rfft2(torch.fft.ifftshift(wide.psf("ALL"))).real
        field = (2 * N, 2 * N)
        want = torch.fft.irfft2(spec * torch.fft.rfft2(res.double(), s=field), s=field)[:N, :N]
        model, st = plan.minor_cycle("single", res, 1e-20 * float(res.norm()), 1)
        want = want * (2 * 2 / st.theta)
        err = float((model.double() - want).norm() / want.norm())
        print(f"{precision} {N}: {err:.2e}")
        assert err <= tol, (N, err)
        plan.close()
        wide.close()
