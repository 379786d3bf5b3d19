"""Device memory of linear-operator plans per channel: one spectrum of the PSF
per partition beside the circular one, at the length of the transforms that
read it, or of the 2N x 2N field where longer ones would take gigabytes."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


def used(npix, channels):
    """bytes that a plan holds"""
    import torch
    import paper_2406_18356_gb300 as ms
    w = synth.tiny(npix=32)
    u, v = (np.repeat(a[:1], channels, axis=0) for a in (w.u, w.v))
    torch.cuda.synchronize()
    before = torch.cuda.mem_get_info()[0]
    plan = ms.Plan(u, v, npix, w.pixel_size * 32 / npix, 0.1 * npix, 3.0, precision="fp32",
                   levels=1, n_bases=1, convolution="linear")
    torch.cuda.synchronize()
    after = torch.cuda.mem_get_info()[0]
    plan.close()
    return before - after


# 2048: L = 2N, 1536: L = 8/3 N; a quarter for the allocations' granularity
# and the rows
@pytest.mark.parametrize("npix,length", [(2048, 4096), (1536, 4096)])
def test_one_spectrum_per_partition(npix, length):
    used(npix, 1)   # (what the library allocates once)
    got = used(npix, 9) - used(npix, 1)
    spectra = 8 * 3 * 4 * (npix * (npix // 2 + 1) + length * (length // 2 + 1))
    assert got <= 1.25 * spectra, (got / spectra)


def test_many_channels_keep_the_short_spectra():
    """80 channels at 1280 px: spectra of length 4096 would take 5 GB more."""
    n, channels = 1280, 80
    used(n, 1)
    got = used(n, channels) - used(n, 1)
    spectra = (channels - 1) * 3 * 4 * (n * (n // 2 + 1) + 2 * n * (n + 1))
    assert got <= 1.25 * spectra + (1 << 30), (got / spectra)
