"""Gains and kernels whose scales cancel, or leave FP32's exponents when squared: the
subtraction of the auto term keeps the range it has in FP64.  Powers of two, so that scaled
inputs give the same roundings."""
import copy

import numpy as np
import pytest

from gpu_helpers import run_gpu, torch_inputs
from paper_2301_09662_gb300 import epic, synth

pytestmark = pytest.mark.gpu


def _scaled(wl, gain, kernel):
    wl = copy.copy(wl)
    wl.gains = (wl.gains * np.float32(2.0 ** gain)).astype(np.complex64)
    wl.kernel = (wl.kernel * np.float32(2.0 ** kernel)).astype(np.complex64)
    return wl


@pytest.mark.parametrize("N,A,P", [(32, 20, 1), (96, 70, 2), (128, 36, 2), (512, 40, 2)])
@pytest.mark.parametrize("e", [66, -66])
def test_scales_that_cancel(N, A, P, e):
    """A_pq is 2^132 times (or 2^-132 of) what it was, the image the same to the bit."""
    wl = synth.random_small(A=A, P=P, C=2, T=9, N=N, K=3, seed=N + A)
    ref, p = run_gpu(wl)
    p.close()
    got, p = run_gpu(_scaled(wl, e, -e))
    p.close()
    assert np.array_equal(got, ref)


@pytest.mark.parametrize("e", [-66, -30, 30, 50])
def test_taper_outside_the_exponents(e):
    """|W^|^2 of 2^(2 e): times sums of the usual size the image is a number of FP32 again.  Bound:
    the FP64 and the pair form of one product differ by a rounding of the result, 2^-24."""
    wl = synth.random_small(A=36, P=2, C=1, T=6, N=64, K=5, seed=8)
    ref, p = run_gpu(wl, flags=epic.EPIC_KERNEL_TAPER)
    p.close()
    got, p = run_gpu(_scaled(wl, 0, e), flags=epic.EPIC_KERNEL_TAPER)
    p.close()
    got = np.ldexp(got.view(np.float64), -2 * e).view(np.complex128)
    assert np.max(np.abs(got - ref)) <= 2.0 ** -23 * np.max(np.abs(ref))


def test_static_entry_point():
    import torch
    wl = synth.random_small(A=24, P=2, C=2, T=5, N=64, K=3, seed=3)
    out = []
    for w in (wl, _scaled(wl, 66, -66)):
        v, g = torch_inputs(w)
        out.append(epic.image_static(w.ant_xy, 2, w.kernel, 64, w.freq_hz, w.du, v, g))
    assert torch.equal(out[0], out[1]) and bool(torch.isfinite(out[0].real).all())
