"""The auto image of per-antenna kernels (auto_rho_kernel and the epilogue's
per-antenna form) at the edges of its blocking: more offsets than threads, one
offset, more antennas than a tile of weights.  The difference between an image
with and without the subtraction against the oracle's; bound: 1e-5 of the
channel peak, the FP32 form's bound everywhere."""
import copy

import numpy as np
import pytest

import oracle
from gpu_helpers import peak_rel_err, run_gpu
from paper_2301_09662_gb300 import epic, synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("A,P,N,K", [
    (20, 2, 128, 15),      # 435 offsets in two rounds
    (30, 2, 96, 11),       # 231 offsets, one antenna at a time
    (33, 1, 64, 1),        # one offset, eight parts of the antennas
    (516, 2, 128, 3),      # two tiles of weights, the second of four antennas
    (24, 2, 32, 5),
    (20, 2, 256, 5),
])
def test_auto_image_edges(A, P, N, K):
    wl = synth.random_small(A=A, P=P, C=2, T=3, N=N, K=K, seed=A + N, full_range=True)
    wl = copy.copy(wl)
    wl.kernel = synth.antenna_kernels(wl.A, wl.K, np.random.default_rng(K))
    got, p = run_gpu(wl, flags=epic.EPIC_ANTENNA_KERNELS)
    p.close()
    assert peak_rel_err(got, oracle.workload_image(wl), wl.grid_n, P).max() < 1e-5


def test_one_antenna():
    """Its kernel is the plan's one kernel, and its image its auto image: nothing is left of it."""
    wl = copy.copy(synth.random_small(A=1, P=2, C=2, T=3, N=64, K=3, seed=1, full_range=True))
    wl.kernel = synth.antenna_kernels(1, 3, np.random.default_rng(3))
    got, p = run_gpu(wl, flags=epic.EPIC_ANTENNA_KERNELS)
    p.close()
    whole, p = run_gpu(wl, flags=epic.EPIC_ANTENNA_KERNELS | epic.EPIC_NO_AUTOSUB)
    p.close()
    ref = oracle.workload_image(wl, flags=epic.EPIC_NO_AUTOSUB)
    assert peak_rel_err(whole, ref, wl.grid_n, 2).max() < 1e-5
    assert np.abs(got).max() < 1e-5 * np.abs(ref).max()
