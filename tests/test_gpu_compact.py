"""The compact FP32 kernel (sides 64, 96, 128 with at most 64 x 64 occupied
cells) against the FP64 oracle at the edges of its range, and against the
per-class kernel just past them.  Bound: 1e-5 of the channel peak, the FP32
form's bound everywhere."""
import numpy as np
import pytest

import oracle
from gpu_helpers import peak_rel_err, run_gpu, torch_inputs
from paper_2301_09662_gb300 import epic, synth

pytestmark = pytest.mark.gpu
TOL = 1e-5


def _span(wl, span, K):
    """Stretch the layout so that its footprints span exactly `span` cells on both axes."""
    cell = synth.C0 / wl.freq_hz[0] * wl.du
    half = (span - K) / 2 * cell
    xy = wl.ant_xy - wl.ant_xy.mean(axis=0)
    xy = xy / np.abs(xy).max(axis=0) * half * 0.98
    xy[0], xy[1] = (-half, -half), (half, half)
    wl.ant_xy = xy - xy[2:].sum(axis=0) / len(xy)      # keep the corners symmetric about the centroid
    return wl


@pytest.mark.parametrize("N,P,A,T,K,span", [
    (128, 2, 60, 5, 5, 64),     # the widest aperture: all 64 rows, lists read through L1
    (128, 2, 60, 5, 5, 67),     # past it: the per-class kernel
    (128, 2, 33, 4, 3, 33),     # one row and column past 32
    (128, 1, 37, 3, 3, 40),     # odd A P: voltages by bytes
    (128, 2, 41, 1, 7, 60),     # one sample, A P mod 4 = 2, widest kernel
    (96, 2, 50, 6, 3, 49),      # folds one position past 48
    (96, 1, 30, 2, 5, 64),
    (64, 2, 24, 7, 3, 40),      # two samples at a time, the last one absent
    (64, 1, 23, 8, 1, 33),      # one tap, odd row: the shared-memory kernel
    (64, 1, 23, 8, 3, 33),
    (64, 2, 40, 3, 5, 60),      # planes of two samples do not fit: the per-class kernel
    (64, 1, 104, 9, 5, 40),     # 65 footprint cells a row: compact with a single polarisation
    (64, 1, 92, 9, 5, 40),      # 57.5: the per-class kernel
    (64, 2, 16, 5, 1, 20),      # few footprint cells: the per-class kernel
])
def test_edges(N, P, A, T, K, span):
    wl = _span(synth.random_small(A=A, P=P, C=3, T=T, N=N, K=K, seed=A + N + T, full_range=True), span, K)
    got, p = run_gpu(wl)
    p.close()
    assert peak_rel_err(got, oracle.workload_image(wl), wl.grid_n, P).max() < TOL


@pytest.mark.parametrize("N,P,T", [(128, 2, 3), (96, 2, 4),     # so few spectra: the per-class kernel
                                   (128, 2, 38), (128, 2, 39), (128, 1, 76), (96, 1, 79), (96, 2, 44),  # and past its line
                                   (64, 1, 5)])
def test_efield_keeps_the_origin_phase(N, P, T):
    wl = synth.random_small(A=36, P=P, C=2, T=T, N=N, K=3, seed=N + T)
    p = epic.Plan.from_workload(wl)
    v, g = torch_inputs(wl)
    got = p.image_efield(v, g).cpu().numpy().astype(np.complex128)
    p.close()
    ref = oracle.workload_efield(wl)
    assert np.max(np.abs(got - ref)) / np.max(np.abs(ref)) < TOL


@pytest.mark.parametrize("N,left,right", [
    (128, 31, 30),     # from the quarter on, 62 cells + the kernel's
    (128, 36, 23),     # begins before the quarter and ends past cell 64: the factor from the table
    (96, 30, 30),      # the same at side 96, from cell 18 - 1
    (64, 20, 26),      # begins before the quarter, fits from the corner
])
def test_efield_placements(N, left, right):
    wl = synth.random_small(A=36, P=2, C=2, T=40, N=N, K=3, seed=left)   # past the per-class kernel's line
    cell = synth.C0 / wl.freq_hz[0] * wl.du
    rng = np.random.default_rng(N + left)
    for axis in (0, 1):
        x = rng.uniform(-8, 8, 36)
        x[0], x[1] = -left, right
        x[2:] -= x.sum() / 34
        wl.ant_xy[:, axis] = x * cell
    p = epic.Plan.from_workload(wl)
    v, g = torch_inputs(wl)
    got = p.image_efield(v, g).cpu().numpy().astype(np.complex128)
    p.close()
    ref = oracle.workload_efield(wl)
    assert np.max(np.abs(got - ref)) / np.max(np.abs(ref)) < TOL


def test_autotuned_long_call():
    """The tuner may keep fewer time chunks than the cost model (FP32 sums of up to 600 spectra)."""
    wl = synth.random_small(A=36, P=2, C=3, T=600, N=128, K=3, seed=11)
    p = epic.Plan.from_workload(wl)
    p.autotune(wl.T)
    got, _ = run_gpu(wl, plan=p)
    p.close()
    assert peak_rel_err(got, oracle.workload_image(wl), wl.grid_n, 2).max() < TOL
