"""The wide FP32 kernels (sides 256 and 512, at most 128 x 128 occupied cells)
against the FP64 oracle at the edges of their range, just past it, in several
time batches, and against the per-class kernel.  Bound: 1e-5 of the channel
peak, the FP32 form's bound everywhere."""
import numpy as np
import pytest

import oracle
from gpu_helpers import peak_rel_err, run_gpu, torch_inputs
from paper_2301_09662_gb300 import epic, synth

pytestmark = pytest.mark.gpu
TOL = 1e-5
WIDE = epic.EPIC_DIAG_ALIAS_BATCH(200)      # small cases take the path too


def _case(N, A, T, K, span_x, span_y, C=2):
    """Footprints that span span_x x span_y cells."""
    wl = synth.random_small(A=A, P=2, C=C, T=T, N=N, K=K, seed=N + A + T, full_range=True)
    cell = synth.C0 / wl.freq_hz[0] * wl.du
    half = np.array([span_x - K, span_y - K]) / 2 * cell
    xy = wl.ant_xy - wl.ant_xy.mean(axis=0)
    xy = xy / np.abs(xy).max(axis=0) * half * 0.98
    xy[0], xy[1] = -half, half
    wl.ant_xy = xy - xy[2:].sum(axis=0) / len(xy)
    return wl


@pytest.mark.parametrize("N,A,T,K,sx,sy,flags", [
    (512, 60, 5, 7, 128, 128, 0),                          # the widest aperture, two full bands
    (512, 60, 3, 7, 131, 128, 0),                          # past it: the fold path
    (512, 44, 2, 5, 63, 65, 0),                            # one row in the second band
    (512, 36, 7, 3, 66, 33, 0),                            # one band, folded columns only
    (512, 40, 4, 5, 100, 120, epic.EPIC_KERNEL_TAPER),     # one tap
    (512, 40, 7, 5, 90, 100, epic.EPIC_DIAG_ALIAS_BATCH(3)),  # three time batches into the same partial images
    (512, 40, 7, 5, 90, 100, epic.EPIC_DIAG_ALIAS_BATCH(1)),  # seven into one
    (256, 60, 9, 5, 128, 127, 0),
    (256, 30, 1, 3, 17, 16, epic.EPIC_STOKES),             # one sample, one block of 16 rows
    (256, 34, 8, 7, 60, 128, epic.EPIC_DIAG_ALIAS_BATCH(3)),   # batches into a partial image each
    (256, 34, 16, 7, 60, 128, epic.EPIC_DIAG_ALIAS_BATCH(1)),  # sixteen into four in turn
])
def test_edges(N, A, T, K, sx, sy, flags):
    wl = _case(N, A, T, K, sx, sy)
    if not flags >> 16:
        flags |= WIDE
    got, p = run_gpu(wl, flags=flags)
    p.close()
    if flags & epic.EPIC_STOKES:
        plain, p = run_gpu(wl, flags=WIDE)
        p.close()
        im = oracle.split_channels(plain, wl.grid_n, 2)
        assert peak_rel_err(plain, oracle.workload_image(wl), wl.grid_n, 2).max() < TOL
        for s, x in zip(oracle.split_channels(got, wl.grid_n, 2), im):
            peak = np.abs(x[:2]).max()
            assert np.max(np.abs(s[0] - (x[0] + x[1]))) / peak < TOL
            assert np.max(np.abs(s[3] - 2 * x[2].imag)) / peak < TOL
        return
    assert peak_rel_err(got, oracle.workload_image(wl), wl.grid_n, 2).max() < TOL


@pytest.mark.parametrize("N", [256, 512])
def test_delays_against_the_per_class_kernel(N):
    import torch
    wl = _case(N, 48, 6, 5, 90, 100)
    d = torch.from_numpy(synth.geometric_delays(wl.ant_xy, wl.T)).cuda()
    v, g = torch_inputs(wl)
    out = []
    for flags in (WIDE, epic.EPIC_DIAG_NO_ALIAS):
        p = epic.Plan.from_workload(wl, flags=flags)
        out.append(p.image(v, g, delays=d).cpu().numpy().astype(np.complex128))
        p.close()
    assert peak_rel_err(out[0], out[1], wl.grid_n, 2).max() < TOL


def test_no_room_for_the_workspace():
    """1.5 GiB of device memory left, the workspace wants 4: the plan is made and images per class."""
    import torch
    wl = _case(256, 60, 3, 5, 100, 90)
    torch.cuda.empty_cache()
    hold = torch.empty(torch.cuda.mem_get_info()[0] - (3 << 29), dtype=torch.uint8, device="cuda")
    p = epic.Plan.from_workload(wl, max_spectra=16384)
    got, _ = run_gpu(wl, plan=p)
    p.close()
    del hold
    torch.cuda.empty_cache()
    assert peak_rel_err(got, oracle.workload_image(wl), wl.grid_n, 2).max() < TOL


def test_two_channel_groups():
    """63 channels x 100 spectra take two turns of the workspace, the second of one channel fewer."""
    wl = _case(512, 24, 2, 3, 126, 120, C=63)
    p = epic.Plan.from_workload(wl, flags=WIDE, max_spectra=100)
    got, _ = run_gpu(wl, plan=p)
    p.close()
    ch = [0, 31, 32, 62]
    got = [oracle.split_channels(got, wl.grid_n, 2)[c] for c in ch]
    ref = oracle.split_channels(oracle.workload_image(wl, channels=ch), wl.grid_n[ch], 2)
    for a, b in zip(got, ref):
        assert np.max(np.abs(a - b)) / np.max(np.abs(b[:2])) < TOL


def test_no_room_for_the_partial_images():
    """44 MiB left: the workspace (16) fits, with its nine partial images (36) it does not, and the
    plan images per class with two (8)."""
    import torch
    wl = _case(512, 40, 64, 3, 30, 28, C=1)
    v, g = torch_inputs(wl)
    out = torch.empty(4 * 512 * 512, dtype=torch.complex64, device="cuda")
    for flags in (WIDE, epic.EPIC_DIAG_NO_ALIAS):        # loads both paths' kernels
        p = epic.Plan.from_workload(wl, flags=flags)
        p.image(v, g, out=out)
        torch.cuda.synchronize()
        p.close()
    torch.cuda.empty_cache()
    hold = torch.empty(torch.cuda.mem_get_info()[0] - (44 << 20), dtype=torch.uint8, device="cuda")
    try:
        p = epic.Plan.from_workload(wl)
        p.image(v, g, out=out)
        torch.cuda.synchronize()
        assert p.status() == epic.EPIC_OK
        p.close()
    finally:
        del hold
        torch.cuda.empty_cache()
    got = out.cpu().numpy().astype(np.complex128)
    assert peak_rel_err(got, oracle.workload_image(wl), wl.grid_n, 2).max() < TOL


@pytest.mark.parametrize("flags", [0, epic.EPIC_DIAG_ALIAS_BATCH(3)])
def test_channels_on_both_sides_of_the_range(flags):
    """Two of three channels span at most 128 cells: a group each, one stage of the side."""
    wl = _case(512, 40, 7, 5, 120, 110, C=3)
    wl.freq_hz = wl.freq_hz[0] * np.array([1.0, 1.2, 0.9])
    p = epic.Plan.from_workload(wl, flags=flags | (WIDE if not flags else 0))
    p.set_profiling()
    got, _ = run_gpu(wl, plan=p)
    times = p.stage_times()
    p.close()
    assert peak_rel_err(got, oracle.workload_image(wl), wl.grid_n, 2).max() < TOL
    assert sorted(times) == ["autopower", "epilogue[N=512]", "image[N=512]"] and min(times.values()) > 0
