"""The gain solver's cluster form (n_ant n_pol <= 1024) at the edges of its row
widths, with few samples and odd rows, and the one-CTA form just past it,
against the FP64 oracle.  FP32 sums of T <= 70 samples and A <= 601 antennas:
relative rounding below 2^-24 sqrt(T A) ~ 1e-5 of the unit RMS gain."""
import numpy as np
import pytest

import oracle
from oracle import calib
from paper_2301_09662_gb300 import epic, synth

from gpu_helpers import torch_inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("A,P,C,T", [
    (64, 2, 3, 70),     # 128 values: one word a lane, exactly full
    (65, 2, 2, 33),     # rows of 130 bytes: read by bytes
    (128, 2, 70, 40),   # 256 values, many channels: small clusters
    (256, 2, 2, 7),     # fewer samples than warps
    (257, 1, 1, 1),     # one sample, odd row
    (512, 2, 1, 50),    # 1024 values
    (513, 2, 1, 20),    # past the widest: the one-CTA form
    # the calls above of fewer than 48 spectra (64 past 512 values) take the one-CTA form; clusters:
    (65, 2, 2, 49),     # rows read by bytes, a sample more than a multiple of the warps
    (128, 2, 70, 48),   # the shortest, many channels: small clusters
    (257, 1, 1, 51),    # odd row
    (512, 2, 1, 67),    # the widest
    (300, 2, 61, 64),   # 600 values: one CTA an SM
    (601, 1, 2, 17),    # past 512 values of one polarisation
])
def test_edges(A, P, C, T):
    wl = synth.random_small(A=A, P=P, C=C, T=T, N=128, K=1, seed=A + T, gains=False)
    rng = np.random.default_rng(A)
    l0, m0 = 0.25, -0.125
    xy = wl.ant_xy - wl.ant_xy.mean(axis=0)
    uv = xy[None] * (wl.freq_hz[:, None, None] / synth.C0)
    ph = np.exp(-2j * np.pi * (uv[..., 0] * l0 + uv[..., 1] * m0))                  # [C][A]
    G = rng.uniform(0.7, 1.3, (C, A, P)) * np.exp(1j * rng.uniform(-1, 1, (C, A, P)))
    s = 2 * (rng.standard_normal((T, C, 1, P)) + 1j * rng.standard_normal((T, C, 1, P)))
    x = s * (ph[..., None] * G)[None] + rng.standard_normal((T, C, A, P)) + 1j * rng.standard_normal((T, C, A, P))
    wl.v = synth.pack_ci4(synth.quantise(x.real), synth.quantise(x.imag))
    p = epic.Plan.from_workload(wl)
    v, _ = torch_inputs(wl)
    got = p.solve_gains(v, l0, m0, 2).cpu().numpy().astype(np.complex128)
    p.close()
    ref = calib.solve_gains(wl.v, oracle.cell_map(wl.ant_xy, wl.freq_hz, wl.grid_n, wl.du), wl.grid_n, l0, m0, wl.du, 2)
    assert np.max(np.abs(got - ref)) < 2e-5
