"""A plan's first call launches directly, later ones replay its graph: the same
image to the bit, also with buffers exchanged in every call, and when the first
call is made while its stream is being captured."""
import numpy as np
import pytest

import oracle
from gpu_helpers import peak_rel_err, torch_inputs
from paper_2301_09662_gb300 import epic, synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,A,P", [(32, 16, 1), (128, 40, 2)])
def test_first_and_later_calls_agree(N, A, P):
    import torch
    wl = synth.random_small(A=A, P=P, C=3, T=20, N=N, K=3, seed=N)
    p = epic.Plan.from_workload(wl)
    v, g = torch_inputs(wl)
    sets = [(v.clone(), g.clone()) for _ in range(3)]
    outs = [p.image(*sets[i % 3]) for i in range(7)] + [p.image(v, g), p.image(v, g)]
    torch.cuda.synchronize()
    assert all(torch.equal(outs[0], o) for o in outs[1:])
    p.close()
    got = outs[0].cpu().numpy().astype(np.complex128)
    assert peak_rel_err(got, oracle.workload_image(wl), wl.grid_n, P).max() < 1e-5


def test_first_call_under_capture():
    import torch
    wl = synth.random_small(A=24, P=2, C=2, T=9, N=64, K=3, seed=2)
    v, g = torch_inputs(wl)
    warm = epic.Plan.from_workload(wl)                  # the kernels are loaded before the capture
    ref = warm.image(v, g)
    torch.cuda.synchronize()
    p = epic.Plan.from_workload(wl)
    out = torch.zeros_like(ref)
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        p.image(v, g, out=out)
    graph.replay()
    torch.cuda.synchronize()
    assert torch.equal(out, ref)
    warm.close()
    p.close()


@pytest.mark.parametrize("flags", [0, epic.EPIC_DIAG_NO_GRAPH])
def test_stage_times_of_direct_and_replayed_calls(flags):
    import torch
    wl = synth.random_small(A=24, P=2, C=2, T=9, N=64, K=3, seed=2)
    v, g = torch_inputs(wl)
    p = epic.Plan.from_workload(wl, flags=flags)
    p.set_profiling()
    for _ in range(3):
        p.image(v, g)
        times = p.stage_times()
        assert len(times) == 3 and all(0 < t < 100 for t in times.values())
    p.close()
