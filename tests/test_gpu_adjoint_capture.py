"""The adjoint captured into a caller's CUDA graph: every replay gives the
eager call's gradient, whatever ran on the handle before it."""
import numpy as np
import pytest

from paper_2006_10142_gb300 import inputs
from helpers import f32

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("every", [12, 6, 4])  # one, two and three segments
def test_replayed_adjoint_matches_eager(every):
    """An eager run leaves w and z of its last segments in the adjoint's
    workspace; a captured adjoint, and one after it, may not count on them.
    The kernels and values are the same either way: equal to the bit."""
    import torch
    from paper_2006_10142_gb300 import api
    dev = torch.device("cuda:0")
    n, steps = 65, 12
    prob, _ = inputs.adjoint_problem(n, steps, seed=3, n_rec=9)
    src = (n // 2, prob.rec[0][1] + 3)
    wav = torch.from_numpy(f32(prob.wavelet)).to(dev)
    m = torch.from_numpy(f32(prob.m)).to(dev)
    zero = torch.zeros(n, n, device=dev)
    gen = np.random.default_rng(5)
    resid = [torch.from_numpy(f32(gen.standard_normal((steps, len(prob.rec))))).to(dev) for _ in range(2)]
    h = api.AdiWave(m, zero, prob.tau, src=src, wavelet=wav)
    h.set_checkpointing(every)

    def run():
        h.reset(zero, src=src, wavelet=wav)
        h.run(steps, src=src, wavelet=wav, rec=prob.rec)

    try:
        want = []
        for r in resid:
            run()
            want.append(h.adjoint(r))
        assert all(w[0].abs().max() > 0 for w in want)
        run()
        fixed = resid[0].clone()
        graph = torch.cuda.CUDAGraph()
        torch.cuda.synchronize()
        with torch.cuda.graph(graph):
            got = h.adjoint(fixed)
        for q in (0, 1, 0, 1):
            fixed.copy_(resid[q])
            graph.replay()
            torch.cuda.synchronize()
            assert torch.equal(got[0], want[q][0]) and torch.equal(got[1], want[q][1]), q
        run()  # eager, then a replay in front of the eager adjoint
        graph.replay()
        gm, gw = h.adjoint(resid[0])
        h.sync_status()
        assert torch.equal(gm, want[0][0]) and torch.equal(gw, want[0][1])
    finally:
        h.close()
