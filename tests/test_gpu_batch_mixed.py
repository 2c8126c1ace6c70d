"""Batches of shots that take the one-launch step and shots that need the
sweeps: both groups advance side by side, replayed from a graph, launched one
by one, or in a caller's graph."""
import pytest

from helpers import oracle_run, rel_l2
from test_gpu_batch_tables import _batch, _states
from test_gpu_tile import _problem

pytestmark = pytest.mark.gpu

# tau = 2h and rows of fewer than 32 columns need the sweeps
SHAPES = [(300, 260, 0.5), (300, 200, 2.0), (17, 40, 0.5), (100, 80, 0.5), (500, 130, 2.0)]


@pytest.mark.parametrize("way", ["graph", "profile", "captured"])
def test_mixed_batch_matches_oracle(way):
    import torch
    probs = [_problem(nx, ny, cfl, nx + ny) for nx, ny, cfl in SHAPES]
    srcs = [(nx // 3, ny // 2) for nx, ny, _ in SHAPES]
    B, t = _batch(probs)
    wavs = [t(p[3]) for p in probs]
    B.profile(way == "profile")
    total = 0

    def run(n):
        B.run(n, srcs=srcs, wavelets=wavs)

    for n in (3, 1, 2):  # pairs and a step left over, one step, pairs; both orientations
        if way == "captured" and n == 2:
            graph = torch.cuda.CUDAGraph()
            torch.cuda.synchronize()
            with torch.cuda.graph(graph):
                run(n)
            graph.replay()
        else:
            run(n)
        total += n
    B.sync_status()
    bound = 4 * total ** 2 * 2.0 ** -24  # as in test_gpu_tile.py
    got = _states(B)
    for b, (m, phi, tau, wav) in enumerate(probs):
        o = oracle_run(m, phi, tau, total, src=srcs[b], wavelet=wav)
        assert B.state(b)[2] == total + 1
        assert rel_l2(got[b][1].double().cpu().numpy(), o["u_cur"]) < bound, SHAPES[b]
        assert rel_l2(got[b][0].double().cpu().numpy(), o["u_prev"]) < bound, SHAPES[b]
    B.close()


@pytest.mark.parametrize("shapes", [SHAPES, [s for s in SHAPES if s[2] < 1 and s[0] >= 32]])
def test_first_run_of_a_handle_may_be_captured(shapes):
    """Its tables are there, and nothing is allocated."""
    import torch
    probs = [_problem(nx, ny, cfl, nx + ny) for nx, ny, cfl in shapes]
    want, t = _batch(probs)
    want.run(3)
    B, _ = _batch(probs)
    graph = torch.cuda.CUDAGraph()
    torch.cuda.synchronize()
    with torch.cuda.graph(graph):
        B.run(3)
    graph.replay()
    B.sync_status()
    for a, b in zip(_states(B), _states(want)):
        assert torch.equal(a[0], b[0]) and torch.equal(a[1], b[1])
    B.close()
    want.close()
