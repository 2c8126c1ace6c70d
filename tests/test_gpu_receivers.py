"""Receiver traces of a run against the fields of the same steps taken one at
a time: the values are copies, equal to the bit, whoever takes them (the step
that starts from a level, or a launch after the step that made it)."""
import numpy as np
import pytest

from helpers import f32
from test_gpu_tile import _problem

pytestmark = pytest.mark.gpu


def _check(nx, ny, cfl, n_rec, tuning, every=0, steps=5):
    import torch
    from paper_2006_10142_gb300 import api
    m, phi, tau, wav = _problem(nx, ny, cfl, nx + ny)
    t = lambda a: torch.from_numpy(f32(a)).to("cuda:0")
    wav = t(np.tile(wav, 2))
    rng = np.random.default_rng(n_rec)
    rec = np.stack([rng.integers(0, nx, n_rec), rng.integers(0, ny, n_rec)], 1).astype(np.int32)
    rec[-1] = nx - 1, ny - 1
    src = (nx // 2, ny // 3)
    h = api.AdiWave(t(m), t(phi), tau)
    if tuning:
        h.set_tuning(**tuning)
    h.set_checkpointing(every)
    want = []
    # steps taken one at a time keep no checkpoints: the sweeps' plan then has to be given
    for _ in range(2 * steps):
        h.step(src=src, wavelet=wav)
        want.append(h.state()[1][rec[:, 1], rec[:, 0]])
    end = h.state()[1]
    h.reset(t(phi))
    got = [h.run(steps, src=src, wavelet=wav, rec=rec) for _ in range(2)]  # both orientations
    assert torch.equal(torch.cat(got), torch.stack(want))
    assert torch.equal(h.state()[1], end)
    h.reset(t(phi))  # other receivers: captured steps hold the list and its length
    assert torch.equal(h.run(steps, src=src, wavelet=wav, rec=rec[3:]), torch.stack(want[:steps])[:, 3:])
    h.sync_status()
    h.close()


@pytest.mark.parametrize("use_graph", [0, 1])
@pytest.mark.parametrize("nx,ny,tuning", [(300, 200, dict(solver=1)), (4100, 60, dict(solver=1)),
                                          (2500, 40, dict(x_stage=5, chunk_x=32, x_cluster=2, rows_per_cta=1))])
def test_sweeps(nx, ny, tuning, use_graph):
    _check(nx, ny, 0.5, 300, dict(tuning, use_graph=use_graph))


@pytest.mark.parametrize("tuning", [dict(solver=1), dict(x_stage=5, chunk_x=32, x_cluster=2, rows_per_cta=1)])
def test_sweeps_with_kept_segments(tuning):
    _check(2500, 40, 0.5, 300, tuning, every=2)


# small patches (256 threads a CTA), patches (256) and bands (128): up to eight
# receivers per thread in the step, more after it
@pytest.mark.parametrize("use_graph", [0, 1])
@pytest.mark.parametrize("nx,ny,n_rec", [(100, 75, 2048), (100, 75, 2049), (1000, 700, 2048), (1000, 700, 9000),
                                         (2305, 2321, 1024), (2305, 2321, 1025)])
def test_one_pass_step(nx, ny, n_rec, use_graph):
    _check(nx, ny, 0.5, n_rec, dict(use_graph=use_graph))


@pytest.mark.parametrize("n_rec", [16384, 16385])
def test_sweeps_with_many(n_rec):
    _check(300, 200, 0.5, n_rec, dict(solver=1))


def test_many_receivers_are_sampled_by_a_launch_of_their_own():
    """Every CTA of a one-pass step would go through the list otherwise."""
    import torch
    from paper_2006_10142_gb300 import api
    dev = torch.device("cuda:0")
    n, steps = 300, 4
    h = api.AdiWave(torch.ones(n, n, device=dev), torch.zeros(n, n, device=dev), 0.5 / (n + 1))
    count = []
    for n_rec in (2048, 2049):
        before = h.launch_count()
        h.run(steps, rec=np.zeros((n_rec, 2), dtype=np.int32))
        count.append(h.launch_count() - before)
    assert count[1] - count[0] == steps - 1  # the last level has one either way
    h.close()


def test_captured_run_keeps_its_receiver_list():
    """The caller's list is gone when the graph is replayed, and the handle has
    since sampled a longer one."""
    import gc
    import torch
    from paper_2006_10142_gb300 import api
    nx, ny, steps = 300, 260, 4
    m, phi, tau, wav = _problem(nx, ny, 0.5, 3)
    t = lambda a: torch.from_numpy(f32(a)).to("cuda:0")
    phi = t(phi)
    h = api.AdiWave(t(m), phi, tau)
    rng = np.random.default_rng(1)
    pick = lambda n: np.stack([rng.integers(0, nx, n), rng.integers(0, ny, n)], 1).astype(np.int32)
    few, many = pick(50), pick(5000)
    want = h.run(steps, rec=few)
    h.reset(phi)
    graph = torch.cuda.CUDAGraph()
    torch.cuda.synchronize()
    with torch.cuda.graph(graph):
        got = h.run(steps, rec=few.copy())
    gc.collect()
    junk = [np.full((50, 2), -7, dtype=np.int32) for _ in range(64)]
    h.run(steps, rec=many)
    for _ in range(2):
        h.reset(phi)
        got.zero_()
        graph.replay()
        assert torch.equal(got, want)
    h.sync_status()
    h.close()
    del junk
