"""The tables of the batch's one-launch step (tensor maps, arguments, CTA
list): in place for the first run, whatever stream it is on, and rebuilt when
a reset changes a plan."""
import pytest

from helpers import f32
from test_gpu_tile import _problem

pytestmark = pytest.mark.gpu

STEPS = 3


def _batch(probs, mode=None):
    import torch
    from paper_2006_10142_gb300 import api
    t = lambda a: torch.from_numpy(f32(a)).to("cuda:0")
    B = api.AdiWaveBatch([t(p[0]) for p in probs], [t(p[1]) for p in probs], [p[2] for p in probs])
    if mode is not None:
        B.set_mode(mode)
    return B, t


def _states(B):
    return [B.state(b)[:2] for b in range(B.n)]


def _shot_by_shot(probs, steps):
    """The same kernels launched per shot: equal to the bit for the halo of 12."""
    B, _ = _batch(probs, mode=1)
    B.run(steps)
    out = _states(B)
    B.sync_status()
    B.close()
    return out


def _equal(a, b):
    import torch
    return all(torch.equal(x[0], y[0]) and torch.equal(x[1], y[1]) for x, y in zip(a, b))


# 256 x 240 and above go by bands, 100 columns by patches
@pytest.mark.parametrize("shapes", [[(2300, 2000), (700, 900), (224, 300)], [(300, 260), (100, 41)]])
def test_first_run_on_a_non_blocking_stream(shapes):
    import torch
    probs = [_problem(nx, ny, 0.5, nx + ny) for nx, ny in shapes]
    want = _shot_by_shot(probs, STEPS)
    side = torch.cuda.Stream()  # non-blocking: not ordered with the legacy stream
    for _ in range(3):
        B, _ = _batch(probs)
        torch.cuda.synchronize()
        B.run(STEPS, stream=side)
        side.synchronize()
        assert _equal(_states(B), want)
        B.close()
