"""The tables of the batch's one-launch step (tensor maps, arguments, CTA
list): in place for the first run, whatever stream it is on, and rebuilt when
a reset changes a plan."""
import pytest

from helpers import f32, rel_l2
from test_gpu_tile import _problem

pytestmark = pytest.mark.gpu

STEPS = 3
BOUND = 4 * STEPS ** 2 * 2.0 ** -24  # two forms of a step, as in test_gpu_tile.py


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
    """The same step launched per shot."""
    B, _ = _batch(probs, mode=1)
    B.run(steps)
    out = _states(B)
    B.sync_status()
    B.close()
    return out


def _near(a, b):
    h = lambda t: t.double().cpu().numpy()
    return all(rel_l2(h(x[q]), h(y[q])) < BOUND for x, y in zip(a, b) for q in (0, 1))


# by bands and, with a shot of 100 columns, by patches
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
        assert _near(_states(B), want)
        B.close()


def test_tables_follow_a_reset_that_changes_a_plan():
    """The second shot's medium moves it from the one-launch step to the sweeps
    and back, then all shots to the halo of 16: the tables are freed and made
    again, as like as not at the same address, with other shots and boxes."""
    import torch
    shapes = [(300, 260), (224, 300), (700, 500)]
    base = [_problem(nx, ny, 0.5, nx + ny) for nx, ny in shapes]
    B, t = _batch(base)
    for scale in ((1, 1, 1), (1, 16, 1), (1, 1, 1), (3.9, 3.9, 3.9), (1, 16, 16), (1, 1, 1)):
        probs = [(s * p[0],) + p[1:] for s, p in zip(scale, base)]
        want = _shot_by_shot(probs, STEPS)
        B.reset([t(p[1]) for p in probs], ms=[t(p[0]) for p in probs])
        B.run(STEPS)
        B.sync_status()
        assert _near(_states(B), want), scale
    B.close()
