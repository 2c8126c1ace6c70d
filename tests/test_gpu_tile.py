"""The one-pass step (adi_tile.cu) at the edges of its tiles against the
separate sweeps of the same handle and against the FP64 oracle.

Both paths solve the same systems in FP32 and differ by rounding only.  A step
adds at most a few units in the last place of max|u| to the state and the
scheme carries a perturbation on at most linearly in the number of steps, so
after S steps the two differ by at most 4 S^2 2^-24 in relative L2 (the
truncated couplings, below 2^-30 per step, are far below that).
"""
import math

import numpy as np
import pytest

from helpers import gpu_run, oracle_run, rel_l2, smooth_state
from paper_2006_10142_gb300 import inputs

pytestmark = pytest.mark.gpu

STEPS = 6
BOUND = 4 * STEPS ** 2 * 2.0 ** -24


def _problem(nx, ny, cfl, seed):
    m = inputs.m_field(nx, ny, seed)
    tau = cfl * min(1.0 / (nx + 1), 1.0 / (ny + 1)) / math.sqrt(m.max())
    wav = inputs.wavelet_samples(STEPS + 2, tau, fp=3.0)
    return m, smooth_state(nx, ny, seed, 1e-2), tau, wav


# small patches (32 x 40 points), patches (96 x 40), bands (strips of 224
# columns, blocks of 16 rows); the halo of 12 (cfl 0.5) and of 16 (cfl 1, 32
# rows to a patch); sources at the corners of patches, chunks and blocks
@pytest.mark.parametrize("nx,ny,src", [(32, 40, (31, 39)), (33, 41, (32, 40)), (95, 7, (0, 0)), (224, 293, (0, 0)),
                                       (225, 304, (32, 40)), (449, 161, (224, 15)),
                                       (1000, 700, (96, 40)), (671, 1025, (479, 1024)), (2049, 200, (95, 39)),
                                       (257, 4099, (16, 32)),
                                       (2305, 2321, (224, 16)), (9000, 1000, (447, 999))])
@pytest.mark.parametrize("cfl", [0.5, 1.0])
def test_one_pass_step_matches_sweeps_and_oracle(nx, ny, src, cfl):
    m, phi, tau, wav = _problem(nx, ny, cfl, nx + ny)
    rec = np.array([[0, 0], [nx - 1, ny - 1], [nx // 2, ny // 3]], dtype=np.int32)
    a = gpu_run(m, phi, tau, STEPS, src=src, wavelet=wav, rec=rec)
    b = gpu_run(m, phi, tau, STEPS, src=src, wavelet=wav, rec=rec, tuning=dict(solver=1))
    o = oracle_run(m, phi, tau, STEPS, src=src, wavelet=wav, rec=rec)
    for f in ("u_cur", "u_prev", "traces"):
        assert rel_l2(a[f], b[f]) < BOUND, f
        assert rel_l2(a[f], o[f]) < 1e-4, f


@pytest.mark.parametrize("shapes", [[(2300, 2000, 0.5), (700, 900, 0.5), (224, 300, 1.0)],   # bands
                                    [(300, 260, 0.5), (33, 41, 0.5), (449, 64, 1.0)],        # patches
                                    [(300, 260, 0.5), (300, 200, 2.0), (120, 90, 5.0), (17, 40, 0.5),
                                     (100, 80, 0.5)]])  # with shots that need the sweeps
def test_batch_in_one_launch_matches_oracle(shapes):
    import torch
    from helpers import f32
    from paper_2006_10142_gb300 import api
    t = lambda a: torch.from_numpy(f32(a)).to("cuda:0")
    probs = [_problem(nx, ny, cfl, nx + ny) for nx, ny, cfl in shapes]
    srcs = [(nx // 3, ny // 2) for nx, ny, _ in shapes]
    B = api.AdiWaveBatch([t(p[0]) for p in probs], [t(p[1]) for p in probs], [p[2] for p in probs])
    for n in (STEPS - 1, 1):  # both orientations of the buffers
        B.run(n, srcs=srcs, wavelets=[t(p[3]) for p in probs])
    B.sync_status()
    for b, (m, phi, tau, wav) in enumerate(probs):
        up, uc, k = B.state(b)
        o = oracle_run(m, phi, tau, STEPS, src=srcs[b], wavelet=wav)
        assert k == STEPS + 1
        assert rel_l2(uc.double().cpu().numpy(), o["u_cur"]) < BOUND, shapes[b]
        assert rel_l2(up.double().cpu().numpy(), o["u_prev"]) < BOUND, shapes[b]
    B.close()


@pytest.mark.parametrize("nx,ny", [(300, 1100), (40, 4500), (1100, 700)])
def test_fp64_elimination_of_long_lines_matches_oracle(nx, ny):
    """The automatic FP64 geometry: 16 and 32 rows per thread over clusters,
    short columns."""
    m, phi, tau, wav = _problem(nx, ny, 6.0, nx + ny)
    a = gpu_run(m, phi, tau, STEPS, src=(nx // 2, ny - 1), wavelet=wav)
    o = oracle_run(m, phi, tau, STEPS, src=(nx // 2, ny - 1), wavelet=wav)
    for f in ("u_cur", "u_prev"):
        assert rel_l2(a[f], o[f]) < BOUND, f


def test_noalloc_step_of_two_sweeps_matches_handle():
    """tau = 2 h / max c: the couplings reach too far for the one-launch step;
    bit for bit the handle's step, as with it."""
    import torch
    from helpers import f32
    from paper_2006_10142_gb300 import api
    nx, ny = 300, 200
    m, phi, tau, wav = _problem(nx, ny, 2.0, 7)
    dev = torch.device("cuda:0")
    pit = lambda a: torch.nn.functional.pad(torch.from_numpy(f32(a)), (0, 320 - nx)).contiguous().to(dev)
    wav = torch.from_numpy(f32(wav)).to(dev)
    h = api.AdiWave(torch.from_numpy(f32(m)).to(dev), torch.from_numpy(f32(phi)).to(dev), tau)
    u0, u1, md = pit(phi), pit(phi), pit(m)
    for k in (1, 2):
        h.step(src=(9, 9), wavelet=wav)
        api.step_noalloc(md, u1, u0, nx, tau, float(f32(m).max()), k, src=(9, 9), wavelet=wav)
        u0, u1 = u1, u0
    assert torch.equal(h.state()[1], u1[:, :nx])
    h.close()


@pytest.mark.parametrize("tuning", [dict(), dict(use_graph=1)])
def test_levels_below_zero_have_no_source(tuning):
    """Levels -2 .. 2: the wavelet starts at level 0; every level is sampled."""
    import torch
    from helpers import f32
    from paper_2006_10142_gb300 import api
    nx, ny = 300, 260
    m, phi, tau, wav = _problem(nx, ny, 0.5, 5)
    t = lambda a: torch.from_numpy(f32(a)).to("cuda:0")
    out = []
    for tun in (tuning, dict(solver=1)):
        h = api.AdiWave(t(m), t(phi), tau)
        h.set_tuning(**tun)
        h.set_state(t(phi), t(phi), -2)
        tr = h.run(5, src=(31, 39), wavelet=t(1e4 * wav + 1e4), rec=[[31, 39], [32, 40], [299, 0]])
        out.append((tr, h.state()[1]))
        h.sync_status()
        h.close()
    for a, b in zip(*out):
        assert rel_l2(a.double().cpu().numpy(), b.double().cpu().numpy()) < BOUND


def test_one_pass_step_reports_non_finite_values():
    import torch
    from paper_2006_10142_gb300 import api
    nx, ny = 603, 500
    dev = torch.device("cuda:0")
    h = api.AdiWave(torch.ones(ny, nx, device=dev), torch.zeros(ny, nx, device=dev), 0.5 / 604)
    for j, i in ((0, 0), (ny - 1, nx - 1), (250, 223), (255, 224)):
        bad = torch.zeros(ny, nx, device=dev)
        bad[j, i] = float("inf")
        h.set_state(torch.zeros_like(bad), bad, 1)
        h.step()
        with pytest.raises(api.AdiError) as ei:
            h.sync_status()
        assert ei.value.code == 4
    h.close()
