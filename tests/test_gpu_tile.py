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
