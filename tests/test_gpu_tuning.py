"""What a tuning selects, refuses and reports."""
import pytest

pytestmark = pytest.mark.gpu


def _handle(nx, ny, cfl, **kw):
    import torch
    from paper_2006_10142_gb300 import api
    dev = torch.device("cuda:0")
    return api.AdiWave(torch.ones(ny, nx, device=dev), torch.zeros(ny, nx, device=dev),
                       cfl / (max(nx, ny) + 1), **kw)


@pytest.mark.parametrize("knobs", [dict(chunk_y=8), dict(cols_per_cta=8), dict(cta_threads_y=256)])
def test_a_given_column_geometry_keeps_the_tree_in_fp64(knobs):
    from paper_2006_10142_gb300 import _lib
    h = _handle(300, 1100, 5.0, fp64="always")
    assert h.tuning()["solver"] == 2  # all automatic: cyclic reduction
    h.set_tuning(**knobs)
    assert h.tuning()["solver"] == 1
    h.close()
    # 64 chunks of a column per 32-lane top system: refused, not taken by the other solver
    h = _handle(64, 8192, 5.0, fp64="always")
    with pytest.raises(_lib.AdiError) as ei:
        h.set_tuning(cols_per_cta=4, chunk_y=4, cta_threads_y=512)
    assert ei.value.code == _lib.ADI_EUNSUPPORTED
    h.close()


def test_adjoint_refuses_more_pieces_of_a_column_than_its_top_system_holds():
    """Cyclic reduction takes a column in 64 pieces, the reverse step's tree
    holds 32."""
    import torch
    from paper_2006_10142_gb300 import _lib
    h = _handle(64, 8192, 0.5)
    h.set_tuning(solver=2, cols_per_cta=4, chunk_y=4, cta_threads_y=512)
    h.set_checkpointing(2)
    tr = h.run(2, rec=[[3, 3]])
    with pytest.raises(_lib.AdiError) as ei:
        h.adjoint(tr)
    assert ei.value.code == _lib.ADI_EUNSUPPORTED
    h.set_tuning(solver=2)
    h.run(2, rec=[[3, 3]])
    gm, _ = h.adjoint(tr)
    h.sync_status()
    assert torch.equal(gm, torch.zeros_like(gm))  # a field at rest
    h.close()


def test_use_graph_reports_what_runs_do():
    import torch
    from paper_2006_10142_gb300 import _lib, api
    h = _handle(300, 200, 0.5)
    for value, reported in ((0, -1), (1, 1), (-1, -1)):
        h.set_tuning(use_graph=value)
        assert h.tuning()["use_graph"] == reported
        assert h.plan()["form"] == "small_patches"  # no knob of the sweeps
    h.close()
    m = torch.ones(40, 40, device="cuda:0")
    B = api.AdiWaveBatch([m, m], [m, m], 0.01)
    t = _lib.Tuning()
    _lib.check(B._lib.adi_wave_get_tuning(B._h, t), B._h)
    assert t.use_graph == 1
    B.close()


@pytest.mark.parametrize("tuning", [dict(solver=1), dict()])
def test_captured_steps_follow_resets_receivers_and_checkpoints(tuning):
    """Step pairs replayed from graphs against chained launches, to the bit:
    a second run, other receivers, a medium that changes nothing in the plan,
    one that takes the systems to FP64 and back, and runs with checkpoints
    (whose steps are the sweeps)."""
    import torch
    from helpers import f32
    from paper_2006_10142_gb300 import api
    from test_gpu_tile import _problem
    nx, ny, steps = 300, 260, 7
    m, phi, tau, wav = _problem(nx, ny, 0.5, 5)
    t = lambda a: torch.from_numpy(f32(a)).to("cuda:0")
    wav = t(wav)
    out = []
    for graph in (1, -1):
        h = api.AdiWave(t(m), t(phi), tau)
        h.set_tuning(use_graph=graph, **tuning)
        got = []

        def run(rec=None):
            tr = h.run(steps, src=(31, 39), wavelet=wav, rec=rec)
            got.extend(([] if tr is None else [tr]) + list(h.state()[:2]))

        run()
        run()
        run(rec=[[31, 39], [299, 0]])
        run(rec=[[5, 6], [7, 8], [31, 39]])
        for scale in (1.3, 100.0, 1.0):
            h.reset(t(phi), m=t(scale * m))
            run(rec=[[5, 6], [7, 8], [31, 39]])
            run()
        h.set_checkpointing(3)
        run(rec=[[5, 6]])
        run()
        h.set_checkpointing(0)
        run()
        h.sync_status()
        out.append(got)
        h.close()
    assert len(out[0]) == len(out[1]) and all(torch.equal(a, b) for a, b in zip(*out))


def test_sweeps_of_long_rows_are_replayed_and_may_be_captured():
    """Rows of the band form on a small grid: graphs by default, launches in a
    caller's graph; the same fields."""
    import torch
    h = _handle(5000, 40, 2.0)
    assert h.tuning()["x_stage"] == 5 and h.tuning()["use_graph"] == 1
    phi = torch.randn(40, 5000, device="cuda:0")
    h.reset(phi)
    h.run(5)
    want = h.state()
    h.reset(phi)
    graph = torch.cuda.CUDAGraph()
    torch.cuda.synchronize()
    with torch.cuda.graph(graph):
        h.run(5)
    graph.replay()
    got = h.state()
    h.sync_status()
    assert torch.equal(got[0], want[0]) and torch.equal(got[1], want[1])
    h.close()


@pytest.mark.parametrize("nx,ny,cfl,form", [(32, 32000, 1.0, "sweeps"), (32, 32000, 0.5, "patches"),
                                            (33, 20000, 1.0, "patches"), (48, 32000, 1.0, "patches")])
def test_narrow_grids_of_many_patches_keep_the_sweeps(nx, ny, cfl, form):
    h = _handle(nx, ny, cfl)
    assert h.plan()["form"] == form
    h.close()
