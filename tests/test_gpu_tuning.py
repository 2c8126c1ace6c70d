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
