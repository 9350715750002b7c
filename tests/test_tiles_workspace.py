"""The workspace of the persistent path's tile engine goes to the grids that it can hold, and to no
others: beyond its cone limit (10,240) a handle never gets it, which gives the size without."""
import pytest

from paper_1405_3331_gb300 import build as cue_build


@pytest.fixture(scope="module")
def cue():
    cue_build.build()
    from paper_1405_3331_gb300 import cue as binding
    return binding


def _extra(cue, nx, ny):
    p = cue.cue_params(2, nx, ny, 1, 1.0, 1.0, 0.01, 0.2, 0)
    return cue.cue_workspace_bytes(p, 8, 10240) - cue.cue_workspace_bytes(p, 8, 10241)


@pytest.mark.parametrize("nx,ny", [(2048, 2048), (2000, 2000), (1800, 1800), (128, 32768), (127, 512), (4096, 900)])
def test_grids_the_engine_cannot_hold_do_without(cue, nx, ny):
    assert abs(_extra(cue, nx, ny)) < 4 << 20            # (the bins of one cone more)


@pytest.mark.parametrize("nx,ny", [(128, 128), (129, 1000), (1024, 1024), (1701, 1701), (9600, 16), (2048, 1024)])
def test_grids_it_can_hold_have_its_packets(cue, nx, ny):
    assert _extra(cue, nx, ny) > 16 * nx * ny
