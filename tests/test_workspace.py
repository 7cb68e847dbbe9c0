"""Bytes of a context's workspace (host only)."""
import pytest

@pytest.fixture(scope="module")
def lbm():
    import __graft_entry__

    __graft_entry__.build()
    from paper_2403_11167_gb300 import lbm as L

    return L


@pytest.mark.parametrize("precision,nx,ny", [(1, 1, 1000000), (1, 200, 100), (1, 4096, 4096), (0, 1, 1000000),
                                             (0, 1022, 770), (0, 4, 5000), (0, 200, 3)])
def test_no_strip_slots_where_no_strip_can_run(lbm, precision, nx, ny):
    """FP64, widths that are not a multiple of 4 and lattices below 8 x 4 run no strip kernel: beside the two
    buffers and the four fields the workspace holds the walls' scratch and less than 32 KB."""
    esz = 8 if precision else 4
    pitch = -(-nx * ny // 64) * 64
    planes = 9 if precision else 10
    base = 2 * planes * pitch * esz + 4 * nx * ny * esz + 14 * nx * esz
    got = lbm.lbm_workspace_bytes(precision, nx, ny)
    assert base <= got < base + 32768
