"""crkdg_get_launch reports the rows a segment has: those that were set, or more
where the room of the seam scratch (256 MiB here) leaves fewer segments."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,ny,rows", [(64, 40, 1), (64, 40, 3), (64, 40, 40), (1024, 400, 8), (1024, 400, 1), (2048, 801, 1)])
def test_rows_in_effect(nx, ny, rows):
    from paper_2307_06471_gb300 import binding as B
    from paper_2307_06471_gb300 import tableaux as T
    mesh = B.make_mesh(2, nx, ny, (0.0, 1.0, 0.0, 1.0), [B.BC_PERIODIC] * 4)
    s = B.Solver(mesh, 2, B.BASIS_P, T.SSPRK3, B.EULER, B.F64)
    s.set_launch(rows, 1)
    # per segment and column: 3 stages and a flux of 3 points x 4 variables, twice, and 24 modes
    seg = nx * (2 * (3 * 12 + 12) + 24) * 8
    most = max(ny * nx * 24 * 8 // 8, 256 << 20) // seg
    nseg = min(-(-ny // rows), most)
    assert s.get_launch() == (max(rows, -(-ny // nseg)), 1)
    got = s.get_launch()[0]
    s.set_launch(got, 1)
    assert s.get_launch()[0] == got
    s.close()
