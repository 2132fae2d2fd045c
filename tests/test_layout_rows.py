"""CPU test of the tile lists of very long rows (host code of liblbm.so)."""
import pytest

from paper_1608_06915_gb300 import build as B


@pytest.fixture(scope="module")
def L():
    B.build()
    from paper_1608_06915_gb300 import lbm
    return lbm


@pytest.mark.parametrize("nx,tiles", [(4194304, True), (4194369, False)])
def test_rows_beyond_the_tile_index_go_node_by_node(L, nx, tiles):
    """A tile entry holds the x-tile in 16 bits, in units of 64 nodes for the
    64-node kernel: rows beyond 65536 such tiles (4194304 nodes) go node by node,
    16 bytes of lists per tile (for both step parities) instead of 56."""
    case = dict(n=(nx, 4, 4), periodic=(1, 1, 1), walls=(0,) * 6, inflow_axis=-1, u_in=(0, 0, 0), boxes=[],
                solid=None, nu0=0.01, accel0=(0, 0, 0), thermal=None)
    g = L.Grid(case, "fp16s", bind=False)
    rows, nxp = 16, -(-nx // 32) * 32
    lists = g.device_bytes - rows * nxp * (2 * 27 * 2 + 1)
    n = rows * -(-nx // 128)
    per_tile = 56 if tiles else 16
    assert abs(lists - per_tile * n) < n, (lists / n, per_tile)
