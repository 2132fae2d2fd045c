"""Rows of any length on the tile passes: periodic rows that do not end on a
16-byte boundary, rows shorter than a tile, a warp or the halo, and rows that
end just before or after a tile (GPU, against the oracle)."""
import numpy as np
import pytest

from gpu_util import pop_diff, twin

pytestmark = pytest.mark.gpu

LENGTHS = [4, 5, 9, 31, 33, 63, 65, 127, 129, 130, 133, 149]


@pytest.fixture(scope="module", autouse=True)
def _lib():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1608_06915_gb300 import build as B
    B.build()


def box(nx, walls=(0,) * 6, thermal=None):
    return dict(name="ragged", n=(nx, 5, 6), periodic=(1, 1, 0 if walls[4] else 1), walls=walls, inflow_axis=-1,
                u_in=(0, 0, 0), boxes=[], solid=None, nu0=0.01, accel0=(0, 0, 0), mirror_lbgk=False, thermal=thermal)


def noisy(seed, thermal=False):
    def fields(x, y, z, p, info):
        shp = tuple(reversed(info["dim"]))
        r = np.random.default_rng(seed)
        out = [1.0 + 0.01 * r.uniform(-1, 1, shp), 0.03 * r.uniform(-1, 1, (3,) + shp)]
        return out + [1.0 / 3.0 + 0.005 * r.uniform(-1, 1, shp)] if thermal else out
    return fields


@pytest.mark.parametrize("nx", LENGTHS)
def test_odd_rows_match_the_oracle_fp64(nx):
    """Every step within 1e-12 of the oracle, for every tile variant."""
    for v in (0, 1, 2):
        g, o = twin(box(nx), "fp64", noisy(nx))
        g.set_variant(v)
        for _ in range(3):
            g.step(1)
            o.step(1)
            assert pop_diff(g, o) < 1e-12, (nx, v)


@pytest.mark.parametrize("storage", ["fp32", "fp16s", "bf16s"])
@pytest.mark.parametrize("nx", LENGTHS)
def test_odd_rows_variants_agree(nx, storage):
    """The five tile kernels (single nodes and node pairs, 128 and 64 node
    tiles) give the same bits; FP32 is within its per-step bound of the oracle
    (2e-6 per collision, three steps)."""
    import torch
    ref = None
    for v in range(5):
        g, o = twin(box(nx), storage, noisy(nx), oracle=v == 0 and storage == "fp32")
        g.set_variant(v)
        g.step(3)
        f = g.get_populations(0)
        if ref is None:
            ref = f
            if o is not None:
                o.step(3)
                assert pop_diff(g, o) < 6e-6
        assert torch.equal(f, ref), (nx, storage, v)


@pytest.mark.parametrize("pr", [0.7, 2.0])
@pytest.mark.parametrize("nx", LENGTHS)
def test_odd_rows_thermal(nx, pr):
    """The two-population model between plates: FP64 within 1e-12 of the
    oracle every step, FP32 within 6e-6 after three (f and g)."""
    th = dict(pr=pr, t0=1 / 3, glambda=1e-3, t_ref=1 / 3, dT=0.01,
              wall_T=(0, 0, 0, 0, 1 / 3 + 0.005, 1 / 3 - 0.005))
    case = box(nx, walls=(0, 0, 0, 0, 1, 1), thermal=th)
    for storage, tol in (("fp64", 1e-12), ("fp32", 6e-6)):
        for v in (0, 1):
            g, o = twin(case, storage, noisy(nx, True))
            g.set_variant(v)
            for _ in range(3):
                g.step(1)
                o.step(1)
                assert pop_diff(g, o) < tol and pop_diff(g, o, 1) < tol, (nx, pr, storage, v)
