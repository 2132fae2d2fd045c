"""Which kernel a grid's stream-collide runs on, and that each route gives the
result of the others or of the oracle at the sizes where the rules change
(GPU).  The route is read from the per-launch timing: "stream_collide_tma" is
the tile pass, "stream_collide" the node-by-node kernels."""
import numpy as np
import pytest

from gpu_util import pop_diff, twin

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1608_06915_gb300 import build as B
    B.build()


def box(n, walls=(0,) * 6, accel0=(0, 0, 0), boxes=(), solid=None, thermal=None, **more):
    return dict(name="routes", n=n, periodic=tuple(int(not walls[2 * a]) for a in range(3)), walls=walls,
                inflow_axis=-1, u_in=(0, 0, 0), boxes=list(boxes), solid=solid, nu0=0.01, accel0=accel0,
                mirror_lbgk=False, thermal=thermal, **more)


def noisy(seed, thermal=False):
    def fields(x, y, z, p, info):
        shp = tuple(reversed(info["dim"]))
        r = np.random.default_rng(seed + p)
        out = [1.0 + 0.01 * r.uniform(-1, 1, shp), 0.03 * r.uniform(-1, 1, (3,) + shp)]
        return out + [1.0 / 3.0 + 0.005 * r.uniform(-1, 1, shp)] if thermal else out
    return fields


def timed_step(g):
    """One step under per-launch timing: {kind: (launches, nodes)}."""
    g.timing(True)
    g.step(1)
    out = {}
    for r in g.timing_report():
        n, m = out.get(r["kind"], (0, 0.0))
        out[r["kind"]] = (n + r["launches"], m + r["nodes"])
    g.timing(False)
    return out


@pytest.mark.parametrize("storage", ["fp32", "fp16s", "bf16s"])
@pytest.mark.parametrize("n,node_by_node", [
    ((24, 24, 24), True), ((25, 9, 7), True), ((119, 25, 24), True), ((200, 6, 5), True), ((128, 8, 9), True),
    ((20, 57, 32), True),   # 1824 tiles, the limit
    ((20, 25, 73), False),  # 1825
    ((129, 50, 25), None),  # 2500: 16-bit rows beyond 64 nodes go to 6080
    ((80, 76, 80), None), ((80, 11, 553), False)])  # 6080, 6083
def test_small_one_level_grids_run_node_by_node(n, node_by_node, storage):
    """Few tiles: node by node by default and after autotune, on the tile
    kernels once a variant is set, with the same bits (periodic, with walls and
    a force)."""
    import torch
    if node_by_node is None:
        node_by_node = storage != "fp32"
    for walls, acc in (((0,) * 6, (0, 0, 0)), ((0, 0, 1, 1, 0, 0), (1e-5, 0, 0)), ((0, 0, 0, 0, 1, 1), (0, 0, 2e-5))):
        if walls != (0,) * 6 and n[1] * n[2] > 2000:
            continue
        case = box(n, walls, acc)
        a, _ = twin(case, storage, noisy(3), oracle=False)
        b, _ = twin(case, storage, noisy(3), oracle=False)
        a.step(2)
        b.set_variant(1)
        b.step(2)
        ta, tb = timed_step(a), timed_step(b)
        assert ("stream_collide_tma" in ta) != node_by_node and "stream_collide_tma" in tb, (ta, tb)
        assert sum(m for _, m in ta.values()) == sum(m for _, m in tb.values()) == n[0] * n[1] * n[2]
        assert torch.equal(a.get_populations(0), b.get_populations(0))
    a.autotune(trials=1)
    assert ("stream_collide_tma" in timed_step(a)) != node_by_node


@pytest.mark.parametrize("storage", ["fp32", "fp64"])
@pytest.mark.parametrize("pr", [0.7, 2.0, None])
def test_float32_moments_are_the_float64_ones_rounded_once(pr, storage):
    """rho, u and T in float32 are the float64 outputs of the same state,
    rounded once (pr None: the isothermal model with a force)."""
    import torch
    if pr is None:
        case = box((37, 20, 31), (0, 0, 0, 0, 1, 1), (1e-3, 2e-3, -1e-3))
    else:
        case = box((37, 20, 31), (0, 0, 0, 0, 1, 1),
                   thermal=dict(pr=pr, t0=1 / 3, glambda=0.02, t_ref=1 / 3 + 1e-3, dT=0.01,
                                wall_T=(0, 0, 0, 0, 1 / 3 + 0.005, 1 / 3 - 0.005)))
    g, _ = twin(case, storage, noisy(5, pr is not None), oracle=False)
    g.step(3)
    wide = g.moments(0, dtype=torch.float64)
    narrow = g.moments(0, dtype=torch.float32)
    for a, b in list(zip(wide, narrow))[:3 if pr is not None else 2]:
        assert torch.equal(a.float(), b)


def plates(pr, n, **more):
    return box(n, (0, 0, 0, 0, 1, 1),
               thermal=dict(pr=pr, t0=1 / 3, glambda=1e-3, t_ref=1 / 3, dT=0.01,
                            wall_T=(0, 0, 0, 0, 1 / 3 + 0.005, 1 / 3 - 0.005)), **more)


@pytest.mark.parametrize("pr", [0.7, 2.0])
@pytest.mark.parametrize("nx", [45, 64, 131])
def test_thermal_tile_passes_refined_fp32_every_step(nx, pr):
    """Both FP32 thermal tile passes on a three-level cell against the oracle.
    A coarse step applies up to six collisions to a value (four fine steps,
    coalesce, explode), each within 2e-6 of f and 5e-6 of g in FP32."""
    boxes = [(lev, (0, 0, lo), (nx - 1, 8, hi)) for lev, lo, hi in
             ((1, 0, 8), (1, 25, 33), (2, 0, 4), (2, 29, 33))]
    case = plates(pr, (nx, 9, 34), boxes=boxes)
    g0, o = twin(case, "fp32", noisy(11, True))
    g1, _ = twin(case, "fp32", noisy(11, True), oracle=False)
    g1.set_variant(1)
    for s in range(1, 4):
        o.step(1)
        for g in (g0, g1):
            g.step(1)
            df, dg = pop_diff(g, o, 0), pop_diff(g, o, 1)
            assert df < 6 * 2e-6 * s and dg < 6 * 5e-6 * s, (s, df, dg)


@pytest.mark.parametrize("pr", [0.7, 2.0])
def test_thermal_inflow_fp64_every_step(pr):
    """FP64 thermal grids go node by node whole, beside an inlet and an outlet
    too; inlet nodes keep their populations.  The inlet's temperature is not an
    input of the model (the library takes T0, the oracle the field's), so both
    step from the library's initial state."""
    case = plates(pr, (64, 6, 8))
    case.update(periodic=(0, 1, 0), inflow_axis=0, u_in=(0.03, 0.0, 0.0))
    for v in (0, 1):
        g, o = twin(case, "fp64", noisy(13, True))
        for which in (0, 1):
            o.set_pop(0, g.get_populations(0, which).cpu().numpy(), which)
        g.set_variant(v)
        for s in range(3):
            g.step(1)
            o.step(1)
            df, dg = pop_diff(g, o, 0), pop_diff(g, o, 1)
            assert df < 1e-12 and dg < 1e-12, (s, df, dg)


def test_batches_of_tile_patches_fp64():
    """Ten level-1 boxes whose rows fill their tiles: more patches with tiles
    than one launch of the tile pass takes (8), so each instant takes two
    launches; populations against the oracle every step."""
    boxes = [(1, (4 + 41 * k, 8, 8), (35 + 41 * k, 16, 16)) for k in range(10)]
    case = box((412, 24, 24), boxes=boxes)
    for v in (0, 1, 2):
        g, o = twin(case, "fp64", noisy(17))
        g.set_variant(v)
        for _ in range(2):
            g.step(1)
            o.step(1)
            assert pop_diff(g, o) < 1e-12
        assert timed_step(g)["stream_collide_tma"][0] == 4  # two instants


@pytest.mark.parametrize("walls", [(0,) * 6, (0, 0, 0, 0, 1, 1)])
@pytest.mark.parametrize("nx", [29, 30, 32, 61, 62, 64, 93, 94, 126, 128, 158, 160, 189, 254, 256])
def test_rows_that_fill_their_lanes_run_on_the_fp64_tile_pass(nx, walls):
    """FP64 rows with at most a tenth of the lanes idle stay on the tiles: every
    step within 1e-12 of the oracle, for every tile kernel."""
    for v in (0, 1, 2):
        g, o = twin(box((nx, 5, 6), walls), "fp64", noisy(nx))
        g.set_variant(v)
        for _ in range(3):
            g.step(1)
            o.step(1)
            assert pop_diff(g, o) < 1e-12, (nx, v)
        t = timed_step(g)
        assert t["stream_collide_tma"] == (1, nx * 5 * 6), t


def test_fixup_nodes_at_a_curved_surface_fp64():
    """A ball with its analytic surface on rows that fill the FP64 tiles: the
    nodes beside it are fix-up nodes, few enough for the warp-per-node kernel;
    populations and drag against the oracle every step."""
    c, r = (30.3, 11.8, 12.1), 6.0
    z, y, x = np.meshgrid(np.arange(24), np.arange(24), np.arange(64), indexing="ij")
    mask = (((x - c[0]) ** 2 + (y - c[1]) ** 2 + (z - c[2]) ** 2) < r * r).astype(np.uint8)
    case = box((64, 24, 24), accel0=(1e-5, 0, 0), solid=dict(level=0, lo=(0, 0, 0), mask=mask),
               wall_shape=dict(kind="sphere", c=c, r=r, solid_inside=True))
    for v in (0, 1, 2):
        g, o = twin(case, "fp64", noisy(19))
        g.set_variant(v)
        for s in range(3):
            g.step(1)
            o.step(1)
            d = pop_diff(g, o)
            assert d < 1e-12, (s, d)
            Fg, Fo = np.array(g.drag()), o.drag()
            assert np.max(np.abs(Fg - Fo)) < 1e-12 * np.linalg.norm(Fo), (Fg, Fo)
        t = timed_step(g)
        assert t["stream_collide_tma"][1] > 0 and 0 < t["stream_collide"][1] < 2000, t


@pytest.mark.parametrize("storage,stored", [("fp32", "float32"), ("fp16s", "float16"), ("bf16s", "bfloat16")])
@pytest.mark.parametrize("nx", [4, 5, 6, 7, 8, 9, 10, 11, 12, 13, 14, 15, 31, 65, 130, 149])
def test_periodic_wrap_at_every_offset_against_the_oracle(nx, storage, stored):
    """One step of every tile kernel from the stored state, every place of the
    row's last node in its 16-byte box: within the FP32 collision's 2e-6 and the
    storage's rounding of the deviation from W_i (half a unit in the last
    place, and half the smallest FP16 step)."""
    import torch
    unit = torch.finfo(getattr(torch, stored)).eps / 2
    W = np.array([np.prod([2 / 3 if c == 1 else 1 / 6 for c in (i % 3, i // 3 % 3, i // 9)]) for i in range(27)])
    for v in range(5):
        g, o = twin(box((nx, 5, 6)), storage, noisy(nx))
        g.set_variant(v)
        o.set_pop(0, g.get_populations(0).cpu().numpy())
        g.step(1)
        o.step(1)
        fo = o.get_pop(0)
        dev = np.abs(fo - W[:, None, None, None])
        err = np.abs(g.get_populations(0).cpu().numpy() - fo)
        assert np.all(err <= 2e-6 + unit * (dev + 2e-6) + 2.0 ** -25), (v, np.max(err))
