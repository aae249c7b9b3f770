"""The 2D classic step of the Roe systems in strength form (roe2d.cuh) against
the CPU oracle: strips of 28 columns per warp (FP64) and 60 (FP32) and their
edges, odd rows, every limiter, order and transverse mode, boundaries,
dimensional splitting, states that cross the sonic points in both directions
(with and without the entropy fix), and the same bits for every tile shape."""
import numpy as np
import pytest

from paper_1111_6583_gb300 import workloads as wl
from tests.gpu_util import (FP32_SMOOTH_TOL, FP64_TOL, gpu_evolve, gpu_fixed_steps,
                            oracle_fixed_steps, rel_maxnorm)

pytestmark = pytest.mark.gpu
SYSTEMS = ["sw_roe"]


@pytest.fixture(scope="module", autouse=True)
def _built():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import __graft_entry__
    __graft_entry__.build()


def _check(orc, spec, dt, n=3, fp32=True):
    qo, co = oracle_fixed_steps(orc, spec, dt, n)
    qg, cg = gpu_fixed_steps(spec, "fp64", dt, n)
    assert rel_maxnorm(qg, qo) <= FP64_TOL
    assert np.allclose(cg, co, rtol=1e-12, atol=0)
    if fp32:
        q32, _ = gpu_fixed_steps(spec, "fp32", dt, n)
        assert rel_maxnorm(q32, qo) <= FP32_SMOOTH_TOL


@pytest.mark.parametrize("rp", SYSTEMS)
@pytest.mark.parametrize("n2", [(4, 4), (28, 11), (29, 10), (56, 9), (60, 31), (61, 33), (120, 9),
                                (121, 8), (249, 5)])
def test_strip_edges(orc, rp, n2):
    spec = wl.random_smooth_2d(rp, *n2)
    spec["bc_lower"], spec["bc_upper"] = ["extrap", "wall"], ["wall", "extrap"]
    _check(orc, spec, 0.1 / max(n2))


@pytest.mark.parametrize("rp", SYSTEMS)
@pytest.mark.parametrize("lim", ["none", "minmod", "superbee", "vanleer", "mc"])
@pytest.mark.parametrize("order,transverse", [(2, 2), (2, 1), (2, 0), (1, 2)])
def test_limiters_and_modes(orc, rp, lim, order, transverse):
    _check(orc, wl.random_smooth_2d(rp, 70, 23, lim=lim, order=order, transverse=transverse),
           0.1 / 70)


def _sonic(rp, nx, ny, seed, swap, **kw):
    """Jumps between states on both sides of the sonic speed, the flow along x
    (y when swap) with both signs."""
    rng = np.random.Generator(np.random.PCG64(seed))
    spec = wl.random_smooth_2d(rp, nx, ny, **kw)
    q = spec["q0"].copy()
    h = rng.uniform(0.8, 1.2, (ny, nx))
    u = rng.uniform(0.6, 1.6, (ny, nx)) * np.where(rng.random((ny, nx)) < 0.5, 1.0, -1.0)
    v = rng.uniform(-1.4, 1.4, (ny, nx))
    if swap:
        u, v = v, u
    q[0], q[1], q[2] = h, h * u, h * v
    if rp != "sw_roe":
        q[3] = rng.uniform(0.7, 1.3, (ny, nx)) / 0.4 + 0.5 * h * (u * u + v * v)
    spec["q0"] = np.ascontiguousarray(q)
    return spec


@pytest.mark.parametrize("rp", SYSTEMS)
@pytest.mark.parametrize("swap", [False, True])
@pytest.mark.parametrize("kw", [{}, {"entropy_fix": 0}, {"transverse": 1}, {"dim_split": 1},
                                {"lim": "superbee"}])
def test_sonic_states(orc, rp, swap, kw):
    for seed in (1, 2):
        _check(orc, _sonic(rp, 61, 37, seed, swap, **kw), 0.05 / 61, n=1, fp32=False)


@pytest.mark.parametrize("rp", SYSTEMS)
@pytest.mark.parametrize("split", [0, 1])
def test_inflow_boundaries(orc, rp, split):
    spec = wl.random_smooth_2d(rp, 65, 37)
    spec["bc_lower"], spec["bc_upper"] = ["inflow", "extrap"], ["extrap", "inflow"]
    spec["inflow"] = list(spec["q0"][:, 3, 3])
    if split:
        spec["dim_split"] = 1
    _check(orc, spec, 0.1 / 65)


@pytest.mark.parametrize("rp", SYSTEMS)
@pytest.mark.parametrize("prec", ["fp32", "fp64"])
@pytest.mark.parametrize("kw", [{}, {"lim": "minmod"}, {"dim_split": 1}])
def test_shapes_bitwise(rp, prec, kw):
    spec = wl.random_smooth_2d(rp, 131, 77, **kw)
    ref, info = gpu_evolve(spec, prec, 0.05, tune=(64, 32))
    for shape in ((64, 8), (64, 1), (128, 8), (128, 41)):
        q, i2 = gpu_evolve(spec, prec, 0.05, tune=shape)
        assert i2["steps"] == info["steps"]
        assert np.array_equal(q, ref), shape


@pytest.mark.parametrize("prec", ["fp32", "fp64"])
@pytest.mark.parametrize("value", [0.0, -1.0, np.nan, np.inf])
def test_non_physical_depth_is_reported(prec, value):
    spec = wl.random_smooth_2d("sw_roe", 40, 40)
    spec["q0"][0, 7, 9] = value
    spec["dt_initial"] = 1e-4
    _, info = gpu_evolve(spec, prec, 1.0, max_steps=4)
    assert info["status"] == 6 and info["steps"] == 0
