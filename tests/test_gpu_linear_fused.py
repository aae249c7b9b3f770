"""The fused steps of the constant-coefficient linear systems (linear.cuh) at
the edges of their tiles, against the CPU oracle: 2D strips of 60 and 124
columns (aligned and odd row lengths, narrow last strips) with the same bits
for every tile shape, 3D blocks of 28 x 12 columns and z segments, every
limiter, first order, both transverse modes, and a non-finite state."""
import numpy as np
import pytest

from paper_1111_6583_gb300 import workloads as wl
from tests.gpu_util import (FP32_SMOOTH_TOL, FP64_TOL, gpu_evolve, gpu_fixed_steps,
                            oracle_fixed_steps, rel_maxnorm)

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import __graft_entry__
    __graft_entry__.build()


def _check(orc, spec, dt, n=3):
    qo, co = oracle_fixed_steps(orc, spec, dt, n)
    qg, cg = gpu_fixed_steps(spec, "fp64", dt, n)
    assert rel_maxnorm(qg, qo) <= FP64_TOL
    assert np.allclose(cg, co, rtol=1e-13, atol=0)
    q32, _ = gpu_fixed_steps(spec, "fp32", dt, n)
    assert rel_maxnorm(q32, qo) <= FP32_SMOOTH_TOL


@pytest.mark.parametrize("rp", ["acoustics", "advection"])
@pytest.mark.parametrize("n2", [(4, 4), (60, 31), (61, 33), (124, 9), (125, 8), (249, 5)])
def test_2d_strip_edges(orc, rp, n2):
    spec = wl.random_smooth_2d(rp, *n2)
    spec["bc_lower"], spec["bc_upper"] = ["extrap", "wall"], ["wall", "extrap"]
    _check(orc, spec, 0.15 / max(n2))


@pytest.mark.parametrize("lim", ["none", "minmod", "superbee", "vanleer", "mc"])
@pytest.mark.parametrize("order,transverse", [(2, 2), (2, 1), (2, 0), (1, 2)])
def test_2d_limiters_and_modes(orc, lim, order, transverse):
    for rp in ("acoustics", "advection"):
        spec = wl.random_smooth_2d(rp, 70, 23, lim=lim, order=order, transverse=transverse)
        if rp == "advection":
            spec["params"] = [-0.7, 0.4]
        _check(orc, spec, 0.15 / 70)


@pytest.mark.parametrize("prec", ["fp32", "fp64"])
@pytest.mark.parametrize("rp,split", [("acoustics", 0), ("acoustics", 1), ("advection", 0)])
def test_2d_shapes_bitwise(prec, rp, split):
    spec = wl.random_smooth_2d(rp, 131, 77)
    if split:
        spec["dim_split"] = 1
    ref, info = gpu_evolve(spec, prec, 0.05, tune=(128, 32))
    for shape in ((64, 8), (64, 41), (128, 8), (128, 128), (64, 1)):
        q, i2 = gpu_evolve(spec, prec, 0.05, tune=shape)
        assert i2["steps"] == info["steps"]
        assert np.array_equal(q, ref), shape


@pytest.mark.parametrize("rp", ["acoustics", "advection"])
@pytest.mark.parametrize("n3", [(28, 12, 5), (29, 13, 4), (27, 25, 65), (57, 11, 130), (4, 4, 4)])
def test_3d_block_edges(orc, rp, n3):
    spec = wl.random_3d(rp, *n3, bc="extrap")
    if rp == "acoustics":
        spec["bc_lower"], spec["bc_upper"] = ["wall", "extrap", "wall"], ["extrap", "wall", "wall"]
    _check(orc, spec, 0.15 / max(n3))


@pytest.mark.parametrize("lim", ["none", "minmod", "superbee", "vanleer", "mc"])
@pytest.mark.parametrize("order,transverse", [(2, 2), (2, 1), (1, 2)])
def test_3d_limiters_and_modes(orc, lim, order, transverse):
    for rp in ("acoustics", "advection"):
        spec = wl.random_3d(rp, 31, 14, 9, lim=lim, order=order, transverse=transverse)
        _check(orc, spec, 0.15 / 31)


@pytest.mark.parametrize("prec", ["fp32", "fp64"])
@pytest.mark.parametrize("value", [np.nan, np.inf])
def test_non_finite_state_is_reported(prec, value):
    for spec in (wl.random_smooth_2d("acoustics", 40, 40), wl.random_3d("acoustics", 12, 12, 12)):
        spec["q0"][(0,) + (5,) * spec["ndim"]] = value
        spec["dt_initial"] = 1e-3
        _, info = gpu_evolve(spec, prec, 1.0, max_steps=4)
        assert info["status"] == 6 and info["steps"] == 0
