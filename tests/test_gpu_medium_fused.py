"""The fused 2D step of acoustics in a varying medium (medium2d.cuh) against
the CPU oracle at the edges of its strips (60 and 124 columns, odd rows), with
and without a capacity, every limiter, order, transverse mode and
boundary, dimensionally split; every tile shape gives the same bits."""
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


def _spec(nx, ny, capacity, **kw):
    spec = wl.random_smooth_2d("acoustics_vc", nx, ny, num_aux=3 if capacity else 2, **kw)
    if capacity:
        spec["capa_index"] = 2
    else:
        spec["aux"] = np.ascontiguousarray(spec["aux"][:2])
    return spec


def _check(orc, spec, dt, n=3):
    qo, co = oracle_fixed_steps(orc, spec, dt, n)
    qg, cg = gpu_fixed_steps(spec, "fp64", dt, n)
    assert rel_maxnorm(qg, qo) <= FP64_TOL
    assert np.allclose(cg, co, rtol=1e-13, atol=0)
    q32, _ = gpu_fixed_steps(spec, "fp32", dt, n)
    assert rel_maxnorm(q32, qo) <= FP32_SMOOTH_TOL


@pytest.mark.parametrize("capacity", [False, True])
@pytest.mark.parametrize("n2", [(4, 4), (60, 31), (61, 33), (124, 9), (125, 8), (249, 5)])
def test_strip_edges(orc, capacity, n2):
    spec = _spec(*n2, capacity)
    spec["bc_lower"], spec["bc_upper"] = ["extrap", "wall"], ["wall", "extrap"]
    _check(orc, spec, 0.2 / max(n2))


@pytest.mark.parametrize("lim", ["none", "minmod", "superbee", "vanleer", "mc"])
@pytest.mark.parametrize("order,transverse", [(2, 2), (2, 1), (2, 0), (1, 2)])
def test_limiters_and_modes(orc, lim, order, transverse):
    for capacity in (False, True):
        _check(orc, _spec(70, 23, capacity, lim=lim, order=order, transverse=transverse), 0.2 / 70)


@pytest.mark.parametrize("split", [0, 1])
def test_inflow_boundaries(orc, split):
    spec = _spec(65, 37, True)
    spec["bc_lower"], spec["bc_upper"] = ["inflow", "extrap"], ["extrap", "inflow"]
    spec["inflow"] = [0.3, 0.1, -0.2]
    if split:
        spec["dim_split"] = 1
    _check(orc, spec, 0.2 / 65)


@pytest.mark.parametrize("prec", ["fp32", "fp64"])
@pytest.mark.parametrize("capacity", [False, True])
def test_shapes_bitwise(prec, capacity):
    spec = _spec(131, 77, capacity)
    ref, info = gpu_evolve(spec, prec, 0.05, tune=(64, 32))
    for shape in ((64, 8), (64, 1), (128, 8), (128, 41)):
        q, i2 = gpu_evolve(spec, prec, 0.05, tune=shape)
        assert i2["steps"] == info["steps"]
        assert np.array_equal(q, ref), shape
