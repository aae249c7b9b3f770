"""Several attempts of a small 1D grid in one cluster launch: the edges of the
warp units (60 cells in FP64, 240 and 120 in FP32) and of the sizes that take
this path, odd (unaligned) rows, every boundary and limiter, runs with rejected
attempts, a run that ends inside a launch, and a failing one, against the CPU
oracle; the systems with explicit rounding give the bits of single attempts."""
import numpy as np
import pytest

from paper_1111_6583_gb300 import workloads as wl
from tests.gpu_util import (FP32_SMOOTH_TOL, FP64_TOL, gpu_evolve, oracle_evolve, rel_maxnorm)

pytestmark = pytest.mark.gpu
SYSTEMS = ["advection", "acoustics", "sw_roe", "euler_roe", "euler_hlle", "euler_tracer",
           "elasticity_fwave"]


@pytest.fixture(scope="module", autouse=True)
def _built():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import __graft_entry__
    __graft_entry__.build()


@pytest.mark.parametrize("rp", SYSTEMS)
@pytest.mark.parametrize("n", [4, 59, 61, 240, 1001])
def test_sizes(orc, rp, n):
    spec = wl.random_1d(rp, n, jump=False)
    t_end = 0.3 / n * 20
    qo, io = oracle_evolve(orc, spec, t_end)
    qg, ig = gpu_evolve(spec, "fp64", t_end)
    assert ig["steps"] == io["steps"] and ig["t"] == t_end and ig["status"] == 0
    assert rel_maxnorm(qg, qo) <= FP64_TOL
    q32, _ = gpu_evolve(spec, "fp32", t_end)
    assert rel_maxnorm(q32, qo) <= FP32_SMOOTH_TOL


@pytest.mark.parametrize("bc", [("wall", "extrap"), ("extrap", "wall"), ("inflow", "extrap"),
                                ("periodic", "periodic")])
@pytest.mark.parametrize("rp", ["acoustics", "sw_roe", "elasticity_fwave"])
def test_boundaries(orc, rp, bc):
    spec = wl.random_1d(rp, 300, bc=bc)
    spec["inflow"] = list(spec["q0"][:, 0])
    qo, io = oracle_evolve(orc, spec, 0.05)
    qg, ig = gpu_evolve(spec, "fp64", 0.05)
    assert ig["steps"] == io["steps"]
    assert rel_maxnorm(qg, qo) <= FP64_TOL


@pytest.mark.parametrize("lim", ["none", "minmod", "superbee", "vanleer", "mc"])
@pytest.mark.parametrize("rp", ["acoustics", "elasticity_fwave", "euler_roe"])
def test_limiters(orc, rp, lim):
    spec = wl.random_1d(rp, 180, lim=lim)
    qo, io = oracle_evolve(orc, spec, 0.05)
    qg, ig = gpu_evolve(spec, "fp64", 0.05)
    assert ig["steps"] == io["steps"]
    assert rel_maxnorm(qg, qo) <= FP64_TOL


@pytest.mark.parametrize("prec", ["fp64", "fp32"])
@pytest.mark.parametrize("rp", ["advection", "acoustics", "elasticity_fwave"])
@pytest.mark.parametrize("n", [4, 500, 5759, 5760, 5761, 7681, 122881])
def test_bits_of_single_attempts(prec, rp, n):
    spec = wl.random_1d(rp, n)
    a, ia = gpu_evolve(spec, prec, 1e30, max_steps=37)
    b, ib = gpu_evolve(spec, prec, 1e30, max_steps=37, tune=(0, 2))
    assert ia["steps"] == ib["steps"] == 37 and ia["t"] == ib["t"] and ia["cfl"] == ib["cfl"]
    assert np.array_equal(a, b)


def test_rejected_attempts(orc):
    spec = wl.random_1d("sw_roe", 400, dt_initial=0.02)
    qo, io = oracle_evolve(orc, spec, 0.1)
    qg, ig = gpu_evolve(spec, "fp64", 0.1)
    assert io["rejects"] >= 1 and ig["rejects"] == io["rejects"] and ig["steps"] == io["steps"]
    assert rel_maxnorm(qg, qo) <= FP64_TOL


def test_failing_run_stops():
    spec = wl.random_1d("sw_roe", 400)
    spec["q0"][0, 123] = -1.0
    spec["dt_initial"] = 1e-4
    q, info = gpu_evolve(spec, "fp64", 1.0)
    assert info["status"] == 6 and info["steps"] == 0
    assert np.array_equal(q, spec["q0"])
