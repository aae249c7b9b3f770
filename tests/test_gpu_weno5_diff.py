"""The WENO5 SharpClaw stage on first differences (sharpclaw.cuh) against the
CPU oracle: every 2D system in FP64 and FP32 (field pairs in packed FP32, odd
counts with a last single one), states around the sonic points (the FP64
pre-test before the entropy fix), and divisors outside the range of the fast
reciprocals."""
import numpy as np
import pytest

from paper_1111_6583_gb300 import workloads as wl
from tests.gpu_util import (FP32_SMOOTH_TOL, FP64_TOL, gpu_fixed_steps, oracle_fixed_steps,
                            rel_maxnorm)

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import __graft_entry__
    __graft_entry__.build()


@pytest.mark.parametrize("rp,char", [("advection", 1), ("acoustics", 1), ("sw_roe", 1),
                                     ("sw_roe", 0), ("euler_roe", 1), ("euler_roe", 0),
                                     ("euler_hlle", 1), ("euler_tracer", 1),
                                     ("elasticity_fwave", 0)])
@pytest.mark.parametrize("n2", [(33, 17), (48, 32)])
def test_systems(orc, rp, char, n2):
    kw = {} if rp == "elasticity_fwave" else dict(scheme="sharpclaw", char_decomp=char)
    spec = wl.random_smooth_2d(rp, *n2, **kw)
    dt = 0.1 / max(n2)
    qo, co = oracle_fixed_steps(orc, spec, dt, 2)
    qg, cg = gpu_fixed_steps(spec, "fp64", dt, 2)
    assert rel_maxnorm(qg, qo) <= FP64_TOL
    assert np.allclose(cg, co, rtol=1e-12, atol=0)
    q32, _ = gpu_fixed_steps(spec, "fp32", dt, 2)
    assert rel_maxnorm(q32, qo) <= FP32_SMOOTH_TOL


@pytest.mark.parametrize("scheme", ["sharpclaw", "classic"])
@pytest.mark.parametrize("rp", ["euler_roe", "euler_tracer"])
@pytest.mark.parametrize("sign", [1.0, -1.0])
def test_sonic_states(orc, scheme, rp, sign):
    spec = wl.random_smooth_2d(rp, 41, 29, scheme=scheme, char_decomp=1)
    q = spec["q0"].copy()
    rng = np.random.Generator(np.random.PCG64(7))
    # velocities spread over the sonic speed (about 1.18) with jumps
    u = sign * rng.uniform(0.9, 1.5, q.shape[1:])
    v = sign * rng.uniform(0.9, 1.5, q.shape[1:])
    p = rng.uniform(0.7, 1.3, q.shape[1:])
    q[1], q[2] = q[0] * u, q[0] * v
    q[3] = p / 0.4 + 0.5 * q[0] * (u * u + v * v)
    spec["q0"] = np.ascontiguousarray(q)
    qo, _ = oracle_fixed_steps(orc, spec, 0.05 / 41, 1)
    qg, _ = gpu_fixed_steps(spec, "fp64", 0.05 / 41, 1)
    assert rel_maxnorm(qg, qo) <= FP64_TOL


@pytest.mark.parametrize("power", [0, 60, 100])
def test_divisor_range(orc, power):
    """The Euler equations scale with the state; at 2^100 the WENO divisors
    leave the fast reciprocals' range (2^-767 .. 2^769)."""
    spec = wl.random_smooth_2d("euler_roe", 24, 16, scheme="sharpclaw", char_decomp=0)
    spec["q0"] = spec["q0"] * 2.0 ** power
    qo, _ = oracle_fixed_steps(orc, spec, 0.1 / 24, 1)
    qg, _ = gpu_fixed_steps(spec, "fp64", 0.1 / 24, 1)
    assert np.isfinite(qo).all()
    assert rel_maxnorm(qg, qo) <= FP64_TOL
