"""The lattice Boltzmann step: overlapping launches over many shapes and sizes,
and the collision at and away from tau = 1."""
import numpy as np
import pytest

import oracle as O
from paper_2110_13055_gb300 import cdi, inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="session", autouse=True)
def built():
    import __graft_entry__ as g
    g.build()


def solve(m, prec, shape, **kw):
    with cdi.Domain(m, precision=prec) as d:
        cdi.set_launch_shapes(d.handle, shape, -1)
        d.solve_flow(tol=0.0, check_every=20, max_steps=40, U_target=0.0, force=1e-6, **kw)
        return d.u_lattice()


@pytest.mark.parametrize("prec", [cdi.FP64, cdi.FP32, cdi.FP32_SPLIT, cdi.BF16_POP])
@pytest.mark.parametrize("shape", [(40, 70), (523, 771), (65, 67, 71)], ids=str)
def test_shapes_and_sizes_same_bits(shape, prec):
    """From fewer sites than one launch's first blocks to many waves; the
    prefetching odd step against one thread a site."""
    m = inputs.grain_pack(shape, 0.7, 2.0, 4.0, seed=3)[0]
    for tau in (1.0, 0.8):
        assert np.array_equal(solve(m, prec, 5, tau=tau), solve(m, prec, 1, tau=tau))


@pytest.mark.parametrize("prec,tol", [(cdi.FP64, 1e-12), (cdi.FP32, 2e-5)])
@pytest.mark.parametrize("tau", [1.0, 0.8])
@pytest.mark.parametrize("shape", [(40, 70), (11, 13, 19)], ids=str)
def test_collision_against_oracle(shape, tau, prec, tol):
    """400 steps of one rounding each (6e-8 in FP32) that the conserved moments
    keep: below 400 roundings."""
    m = inputs.grain_pack(shape, 0.6, 2.0, 4.0, seed=5)[0]
    ref, *_ = O.lbm(m, tau=tau, force=1e-6, tol=0.0, check_every=100, max_steps=400)
    with cdi.Domain(m, precision=prec) as d:
        d.solve_flow(tau=tau, force=1e-6, tol=0.0, check_every=100, max_steps=400, U_target=0.0)
        u = d.u_lattice()
    assert np.linalg.norm(u - ref) < tol * np.linalg.norm(ref)


def test_fp64_collision_conserves_mass_at_every_relaxation_time():
    """Chambers joined by single cells, 2,000 steps: where the collision makes
    or loses mass on average the chambers fill.  Against the same run in 80-bit
    arithmetic unbiased FP64 roundings give 1.8e-15 here, and weights that do
    not add up to 1 give 1.7e-14; the oracle's own roundings come on top."""
    m = np.zeros((40, 64), np.uint8)
    for k, x in enumerate(range(15, 64, 16)):
        m[:, x] = 1
        m[10 if k % 2 == 0 else 30, x] = 0
    ref, *_ = O.lbm(m, tau=0.8, force=1e-6, tol=0.0, check_every=100, max_steps=2000)
    with cdi.Domain(m, precision=cdi.FP64) as d:
        d.solve_flow(tau=0.8, force=1e-6, tol=0.0, check_every=100, max_steps=2000, U_target=0.0)
        u = d.u_lattice()
    assert np.linalg.norm(u - ref) < 6e-15 * np.linalg.norm(ref)
