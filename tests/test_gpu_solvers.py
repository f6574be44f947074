"""The cooperative linear solvers at the edges of their launch shapes: fewer
cells than a warp, one warp a block, several cells a thread."""
import numpy as np
import pytest

import oracle as O
from paper_2110_13055_gb300 import cdi, inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="session", autouse=True)
def built():
    import __graft_entry__ as g
    g.build()


def rel(a, b):
    return float(np.linalg.norm(np.asarray(a) - np.asarray(b)) / np.linalg.norm(b))


def image(shape):
    if shape == (4, 5):
        m = np.zeros(shape, np.uint8)
        m[1, 2] = 1
        return m
    r = 2.0 if len(shape) == 3 else 3.0
    return inputs.grain_pack(shape, 0.6, r, 2 * r, seed=7)[0]


SHAPES = [(4, 5), (61, 83), (18, 21, 25), (64, 61, 70)]


@pytest.mark.parametrize("walls", [False, True])
@pytest.mark.parametrize("mode,lam", [("debye", 1.5e-7), ("debye", 1e-6), ("laplace", 0.0)])
@pytest.mark.parametrize("shape", SHAPES, ids=str)
def test_potential_solver_shapes(shape, mode, lam, walls):
    """Relative residuals of 1e-13 leave an error of the condition number
    (below 1e3 in pores of some ten cells) times that."""
    m = image(shape)
    ref, _, _ = O.psi(m, -0.7, dx=1e-7, c_bulk=10.0, mode=mode, lambda_D=lam or None,
                      tol=1e-14, lateral_walls=walls)
    with cdi.Domain(m, lateral_walls=walls) as d:
        d.solve_flow(tol=0.0, max_steps=0, U_target=0.0)
        it, res = d.set_potential(0.7, c_bulk=10.0, lambda_D=lam, mode=mode, tol=1e-13)
        ps = d.psi()
    assert it > 0 and res < 1e-13
    assert rel(ps, ref) < 1e-10
    assert np.all(ps[m == 1] == 0.0)


def test_potential_beyond_refinement():
    """A tolerance below what a residual in FP64 can show is still reached by
    the FP64 iteration (its residual is a recurrence); too few iterations are
    still an error; no surface potential is a zero field."""
    m = image((61, 83))
    with cdi.Domain(m) as d:
        d.solve_flow(tol=0.0, max_steps=0, U_target=0.0)
        it, res = d.set_potential(0.7, lambda_D=1e-6, tol=1e-18)
        assert it > 0 and res < 1e-18
        a = d.psi()
        d.set_potential(0.7, lambda_D=1e-6, tol=1e-13)
        assert rel(d.psi(), a) < 1e-9      # the condition number, 1.2e3, times tol
        with pytest.raises(cdi.CDIError) as e:
            d.set_potential(0.7, lambda_D=1e-6, tol=1e-13, max_iter=2)
        assert e.value.status == 4
        it, res = d.set_potential(0.0, lambda_D=1e-6, tol=1e-13)
        assert it == 0 and res == 0.0 and not d.psi().any()


@pytest.mark.parametrize("shape,Z,D", [
    ((4, 5), (1,), (1.33e-9,)),
    ((61, 83), (1, -1, 2), (1.33e-9, 2.03e-9, 0.8e-9)),
    ((18, 21, 25), (1, -1, 2, -2), (1.33e-9, 2.03e-9, 0.8e-9, 1.1e-9)),
    ((540, 560), (1, -1), (1.33e-9, 2.03e-9))], ids=str)
def test_implicit_solver_shapes(shape, Z, D):
    """FP64 storage and relative residuals of 1e-13: 1e-9 leaves four orders
    for the conditioning, as in the implicit tests."""
    m = image(shape)
    r = O.run_case(m, flow_tol=0.0, max_flow_steps=200, U_target=1e-4, applied_V=0.3,
                   lambda_D=1.5e-7, n_np_steps=0)
    dt, n = 20 * r["dt"], 3
    Co, Go, Io, Oo = O.np_implicit_run(m, r["u"], r["psi"], Z, D, c0=10.0, dt=dt, n_steps=n)
    with cdi.Domain(m, precision=cdi.FP64) as d:
        d.solve_flow(tol=0.0, max_steps=200, U_target=1e-4)
        d.set_potential(0.3, c_bulk=10.0, lambda_D=1.5e-7, tol=1e-14)
        d.init_transport(Z, D, c0=10.0, Ka=1e-6, dt=dt)
        d.set_implicit(1e-13, 2000)
        d.step(n)
        C = d.C()
        M, G, I, Ou = d.mass_balance()
    assert rel(C, Co) < 1e-9
    np.testing.assert_allclose(G, Go, rtol=1e-9)
    np.testing.assert_allclose(I, Io, rtol=1e-9, atol=1e-9 * np.abs(Io).max())
    np.testing.assert_allclose(Ou, Oo, rtol=1e-9, atol=1e-9 * np.abs(Io).max())


@pytest.mark.parametrize("shift", [-90, -45, 80])
@pytest.mark.parametrize("mode,lam", [("laplace", 0.0), ("debye", 1e-6)])
@pytest.mark.parametrize("shape", [(61, 83), (18, 21, 25)], ids=str)
def test_potential_of_any_size(shape, mode, lam, shift):
    """Eq. 4 is linear: a surface potential 2^shift times as large has the
    same relative field and residual, also where its square leaves FP32's
    range.  Both residuals are below 1e-13, at condition numbers below 1.2e3."""
    m = image(shape)
    with cdi.Domain(m) as d:
        d.solve_flow(tol=0.0, max_steps=0, U_target=0.0)
        it, _ = d.set_potential(0.75, lambda_D=lam, mode=mode, tol=1e-13)
        a = d.psi()
        it2, res = d.set_potential(0.75 * 2.0 ** shift, lambda_D=lam, mode=mode, tol=1e-13)
        b = d.psi() * 2.0 ** -shift
    assert it2 == it and 0.0 < res < 1e-13
    assert rel(b, a) < 2.4e-10


def test_iterations_counted():
    """The timing counts the iterations of every solve; the call returns those
    of the solve that gave the field."""
    m = image((61, 83))

    def counted(**kw):
        d.timing(reset=True)
        it = d.set_potential(0.7, lambda_D=1e-6, **kw)[0]
        return it, d.timing()["psi_iters"]

    with cdi.Domain(m) as d:
        d.solve_flow(tol=0.0, max_steps=0, U_target=0.0)
        it, n = counted(tol=1e-13)
        assert n == it
        it, n = counted(tol=1e-18)       # begun again by the FP64 iteration
        assert n > it > 0
        d.timing(reset=True)
        with pytest.raises(cdi.CDIError):
            d.set_potential(0.7, lambda_D=1e-6, tol=1e-13, max_iter=2)
        assert d.timing()["psi_iters"] == 4


@pytest.mark.parametrize("walls", [False, True])
def test_potential_lateral_differences_beyond_16_bits(walls):
    """Cells whose z neighbours lie more than 32,000 ranks apart (the refinement
    then reads their full ranks); at the bar of test_potential_solver_shapes."""
    m = np.zeros((3, 190, 256), np.uint8)
    m[1, 2:185, :] = 1
    ref, _, _ = O.psi(m, -0.7, dx=1e-7, c_bulk=10.0, mode="laplace", tol=1e-14,
                      lateral_walls=walls)
    with cdi.Domain(m, lateral_walls=walls) as d:
        d.solve_flow(tol=0.0, max_steps=0, U_target=0.0)
        d.set_potential(0.7, c_bulk=10.0, mode="laplace", tol=1e-13)
        ps = d.psi()
    assert rel(ps, ref) < 1e-10
