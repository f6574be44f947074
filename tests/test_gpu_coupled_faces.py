"""A coupled re-solve of the potential that stops at its iteration limit
leaves a valid state (Eq. 3-5): the steps that follow run in the potential it
left, as they do after that state is saved and loaded."""
import numpy as np
import pytest

from paper_2110_13055_gb300 import cdi, inputs

pytestmark = pytest.mark.gpu
Z, D = (1, -1), (1.33e-9, 2.03e-9)


@pytest.fixture(scope="module", autouse=True)
def built():
    import __graft_entry__ as g
    g.build()


@pytest.mark.parametrize("implicit", [False, True])
@pytest.mark.parametrize("prec", [cdi.FP64, cdi.FP32, cdi.FP32_CPAIR])
def test_steps_after_a_solve_that_did_not_converge(prec, implicit):
    """The two runs are the same steps from the same state: equal bits.  (The
    first 70 steps separate the species, so the re-solve's charge and its
    potential differ from the first ones.)"""
    m = inputs.grain_pack((23, 37), 0.6, 2.0, 4.0, seed=3)[0]
    with cdi.Domain(m, dx=2e-8, precision=prec) as d:
        d.solve_flow(tol=0.0, max_steps=200, U_target=1e-4)
        with pytest.raises(cdi.CDIError) as e:
            d.set_potential(0.3, mode="laplace", tol=1e-12, max_iter=2)
        assert e.value.status == 4
        d.init_transport(Z, D, c0=1.0, Ka=1e-5, dt=1e-9)
        if implicit:
            d.set_implicit(1e-12, 1000)
        d.step(70)
        d.set_coupling(70)
        with pytest.raises(cdi.CDIError) as e:
            d.step(1)
        assert e.value.status == 4
        d.set_coupling(0)
        state = d.save_state()
        d.step(70)
        a = d.C(), d.adsorbed()
        d.load_state(state)
        d.step(70)
        b = d.C(), d.adsorbed()
    assert np.array_equal(a[0], b[0]) and np.array_equal(a[1], b[1])
