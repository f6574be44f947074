"""Different domains are independent: they may be driven by different host
threads at the same time."""
import threading

import pytest

from paper_2110_13055_gb300 import cdi, inputs

pytestmark = pytest.mark.gpu
Z, D = (1, -1, 2, -2), (1.33e-9, 2.03e-9, 0.8e-9, 1.1e-9)


@pytest.fixture(scope="module", autouse=True)
def built():
    import __graft_entry__ as g
    g.build()


def test_implicit_steps_of_several_threads():
    """Steps whose solver launches ask for different amounts of shared memory
    beyond the default limit (three and four species, a block's full number of
    threads).  The tolerance is met at once, so a step is little more than its
    launches."""
    m = inputs.grain_pack((540, 560), 0.6, 3.0, 6.0, seed=7)[0]
    doms, errors = [], []
    for ns in (3, 4, 3, 4):
        d = cdi.Domain(m)
        d.solve_flow(tol=0.0, max_steps=0, U_target=0.0)
        d.set_potential(0.3, lambda_D=1.5e-7, tol=1e-10)
        d.init_transport(Z[:ns], D[:ns], c0=10.0, Ka=1e-6)
        d.set_implicit(0.5, 10)
        doms.append(d)

    def run(d):
        try:
            for _ in range(1500):  # (the launch shape is found once a call)
                d.step(1)
        except cdi.CDIError as e:
            errors.append(e)

    threads = [threading.Thread(target=run, args=(d,)) for d in doms]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    for d in doms:
        d.close()
    assert not errors
