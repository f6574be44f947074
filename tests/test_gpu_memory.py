"""Device memory that cannot be had: what the library takes only to be faster
is done without, with the same results; a call that needs more than there is
fails alone.  (No GPU fault is made: the allocator returns NULL.)"""
import numpy as np
import pytest

from paper_2110_13055_gb300 import cdi, inputs

pytestmark = pytest.mark.gpu
Z, D = (1, -1), (1.33e-9, 2.03e-9)


@pytest.fixture(scope="module", autouse=True)
def built():
    import __graft_entry__ as g
    g.build()


class Allocator:
    """Device memory from torch's caching allocator, NULL for a block that
    `refuse(bytes)` names; as the torch_resources of a Domain."""
    stream_handle = None

    def __init__(self, refuse=lambda nbytes: False):
        import torch
        self.refuse, self.live, self.refused = refuse, {}, 0

        def _alloc(nbytes, ctx):
            if self.refuse(nbytes):
                self.refused += 1
                return None
            p = torch.cuda.caching_allocator_alloc(int(nbytes), 0)
            self.live[p] = nbytes
            return p

        def _free(ptr, nbytes, ctx):
            assert self.live.pop(ptr) == nbytes
            torch.cuda.caching_allocator_delete(ptr)

        self._a, self._f = cdi.ALLOC_FN(_alloc), cdi.FREE_FN(_free)
        self.allocator = cdi.cdi_allocator(self._a, self._f, None)

    def total(self):
        return sum(self.live.values())


def pack(shape=(23, 37)):
    return inputs.grain_pack(shape, 0.6, 1.5, 3.0, seed=3)[0]


@pytest.mark.parametrize("prec", [cdi.FP64, cdi.FP32, cdi.FP32_CPAIR])
def test_implicit_species_after_one_another(prec):
    """Without memory for the vectors of all species they are solved in one
    set of vectors: the same bits.  A step whose second species does not
    converge takes nothing, neither concentrations nor accounts."""
    m = pack()

    def run(one_set, limit):
        a = Allocator()
        with cdi.Domain(m, precision=prec, torch_resources=a) as d:
            d.solve_flow(tol=0.0, max_steps=0, U_target=0.0)
            d.set_potential(0.3, lambda_D=1.5e-7, tol=1e-12)
            # dt D / dx^2 is 1e-3 and 20: 3 iterations are enough for the first
            d.init_transport((0, 0), (1e-13, 2e-9), c0=10.0, Ka=1e-6, dt=1e-4)
            d.set_implicit(1e-6, limit)
            if one_set:
                a.refuse = lambda nbytes: True
            if limit == 3:
                C = d.C()
                with pytest.raises(cdi.CDIError) as e:
                    d.step(1)
                assert e.value.status == 4
                assert np.array_equal(d.C(), C)
                M, G, In, Out = d.mass_balance()
                assert not G.any() and not In.any() and not Out.any()
                d.set_implicit(1e-6, 500)
            d.step(3)
            assert (a.refused > 0) == one_set
            return (d.C(),) + d.mass_balance()

    ref = run(False, 500)
    assert np.all(ref[2] > 0.0)
    for one_set, limit in ((True, 500), (False, 3), (True, 3)):
        for x, y in zip(run(one_set, limit), ref):
            assert np.array_equal(x, y)


@pytest.mark.parametrize("fail_at", [1, 2, 3])
def test_implicit_memory_all_or_nothing(fail_at):
    """Every call that cannot have the implicit scheme's memory fails and keeps
    none of it; the first that can, works."""
    m = pack()

    def run(tries):
        a = Allocator()
        with cdi.Domain(m, torch_resources=a) as d:
            d.solve_flow(tol=0.0, max_steps=0, U_target=0.0)
            d.set_potential(0.3, lambda_D=1.5e-7, tol=1e-12)
            d.init_transport(Z, D, c0=10.0, Ka=1e-6)
            before = a.total()
            for _ in range(tries):
                calls = []
                a.refuse = lambda nbytes: calls.append(nbytes) or len(calls) >= fail_at
                with pytest.raises(cdi.CDIError) as e:
                    d.set_implicit(1e-10, 500)
                assert e.value.status == 2
                assert a.total() == before
            a.refuse = lambda nbytes: False
            d.set_implicit(1e-10, 500)
            d.step(2)
            return d.C()

    assert np.array_equal(run(2), run(0))
