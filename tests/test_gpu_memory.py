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
                assert a.total() <= before      # (optional memory was given back for it)
            a.refuse = lambda nbytes: False
            d.set_implicit(1e-10, 500)
            d.step(2)
            return d.C()

    assert np.array_equal(run(2), run(0))


def bern_block(m, ns, prec):
    """Names the block of the stored face coefficients (all species' pairs of
    FP64 or FP32 words on dim + 1 faces a cell; sizes round up to 256 bytes)."""
    size = (m.ndim + 1) * int((m == 0).sum()) * ns * (16 if prec == cdi.FP64 else 8)
    return lambda nbytes: size <= nbytes < size + 256


@pytest.mark.parametrize("prec", [cdi.FP64, cdi.FP32, cdi.FP32_CPAIR])
@pytest.mark.parametrize("ns", [1, 2, 3])
@pytest.mark.parametrize("shape", [(23, 37), (9, 13, 35)], ids=str)
def test_faces_evaluated_at_every_step(shape, ns, prec):
    """Without memory for the stored coefficients a step evaluates every face
    itself, by the same operations: the same bits, alone, in a sweep and in a
    batch (where the first member's coefficients are stored and the second's
    are not)."""
    m = pack(shape)
    z, D3 = (1, -1, 2)[:ns], (1.33e-9, 2.03e-9, 0.7e-9)[:ns]
    combos = [(1e-2, 0.3), (1e-3, 0.2)]

    def run(allowed):
        a = Allocator()
        named, seen = bern_block(m, ns, prec), []
        kw = dict(z=z, D=D3, c0=10.0, Ka=1e-6, n_steps=70, lambda_D=1.5e-7)
        with cdi.Domain(m, precision=prec, torch_resources=a) as d, \
                cdi.Domain(m, precision=prec, lateral_walls=True) as other:
            for x in (d, other):
                x.solve_flow(tol=0.0, max_steps=200, U_target=1e-2)
            d.set_potential(0.3, lambda_D=1.5e-7, tol=1e-12)
            out = []
            for what in ("steps", "sweep", "batch"):
                seen.clear()
                a.refuse = lambda nbytes: named(nbytes) and (seen.append(1) or len(seen) > allowed)
                if what == "steps":
                    d.init_transport(z, D3, c0=10.0, Ka=1e-6)
                    d.step(70)
                    out += [d.C(), *d.mass_balance()]
                elif what == "sweep":
                    out += list(d.sweep(combos, **kw))
                else:
                    p = cdi.cdi_elec_params(298.15, 78.5, 10.0, 1.5e-7, 0, 1e-12, 100000)
                    out += list(cdi.sweep_batch([d.handle, other.handle], combos, p, z, D3, 10.0,
                                                1e-6, 70))
                assert seen
            return out

    ref = run(100)
    for allowed in (0, 1):
        for x, y in zip(run(allowed), ref):
            assert np.array_equal(x, y)


@pytest.mark.parametrize("prec", [cdi.FP64, cdi.FP32])
def test_stored_coefficients_give_way(prec):
    """A domain that holds face coefficients sets up the implicit scheme and the
    coupling in the memory that these need alone, and goes back to explicit
    steps; one that steps implicitly holds none."""
    m = pack((9, 13, 35))
    n = int((m == 0).sum())
    named = bern_block(m, 2, prec)

    def run(short):
        a = Allocator()
        with cdi.Domain(m, precision=prec, torch_resources=a) as d:
            d.solve_flow(tol=0.0, max_steps=200, U_target=1e-2)
            d.set_potential(0.3, lambda_D=1.5e-7, tol=1e-12)
            # operator (10 values a species), one species' vectors, scalars; charges
            need = (4 * 10 + 5) * 8 * n + 8 * m.size + 4 * 256
            cap = a.total() + need
            if short:
                a.refuse = lambda nbytes: a.total() + nbytes > cap
            d.init_transport(Z, D, c0=1e-3, Ka=1e-6)
            d.step(5)
            assert any(named(b) for b in a.live.values())
            d.set_implicit(1e-10, 500)
            d.step(2)
            d.set_coupling(1)
            d.step(1)
            d.set_coupling(0)
            d.step(1)
            if short:
                assert a.refused and not any(named(b) for b in a.live.values())
            d.set_implicit(0.0)
            d.step(70)
            return [d.C(), *d.mass_balance()]

    for x, y in zip(run(True), run(False)):
        assert np.all(np.isfinite(x)) and np.array_equal(x, y)
    a = Allocator()
    with cdi.Domain(m, precision=prec, torch_resources=a) as d:
        d.solve_flow(tol=0.0, max_steps=200, U_target=1e-2)
        d.set_potential(0.3, lambda_D=1.5e-7, tol=1e-12)
        d.set_implicit(1e-10, 500)
        d.init_transport(Z, D, c0=1e-3, Ka=1e-6)
        d.step(2)
        assert not any(named(b) for b in a.live.values())


@pytest.mark.parametrize("prec", [cdi.FP64, cdi.FP32, cdi.FP32_CPAIR])
def test_sweep_members_in_parts(prec):
    """Five members in the memory of two: in parts, with the same bits.  Less
    than one member needs: an error, and nothing kept.  (A member: velocity,
    two concentration buffers and accounts; its face data may be the domain's.)"""
    m = pack((9, 13, 35))
    n, w = int((m == 0).sum()), 8 if prec == cdi.FP64 else 4
    words = 2 if prec == cdi.FP32_CPAIR else 1
    member = sum(-(-b // 256) * 256 for b in (
        3 * w * n, 2 * w * words * n, 2 * w * words * n, 3 * 4 * 8 * (((n + 30) // 31 + 7) // 8 * 8)))
    combos = [(1e-2, 0.3), (1e-3, 0.3), (1e-3, 0.0), (0.0, 0.3), (2e-3, 0.3)]
    p = cdi.cdi_elec_params(298.15, 78.5, 10.0, 1.5e-7, 0, 1e-12, 100000)

    def run(members):
        a = Allocator()
        with cdi.Domain(m, precision=prec, torch_resources=a) as d, \
                cdi.Domain(m[:, :, ::-1].copy(), precision=prec) as other:
            for x in (d, other):
                x.solve_flow(tol=0.0, max_steps=200, U_target=1e-2)
            before = a.total()
            out = []
            for phis, call in ((2, lambda: cdi.sweep_transport(d.handle, combos, p, Z, D, 10.0,
                                                               1e-6, 70)),
                               (4, lambda: cdi.sweep_batch([d.handle, other.handle], combos, p, Z,
                                                           D, 10.0, 1e-6, 70))):
                # the potentials, two small tables, and the members
                cap = before + phis * (-(-8 * n // 256) * 256) + 4096 + int(members * member)
                a.refuse = lambda nbytes: a.total() + nbytes > cap
                if members < 1:
                    with pytest.raises(cdi.CDIError) as e:
                        call()
                    assert e.value.status == 2
                else:
                    out += list(call())
                assert a.total() == before and (a.refused > 0) == (members < 1000)
            return out

    ref = run(1000)
    for members in (1, 2):
        for x, y in zip(run(members), ref):
            assert np.array_equal(x, y)
    assert run(0.5) == []


@pytest.mark.parametrize("prec", [cdi.FP64, cdi.FP32_CPAIR])
def test_allocator_of_looser_alignment(prec):
    """Blocks that start on 8 bytes only: the same bits as on 256."""
    m = pack((9, 13, 35))

    class Loose(Allocator):
        def __init__(self):
            import torch
            self.live = {}

            def _alloc(nbytes, ctx):
                p = torch.cuda.caching_allocator_alloc(int(nbytes) + 8, 0) + 8
                self.live[p] = nbytes
                return p

            def _free(ptr, nbytes, ctx):
                assert self.live.pop(ptr) == nbytes
                torch.cuda.caching_allocator_delete(ptr - 8)

            self._a, self._f = cdi.ALLOC_FN(_alloc), cdi.FREE_FN(_free)
            self.allocator = cdi.cdi_allocator(self._a, self._f, None)

    def run(a):
        with cdi.Domain(m, precision=prec, torch_resources=a) as d:
            d.solve_flow(tol=0.0, max_steps=200, U_target=1e-2)
            d.set_potential(0.3, mode="laplace", tol=1e-12)
            d.init_transport((1, -1, 2), (1.33e-9, 2.03e-9, 0.7e-9), c0=1e-3, Ka=1e-6)
            d.step(70)
            d.set_implicit(1e-10, 500)
            d.step(2)
            out = [d.C(), *d.mass_balance()]
        assert not a.live
        return out

    for x, y in zip(run(Loose()), run(Allocator())):
        assert np.array_equal(x, y)


@pytest.mark.parametrize("prec", [cdi.FP64, cdi.FP32, cdi.FP32_CPAIR])
@pytest.mark.parametrize("shape", [(301, 403), (48, 51, 55)], ids=str)
def test_domain_memory(shape, prec):
    """The most that creating a domain holds, bytes: 2D and 3D packs of
    porosity 0.6 fit where they fitted before the transport step had face data
    and 16-bit links of its own (flow flags, ranks and rank metadata then stood
    beside the fields)."""
    m = pack(shape)
    dim, N, n = m.ndim, m.size, int((m == 0).sum())
    w = 8 if prec == cdi.FP64 else 4
    flow = 2 * n * (9 * w + 4 + 4 + 4) if dim == 2 else 2 * n * (19 * w + 4 + 4 + 8)
    flow += 2 * N * ((2 if dim == 2 else 4) + 4 + 8 * dim)        # flags, ranks, velocity
    transport = n * (4 + 8 + 2 + 8 * (dim - 1) + dim * w + 8)     # lists, links, u, phi
    transport += n * 2 * 4 * w * (2 if prec == cdi.FP32_CPAIR else 1)
    accounts = 3 * 4 * 8 * (((n + 30) // 31 + 7) // 8 * 8)
    before = flow + transport + accounts + N * (1 + 2 + 8 + 32)
    # tile bases, row words, links of the x edges; partials and the rest
    rows = N // m.shape[-1]
    tables = (2 if dim == 2 else 8) * n // 4 + rows * 8 * (-(-m.shape[-1] // 32))
    tables += (8 if dim == 2 else 18) * 4 * 2 * rows + (1 << 18)
    a, peak = Allocator(), []
    a.refuse = lambda nbytes: peak.append(a.total() + nbytes)
    with cdi.Domain(m, precision=prec, torch_resources=a):
        assert max(peak) <= before + tables
