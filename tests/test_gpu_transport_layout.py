"""The FP32 transport step's stored face data, species records and 16-bit
lateral differences against FP64 storage of the same run (which holds planes,
full neighbour ranks and evaluates every face), where they can go wrong:
every species count, faces below and above |P| = 1/2, feed faces, walls, and
differences that do not fit 16 bits."""
import numpy as np
import pytest

from paper_2110_13055_gb300 import cdi, inputs

pytestmark = pytest.mark.gpu
ZS, DS = (1, -1, 2, -1), (1.33e-9, 2.03e-9, 0.7e-9, 1.1e-9)


@pytest.fixture(scope="module", autouse=True)
def built():
    import __graft_entry__ as g
    g.build()


def advance(m, prec, ns, lam, steps, walls=False, U=1e-4, dt=0.0):
    with cdi.Domain(m, precision=prec, lateral_walls=walls) as d:
        d.solve_flow(tol=0.0, max_steps=200, U_target=U)
        d.set_potential(0.3, lambda_D=lam, tol=1e-13)
        dt = d.init_transport(ZS[:ns], DS[:ns], c0=10.0, Ka=1e-6, dt=dt)
        d.step(steps)
        return d.C(), d.adsorbed(), dt


def rel(a, b):
    return float(np.linalg.norm(a - b) / np.linalg.norm(b))


# FP32 rounding of flux and flow: a few 1e-7 a step of the part of C that a
# step moves, over 40 steps; the bar is the FP32 storage's own (1e-4 for C,
# 1e-6 of the total adsorbed amount, 1e-5 of the species')
@pytest.mark.parametrize("prec", [cdi.FP32, cdi.FP32_CPAIR])
@pytest.mark.parametrize("ns", [1, 2, 3, 4])
@pytest.mark.parametrize("lam", [0.0, 1.5e-7])
@pytest.mark.parametrize("shape", [(23, 37), (9, 13, 35)])
def test_species_records_and_faces(prec, ns, lam, shape):
    m = inputs.grain_pack(shape, 0.6, 1.5, 3.0, seed=7 + ns)[0]
    walls = ns % 2 == 0
    C, G, dt = advance(m, cdi.FP64, ns, lam, 40, walls, U=1e-2)
    c, g, _ = advance(m, prec, ns, lam, 40, walls, U=1e-2, dt=dt)
    assert rel(c, C) < 1e-4
    assert np.all(np.abs(g - G) < 1e-6 * np.abs(G).sum() + 1e-5 * np.abs(G))


def test_lateral_differences_beyond_16_bits():
    """Consecutive ranks whose z neighbours lie more than 32,000 ranks apart."""
    m = np.zeros((3, 190, 256), np.uint8)
    m[1, 2:185, :] = 1
    C, G, dt = advance(m, cdi.FP64, 2, 0.0, 6)
    c, g, _ = advance(m, cdi.FP32_CPAIR, 2, 0.0, 6, dt=dt)
    assert rel(c, C) < 1e-6
    assert np.all(np.abs(g - G) < 1e-6 * np.abs(G).sum())


@pytest.mark.parametrize("prec", [cdi.FP32, cdi.FP32_CPAIR])
@pytest.mark.parametrize("ns", [2, 3])
def test_steps_of_a_state_larger_than_l2(ns, prec):
    """1.8 million pore cells: the step asks for its inputs ahead (one and two
    species pairs).  Four steps; the bars of test_species_records_and_faces."""
    m = inputs.grain_pack((120, 125, 171), 0.7, 8.0, 14.0, seed=3)[0]
    C, G, dt = advance(m, cdi.FP64, ns, 0.0, 4)
    c, g, _ = advance(m, prec, ns, 0.0, 4, dt=dt)
    assert rel(c, C) < 1e-4
    assert np.all(np.abs(g - G) < 1e-6 * np.abs(G).sum() + 1e-5 * np.abs(G))
