"""The second difference of a 5-point FVS line in fixed point (af_math.cuh up5): components over
the whole exponent range, exact zeros, mixed signs and jumps, through unlimited stages against the
oracle (dt of order 1: the update is as large as the state)."""
import math
from fractions import Fraction as F

import numpy as np
import pytest

import af_inputs as ai
import oracle

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_2506_04857_gb300 as af  # noqa: E402


DT = 1.0


def stage(pb, U):
    s = af.Solver(pb.nx, pb.ny, pb.gamma, pb.bc, domain=(pb.x0, pb.x1, pb.y0, pb.y1), kappa=0.0, pp_on=False)
    s.set_state([torch.from_numpy(u).cuda() for u in U])
    s.stage(0, DT)
    out = s.get_stage(device=False)
    s.close()
    return out


def oracle_stage(pb, U):
    return oracle.stage(pb, U, U, DT, 0.0, 1.0, kappa=0.0, pp_on=False)


# size of the third components of momentum and field (they enter the others squared only):
# ordinary, exactly zero, at and beyond the smallest exponent of the fixed-point path
# (2^-823), and subnormal
@pytest.mark.parametrize("log2", [0, None, -60, -500, -822, -826, -1060])
@pytest.mark.parametrize("bc", [ai.PERIODIC, ai.OUTFLOW])
def test_small_components(log2, bc):
    pb = ai.random_smooth(33, 9, seed=4, amp=0.3, bc=bc)
    rng = np.random.default_rng(7)
    U = ai.dofs(pb)
    for u in U:
        for k in (3, 6):
            E = 0.5 * u[3] ** 2 / u[0] if k == 3 else 0.5 * u[6] ** 2
            u[7] -= E
            u[k] = 0.0 if log2 is None else np.ldexp(rng.normal(size=u[k].shape), log2)
            u[7] += 0.5 * u[3] ** 2 / u[0] if k == 3 else 0.5 * u[6] ** 2
    G, R = stage(pb, U), oracle_stage(pb, U)
    for a, b in zip(G, R):
        for k in range(8):
            scale = np.abs(b[k]).max()
            # an update below 2^-1000 is at the subnormal spacing times dt/h
            tiny = 64 * 33 * 5e-324
            assert np.abs(a[k] - b[k]).max() <= 1e-12 * scale + tiny, (k, log2)
            if log2 is None and k in (3, 6):
                assert not a[k].any()


# a jump of 2^bits in density, energy and field between neighbouring points, and noise of
# either sign: alignments from 0 to beyond 63 bits.  Compared at the corners, whose lines hold
# corners and faces only (a cell-centre value is itself a difference of such states).
@pytest.mark.parametrize("bits", [0, 5, 6, 7, 31, 32, 33, 57, 58, 59, 63, 64, 70])
def test_jumps(bits):
    pb = ai.random_smooth(20, 7, seed=5, amp=0.2)
    rng = np.random.default_rng(bits)
    U = ai.dofs(pb)
    for u in U:
        big = rng.random(u[0].shape) < 0.3
        f = np.where(big, 2.0 ** bits, 1.0)
        u[1:4] *= rng.choice([-1.0, 1.0], size=u[1:4].shape) * 0.1
        u[4:7] *= rng.choice([-1.0, 1.0], size=u[4:7].shape) * 0.1
        u[[0, 1, 2, 3, 7]] *= f
        u[4:7] *= np.sqrt(f)
        u[7] = 2.0 * f + 0.5 * (u[1:4] ** 2).sum(0) / u[0] + 0.5 * (u[4:7] ** 2).sum(0)
    a, b = stage(pb, U)[3], oracle_stage(pb, U)[3]
    for k in range(8):
        assert np.abs(a[k] - b[k]).max() <= 1e-12 * np.abs(b[k]).max(), (k, bits)


# The sum itself to its own error bound.  Gas at rest under one pressure without a field: every flux
# difference is 0 and a corner's density becomes rho - c alpha up, up = u0 + u4 - 4 (u1 + u3) + 6 u2 of
# its x line (its y line is constant), c a power of two.  up may be off by a quarter of a unit of
# the largest term's last place (the bits dropped in the alignment) and half of one of its own
# (rounding); alpha (two square roots, a reciprocal, three products), its product with up and the
# update add at most 8 half units of the result's.  Lines: ordinary values, jumps of 2^bits, and
# lines of equal or exactly cancelling values, where up is 0 and the density must not change.
@pytest.mark.parametrize("kind", ["smooth", "cancel", 0, 1, 5, 6, 7, 31, 52, 58, 59, 64, 70])
def test_error_bound(kind):
    nx, ny, p, gamma = 64, 4, 1.0, 1.5
    rng = np.random.default_rng(11)
    x = np.arange(2 * nx) / (2 * nx)   # corners at the even places, y-faces at the odd ones
    if kind == "smooth":
        rho = 1.0 + 0.3 * np.sin(2 * np.pi * x) + 0.1 * np.cos(6 * np.pi * x)
    elif kind == "cancel":   # cubics with coefficients of a few bits, and constant stretches
        k = np.arange(2 * nx)
        rho = np.where(k % 32 < 16, 1.0 + ((k % 16) - 8.0) ** 3 / 4096.0, 1.375)
    else:
        rho = (1.0 + rng.random(2 * nx)) * np.where(rng.random(2 * nx) < 0.3, 2.0 ** kind, 1.0)
    C, Y = rho[0::2], rho[1::2]
    U = []
    for r in (Y, C, Y, C):   # averages and x-faces lie on other lines; x-faces as the corners above and below
        u = np.zeros((8, ny, nx))
        u[0], u[7] = r, p / (gamma - 1.0)
        U.append(u)
    s = af.Solver(nx, ny, gamma, ai.PERIODIC, domain=(0.0, 1.0, 0.0, 1.0), kappa=0.0, pp_on=False)
    s.set_state([torch.from_numpy(u).cuda() for u in U])
    s.stage(0, 2.0 ** 20)
    got = s.get_stage(device=False)[3][0]
    s.close()
    c = F(2) ** 25
    zeros = 0
    for i in range(nx):
        u = [C[i - 1], Y[i - 1], C[i], Y[i], C[(i + 1) % nx]]
        up = F(u[0]) + F(u[4]) - 4 * (F(u[1]) + F(u[3])) + 6 * F(u[2])
        al = F(math.sqrt(gamma * p / min(u)))
        want = F(u[2]) - c * al * up
        bound = c * al * (F(1, 4) * F(np.spacing(max(u))) + F(1, 2) * F(np.spacing(abs(float(up)))))
        bound += 8 * F(1, 2) * F(np.spacing(abs(float(want))))
        for j in range(ny):
            if up == 0:
                zeros += 1
                assert got[j, i] == u[2]
            else:
                assert abs(F(got[j, i]) - want) <= bound, (i, j, float(up))
    assert kind != "cancel" or zeros > nx
