"""Quiet tiles: large grids whose gas is uniform outside a disturbance, against the same run
without the levels (a batch; a short 1D grid), bitwise and with equal counters."""
from fractions import Fraction as F

import numpy as np
import pytest

import af_inputs as ai

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_2506_04857_gb300 as af  # noqa: E402


def disturbed(nx, ny, bc, x, y, strong, V=(1.0, 0.3, -0.2, 0.0, 0.5, 0.4, 0.0, 1.0)):
    """Uniform gas but for a patch of 9 x 9 index points around (x, y) (wrapped)."""
    rng = np.random.default_rng(nx + ny)
    out = []
    for ex, ey in ai.class_extents(nx, ny, bc):
        w = [np.full((ey, ex), v) for v in V]
        i, j = np.meshgrid((np.arange(-4, 5) + x) % ex, (np.arange(-4, 5) + y) % ey)
        for k in range(8):
            w[k][j, i] += 0.05 * rng.normal(size=i.shape)
        if strong:
            w[7][j, i] += 100.0
        out.append(ai.prim_to_cons(w, 1.4))
    return out


# last tiles of one column or row (periodic: 1025, 1021 + 4; outflow index grids are one larger),
# the disturbance inside, at a corner (through the wrap) and next to the last tile
@pytest.mark.parametrize("nx,ny,bc", [(1025, 517, ai.PERIODIC), (1024, 516, ai.OUTFLOW), (996, 600, ai.PERIODIC)])
@pytest.mark.parametrize("where", ["inside", "corner", "end"])
@pytest.mark.parametrize("kappa,cfl", [(1.0, 0.2), (0.0, 0.9)])
def test_quiet_equals_batch(nx, ny, bc, where, kappa, cfl):
    x, y = {"inside": (nx // 2, ny // 2), "corner": (1, 1), "end": (nx - 5, ny - 6)}[where]
    U = [torch.from_numpy(u).cuda() for u in disturbed(nx, ny, bc, x, y, strong=kappa > 0)]
    s = af.Solver(nx, ny, 1.4, bc, kappa=kappa, cfl=cfl)
    s.set_state(U)
    b = af.af_batch_create([nx], [ny], [1.4], [bc])
    af.af_batch_set_params(b, 0, kappa=kappa, cfl=cfl)
    af.af_batch_set_state(b, 0, U)
    for _ in range(2):
        s.step(False)
    af.af_batch_step(b, 2)
    got = af.af_batch_get_state(b, 0, [torch.empty_like(u) for u in U])
    for p, q in zip(s.get_state(), got):
        assert torch.equal(p, q)
    assert s.status()[1] == af.af_batch_status(b)[1]
    s.close()
    af.af_batch_destroy(b)


def test_uniform_gas_takes_its_dt_and_stays():
    V = (1.0, 0.3, -0.2, 0.1, 0.5, 0.4, 0.2, 1.0)
    dts = []
    for n in (64, 768):   # without and with the levels
        pb = ai.constant(n, n, bc=ai.OUTFLOW, gamma=1.4, w=V)
        U = [torch.from_numpy(u).cuda() for u in ai.dofs(pb, quad=1)]
        s = af.Solver(n, n, 1.4, pb.bc, domain=(0.0, n / 1024.0, 0.0, n / 1024.0))
        s.set_state(U)
        dts.append(s.step())
        for p, q in zip(s.get_state(), U):
            assert float((p - q).abs().max()) <= 1e-15
        s.close()
    assert dts[0] == dts[1]


# a long grid (levels) against a short one with the same cells around the disturbance
@pytest.mark.parametrize("n,at", [((1 << 20) + 1, 500000), ((1 << 20) + 130, 700)])
@pytest.mark.parametrize("kappa", [0.0, 1.0])
def test_1d_quiet_equals_short_grid(n, at, kappa):
    m, off = 6000, at - 600   # the short grid holds the long one's cells off .. off + m - 1
    rng = np.random.default_rng(3)
    w = [np.full(n + 1, v) for v in (1.0, 0.3, -0.2, 0.1, 0.5, 0.4, 0.2, 1.0)]
    for k in range(8):
        w[k][at:at + 40] += 0.05 * rng.normal(size=40)
    w[7][at:at + 40] += 50.0
    P = ai.prim_to_cons(w, 1.4)
    A = 0.5 * (P[:, :-1] + P[:, 1:])
    states = []
    for U, c0, c1 in (([A, P], 0, n), ([A[:, off:off + m], P[:, off:off + m + 1]], off, off + m)):
        s = af.Solver1D(c1 - c0, 1.4, af.AF_BC_OUTFLOW, domain=(c0 / 1024.0, c1 / 1024.0), kappa=kappa)
        s.set_state([torch.from_numpy(np.ascontiguousarray(u)).cuda() for u in U])
        for st in range(6):
            s.stage(st % 3, 2e-5)
        states.append((s.get_state(), s.status()[1]))
        s.close()
    (L, cl), (S, cs) = states
    assert torch.equal(L[0][:, off:off + m], S[0]) and torch.equal(L[1][:, off:off + m + 1], S[1])
    assert cl == cs


def centre_misses(v):
    """Whether 36/16 v - 4 4/16 v - 4/16 v, rounded as the centre value is, is not v."""
    r = float(F(-5, 4) * F(v))
    return float(F(9, 4) * F(v) + F(r)) != v


# Uniform gas whose zeros are of either sign, and whose centre value would not be the state itself
# were it formed from the nine states: uniform bit for bit, so it takes the state, and the quiet
# tiles and the others (here: a batch) agree.
@pytest.mark.parametrize("nx,ny,bc", [(1025, 517, ai.PERIODIC), (1024, 516, ai.OUTFLOW)])
def test_zeros_of_either_sign(nx, ny, bc):
    rng = np.random.default_rng(1)
    V = np.array([1.0, 0.3, -0.2, 0.0, 0.5, 0.4, 0.0, 3.0])
    for k in (0, 1, 4, 7):
        while not centre_misses(V[k]):
            V[k] += 1e-3 * rng.random()
    U = []
    for ex, ey in ai.class_extents(nx, ny, bc):
        u = np.empty((8, ey, ex))
        for k in range(8):
            u[k] = V[k]
        for k in (3, 6):
            u[k] = np.copysign(0.0, rng.random((ey, ex)) - 0.5)
        u[7, ey // 2: ey // 2 + 9, ex // 2: ex // 2 + 9] += 0.01 * rng.random((9, 9))
        U.append(torch.from_numpy(u).cuda())
    s = af.Solver(nx, ny, 1.4, bc, kappa=1.0, cfl=0.9)
    s.set_state(U)
    s.stage(0, 2e-4)   # the forward-Euler stage leaves the state, and the tiles near the disturbance do too
    for p in s.get_stage():
        assert torch.equal(p[:, :248], torch.from_numpy(V).cuda()[:, None, None].expand_as(p[:, :248]))
    s.set_state(U)
    b = af.af_batch_create([nx], [ny], [1.4], [bc])
    af.af_batch_set_params(b, 0, kappa=1.0, cfl=0.9)
    af.af_batch_set_state(b, 0, U)
    s.step(False)
    af.af_batch_step(b, 1)
    got = af.af_batch_get_state(b, 0, [torch.empty_like(u) for u in U])
    for p, q in zip(s.get_state(), got):
        assert torch.equal(p, q)
    s.close()
    af.af_batch_destroy(b)


# A NaN anywhere makes the time step NaN and with it every degree of freedom, in the quiet tiles too;
# the counters and the error are those of the run without tiles.
@pytest.mark.parametrize("nx,ny,bc", [(1024, 516, ai.OUTFLOW)])
def test_poisoned_state(nx, ny, bc):
    U = [torch.from_numpy(u).cuda() for u in disturbed(nx, ny, bc, nx // 2, ny // 2, strong=False)]
    U[3][7, ny // 2, nx // 2] = float("nan")
    s = af.Solver(nx, ny, 1.4, bc, kappa=1.0)
    s.set_state(U)
    b = af.af_batch_create([nx], [ny], [1.4], [bc])
    af.af_batch_set_params(b, 0, kappa=1.0)
    af.af_batch_set_state(b, 0, U)
    s.step(False)
    af.af_batch_step(b, 1)
    got = af.af_batch_get_state(b, 0, [torch.empty_like(u) for u in U])
    for p, q in zip(s.get_state(), got):
        assert bool(torch.isnan(p).all()) and bool(torch.isnan(q).all())
    rc, cnt = s.status()
    assert (rc, cnt) == tuple(af.af_batch_status(b)) and rc == af.AF_EBOUNDS   # the repair list overflowed
    s.close()
    af.af_batch_destroy(b)


def test_poisoned_state_1d():
    n = 1 << 20
    P = ai.prim_to_cons([np.full(n + 1, v) for v in (1.0, 0.3, -0.2, 0.1, 0.5, 0.4, 0.2, 1.0)], 1.4)
    A = np.ascontiguousarray(P[:, :-1])
    P[7, n // 2] = np.nan
    s = af.Solver1D(n, 1.4, af.AF_BC_OUTFLOW, domain=(0.0, n / 1024.0))
    s.set_state([torch.from_numpy(u).cuda() for u in (A, P)])
    s.step(False)
    for p in s.get_state():
        assert bool(torch.isnan(p).all())
    rc, cnt = s.status()
    assert rc == af.AF_EBOUNDS and cnt["nonadmissible"] >= 3 * (n + 1)
    s.close()
