"""The one-launch 1D step of short grids against the pass-by-pass kernels (which run while the
per-kernel timing is on, and on longer grids): bitwise equal states and equal counters."""
import numpy as np
import pytest

import af_inputs as ai

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_2506_04857_gb300 as af  # noqa: E402


# the smallest grid, remainders of the 32-thread roles of 16 CTAs, one and two rounds of the
# 16 x 128 threads of a role, and the longest grid of the one-launch step (4096 indices)
@pytest.mark.parametrize("n", [4, 5, 31, 33, 511, 512, 513, 800, 2047, 2048, 2049, 4095, 4096, 4097])
@pytest.mark.parametrize("bc", [ai.PERIODIC, ai.OUTFLOW])
@pytest.mark.parametrize("kappa,pp_on", [(1.0, True), (0.0, False)])
def test_step_equals_passes(n, bc, kappa, pp_on):
    pb = ai.blast1d(n)
    rng = np.random.default_rng(n)
    U = ai.dofs1(pb)
    U = [np.ascontiguousarray(u[:, :n] if bc == ai.PERIODIC else u) for u in U]
    for u in U:
        u[1:4] += 1e-2 * rng.normal(size=u[1:4].shape)
        u[7] += 0.5 * (u[1:4] ** 2).sum(0) / u[0]
        if not pp_on:
            u[7] += 2000.0
    a, b = [af.Solver1D(n, pb.gamma, bc, domain=(pb.x0, pb.x1), kappa=kappa, pp_on=pp_on) for _ in range(2)]
    a.set_state(U)
    b.set_state(U)
    b.timing(True)
    for _ in range(2):
        a.step(False)
        b.step(False)
    b.timing(False)
    for s in range(2):   # and stage by stage
        a.stage(s, 1e-3 / n)
        b.stage(s, 1e-3 / n)
    for x, y in zip(a.get_stage() + a.get_state(), b.get_stage() + b.get_state()):
        assert torch.equal(x, y)
    assert a.status()[1] == b.status()[1]
    a.close()
    b.close()


# Beyond one index per thread (16 CTAs of 128) a second round of indices costs more than the launches it
# saves: the step of 3000 cells runs pass by pass, in little more time than that of 2047.  (In two
# rounds: 1.57 times; pass by pass both: 1.05; a launch for each pass against one: at most 1.25.)
def test_longer_grids_do_not_take_a_second_round():
    t = []
    for n in (2047, 3000):
        x = np.linspace(0.0, 1.0, n + 1)
        w = [1.0 + 0.1 * np.sin(2.0 * np.pi * x)] + [np.full(n + 1, v) for v in (0.3, -0.2, 0.1, 0.5, 0.4, 0.2, 1.0)]
        P = ai.prim_to_cons(w, 1.4)
        s = af.Solver1D(n, 1.4, af.AF_BC_OUTFLOW, kappa=1.0)
        s.set_state([torch.from_numpy(np.ascontiguousarray(u)).cuda() for u in (0.5 * (P[:, :-1] + P[:, 1:]), P)])
        best = 1e9
        for _ in range(5):
            e = [torch.cuda.Event(enable_timing=True) for _ in range(2)]
            e[0].record()
            for _ in range(20):
                s.step(False)
            e[1].record()
            torch.cuda.synchronize()
            best = min(best, e[0].elapsed_time(e[1]))
        t.append(best)
        s.close()
    assert t[1] < 1.4 * t[0]
