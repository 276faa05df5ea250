"""Work lists of the runs of a batch: limited runs of several sizes, with every tile shape the
autotuner may choose (one is narrower than a warp), bitwise and in every counter as single runs."""
import numpy as np
import pytest

import af_inputs as ai

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_2506_04857_gb300 as af  # noqa: E402


# without and with the autotuner's tiles (its choice varies; a few draws)
@pytest.mark.parametrize("tuned", [0, 1, 2, 3])
def test_limited_runs(tuned):
    pbs = [ai.rarefaction_lattice(96, periods=12, kappa=0.0), ai.blast(40), ai.rarefaction_lattice(33, periods=2, kappa=0.0),
           ai.double_rarefaction(64, speed=6.0, kappa=0.0), ai.orszag_tang(17, 29)]
    pbs[1].kappa = 0.0
    U = [[torch.from_numpy(u).cuda() for u in ai.dofs(p)] for p in pbs]
    b = af.af_batch_create([p.nx for p in pbs], [p.ny for p in pbs], [p.gamma for p in pbs], [p.bc for p in pbs])
    for r, p in enumerate(pbs):
        af.af_batch_set_domain(b, r, p.x0, p.x1, p.y0, p.y1)
        af.af_batch_set_params(b, r, cfl=p.cfl, kappa=p.kappa, pp_on=(r != 4))
        af.af_batch_set_state(b, r, U[r])
    if tuned:
        af.af_batch_autotune(b, reps=1)
    af.af_batch_status(b, reset=True)
    af.af_batch_step(b, 3)
    total = None
    for r, p in enumerate(pbs):
        s = af.Solver(p.nx, p.ny, p.gamma, p.bc, domain=(p.x0, p.x1, p.y0, p.y1), cfl=p.cfl, kappa=p.kappa, pp_on=(r != 4))
        s.set_state(U[r])
        for _ in range(3):
            s.step(False)
        got = af.af_batch_get_state(b, r, [torch.empty_like(u) for u in U[r]])
        for x, y in zip(s.get_state(), got):
            assert torch.equal(x, y), p.name
        c = s.status()[1]
        if total is None:
            total = dict(c)
        else:
            total = {k: max(total[k], v) if k == "newton_maxit" else total[k] + v for k, v in c.items()}
        s.close()
    assert total["point_limited"] > 0 and total["lambda_lt1"] > 0
    assert af.af_batch_status(b)[1] == total
    af.af_batch_destroy(b)


# One limited run has the whole chip for its lists in a batch too: alone, with a second one, and among
# small runs that nothing limits.  The batch runs the same passes without the overlap of the two lists
# with the others: less than twice the time is expected, three times is allowed.
@pytest.mark.parametrize("others", ["none", "same", "small"])
def test_one_limited_run_has_the_whole_chip(others):
    big = ai.rarefaction_lattice(512, periods=16, kappa=0.0)
    pbs = [big] + {"none": [], "same": [big], "small": [ai.orszag_tang(32)] * 15}[others]
    U = {id(p): [torch.from_numpy(u).cuda() for u in ai.dofs(p)] for p in pbs}
    b = af.af_batch_create([p.nx for p in pbs], [p.ny for p in pbs], [p.gamma for p in pbs], [p.bc for p in pbs])
    runs = []
    for r, p in enumerate(pbs):
        af.af_batch_set_domain(b, r, p.x0, p.x1, p.y0, p.y1)
        af.af_batch_set_params(b, r, cfl=p.cfl, kappa=p.kappa)
        af.af_batch_set_state(b, r, U[id(p)])
        runs.append(af.Solver(p.nx, p.ny, p.gamma, p.bc, domain=(p.x0, p.x1, p.y0, p.y1), cfl=p.cfl, kappa=p.kappa))
        runs[-1].set_state(U[id(p)])

    def best(step):
        times = []
        for _ in range(4):
            t = [torch.cuda.Event(enable_timing=True) for _ in range(2)]
            t[0].record()
            step()
            t[1].record()
            torch.cuda.synchronize()
            times.append(t[0].elapsed_time(t[1]))
        return min(times[1:])

    t_batch = best(lambda: af.af_batch_step(b, 1))
    t_runs = best(lambda: [s.step(False) for s in runs])
    assert runs[0].status()[1]["point_limited"] > 100000
    for s in runs:
        s.close()
    af.af_batch_destroy(b)
    assert t_batch < 3.0 * t_runs


def test_memory_of_a_batch():
    """What a batch holds per index point: three states (8 components of 4 classes) and 163 doubles of
    stage work arrays; the limiter lists take none of their own."""
    n = 1024
    args = lambda m: ([m], [m], [1.4], [af.AF_BC_PERIODIC])   # noqa: E731
    af.af_batch_destroy(af.af_batch_create(*args(8)))
    torch.cuda.synchronize()
    free = torch.cuda.mem_get_info()[0]
    b = af.af_batch_create(*args(n))
    used = free - torch.cuda.mem_get_info()[0]
    af.af_batch_destroy(b)
    assert 0 < used <= n * n * (3 * 32 + 163) * 8 + (32 << 20)
