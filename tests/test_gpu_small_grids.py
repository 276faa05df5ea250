"""The small-grid build of the stage kernels against the large-grid one (bitwise), and the list
passes of the limiters against the oracle with short and long lists."""
import numpy as np
import pytest

import af_inputs as ai
import oracle
from test_gpu_parity import rel_err

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_2506_04857_gb300 as af  # noqa: E402


# the smallest grid, remainders of a 32-wide tile, and both sides of the line between the two
# builds (1216 row tiles of 32 points: 128 x 304 and 128 x 305); batches always run the large build
@pytest.mark.parametrize("nx,ny", [(4, 4), (31, 9), (33, 17), (128, 304), (128, 305)])
@pytest.mark.parametrize("bc", [ai.PERIODIC, ai.OUTFLOW])
def test_builds_agree(nx, ny, bc):
    pb = ai.random_smooth(nx, ny, seed=nx + ny, amp=0.3, bc=bc)
    pb.kappa = 1.0
    U = [torch.from_numpy(u).cuda() for u in ai.dofs(pb)]
    s = af.Solver(pb.nx, pb.ny, pb.gamma, pb.bc, domain=(pb.x0, pb.x1, pb.y0, pb.y1), kappa=pb.kappa)
    s.set_state(U)
    b = af.af_batch_create([nx], [ny], [pb.gamma], [pb.bc])
    af.af_batch_set_domain(b, 0, pb.x0, pb.x1, pb.y0, pb.y1)
    af.af_batch_set_params(b, 0, kappa=pb.kappa)
    af.af_batch_set_state(b, 0, U)
    for _ in range(3):
        s.step(False)
    af.af_batch_step(b, 3)
    got = af.af_batch_get_state(b, 0, [torch.empty_like(u) for u in U])
    for x, y in zip(s.get_state(), got):
        assert torch.equal(x, y)
    s.close()
    af.af_batch_destroy(b)


# cells on the list: a few (a half-warp each) and more than a launch takes half-warps for, in
# both builds; every counter as the oracle's
@pytest.mark.parametrize("n,periods", [(96, 2), (128, 16), (160, 2), (224, 28)])
def test_limiter_lists(n, periods):
    pb = ai.rarefaction_lattice(n, periods=periods, kappa=0.0)
    U = ai.dofs(pb)
    U, _ = oracle.step(pb, U)
    dt = oracle.dt(pb, U)
    st = np.zeros(oracle.NSTATS, dtype=np.int64)
    R = oracle.stage(pb, U, U, dt, 0.0, 1.0, stats=st)
    s = af.Solver(pb.nx, pb.ny, pb.gamma, pb.bc, domain=(pb.x0, pb.x1, pb.y0, pb.y1), cfl=pb.cfl, kappa=0.0)
    s.set_state([torch.from_numpy(u).cuda() for u in U])
    s.stage(0, dt)
    G = s.get_stage()
    rc, cnt = s.status()
    assert rc == af.AF_OK
    assert rel_err(G, R) <= 1e-12
    ref = dict(zip(oracle.STAT_NAMES, st))
    for name in ("src_limited", "lambda_lt1", "face_theta_lt1", "newton_solves", "point_limited", "center_limited"):
        assert cnt[name] == ref[name], (name, cnt[name], ref[name])
    assert cnt["lambda_lt1"] > 0
    s.close()


# af_timing reports what is launched, kernel by kernel: two steps (six stages) of a large grid have
# launches of their own for everything, of a small one three kernels hold more than one part
@pytest.mark.parametrize("n", [64, 256])
def test_timing_counts_every_launch(n):
    pb = ai.random_smooth(n, n, seed=1, amp=0.3)
    s = af.Solver(n, n, pb.gamma, pb.bc, domain=(pb.x0, pb.x1, pb.y0, pb.y1), kappa=1.0)
    s.set_state([torch.from_numpy(u).cuda() for u in ai.dofs(pb)])
    s.timing(True)
    for _ in range(2):
        s.step(False)
    t = s.timing(False)
    s.close()
    own = 0 if n == 64 else 6
    want = {"k_pointdata": 6, "k_dt": own // 3, "k_points": 6, "k_faces": 6, "k_cells": 6, "k_final": 6, "k_repair": own,
            "k_points_slow": own, "k_cells_slow": 6}
    assert {k: v[1] for k, v in t.items()} == want
    assert all((v[0] > 0.0) == (v[1] > 0) for v in t.values())


# A long point list does not delay the passes: a step of the smaller of two limited grids is the shorter
# one (about 0.8 by its points).
def test_a_smaller_limited_grid_is_faster():
    t = []
    for n in (224, 256):
        pb = ai.rarefaction_lattice(n, periods=n // 32, kappa=0.0)
        s = af.Solver(n, n, pb.gamma, pb.bc, domain=(pb.x0, pb.x1, pb.y0, pb.y1), cfl=pb.cfl, kappa=0.0)
        s.set_state([torch.from_numpy(u).cuda() for u in ai.dofs(pb)])
        for _ in range(6):
            s.step(False)
        best = 1e9
        for _ in range(3):
            e = [torch.cuda.Event(enable_timing=True) for _ in range(2)]
            e[0].record()
            for _ in range(5):
                s.step(False)
            e[1].record()
            torch.cuda.synchronize()
            best = min(best, e[0].elapsed_time(e[1]))
        t.append(best)
        s.close()
    assert t[0] < t[1]
