"""A user's CUDA graph around the steps of one run: programmatic launches, the fork to the second
stream and the one-launch 1D step are captured, and a replay gives what direct calls give."""
import pytest

import af_inputs as ai

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_2506_04857_gb300 as af  # noqa: E402


def solver2d(pb):
    return lambda stream: af.Solver(pb.nx, pb.ny, pb.gamma, pb.bc, domain=(pb.x0, pb.x1, pb.y0, pb.y1), cfl=pb.cfl,
                                    kappa=pb.kappa, stream=stream), ai.dofs(pb)


def solver1d(pb, n):
    return lambda stream: af.Solver1D(n, pb.gamma, pb.bc, domain=(pb.x0, pb.x1), kappa=1.0, stream=stream), ai.dofs1(pb)


# a small grid, a larger one with both limiter lists, one with quiet tiles, 1D in one launch and in passes
CASES = {"small": lambda: solver2d(ai.blast(64)), "lists": lambda: solver2d(ai.rarefaction_lattice(256, periods=8, kappa=0.0)),
         "quiet": lambda: solver2d(ai.blast(768)), "1d": lambda: solver1d(ai.blast1d(800), 800),
         "1d_passes": lambda: solver1d(ai.blast1d(5000), 5000)}


@pytest.mark.parametrize("case", sorted(CASES))
def test_replay_equals_calls(case):
    make, U = CASES[case]()
    U = [torch.from_numpy(u).cuda() for u in U]
    stream = torch.cuda.Stream()
    stream.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(stream):
        s, r = make(stream), make(stream)
        s.set_state(U)
        r.set_state(U)
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=stream):
        for _ in range(3):   # the states rotate through three buffers
            s.step(False)
    with torch.cuda.stream(stream):
        for _ in range(2):
            g.replay()
        for _ in range(6):
            r.step(False)
        torch.cuda.synchronize()
        for x, y in zip(s.get_state(), r.get_state()):
            assert torch.equal(x, y)
    assert s.status() == r.status()
    s.close()
    r.close()
