"""Norms after a handle was used on two streams at once, against its contract: the calls that
overlap (a replayed graph with a residual in it beside eager residuals) may return wrong
norms, but the residuals are right and every norm after them is right again, eager, captured
and in a solve."""
import numpy as np
import pytest

from tests.gpu_common import need_gpu, problem_for, rel, small_scene, to_dev, torch

pytestmark = pytest.mark.gpu


@pytest.fixture(autouse=True)
def _gpu():
    need_gpu()


def test_norms_after_overlapping_calls():
    import paper_2405_12380_gb300 as hm
    s = small_scene(3, 64)
    P = problem_for(s)
    f, x = to_dev(s["b"]), to_dev(s["rng"].standard_normal(s["b"].size) + 1j * s["rng"].standard_normal(s["b"].size))
    ref = s["b"] - s["A"] @ x.cpu().numpy()
    n2 = np.vdot(ref, ref).real
    f32, x32 = f.to(torch.complex64), x.to(torch.complex64)
    a, b = torch.cuda.Stream(), torch.cuda.Stream()
    torch.cuda.synchronize()
    P.set_stream(a)
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=a):
        got = [P.residual(f, x) for _ in range(40)]
    P.set_stream(b)
    torch.cuda.synchronize()
    for _ in range(30):
        with torch.cuda.stream(a):
            g.replay()
        with torch.cuda.stream(b):
            r = [(P.residual(f, x)[0], P.residual(f32, x32)[0]) for _ in range(50)]
    torch.cuda.synchronize()
    assert rel(r[-1][0].cpu().numpy(), ref) < 1e-13 and rel(got[-1][0].cpu().numpy(), ref) < 1e-13
    for k in range(130):
        with torch.cuda.stream(b):
            n64, n32 = P.residual(f, x)[1], P.residual(f32, x32)[1]
        assert abs(n64.item() - n2) <= 1e-12 * n2 and abs(n32.item() - n2) <= 1e-5 * n2, k
    for _, n in got:
        n.zero_()
    torch.cuda.synchronize()
    g.replay()
    torch.cuda.synchronize()
    assert all(abs(n.item() - n2) <= 1e-12 * n2 for _, n in got)
    st = P.solve(f, None, hm.opts("fgmres", "jacobi", 1, correction="none", tol=1e-10, restart=5, maxit=5))[1]
    assert abs(st["hist"][0] - 1) < 1e-12 and np.all(np.diff(st["hist"]) <= 0)
