"""The passes of a solve start while the stream's previous kernel drains
(programmatic dependent launch).  Each must still see all that was enqueued
before it: chains of solves and of other kernels that write their sources and
read their potentials, without a synchronisation in between, give bitwise
what the same steps give one at a time on a plan that records events between
its passes, which keeps them from overlapping."""
import numpy as np
import pytest

from paper_1106_0557_gb300 import native

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

TDT = {"f32": torch.float32, "f64": torch.float64, "df64": torch.float64}


def _chain(plan, src, steps, wait):
    x, outs = src.clone(), []
    for k in range(steps):
        x.mul_(0.5).add_(src, alpha=1.0 / (k + 1))  # the source is written by a kernel just before the solve
        phi = plan.solve(x)
        if wait:
            torch.cuda.synchronize()
        outs.append(phi + 1.0)                       # ... and the potential read just after it
        x = plan.solve(phi, out=phi)                 # in place
        if wait:
            torch.cuda.synchronize()
    return outs + [x]


# one CTA per pass, ragged, several waves, the streamed y form, paired z tiles
@pytest.mark.parametrize("N,dtype,flags", [
    ((8, 8, 8), "f32", 0), ((37, 20, 13), "df64", 0), ((128, 96, 64), "f32", 0), ((40, 36, 24), "f64", 0),
    ((64, 256, 40), "f32", native.IPF_FLAG_Y_STREAM), ((20, 12, 1100), "f32", 0)])
def test_chained_solves_match_solves_one_at_a_time(N, dtype, flags):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1106_0557_gb300 import Plan
    g = np.random.default_rng(sum(N))
    src = torch.from_numpy(g.uniform(0.0, 1.0, (N[2], N[1], N[0]))).to("cuda", TDT[dtype])
    with Plan(N, (1.0, 0.5, 1.0), dtype, flags=flags | native.IPF_FLAG_PASS_EVENTS) as p:
        want = _chain(p, src, 6, wait=True)
    with Plan(N, (1.0, 0.5, 1.0), dtype, flags=flags) as p:
        for _ in range(3):
            got = _chain(p, src, 6, wait=False)
            torch.cuda.synchronize()
            assert all(torch.equal(a, b) for a, b in zip(got, want))
        p.check()


def test_host_solves_in_flight_match_solves_without_overlap():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1106_0557_gb300 import Plan
    N, h = (60, 44, 37), (1.0, 0.5, 1.0)
    g = np.random.default_rng(3)
    srcs = [torch.from_numpy(g.uniform(0.0, 1.0, (N[2], N[1], N[0])).astype(np.float32)).pin_memory() for _ in range(6)]
    outs = [torch.empty_like(s).pin_memory() for s in srcs]
    with Plan(N, h, "f32", flags=native.IPF_FLAG_PASS_EVENTS) as p:
        want = [p.solve(s.cuda()).cpu() for s in srcs]
    with Plan(N, h, "f32") as p:
        for s, o in zip(srcs, outs):  # uploads, passes and downloads of neighbours overlap
            p.solve_host_async(s, o)
        p.host_wait()
        assert all(torch.equal(a, b) for a, b in zip(outs, want))
        for s, w in zip(srcs, want):  # eight chunks each
            assert np.array_equal(p.solve_host(s.numpy()), w.numpy())
