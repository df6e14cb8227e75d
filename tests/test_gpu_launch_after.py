"""The kernels of a Lanczos iteration that start before the one ahead of them ends: solves and products enqueued back to
back, on buffers that are written again between them, give what calls with a synchronisation around each give, bit
for bit, at the edges of the sizes that do so."""
import pytest

from paper_1612_00474_gb300 import inputs

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,precision,period", [(256, "fp32", 0.0), (300, "fp32", 90.0), (1400, "fp32", 200.0),
                                                (4096, "fp32", 0.0), (4097, "fp32", 0.0), (33, "fp64", 0.0),
                                                (1000, "fp64", 0.0), (4096, "fp64", 0.0), (4097, "fp64", 0.0)])
def test_back_to_back(gpu_lib, N, precision, period):
    def dev(x):
        return torch.tensor(inputs.to_soa(x), dtype=torch.float64, device="cuda")

    pos = [dev(inputs.monolayer(N, seed=k)) for k in range(3)]
    vec = [dev(inputs.vectors(N, 40 + k)) for k in range(3)]
    ctx = gpu_lib.Context(max_N=N, precision=precision, max_iter=40)

    def calls(p, w):
        g, m, _, _ = ctx.lanczos_sqrt_apply(p, w, tol=1e-4)
        return g, ctx.mobility_apply(p, w), ctx.mobility_apply(p, w, w), m

    try:
        if period:
            ctx.set_periodic(period, period)
        alone = []
        for p, w in zip(pos, vec):
            torch.cuda.synchronize()
            alone.append(calls(p, w))
            torch.cuda.synchronize()
        q, W, out = torch.empty_like(pos[0]), torch.empty_like(vec[0]), []
        for p, w in zip(pos, vec):
            q.copy_(p)
            W.copy_(w)
            out.append(calls(q, W))
        q.zero_()
        W.zero_()
        torch.cuda.synchronize()
    finally:
        ctx.close()
    for a, b in zip(alone, out):
        assert a[3] == b[3]
        for x, y in zip(a[:3], b[:3]):
            assert torch.equal(x, y)
