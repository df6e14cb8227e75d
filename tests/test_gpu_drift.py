"""A drift's two products on two streams: calls enqueued one after another, on buffers that are written again between
them, give what calls with a synchronisation around each give, bit for bit."""
import pytest

from paper_1612_00474_gb300 import inputs

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


# one-way and symmetric products of both precisions, the largest float64 size beside and the first alone, several
# waves of blocks
@pytest.mark.parametrize("N,precision,wall,period", [(100, "fp32", True, 0.0), (300, "fp32", True, 90.0), (3001, "fp32", False, 0.0),
                                                     (5000, "fp32", True, 0.0), (1024, "fp64", True, 0.0),
                                                     (1025, "fp64", True, 0.0)])
def test_back_to_back(gpu_lib, N, precision, wall, period):
    def dev(x):
        return torch.tensor(inputs.to_soa(x), dtype=torch.float64, device="cuda")

    pos = [dev(inputs.monolayer(N, seed=k)) for k in range(4)]
    noise = [dev(inputs.vectors(N, 40 + k)) for k in range(4)]
    ctx = gpu_lib.Context(max_N=N, precision=precision, max_iter=2, wall=wall)
    try:
        if period:
            ctx.set_periodic(period, period)
        alone = []
        for p, w in zip(pos, noise):
            torch.cuda.synchronize()
            alone.append(ctx.rfd_drift(p, w, delta=5e-3).clone())
            torch.cuda.synchronize()
        stream = torch.cuda.Stream()
        stream.wait_stream(torch.cuda.current_stream())
        with torch.cuda.stream(stream):
            q, W, out = torch.empty_like(pos[0]), torch.empty_like(noise[0]), []
            for p, w in zip(pos, noise):
                q.copy_(p)
                W.copy_(w)
                out.append(ctx.rfd_drift(q, W, delta=5e-3))
            q.zero_()
            W.zero_()
        stream.synchronize()
    finally:
        ctx.close()
    for a, b in zip(alone, out):
        assert torch.equal(a, b)
