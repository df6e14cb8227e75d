"""Device memory of float64 contexts: the pairs' blocks are taken by the first Lanczos solve that reads them, for its own
size, and a solve gives the same bits in every context that holds them."""
import gc

import pytest

from paper_1612_00474_gb300 import inputs

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

MB = 1 << 20


def _dev(x):
    return torch.tensor(inputs.to_soa(x), dtype=torch.float64, device="cuda")


def _used():
    gc.collect()  # contexts that earlier tests left behind
    torch.cuda.synchronize()
    free, total = torch.cuda.mem_get_info()
    return total - free


def _blocks(N):
    nb = -(-N // 32)
    return nb * (nb + 1) // 2 * 1024 * 64


def _solve(ctx, N):
    return ctx.lanczos_sqrt_apply(_dev(inputs.monolayer(N, seed=2)), _dev(inputs.vectors(N, 3)), tol=1e-3)[0]


def _alone(gpu_lib, N):
    ctx = gpu_lib.Context(max_N=N, precision="fp64", max_iter=20)
    try:
        return _solve(ctx, N)
    finally:
        ctx.close()


def test_only_solves_that_read_them(gpu_lib):
    N = 8192  # blocks of 2.1 GB
    pos, F = _dev(inputs.monolayer(700, seed=1)), _dev(inputs.vectors(700, 1))
    ref = _alone(gpu_lib, 700)
    assert torch.equal(ref, ref.clone())  # the comparison's own kernels are loaded before memory is counted
    before = _used()
    ctx = gpu_lib.Context(max_N=N, precision="fp64", max_iter=20)
    try:
        ctx.mobility_apply(pos, F)
        ctx.forces(pos)
        ctx.rfd_drift(pos, F)
        ctx.set_periodic(200.0, 200.0)
        ctx.lanczos_sqrt_apply(pos, F, tol=1e-3)
        ctx.set_periodic(0.0, 0.0)
        ctx.lanczos_sqrt_apply(pos, F, tol=0.0, max_iter=1, raise_on_noconv=False)
        plain = _used() - before
        assert plain < 300 * MB
        g = _solve(ctx, 700)
        assert torch.equal(g, ref)
        assert _used() - before < plain + _blocks(700) + 64 * MB
    finally:
        ctx.close()
    assert _used() - before < 64 * MB


def test_sized_by_the_solve(gpu_lib):
    """Solves of growing and shrinking sizes in a context too large for all of its pairs' blocks (17000 spheres)."""
    sizes = (500, 3000, 600, 3100, 4096, 33)
    refs = [_alone(gpu_lib, N) for N in sizes]
    before = _used()
    ctx = gpu_lib.Context(max_N=17000, precision="fp64", max_iter=20)
    try:
        plain = _used()
        for N, ref in zip(sizes, refs):
            assert torch.equal(_solve(ctx, N), ref)
        taken = _used() - plain
        assert _blocks(4096) <= taken + 2 * MB and taken < 2 * _blocks(4096)
    finally:
        ctx.close()
    assert _used() - before < 64 * MB
