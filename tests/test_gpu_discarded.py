"""Products that a host-driven Lanczos solve enqueues ahead and discards: none on the routes that cannot leave early where
a product takes longer than the host's answers of a solve, and no error of a discarded one."""
import pytest

from paper_1612_00474_gb300 import inputs

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


def _dev(x):
    return torch.tensor(inputs.to_soa(x), dtype=torch.float64, device="cuda")


# float64 pseudo-periodic products evaluate every image and do not read the stop word: a solve that stops by itself
# launches what a solve of as many iterations does
@pytest.mark.parametrize("N", [300, 500, 830])
def test_periodic_float64_solve_discards_nothing(gpu_lib, N):
    pos, W = _dev(inputs.monolayer(N, seed=3)), _dev(inputs.vectors(N, 4))
    ctx = gpu_lib.Context(max_N=N, precision="fp64", max_iter=40)
    try:
        ctx.set_periodic(120.0, 120.0)
        counts = []
        _, m, _, _ = ctx.lanczos_sqrt_apply(pos, W, tol=1e-3)
        for kw in (dict(tol=1e-3), dict(tol=0.0, max_iter=m)):
            before = gpu_lib.launch_count()
            ctx.lanczos_sqrt_apply(pos, W, **kw)
            counts.append(gpu_lib.launch_count() - before)
    finally:
        ctx.close()
    assert counts[0] == counts[1]


# a caller's product: one call an iteration (for short ones, one more), and the error of a call that the solve does not
# need does not reach it
@pytest.mark.parametrize("N,precision,more", [(100, "fp64", 1), (300, "fp32", 1), (850, "fp64", 0), (2400, "fp64", 0)])
def test_hook_calls(gpu_lib, N, precision, more):
    pos, W = _dev(inputs.monolayer(N, seed=5)), _dev(inputs.vectors(N, 6))
    ctx = gpu_lib.Context(max_N=N, precision=precision, max_iter=40)
    inner = gpu_lib.Context(max_N=N, precision=precision, max_iter=2)
    calls, allowed = [], [40]

    def product(n, p, f, t, u):
        calls.append(n)
        if len(calls) > allowed[0]:
            return gpu_lib.RPB_ECUDA
        return gpu_lib.load().rpb_mobility_apply(inner._h, n, p, f or None, t or None, u)

    try:
        inner._bind_stream()
        ref, m, _, _ = ctx.lanczos_sqrt_apply(pos, W, tol=1e-3)
        ctx.set_product_hook(product)
        _, mh, _, _ = ctx.lanczos_sqrt_apply(pos, W, tol=1e-3)
        assert mh == m and len(calls) == m + more
        calls.clear()
        allowed[0] = m
        g, mh, _, _ = ctx.lanczos_sqrt_apply(pos, W, tol=1e-3)
        # the same products but for the roundings of stored and evaluated pairs
        assert mh == m and float((g - ref).norm()) <= (1e-10 if precision == "fp64" else 1e-5) * float(ref.norm())
        calls.clear()
        allowed[0] = m - 1
        with pytest.raises(gpu_lib.RpbError):  # the last one that it needs
            ctx.lanczos_sqrt_apply(pos, W, tol=1e-3)
        ctx.set_product_hook(None)
    finally:
        ctx.close()
        inner.close()
