"""The float64 symmetric pass against the one-way kernels (the row-range product) and the oracle."""
import numpy as np
import pytest

import oracle as O
from paper_1612_00474_gb300 import inputs

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


def _dev(x):
    return torch.tensor(inputs.to_soa(x), dtype=torch.float64, device="cuda")


def _config(N):
    """A monolayer with spheres in the wall, below it, overlapping and coincident."""
    pos = inputs.monolayer(N, seed=7)
    if N > 3:
        pos[1] = pos[0]
        pos[2] = pos[0] + [1.1, 0.4, 0.2]
        pos[3, 2] = 0.4
        pos[N // 2, 2] = -0.2
    return pos


# tile edges, one run a row and several, units shared by 8, 4, 2 and 1 CTAs
@pytest.mark.parametrize("N", [1, 2, 31, 32, 33, 64, 65, 100, 257, 300, 520, 1000, 2049])
@pytest.mark.parametrize("wall", [True, False])
@pytest.mark.parametrize("torque", [True, False])
def test_against_one_way(gpu_lib, N, wall, torque):
    pos, F = _dev(_config(N)), _dev(inputs.vectors(N, 1))
    T = _dev(inputs.vectors(N, 2)) if torque else None
    ctx = gpu_lib.Context(max_N=N + 5, precision="fp64", max_iter=2, wall=wall)
    try:
        U = ctx.mobility_apply(pos, F, T)
        R = ctx.mobility_apply_rows(pos, F, T, 0, N)
        again = ctx.mobility_apply(pos, F, T)
    finally:
        ctx.close()
    assert torch.equal(U, again)
    # sums of N float64 terms in another order: N eps at most, far less in the norm
    assert float((U - R).norm()) <= 1e-14 * float(R.norm())


def test_against_oracle_long_rows(gpu_lib):
    """More tiles than runs of one tile: every row in several runs (a context of 4600 spheres)."""
    N = 4600
    pos, F, T = _config(N), inputs.vectors(N, 1), inputs.vectors(N, 2)
    ctx = gpu_lib.Context(max_N=N, precision="fp64", max_iter=2)
    try:
        U = inputs.from_soa(ctx.mobility_apply(_dev(pos), _dev(F), _dev(T)).cpu().numpy(), N)
    finally:
        ctx.close()
    rows = (4096, N)
    assert O.rel_err(U[rows[0]:], O.mobility_apply(pos, F, T, rows=rows)) <= 1e-10  # the float64 path's bound


def test_not_finite(gpu_lib):
    """A position that is not a number reaches the whole product, an infinite force every sphere, as one-way."""
    N = 70
    pos, F = _dev(inputs.monolayer(N, seed=8)), _dev(inputs.vectors(N, 1))
    ctx = gpu_lib.Context(max_N=N, precision="fp64", max_iter=2)
    try:
        for v, k, bad in ((pos, 40, float("nan")), (F, 69, float("inf"))):
            x = v.clone()
            x[k] = bad
            args = (x, F) if v is pos else (pos, x)
            U, R = ctx.mobility_apply(*args), ctx.mobility_apply_rows(*args, None, 0, N)
            assert torch.equal(torch.isfinite(U), torch.isfinite(R))
    finally:
        ctx.close()


# the products of a solve after the first read the blocks that it stored
@pytest.mark.parametrize("N", [1, 2, 31, 33, 64, 100, 300, 1000])
@pytest.mark.parametrize("wall", [True, False])
def test_lanczos_from_stored_blocks(gpu_lib, N, wall):
    pos, W = _config(N), inputs.vectors(N, 3)
    ctx = gpu_lib.Context(max_N=N + 40, precision="fp64", max_iter=16, wall=wall)
    try:
        ctx.lanczos_sqrt_apply(_dev(inputs.monolayer(N, seed=1)), _dev(W), tol=0.0, max_iter=3, raise_on_noconv=False)
        g, m, _, _ = ctx.lanczos_sqrt_apply(_dev(pos), _dev(W), tol=0.0, max_iter=5, raise_on_noconv=False)
    finally:
        ctx.close()
    ref, mr, _, _ = O.lanczos_sqrt(pos, W, exact_iters=5, wall=wall)
    assert m == mr and O.rel_err(inputs.from_soa(g.cpu().numpy(), N), ref) <= 1e-10  # the float64 path's bound
