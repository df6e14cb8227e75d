"""The tridiagonal square root of the Lanczos step on the GPU: dimensions at the edges of its row blocks, and
mobilities that are only semi-definite (the eigen-decomposition path)."""
import numpy as np
import pytest

import oracle as O
from paper_1612_00474_gb300 import inputs

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


def _dev(x):
    return torch.tensor(inputs.to_soa(x), dtype=torch.float64, device="cuda")


@pytest.mark.parametrize("m", [1, 2, 15, 16, 17, 32, 33, 48, 64])
def test_forced_dimension(gpu_lib, m):
    N = 40
    pos, W = inputs.monolayer(N, seed=3), inputs.vectors(N, 4)
    ctx = gpu_lib.Context(max_N=N, precision="fp64", max_iter=64)
    try:
        g, it, _, _ = ctx.lanczos_sqrt_apply(_dev(pos), _dev(W), tol=0.0, max_iter=m, raise_on_noconv=False)
    finally:
        ctx.close()
    ref, mr, _, _ = O.lanczos_sqrt(pos, W, exact_iters=m)
    assert it == mr
    assert O.rel_err(inputs.from_soa(g.cpu().numpy(), N), ref) <= 1e-10  # the float64 path's bound


@pytest.mark.parametrize("precision,tol", [("fp64", 1e-6), ("fp32", 3e-3)])
def test_semi_definite(gpu_lib, precision, tol):
    """Spheres in coincident pairs and some below the wall: half of the spectrum is zero.  A zero eigenvalue
    that rounding moves by r leaves sqrt(r) in the result: 1e-8 in float64, 1e-3.5 with float32 pairs,
    a few times that over the vector."""
    N = 60
    half = inputs.monolayer(N // 2, seed=5)
    half[:5, 2] = -0.3
    pos, W = np.concatenate([half, half]), inputs.vectors(N, 6)
    ctx = gpu_lib.Context(max_N=N, precision=precision, max_iter=64)
    try:
        g, _, _, _ = ctx.lanczos_sqrt_apply(_dev(pos), _dev(W), tol=1e-5, raise_on_noconv=False)
        gf, _, _, _ = ctx.lanczos_sqrt_apply(_dev(pos), _dev(W), tol=0.0, max_iter=64, raise_on_noconv=False)
    finally:
        ctx.close()
    e, Q = np.linalg.eigh(O.dense(pos)[0])
    ref = (Q @ (np.sqrt(np.maximum(e, 0.0)) * (Q.T @ W.ravel()))).reshape(N, 3)
    assert O.rel_err(inputs.from_soa(gf.cpu().numpy(), N), ref) <= tol
    assert O.rel_err(inputs.from_soa(g.cpu().numpy(), N), ref) <= max(tol, 1e-4)
