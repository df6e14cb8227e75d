"""A step against its parts called one by one, on both sides of the sizes up to which the drift runs beside the
Lanczos iterations (1024 spheres in float64, 4096 in float32)."""
import math

import pytest

from paper_1612_00474_gb300 import inputs

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision,N", [("fp64", 33), ("fp64", 1024), ("fp64", 1025), ("fp32", 200), ("fp32", 4096),
                                         ("fp32", 4097)])
@pytest.mark.parametrize("periodic", [False, True])
def test_step_is_its_parts(gpu_lib, precision, N, periodic):
    if periodic and N > 1100:
        pytest.skip("nine times the pair work")
    dt, seed, delta = 0.01, 9, 1e-4 if precision == "fp64" else 5e-3
    q0 = torch.tensor(inputs.to_soa(inputs.monolayer(N, seed=2)), dtype=torch.float64, device="cuda")
    ctx = gpu_lib.Context(max_N=N + 3, precision=precision, max_iter=32)
    try:
        if periodic:
            L = math.sqrt(N * math.pi / 0.4) + 5.0
            ctx.set_periodic(L, L)
        q, U = q0.clone(), torch.zeros_like(q0)
        for k in range(3):  # the same step again and again: nothing is left over from one to the next
            q.copy_(q0)
            st = ctx.ab_step(q, U, 0, seed, dt=dt, delta=delta, tol=1e-3)
        T = torch.zeros_like(q0)
        T[N:2 * N] = 1.0
        Un = ctx.mobility_apply(q0, ctx.forces(q0), T)
        g, m, _, _ = ctx.lanczos_sqrt_apply(q0, ctx.philox_normal(N, seed, 0, 0), tol=1e-3)
        d = ctx.rfd_drift(q0, ctx.philox_normal(N, seed, 0, 1), delta=delta)
    finally:
        ctx.close()
    assert st["m"] == m
    # the same kernels on the same inputs, up to the order of float64 sums; a float32 step of 256 spheres and more
    # takes the velocity and the first Lanczos product in one pass, whose float32 rounding is its own (a product's
    # relative rounding is below 1e-6)
    shared = precision == "fp32" and N >= 256 and not periodic
    assert float((U - Un).abs().max()) <= (1e-6 if shared else 1e-12) * float(Un.abs().max())
    ref = dt * Un + math.sqrt(2.0 * dt) * g + dt * d
    # the drift amplifies a product's rounding by 1/delta
    bound = 1e-6 if shared else 1e-11 + 1e-15 / delta
    assert float((q - q0 - ref).abs().max()) <= bound * float(ref.abs().max())
