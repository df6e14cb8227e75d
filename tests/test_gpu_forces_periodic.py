"""Steric forces of large pseudo-periodic cells: right in both kernels' ranges, and no step in their cost at 8192 spheres,
from where on the slower of the two took them."""
import math

import numpy as np
import pytest

import oracle as O
from paper_1612_00474_gb300 import inputs

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


def _cell(gpu_lib, N):
    L = math.sqrt(N * math.pi / 0.25)
    pos = inputs.monolayer(N, seed=21)
    pos[:, :2] *= math.sqrt(0.4 / 0.25)  # the cell's area fraction: as many near pairs at every N
    ctx = gpu_lib.Context(max_N=N, precision="fp32", max_iter=2)
    ctx.set_periodic(L, L)
    return ctx, torch.tensor(inputs.to_soa(pos), dtype=torch.float64, device="cuda"), pos, L


@pytest.mark.parametrize("N", [8192, 8193, 10007, 40000, 40001])
def test_against_oracle(gpu_lib, N):
    ctx, q, pos, L = _cell(gpu_lib, N)
    try:
        F = inputs.from_soa(ctx.forces(q).cpu().numpy(), N)
    finally:
        ctx.close()
    R = O.forces(pos, periodic=(L, L))
    # float64 sums of a few hundred terms of the size of the largest force, and the cut-off's e^-40
    assert np.max(np.abs(F - R)) <= 1e-12 * np.max(np.abs(R))


def test_cost_grows_with_the_pairs(gpu_lib):
    """One sphere more costs one sphere more."""
    times = {}
    for N in (8192, 8193):
        ctx, q, _, _ = _cell(gpu_lib, N)
        try:
            out, best = torch.empty_like(q), []
            for _ in range(12):
                a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
                a.record()
                for _ in range(5):
                    ctx.forces(q, out=out)
                b.record()
                torch.cuda.synchronize()
                best.append(a.elapsed_time(b))
            times[N] = min(best)
        finally:
            ctx.close()
    assert times[8193] <= 1.5 * times[8192]
