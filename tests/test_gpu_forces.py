"""Steric forces at the edges of the two kernels' ranges: all pairs by groups of sixteen spheres and chunks of 1024
sources up to 4096 spheres (8192 pseudo-periodic), hashed cells beyond, and its all-pairs fallback."""
import math

import numpy as np
import pytest

import oracle as O
from paper_1612_00474_gb300 import inputs

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


def _forces(gpu_lib, pos, period=None):
    N = pos.shape[0]
    ctx = gpu_lib.Context(max_N=N, precision="fp32", max_iter=2)
    try:
        if period:
            ctx.set_periodic(period, period)
        q = torch.tensor(inputs.to_soa(pos), dtype=torch.float64, device="cuda")
        F, G = ctx.forces(q), ctx.forces(q)
        assert torch.equal(F, G)
        return inputs.from_soa(F.cpu().numpy(), N)
    finally:
        ctx.close()


def _close(F, R):
    # float64 sums of a few hundred terms of the size of the largest force, and the cut-off's e^-40
    assert np.max(np.abs(F - R)) <= 1e-12 * np.max(np.abs(R))


def _dense(N, many):
    """A monolayer whose first `many` spheres sit in one small heap (lists of the whole chunk)."""
    pos = inputs.monolayer(N, seed=11)
    rng = np.random.default_rng(1)
    pos[:many] = pos[0] + rng.uniform(0.0, 1.5, (many, 3))
    if many > 1:
        pos[1] = pos[0]
    return pos


@pytest.mark.parametrize("N,many", [(1, 0), (2, 2), (15, 4), (16, 16), (17, 17), (257, 200), (1023, 0), (1024, 1024),
                                    (1025, 1025), (2050, 300), (8192, 40), (8193, 40), (9000, 700)])
def test_open(gpu_lib, N, many):
    pos = _dense(N, many)
    _close(_forces(gpu_lib, pos), O.forces(pos))


@pytest.mark.parametrize("N,many", [(1, 0), (16, 4), (33, 33), (1025, 200), (8300, 30)])
def test_periodic(gpu_lib, N, many):
    L = max(5.0, math.sqrt(N * math.pi / 0.4))
    pos = _dense(N, many)
    pos[:, 0] += 3.0 * L
    _close(_forces(gpu_lib, pos, L), O.forces(pos, periodic=(L, L)))


def test_far_clusters_share_buckets(gpu_lib):
    """Clusters many grid periods apart fall into the same hashed buckets."""
    pos = inputs.monolayer(9000, seed=12)
    pos[3000:6000, 0] += 256 * 6.07 * 40
    pos[6000:, 1] -= 256 * 6.07 * 77
    _close(_forces(gpu_lib, pos), O.forces(pos))
