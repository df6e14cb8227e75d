"""The pseudo-periodic float32 product of small cells, a cluster of blocks per tile, against the oracle."""
import numpy as np
import pytest

import oracle as O
from paper_1612_00474_gb300 import inputs

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


def _dev(x):
    return torch.tensor(inputs.to_soa(x), dtype=torch.float64, device="cuda")


# a last tile of one sphere, of an odd number, of a step of sources and one more, a whole one; the largest cell
# of the rule (55 tiles at 152 SMs) and the first beyond it
@pytest.mark.parametrize("N", [256, 257, 263, 264, 265, 300, 383, 384, 700, 1280, 1281])
@pytest.mark.parametrize("torque", [False, True])
def test_against_oracle(gpu_lib, N, torque):
    L = float(np.sqrt(N * np.pi / 0.25))
    pos, F = inputs.monolayer(N, seed=3), inputs.vectors(N, 1)
    pos[:, :2] = np.random.default_rng(5).uniform(0.0, L, (N, 2))  # overlapping pairs, also across the borders
    pos[N - 1] = pos[0]  # coincident, in different tiles
    pos[2, 2], pos[N // 2, 2] = 0.4, -0.2
    T = inputs.vectors(N, 2) if torque else None
    ctx = gpu_lib.Context(max_N=N, precision="fp32", max_iter=2)
    try:
        ctx.set_periodic(L, 1.1 * L)
        U = ctx.mobility_apply(_dev(pos), _dev(F), None if T is None else _dev(T))
        again = ctx.mobility_apply(_dev(pos), _dev(F), None if T is None else _dev(T))
    finally:
        ctx.close()
    assert torch.equal(U, again)
    ref = O.mobility_apply(pos, F, T, periodic=(L, 1.1 * L))
    assert O.rel_err(inputs.from_soa(U.cpu().numpy(), N), ref) <= 1e-5  # the float32 path's bound
