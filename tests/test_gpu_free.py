"""The float32 products without the wall, packed kernel and tile sums, against the oracle."""
import numpy as np
import pytest

import oracle as O
from paper_1612_00474_gb300 import inputs

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


def _dev(x):
    return torch.tensor(inputs.to_soa(x), dtype=torch.float64, device="cuda")


# the scalar kernel's last size and the packed one's first (one sphere in the last tile, half a tile, a whole
# one, one short of it); chunks of two and three tiles with a short last chunk; tile sums and (from 39 rows
# of tiles) chunks
@pytest.mark.parametrize("N", [2048, 2049, 2112, 2113, 2176, 2303, 3001, 4200, 4865, 5000])
@pytest.mark.parametrize("torque", [False, True])
def test_against_oracle(gpu_lib, N, torque):
    pos, F = inputs.monolayer(N, seed=3), inputs.vectors(N, 1)
    pos[1] = pos[0] + [0.3, 0.2, 0.1]  # overlapping, and coincident
    pos[N - 1] = pos[2]
    T = inputs.vectors(N, 2) if torque else None
    ctx = gpu_lib.Context(max_N=N, precision="fp32", max_iter=2, wall=False)
    try:
        U = ctx.mobility_apply(_dev(pos), _dev(F), None if T is None else _dev(T))
        again = ctx.mobility_apply(_dev(pos), _dev(F), None if T is None else _dev(T))
    finally:
        ctx.close()
    assert torch.equal(U, again)
    got = inputs.from_soa(U.cpu().numpy(), N)
    for r0, r1 in ((0, 130), (max(N - 130, 0), N)):
        ref = O.mobility_apply(pos, F, T, wall=False, rows=(r0, r1))
        assert O.rel_err(got[r0:r1], ref) <= 1e-5  # the float32 path's bound
