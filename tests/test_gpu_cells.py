"""Steric forces by cell lists: lists longer than a group's queue, the range of the exponential, batches whose
suspensions share cells, against the oracle and the single-suspension path."""
import numpy as np
import pytest

import oracle as O
from paper_1612_00474_gb300 import inputs

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


def _dev(x):
    return torch.tensor(inputs.to_soa(x), dtype=torch.float64, device="cuda")


def _heap(N, many, seed):
    """A monolayer whose first `many` spheres sit in one small heap, two of them coincident."""
    pos = inputs.monolayer(N, seed=seed)
    rng = np.random.default_rng(seed)
    pos[:many] = pos[0] + rng.uniform(0.0, 2.5, (many, 3))
    if many > 1:
        pos[1] = pos[0]
    return pos


# lists of the queue's length and one more, of several queues, of the fullest bucket and beyond; b from contacts
# far apart (exponents beyond the short form's range) to a repulsion over many cells of neighbours
@pytest.mark.parametrize("N,many,b", [(4096, 65, 0.1), (4097, 40, 0.1), (8193, 61, 0.1), (8193, 64, 0.1), (8193, 65, 0.1),
                                      (9001, 400, 0.1), (9001, 513, 0.1), (300, 40, 1e-5), (9000, 40, 1e-5),
                                      (300, 3, 0.7), (9000, 3, 0.7)])
def test_single(gpu_lib, N, many, b):
    pos = _heap(N, many, 21)
    ctx = gpu_lib.Context(max_N=N, precision="fp32", max_iter=2)
    try:
        F = ctx.forces(_dev(pos), b=b)
        assert torch.equal(F, ctx.forces(_dev(pos), b=b))
    finally:
        ctx.close()
    R = O.forces(pos, b=b)
    # sums of float64 terms, each with the rounding of (2a - r) / b in its exponent
    tol = 1e-12 + 8 * 2.0 ** -52 * 2.0 / b
    assert np.max(np.abs(inputs.from_soa(F.cpu().numpy(), N) - R)) <= tol * np.max(np.abs(R))


def test_batch_shares_cells(gpu_lib):
    """Suspensions on top of one another, dense ones among them: each velocity is the single path's, and bit for bit
    the same beside other companions."""
    sizes, many = [300, 64, 1, 1500, 130, 700], [200, 64, 1, 90, 2, 0]
    pos = [_heap(N, m, 30 + k) for k, (N, m) in enumerate(zip(sizes, many))]
    bt = gpu_lib.BatchContext(max_total_N=sum(sizes), max_B=len(sizes), precision="fp64", max_iter=32)
    ctx = gpu_lib.Context(max_N=max(sizes), precision="fp64", max_iter=32)

    def step(which):
        q, U = [_dev(pos[k]) for k in which], [torch.zeros(3 * sizes[k], dtype=torch.float64, device="cuda") for k in which]
        bt.ab_step(q, U, [0] * len(which), [5 + k for k in which], dt=1e-3, delta=1e-6, tol=1e-3)
        return U

    try:
        U = step(range(len(sizes)))
        alone = step([3])[0]
        for k, N in enumerate(sizes):
            qs, Us = _dev(pos[k]), torch.zeros(3 * N, dtype=torch.float64, device="cuda")
            ctx.ab_step(qs, Us, 0, 5 + k, dt=1e-3, delta=1e-6, tol=1e-3)
            # the batch takes pairs beyond 2a + 20 b in float32: 1e-14 U0 / b
            assert float((U[k] - Us).norm()) <= 1e-10 * float(Us.norm()), k
    finally:
        bt.close()
        ctx.close()
    assert torch.equal(U[3], alone)
