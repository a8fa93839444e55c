"""GPU: the tensor-map permutation pipeline where its producer looks at many tiles in a turn, bit-exact.

The number of candidate tiles a turn grows with the state: 4 at 25 qubits, 32 at 28 where tiles move in
pairs (in place 4 at most).  Each amplitude holds its own index; the check runs on the device.
"""
import random

import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pkg():
    from paper_1910_09534_gb300 import build
    build.build()
    import paper_1910_09534_gb300 as p
    return p


def swaps(n, pairs):
    p = list(range(n))
    for a, b in pairs:
        p[a], p[b] = b, a
    return p


KINDS = {
    "high_and_low_4": lambda n: swaps(n, [(n - 1, n - 7), (n - 2, n - 9)] + [(i, n - 3 - i) for i in range(4)]),
    "high_5_low_5": lambda n: swaps(n, [(n - 1 - i, n - 11 - i) for i in range(5)] + [(i, n - 6 - i) for i in range(5)]),
    "high_1_low_1": lambda n: swaps(n, [(12, 18), (2, 15)]),
    "low_5": lambda n: swaps(n, [(i, n - 1 - i) for i in range(5)]),
    "reverse": lambda n: list(range(n))[::-1],
    "random_0": lambda n: random.Random(n).sample(range(n), n),
    "random_1": lambda n: random.Random(n + 1).sample(range(n), n),
}


@pytest.mark.parametrize("kind", sorted(KINDS))
@pytest.mark.parametrize("n", [25, 28])
def test_many_candidates_a_turn(pkg, n, kind):
    import torch
    perm = KINDS[kind](n)
    psi = torch.empty(1 << n, 2, dtype=torch.float32, device="cuda")
    torch.cuda.synchronize()
    h = pkg.sim_create(n, ext_state=psi.data_ptr(), ext_bytes=8 << n)
    try:
        pkg.sim_sync(h)  # |0..0> written
        step = 1 << 22
        low = torch.arange(step, device="cuda")
        for first in range(0, 1 << n, step):
            psi[first:first + step, 0] = low + (first & 0x7fffff)  # below 2^23: exact in FP32
            psi[first:first + step, 1] = first >> 23
        torch.cuda.synchronize()
        pkg.sim_permute(h, perm)
        pkg.sim_sync(h)  # a bounded wait that ran out would be reported here
        for first in range(0, 1 << n, step):
            index = first + low
            source = torch.zeros_like(index)
            for q, p in enumerate(perm):
                source |= ((index >> p) & 1) << q
            assert torch.equal(psi[first:first + step, 0], (source & 0x7fffff).float()), (kind, first)
            assert torch.equal(psi[first:first + step, 1], (source >> 23).float()), (kind, first)
    finally:
        pkg.sim_destroy(h)
