"""GPU: qubit-bit permutations through each kernel that an involution pass can take, bit-exact.

In-place tiles of at most 3 row bits (bulk copies), tile pairs and tiles of 4-5 row bits (the
tensor-map pipeline: rows next to each other and apart, so that a tile takes 1, 2 or 4 copies; tiles of
2^9, 2^10 and 2^11 amplitudes), states below 2^11 amplitudes (thread copies), whole random
permutations, and two handles permuting at once.
"""
import numpy as np
import pytest

import syc_inputs as si

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
        p[a], p[b] = p[b], p[a]
    return p


def permuted(psi, perm):
    i = np.arange(psi.size)
    j = np.zeros_like(i)
    for q, b in enumerate(perm):
        j |= ((i >> q) & 1) << b
    out = np.empty_like(psi)
    out[j] = psi
    return out


def check(pkg, n, perm, seed):
    psi = si.random_state(n, seed)
    h = pkg.sim_create(n)
    try:
        pkg.sim_load_amplitudes(h, psi)
        pkg.sim_permute(h, perm)
        got = pkg.sim_amplitudes(h, physical_order=True)
        pkg.sim_sync(h)  # a bounded wait that ran out would be reported here
    finally:
        pkg.sim_destroy(h)
    assert np.array_equal(got.view(np.uint32), permuted(psi, perm).view(np.uint32)), (n, perm)


KINDS = {
    "low_low": lambda n: [(0, 3), (1, 4)],
    "low_1": lambda n: [(2, n - 1)],
    "low_3": lambda n: [(0, n - 3), (1, n - 2), (2, n - 1)],
    "low_4": lambda n: [(i, n - 4 + i) for i in range(4)],
    "low_5": lambda n: [(i, n - 5 + i) for i in range(5)],
    "high_1": lambda n: [(n - 2, n - 1)],
    "reverse": lambda n: [(i, n - 1 - i) for i in range(n // 2)],
    "mixed": lambda n: [(0, 7), (4, 9), (5, n - 1), (6, n - 2)],
    "apart": lambda n: [(0, 6), (1, 8), (2, 10), (3, n - 1), (5, 9)],
}


@pytest.mark.parametrize("kind", KINDS)
@pytest.mark.parametrize("n", [10, 11, 12, 14, 19, 22])
def test_one_involution(pkg, n, kind):
    pairs = [(a, b) for a, b in KINDS[kind](n) if a != b]
    flat = [x for ab in pairs for x in ab]
    if len(set(flat)) != len(flat) or min(flat) < 0:
        pytest.skip("not an involution at this size")
    check(pkg, n, swaps(n, pairs), seed=n)


def test_rows_apart_four_copies_a_tile(pkg):
    # five row bits, none next to another, and high pairs: two tile bits are looped over
    check(pkg, 20, swaps(20, [(0, 7), (1, 9), (2, 11), (3, 13), (4, 15), (6, 19), (8, 18)]), seed=20)


@pytest.mark.parametrize("n", [5, 9, 11, 13, 16, 18, 21, 23])
def test_random(pkg, n):
    for seed in range(6):
        check(pkg, n, si.random_permutation(n, 100 * n + seed), seed)


def test_two_handles_at_once(pkg):
    n = 20
    perms = [si.random_permutation(n, s) for s in (1, 2)]
    psis = [si.random_state(n, s) for s in (3, 4)]
    hs = [pkg.sim_create(n) for _ in perms]
    try:
        for h, psi in zip(hs, psis):
            pkg.sim_load_amplitudes(h, psi)
        want = list(psis)
        for _ in range(10):
            for i, h in enumerate(hs):
                pkg.sim_set_layout(h, list(range(n)))
                pkg.sim_permute(h, perms[i])
                want[i] = permuted(want[i], perms[i])
        for h, w in zip(hs, want):
            assert np.array_equal(pkg.sim_amplitudes(h, physical_order=True), w)
    finally:
        for h in hs:
            pkg.sim_destroy(h)
