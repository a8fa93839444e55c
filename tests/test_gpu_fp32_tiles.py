"""GPU: FP32 blocks over every arrangement of low targets, against the oracle.

k = 5 and 6 run register tiles over shared-memory tiles of 64 groups (n >= k + 6): one tile, several
tiles a CTA, bit 0 a target or not, targets on any of bits 1-3 (which the tile's swizzle feeds from
higher bits), n one below the rule (the tiled kernel).  k <= 4 exchange their targets below bit 5
through shared memory (n >= k + 5): every number of them.  FP32 sums of 2^k complex products keep the
FP32 bound of the repository, ‖Δψ‖₂ <= 1e-5.
"""
import itertools

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


def check(pkg, oracle_mod, n, targets, seed):
    psi = si.random_state(n, seed)
    u = si.random_unitary(len(targets), seed + 1)
    h = pkg.sim_create(n)
    try:
        pkg.sim_load_amplitudes(h, psi)
        pkg.sim_apply_fused(h, targets, u, precision=pkg.SIM_FP32)
        got = pkg.sim_amplitudes(h, dtype=pkg.SIM_C128)
    finally:
        pkg.sim_destroy(h)
    want = psi.astype(np.complex128)
    oracle_mod.apply_kq(want, targets, u)
    err = np.linalg.norm(got - want)
    assert err <= 1e-5, (n, targets, err)


WIDE = [(10, [9, 3, 0, 5, 7]), (11, [0, 1, 2, 3, 4]), (11, [6, 10, 8, 7, 9]), (12, [1, 2, 3, 9, 11]), (13, [0, 12, 6, 4, 9]),
        (14, [2, 13, 5, 7, 3]), (18, [17, 1, 9, 12, 3]), (21, [0, 2, 20, 11, 15]), (22, [21, 5, 13, 8, 17]),
        (11, [0, 2, 4, 6, 8, 10]), (12, [0, 1, 2, 3, 4, 5]), (12, [11, 10, 9, 8, 7, 6]), (13, [3, 12, 1, 7, 5, 9]),
        (15, [14, 2, 8, 0, 11, 5]), (20, [1, 19, 3, 7, 16, 12]), (22, [21, 16, 12, 10, 9, 8])]


@pytest.mark.parametrize("n,targets", WIDE)
def test_wide_blocks(pkg, oracle_mod, n, targets):
    check(pkg, oracle_mod, n, targets, seed=n)


@pytest.mark.parametrize("k", [1, 2, 3, 4])
@pytest.mark.parametrize("n", [9, 16])
def test_every_set_of_low_targets(pkg, oracle_mod, n, k):
    for j in range(1, k + 1):
        for low in itertools.combinations(range(5), j):
            high = list(range(n - 1, n - 1 - (k - j), -1))
            targets = high + list(reversed(low))
            check(pkg, oracle_mod, n, targets, seed=100 * j + sum(low))


@pytest.mark.parametrize("k,n", [(k, n) for k in (5, 6) for n in range(k, k + 6)])
def test_wide_blocks_of_a_small_state(pkg, oracle_mod, k, n):
    # one CTA: from one group, whose rows 8 or 16 threads share, to 32 groups
    rng = np.random.default_rng(n)
    for seed in range(3):
        check(pkg, oracle_mod, n, [int(q) for q in rng.permutation(n)[:k]], seed=10 * n + seed)
