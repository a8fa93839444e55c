"""GPU: the contraction at the edges of its tiles.

Sides below, at and above the tiles of the FP32 and the tensor-core kernel, more tiles than CTAs
run at a time, one to 64 entanglement values (less than, one and several staged chunks), into the
identity and into a permuted layout; against the oracle's plain simulation, within the bound that
the other contractions are held to.
"""
import random

import numpy as np
import pytest

pytestmark = pytest.mark.gpu
TOL = 1e-5


@pytest.fixture(scope="module")
def pkg():
    from paper_1910_09534_gb300 import build
    build.build()
    import paper_1910_09534_gb300 as p
    return p


def bridged(n1, n2, pairs, rng):
    """Single-qubit layers around `pairs` fSim gates that bridge the sides."""
    n, gates, prev = n1 + n2, [], {}

    def layer():
        for q in range(n):
            prev[q] = rng.choice([g for g in range(3) if g != prev.get(q)])
            gates.append((prev[q], q, -1, 0.0, 0.0))

    for i in range(pairs):
        layer()
        gates.append((3, (5 * i) % n1, n1 + (3 * i) % n2, rng.uniform(0.3, 1.5), rng.uniform(0.1, 0.6)))
    layer()
    return gates


@pytest.mark.parametrize("n1,n2", [(1, 1), (1, 8), (9, 1), (5, 7), (6, 6), (7, 7), (8, 9), (12, 9), (9, 12)])
@pytest.mark.parametrize("pairs", [0, 1, 2, 3])
def test_contraction_at_tile_edges(pkg, oracle_mod, n1, n2, pairs):
    n = n1 + n2
    rng = random.Random(100 * n1 + 10 * n2 + pairs)
    gates = bridged(n1, n2, pairs, rng)
    want = oracle_mod.run_circuit(gates, n_qubits=n)
    perm = list(range(n))
    rng.shuffle(perm)
    s = pkg.sim_split_create(n, pkg.gates_array(gates), [0] * n1 + [1] * n2)
    try:
        _, n_wires, n_pairs, _ = pkg.sim_split_info(s)
        assert n_pairs == pairs
        for precision in (pkg.SIM_FP32, pkg.SIM_FP16X3_TMEM):
            for layout in (None, perm):
                hs = [pkg.sim_create(w) for w in n_wires] + [pkg.sim_create(n)]
                try:
                    for t in range(2):
                        plan = pkg.sim_plan_create(n_wires[t], pkg.sim_split_gates(s, t), kmax=4,
                                                   precision=pkg.SIM_FP32)
                        pkg.sim_apply_plan(hs[t], plan)
                        pkg.sim_plan_destroy(plan)
                    if layout:
                        pkg.sim_set_layout(hs[2], layout)
                    pkg.sim_contract(hs[2], hs[0], hs[1], s, precision)
                    got = pkg.sim_amplitudes(hs[2])
                finally:
                    for h in hs:
                        pkg.sim_destroy(h)
                assert np.linalg.norm(got.astype(np.complex128) - want) <= TOL, (precision, layout)
    finally:
        pkg.sim_split_destroy(s)
