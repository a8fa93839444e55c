"""GPU: plans on small states, applied by one thread-block cluster.

sim_apply_plan in FP32 on up to 15-17 qubits runs a plan's blocks on one cluster, several blocks a
launch (14 of 4 qubits, 3 of 5).  Its products are summed in the order of the kernels that
sim_apply_fused launches, so the two give the same amplitudes bit for bit: checked at states smaller
than a block's share per CTA, at the sizes where several threads share a group, above them, and at the
first sizes that take separate launches; and against the oracle (‖Δψ‖₂ <= 1e-5, FP32).
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


@pytest.mark.parametrize("n,kmax,cycles", [(2, 2, 3), (3, 2, 4), (4, 4, 8), (5, 5, 8), (6, 3, 8), (7, 5, 8), (9, 4, 10),
                                           (11, 5, 10), (12, 2, 8), (12, 4, 8), (13, 5, 16), (14, 4, 20), (15, 3, 8),
                                           (15, 5, 20), (16, 4, 12), (17, 5, 8), (17, 4, 8), (18, 5, 8)])
def test_same_amplitudes_as_one_launch_per_block(pkg, oracle_mod, n, kmax, cycles):
    circ = si.sycamore_circuit(si.near_square_grid(n), cycles, seed=n + kmax)
    plan = pkg.sim_plan_create(n, pkg.gates_array(circ), kmax=kmax)
    perm = [(q * 5 + 3) % n if n % 5 else (q + 2) % n for q in range(n)]  # not the identity layout
    blocks = [pkg.sim_plan_block(plan, i) for i in range(pkg.sim_plan_info(plan)[0])]
    got = []
    for whole in (True, False):
        h = pkg.sim_create(n)
        try:
            pkg.sim_set_layout(h, perm)
            pkg.sim_reset(h)
            for _ in range(2):  # twice: the second run starts from a dense state
                if whole:
                    pkg.sim_apply_plan(h, plan)
                else:
                    for t, m in blocks:
                        pkg.sim_apply_fused(h, t, m)
                got.append(pkg.sim_amplitudes(h))
        finally:
            pkg.sim_destroy(h)
    pkg.sim_plan_destroy(plan)
    assert np.array_equal(got[0], got[2]) and np.array_equal(got[1], got[3])
    assert np.linalg.norm(got[0] - oracle_mod.run_circuit(circ)) <= 1e-5


def test_plans_on_two_streams(pkg):
    # the block tables travel with the launches: two handles' plans in flight do not disturb each other
    n = 12
    circs = [si.workload_circuit("syc12_3x4_d8", seed=s) for s in (1, 2)]
    plans = [pkg.sim_plan_create(n, pkg.gates_array(c), kmax=4) for c in circs]
    hs = [pkg.sim_create(n) for _ in circs]
    try:
        want = []
        for h, p in zip(hs, plans):
            pkg.sim_apply_plan(h, p)
            want.append(pkg.sim_amplitudes(h))
        for _ in range(20):
            for h, p in zip(hs, plans):
                pkg.sim_reset(h)
                pkg.sim_apply_plan(h, p)
        for h, w in zip(hs, want):
            assert np.array_equal(pkg.sim_amplitudes(h), w)
    finally:
        for h in hs:
            pkg.sim_destroy(h)
        for p in plans:
            pkg.sim_plan_destroy(p)
