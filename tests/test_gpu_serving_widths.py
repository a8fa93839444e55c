"""GPU: packed circuits on either width of cluster.

Alone they run on the widest clusters the device places, beside a circuit of the large lane on
clusters of 8.  Every amplitude is the same sum of products on either, and the reduced pair is
added up in parts that do not depend on the width: the results agree bit for bit.  The bound
against the oracle is the one of the other served FP32 circuits.
"""
import numpy as np
import pytest

import syc_inputs as si

pytestmark = pytest.mark.gpu
TOL_FP32 = 1e-5


@pytest.fixture(scope="module")
def pkg():
    from paper_1910_09534_gb300 import build
    build.build()
    import paper_1910_09534_gb300 as p
    return p


@pytest.mark.parametrize("kmax", [3, 5])
def test_packed_beside_a_large_circuit_equals_alone(pkg, oracle_mod, kmax):
    sizes = (1, 2, 7, 11, 12, 13, 16, 18)
    small = [si.sycamore_circuit(si.near_square_grid(n), 6, seed=40 + n) for n in sizes]
    large = si.sycamore_circuit(si.near_square_grid(26), 24, seed=39)
    runs = []
    for beside in (False, True):
        srv = pkg.srv_create(small_n=18, slots=2, kmax=kmax)
        try:
            big = pkg.srv_submit(srv, large.n_qubits, pkg.gates_array(large)) if beside else None
            outs = [np.zeros(1 << c.n_qubits, dtype=np.complex64) for c in small]
            tickets = [pkg.srv_submit(srv, c.n_qubits, pkg.gates_array(c), o) for c, o in zip(small, outs)]
            sums = [pkg.srv_wait(srv, t, 60000)[:2] for t in tickets]
            if beside:
                assert abs(pkg.srv_wait(srv, big, 60000)[0] - 1) < 1e-5
        finally:
            pkg.srv_destroy(srv)
        runs.append((outs, sums))
    for c, a, b, sa, sb in zip(small, runs[0][0], runs[1][0], runs[0][1], runs[1][1]):
        assert np.array_equal(a.view(np.uint64), b.view(np.uint64)) and sa == sb, c.n_qubits
        want = oracle_mod.run_circuit(c)
        assert np.linalg.norm(a.astype(np.complex128) - want) <= TOL_FP32
        norm, s2, _ = oracle_mod.reduce(want)
        assert abs(sa[0] - norm) < 1e-5 and abs(sa[1] - s2) < 1e-3 * s2
