"""GPU: which FP32 plans one cluster runs, several blocks a launch, and which take a launch a block: both
sides of the line at every block width (the line's measurements stand beside plan_cluster_eligible)."""
import pytest

import syc_inputs as si

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pkg():
    from paper_1910_09534_gb300 import build
    build.build()
    import paper_1910_09534_gb300 as p
    return p


@pytest.mark.parametrize("kmax,n,cluster", [(2, 13, True), (2, 15, False), (3, 13, True), (3, 15, False), (4, 14, True),
                                            (4, 16, False), (5, 12, True), (5, 14, False), (5, 17, False),
                                            (6, 12, False)])
def test_launches_of_a_plan(pkg, kmax, n, cluster):
    p = pkg.sim_plan_create(n, pkg.gates_array(si.sycamore_circuit(si.near_square_grid(n), 20, seed=n)), kmax=kmax)
    blocks = pkg.sim_plan_info(p)[0]
    h = pkg.sim_create(n)
    try:
        before = pkg.sim_launch_count(h)
        pkg.sim_apply_plan(h, p)
        launches = pkg.sim_launch_count(h) - before
    finally:
        pkg.sim_destroy(h)
        pkg.sim_plan_destroy(p)
    assert launches < blocks if cluster else launches == blocks, (launches, blocks)
