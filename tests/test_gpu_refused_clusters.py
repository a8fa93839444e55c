"""GPU: cluster launches that the device refuses (here: a host function in the launch call's place).

Packed serving goes on with clusters of 8 where wider ones are refused, with the same bits; where those
are refused too, the requests end with an error that names the reason, other circuits are served
still, and the server can be destroyed.  Plans go on with clusters of 8, and where those are refused,
at the first launch or a later one, with one launch a block: the same bits.
"""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)


@pytest.fixture(scope="module")
def refusing_lib(tmp_path_factory):
    """The library with the launch call of its cluster kernels replaced."""
    from paper_1910_09534_gb300 import build
    build.build()
    d = tmp_path_factory.mktemp("refused")
    swapped = {"serve.cu", "plan_cluster.cu"}
    flags = build.CFLAGS + ["-DSYCSIM_CLUSTER_LAUNCH=refused_launch", "-include", os.path.join(HERE, "refused_launch.cuh")]
    jobs = [subprocess.Popen([build.nvcc()] + flags + ["-c", os.path.join(build.CSRC, f), "-o", str(d / (f + ".o"))])
            for f in sorted(swapped)]
    assert all(j.wait() == 0 for j in jobs)
    objs = [str(d / (s + ".o")) if s in swapped else os.path.join(build.BUILD, s + ".o") for s in build.SOURCES]
    lib = str(d / "libsycsim.so")
    subprocess.run([build.nvcc()] + build.ARCH + ["-shared", "-o", lib] + objs + ["-lcuda"], check=True)
    return lib


def run(lib, body, above, after=0):
    """body in a process of its own, on that library; its output, or a failure if it does not end."""
    head = (f"import sys; sys.path.insert(0, {ROOT!r})\n"
            "import hashlib\nimport numpy as np\nimport paper_1910_09534_gb300 as pkg\nimport syc_inputs as si\n"
            "from paper_1910_09534_gb300 import _native\n"
            f"_native.LIB_PATH = {lib!r}\n")
    r = subprocess.run([sys.executable, "-c", head + body], capture_output=True, text=True, timeout=60,
                       env=dict(os.environ, REFUSE_ABOVE=str(above), REFUSE_AFTER=str(after)))
    assert r.returncode == 0, r.stdout + r.stderr
    return r.stdout


SERVE = """
c = [si.sycamore_circuit(si.near_square_grid(n), 6, seed=n) for n in (3, 9, 12, 14, 9)]
big = si.sycamore_circuit(si.near_square_grid(19), 6, seed=1)
srv = pkg.srv_create(small_n=18, slots=2)
outs = [np.zeros(1 << x.n_qubits, dtype=np.complex64) for x in c]
tickets = [pkg.srv_submit(srv, x.n_qubits, pkg.gates_array(x), o) for x, o in zip(c, outs)]
for t, o in zip(tickets, outs):
    try:
        norm, s2, _ = pkg.srv_wait(srv, t, 5000)
        print("ok", norm.hex(), s2.hex(), hashlib.sha256(o.tobytes()).hexdigest())
    except pkg.SimError as e:
        print("error", e)
print("large", abs(pkg.srv_wait(srv, pkg.srv_submit(srv, 19, pkg.gates_array(big)), 20000)[0] - 1) < 1e-5)
pkg.srv_destroy(srv)
print("destroyed")
"""


def test_packed_serving_goes_on_with_narrower_clusters(refusing_lib):
    wide, narrow = run(refusing_lib, SERVE, 16), run(refusing_lib, SERVE, 8)
    assert wide == narrow and wide.count("ok") == 5 and wide.endswith("large True\ndestroyed\n")


@pytest.mark.parametrize("after", [0, 1])
def test_packed_serving_reports_a_refused_launch(refusing_lib, after):
    out = run(refusing_lib, SERVE, 0, after)
    assert out.count("ok") + out.count("error") == 5 and out.endswith("large True\ndestroyed\n")
    assert all("worker launch: too many resources" in x for x in out.splitlines() if x.startswith("error"))
    if after == 0:
        assert out.count("error") == 5


PLAN = """
for n, kmax in ((6, 3), (12, 4), (13, 5), (15, 4)):
    c = si.sycamore_circuit(si.near_square_grid(n), 20, seed=n)
    p = pkg.sim_plan_create(n, pkg.gates_array(c), kmax=kmax)
    h = pkg.sim_create(n)
    pkg.sim_apply_plan(h, p)
    out = pkg.sim_amplitudes(h)
    pkg.sim_sync(h)
    print(n, hashlib.sha256(out.tobytes()).hexdigest(), abs(pkg.sim_reduce(h)[0] - 1) < 1e-5)
    pkg.sim_destroy(h)
    pkg.sim_plan_destroy(p)
"""


def test_plans_go_on_where_clusters_are_refused(refusing_lib):
    want = run(refusing_lib, PLAN, 16)
    assert want.count("True") == 4
    assert run(refusing_lib, PLAN, 8) == want
    for after in (0, 1, 2, 3):
        assert run(refusing_lib, PLAN, 0, after) == want
