"""GPU: the library's kernels behind a kernel of the caller's that lets them start early and runs on for
longer than their bounded waits (4 s): the waits count from the end of the work before, so the pass
is neither given up nor begun too soon."""
import ctypes
import subprocess

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


@pytest.fixture(scope="module")
def trigger(tmp_path_factory):
    import os
    from paper_1910_09534_gb300 import build
    lib = str(tmp_path_factory.mktemp("early") / "libtrigger.so")
    src = os.path.join(os.path.dirname(os.path.abspath(__file__)), "early_trigger.cu")
    r = subprocess.run([build.nvcc()] + build.ARCH + ["-O2", "-Xcompiler", "-fPIC", "-shared", src, "-o", lib],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    f = ctypes.CDLL(lib).trigger_then_run
    f.argtypes = [ctypes.c_void_p, ctypes.c_double, ctypes.c_void_p, ctypes.c_ulonglong, ctypes.c_float]
    return f


def test_permutation_pipeline_behind_long_kernel(pkg, trigger):
    n = 12
    psi = si.random_state(n, 3)
    perm = list(range(n))
    for i in range(5):  # five low bits with the five highest: the tensor-map pipeline, one tile
        perm[i], perm[n - 5 + i] = n - 5 + i, i
    h = pkg.sim_create(n)
    try:
        pkg.sim_load_amplitudes(h, psi)
        ptr, stream = pkg.sim_state_ptr(h)
        pkg.sim_sync(h)
        assert trigger(stream, 4.6, ptr, 1 << n, 2.0) == 0
        pkg.sim_permute(h, perm)
        got = pkg.sim_amplitudes(h, physical_order=True)
        pkg.sim_sync(h)  # a wait that ran out would be reported here
    finally:
        pkg.sim_destroy(h)
    i = np.arange(psi.size)
    j = np.zeros_like(i)
    for q, b in enumerate(perm):
        j |= ((i >> q) & 1) << b
    want = np.empty_like(psi)
    want[j] = 2 * psi  # exact: a power of two
    assert np.array_equal(got.view(np.uint32), want.astype(np.complex64).view(np.uint32))
