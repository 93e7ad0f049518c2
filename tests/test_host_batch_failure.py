"""A batch that runs job by job and fails on the way, on a CUDA runtime whose calls can
be made to fail (no GPU): without memory for a job's graphs nothing has been launched
and no job has moved; a launch that fails inside a job's run leaves that job flagged,
so that its stale populations are not taken for a state."""
import ctypes as ct

import numpy as np
import pytest

import host

UNSTABLE = 5


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    return host.build(tmp_path_factory.mktemp("host"))


def _batch(lib, n_jobs, edge=45):
    from paper_2007_12266_gb300 import _params
    lab, phi = np.zeros((edge,) * 3, np.uint16), np.zeros((edge,) * 3, np.float32)
    b = ct.c_void_p()
    assert lib.lbpm_batch_create(ct.byref(b), 0, None) == 0
    jobs = []
    for _ in range(n_jobs):
        c = ct.c_void_p()
        assert lib.lbpm_create(ct.byref(c), 0, None) == 0
        p = _params(0.7, 0.7, 0.005, 0.95, (0, 0, 1e-5), "fp32", (1, 1, 1), 0, 1.0, 1.0)
        assert lib.lbpm_set_params(c, ct.byref(p)) == 0
        assert lib.lbpm_load_image(c, lab.ctypes.data, edge, edge, edge) == 0
        assert lib.lbpm_init_fluids(c, phi.ctypes.data) == 0
        assert lib.lbpm_batch_add(b, c) == 0
        jobs.append(c)
    return b, jobs


def _steps(lib, jobs):
    out = []
    for c in jobs:
        n = ct.c_longlong()
        assert lib.lbpm_step_count(c, ct.byref(n)) == 0
        out.append(n.value)
    return out


@pytest.mark.parametrize("nth", [1, 2, 3, 4, 5, 6])      # two graphs for each of three jobs
def test_no_memory_for_a_graph(lib, nth):
    b, jobs = _batch(lib, 3)
    before = lib.fake_launches()
    lib.fake_fail(0, nth)
    assert lib.lbpm_batch_advance(b, 24) != 0
    assert lib.lbpm_batch_last_error(b)
    captured = lib.fake_launches() - before              # kernels seen by the captures, of the graphs up to this one
    assert captured == sum((32, 4)[k % 2] for k in range(nth))
    assert _steps(lib, jobs) == [0, 0, 0]
    assert lib.lbpm_batch_advance(b, 24) == 0
    assert _steps(lib, jobs) == [24, 24, 24]


@pytest.mark.parametrize("nth", [1, 4, 9])               # graphs of 16, 2 and 2 steps for each of three jobs
def test_a_launch_that_fails(lib, nth):
    b, jobs = _batch(lib, 3)
    lib.fake_fail(1, nth)
    assert lib.lbpm_batch_advance(b, 24) != 0
    failed = (nth - 1) // 3
    steps = _steps(lib, jobs)
    assert steps[:failed] == [24] * failed and steps[failed + 1:] == [0] * (2 - failed)
    assert lib.lbpm_batch_advance(b, 24) == UNSTABLE
    assert _steps(lib, jobs) == steps
    lib.lbpm_init_fluids(jobs[failed], np.zeros((45,) * 3, np.float32).ctypes.data)
    assert lib.lbpm_batch_advance(b, 24) == 0
