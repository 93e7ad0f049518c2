"""The served jobs' memory estimate and budget, with the library's host code on a CUDA
runtime that counts what is allocated (no GPU): a job never holds more than its
footprint, at any porosity and in both storages, and the jobs together never more than
the budget; one that the device refuses waits, and is not built again before
another has given its memory back."""
import ctypes as ct

import numpy as np
import pytest

import host

RUNNING, DONE = 1, 2


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    return host.build(tmp_path_factory.mktemp("host"))


def _image(edge, porosity, seed=1):
    lab = (np.random.default_rng(seed).random((edge,) * 3) >= porosity).astype(np.uint16)
    lab[0, 0, 0] = 0
    return lab


def _server(lib, budget=0):
    s = ct.c_void_p()
    assert lib.lbpm_server_create(ct.byref(s), 0, None, budget, 64, 10) == 0
    return s


def _submit(lib, s, lab, precision="fp32", reservoir_z=0, max_steps=20):
    from paper_2007_12266_gb300 import JobSpec, _params
    nz, ny, nx = lab.shape
    zero = np.zeros(lab.shape, np.float32)
    sp = JobSpec()
    sp.labels, sp.nx, sp.ny, sp.nz = lab.ctypes.data, nx, ny, nz
    sp.affinity = sp.phi0 = zero.ctypes.data
    sp.params = _params(0.7, 0.7, 0.005, 0.95, (0, 0, 1e-5), precision, (1, 1, 0), reservoir_z, 1.0, 1.0)
    sp.max_steps, sp.flux_tol, sp.sw_tol = max_steps, 1e-4, 1e-4
    t = ct.c_longlong()
    return lib.lbpm_server_submit(s, ct.byref(sp), ct.byref(t)), t.value


def _poll(lib, s, ticket):
    from paper_2007_12266_gb300 import JobStatus
    st = JobStatus()
    assert lib.lbpm_server_poll(s, ticket, ct.byref(st)) == 0
    return st


def _run(lib, s):
    r, q, f = ct.c_int(), ct.c_int(), ct.c_int()
    assert lib.lbpm_server_run(s, ct.byref(r), ct.byref(q), ct.byref(f)) == 0
    return r.value, q.value


@pytest.mark.parametrize("reservoir_z", [0, 1, 3])
@pytest.mark.parametrize("precision", ["fp32", "fp16"])
@pytest.mark.parametrize("porosity", [0.02, 0.2, 0.35, 1.0])
@pytest.mark.parametrize("edge", [20, 96])
def test_footprint_covers_the_job(lib, edge, porosity, precision, reservoir_z):
    s = _server(lib)
    base = lib.fake_live()
    lib.fake_reset_peak()
    st, t = _submit(lib, s, _image(edge, porosity), precision, reservoir_z)
    assert st == 0
    while _run(lib, s)[0]:
        pass
    held = lib.fake_peak() - base
    footprint = _poll(lib, s, t).footprint
    assert held <= footprint
    if edge == 96:                               # and by little more than its MiB
        assert footprint <= 1.12 * held + (1 << 20)
    assert lib.lbpm_server_destroy(s) == 0


@pytest.mark.parametrize("precision", ["fp32", "fp16"])
@pytest.mark.parametrize("porosity", [0.22, 0.35, 1.0])
def test_budget_holds(lib, porosity, precision):
    lab = _image(64, porosity)
    probe = _server(lib)
    _, t = _submit(lib, probe, lab, precision)
    footprint = _poll(lib, probe, t).footprint
    assert lib.lbpm_server_destroy(probe) == 0
    budget = int(2.5 * footprint)
    s = _server(lib, budget)
    base = lib.fake_live()
    lib.fake_reset_peak()
    tickets = [_submit(lib, s, lab, precision)[1] for _ in range(5)]
    most = 0
    for _ in range(50):
        running, queued = _run(lib, s)
        most = max(most, running)
        if not running and not queued:
            break
    assert [_poll(lib, s, t).state for t in tickets] == [DONE] * 5
    assert most == 2 and lib.fake_peak() - base <= budget
    assert lib.lbpm_server_destroy(s) == 0


@pytest.mark.parametrize("release", [False, True])     # the first job's result: left to the server, or released
def test_a_refused_job_is_not_built_again_and_again(lib, release):
    lab = _image(64, 0.3)
    s = _server(lib)
    t1 = _submit(lib, s, lab, max_steps=200)[1]
    t2 = _submit(lib, s, lab, max_steps=20)[1]
    lib.fake_memory_limit(lib.fake_live() + int(1.5 * _poll(lib, s, t1).footprint))
    try:
        refused, uploads = [lib.fake_refused()], []
        for _ in range(19):                            # 190 of the first job's 200 steps
            assert _run(lib, s) == (1, 1)
            refused.append(lib.fake_refused())
            uploads.append(lib.fake_uploads())
        assert refused[1] > refused[0] and set(refused[1:]) == {refused[1]}   # tried once
        assert len(set(np.diff(uploads[1:]))) == 1     # every round's own few
        assert _run(lib, s) == (0, 1)
        assert _poll(lib, s, t1).state == DONE
        if release:
            assert lib.lbpm_server_release(s, t1) == 0
        assert _run(lib, s) == (1, 0)
        assert _run(lib, s) == (0, 0)
        assert _poll(lib, s, t2).state == DONE
        assert lib.fake_refused() == refused[1]
    finally:
        lib.fake_memory_limit(2 ** 63)
    assert lib.lbpm_server_destroy(s) == 0


def test_a_job_the_device_cannot_hold_alone_fails(lib):
    lab = _image(64, 0.3)
    s = _server(lib)
    t = _submit(lib, s, lab)[1]
    lib.fake_memory_limit(lib.fake_live() + _poll(lib, s, t).footprint // 2)
    try:
        assert _run(lib, s) == (0, 0)
    finally:
        lib.fake_memory_limit(2 ** 63)
    assert _poll(lib, s, t).state == 3                 # failed
    assert lib.lbpm_server_destroy(s) == 0
