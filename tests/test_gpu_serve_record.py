"""Serving jobs that record into the caller's buffer: the record of a job submitted the ordinary way,
bit for bit, alone and beside one, and the call's argument errors."""
import ctypes

import numpy as np
import pytest
import torch

from paper_2410_14117_gb300 import inputs as I
from paper_2410_14117_gb300._lib import JobSpec, MGError, Ranges, ServerConfig, call
from paper_2410_14117_gb300.serve import NativeServer, Pool, Request

pytestmark = pytest.mark.gpu


def _server(pool, record=1):
    h = ctypes.c_void_p()
    cfg = ServerConfig(1e9, 20, 2, record, 0, 1, 0, 10.0)
    call("mg_server_create", pool._h, ctypes.byref(cfg), ctypes.byref(h))
    return h


def _spec(n, horizon, seed):
    return JobSpec(n, 0, 7, horizon, 0, seed, seed + 1, Ranges(0.8, 1.2, 0.2, 0.3, 0))


def _drain(h):
    c = [ctypes.c_int32() for _ in range(3)]
    while True:
        call("mg_server_poll", h, *[ctypes.byref(x) for x in c])
        if not any(x.value for x in c):
            return


def test_caller_record_equals_the_servers_own():
    pool = Pool(4096, I.fleet_vehicles())
    h = _server(pool)
    n, T = 333, 50
    mine = torch.full((T, 13, n), -1.0, device="cuda")
    a, b = ctypes.c_int64(), ctypes.c_int64()
    call("mg_server_submit_record", h, ctypes.byref(_spec(n, T, 5)), None, mine.data_ptr(),
         ctypes.byref(a))
    call("mg_server_submit", h, ctypes.byref(_spec(n, T, 5)), ctypes.byref(b))
    _drain(h)
    got = [torch.empty_like(mine) for _ in range(2)]
    st = [torch.empty((n, 21), device="cuda") for _ in range(2)]
    for t, g, s in zip((a, b), got, st):
        call("mg_server_job_result", h, t.value, s.data_ptr(), g.data_ptr())
        call("mg_server_release", h, t.value)
    pool.sync()
    assert torch.equal(mine, got[0]) and torch.equal(got[0], got[1]) and torch.equal(st[0], st[1])
    # the buffer outlives the job and the server
    call("mg_server_destroy", h)
    assert torch.equal(mine, got[1])
    pool.close()


def test_record_argument_errors():
    pool = Pool(4096, I.fleet_vehicles())
    h, plain = _server(pool), _server(pool, record=0)
    n, T = 64, 20
    t = ctypes.c_int64()
    dev = torch.empty((T, 13, n), device="cuda")
    host = np.empty((T, 13, n), np.float32)
    for srv, ptr in ((h, None), (h, host.ctypes.data), (plain, dev.data_ptr())):
        with pytest.raises(MGError) as e:
            call("mg_server_submit_record", srv, ctypes.byref(_spec(n, T, 1)), None, ptr,
                 ctypes.byref(t))
        assert e.value.code == "MG_EINVAL"
    for srv in (h, plain):
        call("mg_server_destroy", srv)
    pool.close()


def test_results_on_another_stream():
    """run() called under a stream other than the pool's: the records are complete when it returns."""
    srv = NativeServer(I.fleet_vehicles(), budget_bytes=1e9, capacity_envs=1 << 14, k=20,
                       keep_results=True)
    out = []
    for s in (torch.cuda.current_stream(), torch.cuda.Stream()):
        with torch.cuda.stream(s):
            done, _ = srv.run([Request(0.0, 500 + 100 * i, 60, i % 2, 3 + i, 9 + i)
                               for i in range(5)], realtime=False)
            out.append([(r.traj.sum(dim=0).cpu(), r.final_state.cpu()) for r in done])
    for x, y in zip(*out):
        assert torch.equal(x[0], y[0]) and torch.equal(x[1], y[1])
    srv.close()


def test_final_states_wait_for_the_memorys_earlier_use():
    """run() under a stream with work still queued: the final states come in memory that this work
    may yet write, and are written on the pool's stream after it."""
    n = 4001
    srv = NativeServer(I.fleet_vehicles(), budget_bytes=1e9, capacity_envs=1 << 14, k=20,
                       record=False, keep_results=True)
    req = lambda: [Request(0.0, n, 40, 0, 3, 9)]  # noqa: E731
    want = srv.run(req(), realtime=False)[0][0].final_state.cpu()
    s = torch.cuda.Stream()
    with torch.cuda.stream(s):
        x = torch.empty((n, 21), device="cuda")
        torch.cuda._sleep(400_000_000)  # 0.2 s, longer than the job takes
        x.fill_(7.0)
        at = x.data_ptr()
        del x
        got = srv.run(req(), realtime=False)[0][0].final_state
        assert got.data_ptr() == at
        s.synchronize()
        assert torch.equal(got.cpu(), want)
    srv.close()
