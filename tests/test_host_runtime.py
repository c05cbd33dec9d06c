"""Host code of the library against a stand-in runtime (tests/host_runtime.py)."""
import ctypes as C
import shutil
import threading
import time

import numpy as np
import pytest

import host_runtime

pytestmark = pytest.mark.skipif(shutil.which("g++") is None, reason="g++ not found")


@pytest.fixture(scope="module")
def so(tmp_path_factory):
    return host_runtime.build_library(tmp_path_factory.mktemp("host"))


def scenario_upload(so, precision, beta):
    """A handle's tables reach the device as they were, however late the copy is made."""
    H = host_runtime.Host(so)
    s = H.state(5000)
    h = H.handle(s, offsets=[0, 1200, 5000], precision=precision, cell_beta=0.15 * beta)
    H.abi.sph_destroy(h)
    return H.L.fake_copied() > 0, H.L.fake_changed()


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("beta", [0, 1])
def test_uploads_outlive_their_copies(so, precision, beta):
    assert host_runtime.run(so, "test_host_runtime:scenario_upload", precision, beta) == "(True, 0)"


def scenario_devices(so):
    """The totals and the parameter adjoints on a device that is not the first one used: launch errors, clusters."""
    H = host_runtime.Host(so)
    n, got = 70000, []
    for dev in (0, 1, 70, 71, 0):
        H.L.fake_set_device(dev)
        s = H.state(n)
        h = H.handle(s)
        out = H.array(5)
        H.launches()
        rc = [H.L.sph_conservation(h, C.byref(s), out.ctypes.data, None)]
        ck = H.abi.sph_ckpt(state=s, dt=H.array(1).ctypes.data)
        adj = H.state(n)
        rc.append(H.L.sph_step_adjoint(h, C.byref(ck), 1, C.byref(adj), C.byref(adj), H.array(2).ctypes.data, None))
        got.append(rc + [c for name, blocks, c in H.launches() if c > 1])
        H.abi.sph_destroy(h)
    return got


def test_clusters_on_every_device(so):
    assert host_runtime.run(so, "test_host_runtime:scenario_devices") == str([[0, 0, 16, 16]] * 5)


def scenario_first_use(so, beta):
    """Two threads that need a kernel's grid for the first time at once: both launch, the same blocks."""
    H = host_runtime.Host(so)
    s = H.state(50000)
    hs = [H.handle(s, cell_beta=0.15 * beta) for _ in range(2)]
    for h in hs:
        H.L.sph_hold_rates(h)
    H.launches()
    H.L.fake_query_ms(400)          # the occupancy query takes this long
    rc = [None, None]

    def step(k):
        rc[k] = H.L.sph_step(hs[k], C.byref(s), 1, None, None)

    threads = [threading.Thread(target=step, args=(k,)) for k in (0, 1)]
    threads[0].start()
    time.sleep(0.1)
    threads[1].start()
    for t in threads:
        t.join()
    grids = {}
    for name, blocks, _ in H.launches():
        if "k_pair" in name or "k_list_build" in name:
            grids.setdefault(name, []).append(blocks)
    return rc, sorted(len(g) for g in grids.values()), all(len(set(g)) == 1 for g in grids.values())


@pytest.mark.parametrize("beta", [0, 1])
def test_first_use_by_two_threads(so, beta):
    assert host_runtime.run(so, "test_host_runtime:scenario_first_use", beta) == str(([0, 0], [2] * (1 + beta), True))


def scenario_counter(so):
    """The calls whose count of kernel launches (sph_profile_read) is not the number of launches made."""
    H = host_runtime.Host(so)
    abi, L, n = H.abi, H.L, 5000
    out, gen, dts = H.array(6 * n), H.array(3 * 8), H.array(16)
    ints = H.array(2 * n, np.int32)
    bp, cnt = abi.sph_balance_params(), C.c_int64()
    units = dict(n_units=8, unit_dim=3, n_upd=2, generators=gen.ctypes.data)
    handles = {"search": {}, "fp64": dict(precision=0), "lists": dict(cell_beta=0.15), "order2": dict(order=2),
               "units": units, "units lists": dict(units, cell_beta=0.15),
               "units sched": dict(units, cell_beta=0.15, unit_sched=1), "batched": dict(offsets=[0, 700, n]),
               "batched lists": dict(offsets=[0, 700, n], cell_beta=0.15)}
    wrong = []
    for name, kw in handles.items():
        s, adj = H.state(n), H.state(n)
        h = H.handle(s, **kw)
        ck = abi.sph_ckpt(state=s, dt=dts.ctypes.data, rates_from_state=1)
        ck64 = abi.sph_ckpt(state=s, dt=dts.ctypes.data, reverse_fp64=1)
        S, o = C.byref(s), out.ctypes.data
        calls = {"eval": lambda: L.sph_eval_rates(h, S, None), "step": lambda: L.sph_step(h, S, 1, None, None),
                 "3 steps": lambda: L.sph_step(h, S, 3, o, None), "2 given steps": lambda: L.sph_step_dt(h, S, 2, dts.ctypes.data, o, None),
                 "build": lambda: L.sph_build_cells(h, S, None), "cfl": lambda: L.sph_cfl_dt(h, S, o, None),
                 "totals": lambda: L.sph_conservation(h, S, o, None), "cells": lambda: L.sph_cell_index(h, S, ints.ctypes.data, None, None),
                 "pairs": lambda: L.sph_pair_list(h, S, n, ints.ctypes.data, ints.ctypes.data, C.byref(cnt), None)}
        if name in ("search", "fp64", "lists"):
            calls["adjoint"] = lambda: L.sph_step_adjoint(h, C.byref(ck), 3, C.byref(adj), C.byref(adj), o, None)
            calls["adjoint fp64"] = lambda: L.sph_step_adjoint(h, C.byref(ck64), 3, C.byref(adj), C.byref(adj), o, None)
        if "units" in name:
            calls["assign"] = lambda: L.voronoi_assign(h, S, gen.ctypes.data, 8, 3, ints.ctypes.data, None, None)
            calls["balance"] = lambda: L.voronoi_balance(h, S, gen.ctypes.data, 8, 3, None, C.byref(bp), None, None)
        for call, f in calls.items():
            L.sph_profile(h, 0)
            H.launches()
            rc, counted = f(), C.c_int64()
            made = len(H.launches())
            L.sph_profile_read(h, None, None, C.byref(counted))
            if rc != 0 or counted.value != made or made == 0:
                wrong.append((name, call, rc, counted.value, made))
        abi.sph_destroy(h)
    return wrong


def test_launch_counter(so):
    assert host_runtime.run(so, "test_host_runtime:scenario_counter") == "[]"


def scenario_host_memory(so, reverse_fp64):
    """sph_step_adjoint with the k-th host allocation refused, k = 0, 1, ...: an error code each time, then success."""
    H = host_runtime.Host(so)
    s, adj = H.state(3000), H.state(3000)
    ck = H.abi.sph_ckpt(state=s, dt=H.array(3).ctypes.data, reverse_fp64=reverse_fp64)
    par, codes = H.array(2), []
    for k in range(200):
        h = H.handle(s)
        H.launches()
        H.L.fake_fail_new(k)
        codes.append(H.L.sph_step_adjoint(h, C.byref(ck), 3, C.byref(adj), C.byref(adj), par.ctypes.data, None))
        H.L.fake_fail_new(-1)
        again = H.L.sph_step_adjoint(h, C.byref(ck), 3, C.byref(adj), C.byref(adj), par.ctypes.data, None)
        H.abi.sph_destroy(h)
        if again != 0:
            return k, again
        if codes[-1] == 0:
            break
    return len(codes) > 3, set(codes[:-1]) == {H.abi.SPH_ERR_CUDA}, codes[-1]


@pytest.mark.parametrize("reverse_fp64", [0, 1])
def test_no_exception_leaves_the_adjoint(so, reverse_fp64):
    assert host_runtime.run(so, "test_host_runtime:scenario_host_memory", reverse_fp64) == "(True, True, 0)"
