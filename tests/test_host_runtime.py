"""Host code of the library against a stand-in runtime (tests/host_runtime.py)."""
import ctypes as C
import shutil
import threading
import time

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
