"""Host code of the library against a stand-in runtime (tests/host_runtime.py)."""
import shutil

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
