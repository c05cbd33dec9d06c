"""Every plan of the list evaluation, and the cell scan with more tiles than
blocks, each with a check that the size meant is the size that ran."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
from test_gpu_group_plans import RATES  # noqa: E402
from test_gpu_pair_groups import _check, _gas, _lattice  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1805_05128_gb300 import build
    build.build()


def _sms():
    return torch.cuda.get_device_properties(0).multi_processor_count


def _plan(n, blocks):
    """Slots of a group, first and last, of the list evaluation with `blocks` resident blocks of 4 warps per SM."""
    warps = 4 * blocks * _sms()
    big = 32 if n > 27 * warps else 16
    if n <= 16 * warps:
        return 8, 8
    if big == 32 and (n + 31) % (32 * warps) >= 32 * warps * 5 // 6:
        return 32, 32
    return big, 8


DIMS = [(25, 23, 22), (33, 33, 33), (45, 33, 31)]


def test_every_plan_is_run():
    plans = {tuple(_plan(int(np.prod(d)), b) for b in (1, 2, 3)) for d in DIMS}
    assert all(len(set(p)) > 1 for p in plans)              # each size runs under several
    assert set().union(*plans) == {(8, 8), (16, 8), (32, 8), (32, 32)}


@pytest.mark.parametrize("precision", ["mixed", "fp64"])
@pytest.mark.parametrize("dims", DIMS)
def test_list_plans_same_bits(dims, precision):
    from paper_1805_05128_gb300 import Simulation
    prob, ref = _gas(_lattice(dims)), None
    for blocks in (1, 2, 3):
        sim = Simulation(prob, precision=precision, units=0, cell_beta=0.15, pair_blocks_per_sm=blocks)
        sim.step(2)
        g = sim.numpy()
        assert sim.read_status() == 0
        ref = ref or g
        for k in RATES + ("x", "rho", "E"):
            assert np.any(g[k]) and np.array_equal(g[k], ref[k]), (blocks, k)
        sim.close()


def test_scan_tiles_outnumber_blocks():
    """Small clusters over a box of 1,601,613 cells: 1,565 tiles of 1,024 for 8 blocks per SM."""
    from paper_1805_05128_gb300 import Simulation
    far = [0.0, 150.0, 301.0]
    pos = np.concatenate([_lattice((4, 3, 3)) + np.array([[a], [b], [c]]) for a in far for b in far for c in far], axis=1)
    prob = _gas(pos)
    sim = Simulation(prob, precision="fp64", units=0)
    cells = sim.cell_index()[1][0][7]
    sim.close()
    assert cells == 1601613 and -(-cells // 1024) > 8 * _sms()
    _check(prob, "fp64", 1e-10)
