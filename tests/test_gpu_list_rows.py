"""What the rows of the Verlet lists of an FP64 handle hold: the particles
within (1 + beta) kappa h_ij at the build and no others, however far the
particle sizes lie apart, so that a list_cap that suffices for the radius is
enough.  (Mixed handles list a margin of 1e-4 of the cell edge more.)"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
from test_gpu_pair_groups import _check_step, _gas, _lattice  # noqa: E402

pytestmark = pytest.mark.gpu
BETA = 0.15


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1805_05128_gb300 import build
    build.build()


def _with_large(dims, ratio, at):
    """A lattice of unit particles and two large ones that set the cell edge."""
    p = np.concatenate([_lattice(dims), np.array([[a] + [0.0] * (len(dims) - 1) for a in at]).T], axis=1)
    return _gas(p, np.concatenate([np.ones(p.shape[1] - 2), [ratio, ratio]]))


CASES = {
    "line": lambda: _gas(_lattice((700,))),
    "line_200": lambda: _with_large((700,), 200.0, (3000.0, 3400.0)),
    "line_600": lambda: _with_large((2500,), 600.0, (9000.0, 10500.0)),
    "plane_12": lambda: _with_large((31, 29), 12.0, (90.0, 130.0)),
    "box": lambda: _gas(_lattice((11, 9, 8))),
    "box_3": lambda: _with_large((11, 10, 9), 3.0, (30.0, 45.0)),
}


def _row_lengths(g, dim, khl):
    """Neighbours of each particle within khl (d_i + d_j), the oracle's operation order."""
    n, d = len(g["d"]), g["d"]
    out = np.zeros(n, dtype=np.int64)
    for i in range(n):
        r2 = (g["x"] - g["x"][i]) ** 2
        for k in "yz"[: dim - 1]:
            r2 = r2 + (g[k] - g[k][i]) ** 2
        R = khl * (d[i] + d)
        out[i] = np.count_nonzero(r2 < R * R) - 1
    return out


@pytest.mark.parametrize("name", list(CASES))
def test_rows_hold_the_radius(name):
    from paper_1805_05128_gb300 import Simulation
    prob = CASES[name]()
    need = 0
    for cap in (0, 1):                                    # the default capacity, then the least that holds the rows
        sim = Simulation(prob, precision="fp64", units=0, cell_beta=BETA, list_cap=cap and max(32, need))
        sim.step(1)
        g = sim.numpy()                                   # positions and sizes of the build: the step's predicted ones
        khl = sim.params.kappa * 0.5 * sim.params.eta * (1.0 + BETA)
        rows = _row_lengths(g, prob.dim, khl)
        need = int(-(-rows.max() // 32) * 32)
        assert sim.pair_counts()[1] == rows.sum()         # entries of all rows
        assert sim.read_status() == 0
        sim.close()
    _check_step(prob, BETA)
