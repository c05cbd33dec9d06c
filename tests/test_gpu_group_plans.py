"""Choices that follow from the size of a system and must not show in its
results: lanes per slot of the cell search, group sizes of the list
evaluation, blocks per sum, tiles per block of the cell scan."""
import math

import numpy as np
import pytest

import synth

torch = pytest.importorskip("torch")
from test_gpu_pair_groups import SHAPES, _check, _check_step, _gas, _lattice  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1805_05128_gb300 import build
    build.build()


RATES = ("ax", "ay", "az", "drho", "dE")


@pytest.mark.parametrize("order,solver", [(1, "acoustic"), (2, "acoustic"), (1, "hll")])
@pytest.mark.parametrize("dims", [(41, 31, 27), (181, 113)])
def test_mixed_search_lanes_same_bits(dims, order, solver):
    """An instance alone (four lanes a slot) and four times in one handle (one lane a slot)."""
    from paper_1805_05128_gb300 import Simulation
    prob = _gas(_lattice(dims))
    out = []
    for copies in (1, 4):
        sim = Simulation([prob] * copies, units=0, order=order, solver=solver)
        sim.eval_rates()
        g = sim.numpy()
        assert sim.read_status() == 0
        out.append({k: g[k].reshape(copies, -1) for k in RATES if k in g})
        sim.close()
    for k, one in out[0].items():
        assert np.any(one) and all(np.array_equal(one[0], row) for row in out[1][k]), k


@pytest.mark.parametrize("precision", ["mixed", "fp64"])
@pytest.mark.parametrize("dims", [(33, 33, 33), (17, 16, 15)])
def test_list_group_plans_same_bits(dims, precision):
    """Groups of 8, of 16 and 8, of 32 and 8 slots: the resident warps decide."""
    from paper_1805_05128_gb300 import Simulation
    prob = _gas(_lattice(dims))
    ref = None
    for blocks in (0, 1, 2, 3, 5):
        sim = Simulation(prob, precision=precision, units=0, cell_beta=0.15, pair_blocks_per_sm=blocks)
        sim.step(2)
        g = sim.numpy()
        assert sim.read_status() == 0
        ref = ref or g
        for k in RATES + ("x", "rho", "E"):
            assert np.any(g[k]) and np.array_equal(g[k], ref[k]), (blocks, k)
        sim.close()


@pytest.mark.parametrize("n", [1, 31, 1025, 4096, 4097, 16385, 66001])
def test_conservation_sums_any_size(n):
    """Against exactly rounded sums: a thread adds at most 8 terms here, its block and cluster 14 more levels, so 32 roundings of the sum of the magnitudes."""
    from paper_1805_05128_gb300 import Simulation
    prob = _gas(_lattice((n,)))
    sim = Simulation(prob, precision="fp64", units=0)
    c = sim.conservation().cpu().numpy()[0]
    g = sim.numpy()
    for col, f in ((0, np.ones(n)), (1, g["vx"]), (4, g["E"])):
        terms = g["m"] * f
        assert abs(c[col] - math.fsum(terms)) <= 32 * 2.0 ** -53 * math.fsum(np.abs(terms)), col
    assert c[2] == 0 and c[3] == 0
    sim.close()


def test_more_scan_tiles_than_blocks():
    """Small clusters in the corners and the middle of a box of over two million cells."""
    base = _lattice((4, 3, 3))
    far = [0.0, 150.0, 301.0]
    at = [(a, b, c) for a in far for b in far for c in far]
    pos = np.concatenate([base + np.array(o)[:, None] for o in at], axis=1)
    _check(_gas(pos), "fp64", 1e-10)


def _hundred_a_cell():
    """Two larger particles far off make cells of about a hundred: several groups of 32 home particles."""
    p = np.concatenate([_lattice((13, 12, 11)), [[60.0, 75.0], [0.0, 0.0], [0.0, 0.0]]], axis=1)
    return _gas(p, np.concatenate([np.ones(p.shape[1] - 2), [1.6, 1.6]]))


LISTED = {**{k: v for k, v in SHAPES.items() if k != "crowded"}, "hundred": _hundred_a_cell}


@pytest.mark.parametrize("name", list(LISTED))
def test_list_build_shapes(name):
    """Lists of few, of sparse and of many candidates a group against the oracle's pairs and steps."""
    _check_step(LISTED[name](), 0.15)
