"""The pair kernel's groups of slots at the shapes where a group can go wrong:
fewer slots than a group, groups that span many rows of cells or many sparse
cells of one row, rows too crowded for one segment, instances sharing a
group, and length units far outside FP32's range (FP64 handles).  The pair
set is bit-exact and the rates agree with the oracle at 1e-10 (FP64) and 1e-4
(mixed)."""
import numpy as np
import pytest

import oracle as O
import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1805_05128_gb300 import build
    build.build()


def _gas(pos, sizes=1.0, seed=5):
    """Ideal gas at the given positions (dim x n), d = sizes, random velocities and energies."""
    dim, n = pos.shape
    u = synth.uniform(seed, 4 * n).reshape(4, n)
    rho = 1.0 + 0.2 * u[3]
    arrays = dict(rho=rho, m=rho * np.broadcast_to(sizes, n) ** dim, E=2.0 + 0.5 * (u[:dim] ** 2).sum(0))
    for k, a in enumerate("xyz"[:dim]):
        arrays[a] = pos[k].copy()
        arrays["v" + a] = 0.3 * (u[k] - 0.5)
    return synth.Problem("gas", dim, arrays, [synth.MaterialSpec("ideal", 1.4)], units=0)


def _lattice(dims, jitter=0.2, seed=3):
    g = np.meshgrid(*[np.arange(k, dtype=float) for k in dims], indexing="ij")
    p = np.stack([a.ravel() for a in g])
    return p + jitter * (synth.uniform(seed, p.size).reshape(p.shape) - 0.5)


def _sparse():
    """Clusters far apart along x: a row of cells with long empty runs."""
    p = _lattice((5, 4, 3))
    return np.concatenate([p + np.array([[s], [0.0], [0.0]]) for s in (0.0, 40.0, 300.0, 311.0, 5000.0)], axis=1)


def _crowded():
    """Small particles beside two large ones that set the cell edge: 1,836 particles in a cell (at most 2048 are accepted), rows over 2048 slots."""
    p = np.concatenate([_lattice((30, 12, 9)), [[200.0, 230.0], [0.0, 0.0], [0.0, 0.0]]], axis=1)
    return p, np.concatenate([np.ones(p.shape[1] - 2), [6.5, 6.5]])


SHAPES = {
    "three": lambda: _gas(np.array([[0.0, 0.9, 2.1], [0.0, 0.2, 0.1], [0.0, 0.0, 0.3]])),
    "thirty_three_1d": lambda: _gas(_lattice((33,))),
    "column": lambda: _gas(_lattice((2, 3, 61))),          # a few slots per row of cells
    "long_row": lambda: _gas(_lattice((257, 2, 2))),
    "sparse": lambda: _gas(_sparse()),
    "crowded": lambda: _gas(*_crowded()),
    "plane": lambda: _gas(_lattice((37, 29))),
}


def _check(prob, precision, tol):
    from paper_1805_05128_gb300 import Simulation
    sim = Simulation(prob, precision=precision, units=0)
    gi, gj = sim.pair_list()
    g = sim.numpy()
    assert sim.read_status() == 0
    p, s = O.from_problem(prob)
    O.eval_rates(p, s)
    _, sd = O.from_problem(prob)
    sd.d[:] = g["d"]
    oi, oj = O.pairs(p, sd, "cells")
    assert np.array_equal(gi, oi) and np.array_equal(gj, oj) and len(gi) > 0
    for k in ["drho", "dE"] + ["a" + c for c in "xyz"[: prob.dim]]:
        ref = getattr(s, k)
        assert np.max(np.abs(g[k] - ref)) <= tol * np.max(np.abs(ref)), k
    sim.close()


@pytest.mark.parametrize("precision,tol", [("fp64", 1e-10), ("mixed", 1e-4)])
@pytest.mark.parametrize("name", list(SHAPES))
def test_group_shapes(name, precision, tol):
    _check(SHAPES[name](), precision, tol)


@pytest.mark.parametrize("scale", [2.0 ** -90, 2.0 ** 90])
def test_length_units_far_outside_fp32(scale):
    """FP64 handles hold any length unit: the search's FP32 frame is scaled by the cell edge."""
    pos = _lattice((9, 8, 7)) * scale
    _check(_gas(pos, sizes=scale), "fp64", 1e-10)


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
def test_instances_share_groups(precision):
    """Instances of 5 to 70 particles in one handle: the same bits as each alone."""
    from paper_1805_05128_gb300 import Simulation
    probs = [_gas(_lattice(d, seed=k + 1), seed=k) for k, d in enumerate([(5, 1, 1), (3, 3, 2), (7, 5, 2), (2, 2, 2), (4, 4, 4)])]
    sim = Simulation(probs, precision=precision, units=0, cell_cap=1 << 16)
    sim.eval_rates()
    g = sim.numpy()
    for b, q in enumerate(probs):
        one = Simulation(q, precision=precision, units=0)
        one.eval_rates()
        o = one.numpy()
        lo, hi = sim.inst_offsets[b], sim.inst_offsets[b + 1]
        for k in ("ax", "ay", "az", "drho", "dE"):
            if precision == "fp64":
                assert np.array_equal(g[k][lo:hi], o[k]), (b, k)
            else:   # the volume scale of the mixed packs follows the largest particle of the handle
                assert np.allclose(g[k][lo:hi], o[k], rtol=0, atol=1e-5 * np.max(np.abs(o[k]))), (b, k)
        one.close()
    sim.close()


def _check_step(prob, beta):
    """One FP64 step with lists against the oracle's."""
    from paper_1805_05128_gb300 import Simulation
    sim = Simulation(prob, precision="fp64", units=0, cell_beta=beta)
    sim.step(2)
    g = sim.numpy()
    assert sim.read_status() == 0
    half = sim.pair_counts()[0]
    p, s = O.from_problem(prob)
    O.step(p, s, 2)
    for k in ("x", "vx", "rho", "E", "ax", "drho", "dE"):
        ref = getattr(s, k)
        assert np.max(np.abs(g[k] - ref)) <= 1e-10 * np.max(np.abs(ref)), k
    _, sd = O.from_problem(prob)
    for k in "xyz"[: prob.dim]:
        getattr(sd, k)[:] = g[k]
    sd.d[:] = g["d"]
    assert half == len(O.pairs(p, sd, "cells")[0])
    sim.close()


@pytest.mark.parametrize("beta", [0.01, 0.15, 0.4])
def test_fp64_lists_longer_than_one_segment(beta):
    """Lists of up to several hundred entries (256 to a segment of the evaluation), most of them rejected at beta = 0.4."""
    prob = _gas(_lattice((11, 10, 9)))
    prob.eta = 2.15
    _check_step(prob, beta)


@pytest.mark.parametrize("scale", [2.0 ** -90, 2.0 ** 90])
def test_fp64_lists_in_any_length_unit(scale):
    _check_step(_gas(_lattice((7, 6, 5)) * scale, sizes=scale), 0.15)
