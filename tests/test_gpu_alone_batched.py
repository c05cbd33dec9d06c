"""What an instance of a batched handle gets is what it gets alone, bit for
bit, where the instances sharing the handle could show: the totals of
instances of any sizes, the list evaluation, whose warps form the rates of
slots of several groups and instances together, and the FP64 sums of
particles with so many neighbours that a group's lists are flushed in the
middle of its scan."""
import numpy as np
import pytest

import synth

torch = pytest.importorskip("torch")
from test_gpu_pair_groups import _gas, _lattice  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1805_05128_gb300 import build
    build.build()


@pytest.mark.parametrize("sizes", [(60, 9000), (31, 4096, 4097, 70000), (140000, 5, 20000, 8193, 33000)])
def test_totals_alone_and_batched(sizes):
    from paper_1805_05128_gb300 import Simulation
    probs = [_gas(_lattice((n,), seed=k + 1), seed=k) for k, n in enumerate(sizes)]
    sim = Simulation(probs, precision="fp64", units=0)
    got = sim.conservation().cpu().numpy()
    sim.close()
    for b, q in enumerate(probs):
        one = Simulation(q, precision="fp64", units=0)
        assert np.array_equal(one.conservation().cpu().numpy()[0], got[b]), sizes[b]
        one.close()


@pytest.mark.parametrize("order,solver", [(1, "acoustic"), (1, "hll"), (2, "acoustic")])
@pytest.mark.parametrize("before", [(1,), (5, 3), (7,) * 9])
def test_many_neighbours_alone_and_batched(before, order, solver):
    """Up to 330 neighbours, more than a list holds between two flushes (224)."""
    from paper_1805_05128_gb300 import Simulation
    probs = [_gas(_lattice((n, 1, 1), seed=n), seed=n) for n in before] + [_gas(_lattice((11, 9, 8)))]
    for q in probs:
        q.eta = 2.15
    pos = np.stack([probs[-1].arrays[k] for k in "xyz"])
    d = np.cbrt(probs[-1].arrays["m"] / probs[-1].arrays["rho"])
    near = np.linalg.norm(pos[:, :, None] - pos[:, None], axis=0) < 2.15 * (d[:, None] + d)
    assert near.sum(0).max() > 224
    kw = dict(precision="fp64", units=0, order=order, solver=solver)
    sim, one = Simulation(probs, cell_cap=1 << 18, **kw), Simulation(probs[-1], **kw)
    sim.eval_rates()
    one.eval_rates()
    g, o, lo = sim.numpy(), one.numpy(), sum(before)
    assert sim.read_status() == 0
    for k in ("ax", "ay", "az", "drho", "dE"):
        assert np.any(o[k]) and np.array_equal(g[k][lo:], o[k]), k
    sim.close()
    one.close()


@pytest.mark.parametrize("steps", [1, 4])
@pytest.mark.parametrize("blocks", [0, 1])
@pytest.mark.parametrize("small,large", [((3, 3, 2), (29, 27, 19)), ((5, 1, 1), (9, 8, 7)), ((1, 1, 1), (2, 2, 2))])
def test_lists_alone_and_batched(small, large, blocks, steps):
    """Small instances around a larger one: states, rates and times after steps with their own dt."""
    from paper_1805_05128_gb300 import Simulation
    probs = [_gas(_lattice(small, seed=k + 1), seed=k) for k in range(40)] + [_gas(_lattice(large))]
    probs += [_gas(_lattice(small, seed=k + 50), seed=k) for k in range(7)]
    kw = dict(precision="fp64", units=0, cell_beta=0.15, pair_blocks_per_sm=blocks)
    sim = Simulation(probs, cell_cap=1 << 20, **kw)
    sim.step(steps)
    g, t, entries = sim.numpy(), sim.time.cpu().numpy(), 0
    assert sim.read_status() == 0
    for b, q in enumerate(probs):
        one = Simulation(q, **kw)
        one.step(steps)
        o, lo, hi = one.numpy(), sim.inst_offsets[b], sim.inst_offsets[b + 1]
        assert t[b] == one.time.cpu().numpy()[0] > 0
        for k in ("x", "vx", "rho", "E", "ax", "ay", "az", "drho", "dE"):
            assert np.array_equal(g[k][lo:hi], o[k]), (b, k)
        entries += one.pair_counts()[1]
        one.close()
    assert sim.pair_counts()[1] == entries
    sim.close()
