"""What an instance of a batched handle gets is what it gets alone, bit for
bit, where the instances sharing the handle could show: the totals of
instances of any sizes."""
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
