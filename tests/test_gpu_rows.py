"""Evaluation over neighbour rows: sums, capacities and state that one small
evaluation against the oracle does not show."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2107_11311_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def gpu_mod():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2107_11311_gb300 import aenet
    return aenet


def _dimers(k, d=(0.5625, 0.625, 0.40625)):
    """k^3 O-H pairs, all at the same place of a cell of 6 A (the water basis' cutoff)
    and out of reach of one another, in coordinates that FP32 holds exactly."""
    at = 12.0 * np.stack(np.meshgrid(*[np.arange(k)] * 3, indexing="ij"), -1).reshape(-1, 1, 3) + 2.0
    pos = np.concatenate([at, at + np.array(d)], 1).reshape(-1, 3)
    return pos, np.tile(np.array([0, 1], np.int32), k ** 3), np.full(3, 12.0 * k)


@pytest.mark.parametrize("precision", ["fp32", "bf16x3"])
def test_virial_is_summed_in_fp64(gpu_mod, precision):
    """21,296 atoms, seven a warp: every pair has the same virial, a sum of two FP32
    numbers, so the total in FP64 is exactly their number times it (24 + 15 bits).
    Sums that a warp carries in FP32 from atom to atom round at 2^-24."""
    k = 22
    pos, types, box = _dimers(k)
    g = gpu_mod.AenetGPU(inputs.make_model("water", hidden=(20, 20)), precision)
    g.fuse_network(False)
    total, one = g.compute(pos, types, box), g.compute(pos[:2], types[:2], box)
    assert np.abs(one["virial"]).min() > 1e-4
    assert np.array_equal(total["virial"], k ** 3 * one["virial"])
