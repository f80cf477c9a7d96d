"""The list build and the list-driven potential kernel at the sizes where they
can go wrong, against the oracle: angular neighbour counts around the 32-entry
blocks, atom counts around one warp and one block, boxes shorter than the cutoff
(self-images, several staging chunks), every kernel form of the basis, and rows
evaluated in slices."""
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


def _compare(g, m, pos, types, box):
    """FP32 against FP64: the error of a sum of products is a small multiple of
    2^-24 of the terms' magnitude; 300 units (2e-5) of the RMS force, and the
    absolute parity bounds for small forces."""
    ref = O.compute(m, pos, types, box)
    out = g.compute(pos, types, box)
    n = len(pos)
    rms = float(np.sqrt((ref["forces"] ** 2).mean()))
    scale = max(1.0, float(np.abs(ref["e_atom"]).max()))
    assert np.abs(out["e_atom"] - ref["e_atom"]).max() <= 2e-5 * scale
    assert abs(out["energy"] - ref["energy"]) <= 2e-5 * scale * n
    assert np.sqrt(((out["forces"] - ref["forces"]) ** 2).mean()) <= max(1e-4, 2e-5 * rms)
    wmax = max(1.0, np.abs(ref["virial"]).max())
    np.testing.assert_allclose(out["virial"], ref["virial"], atol=1e-4 * wmax)
    return ref


def _cluster(k, n_species, seed):
    """k atoms in a ball of radius 1.9 A (all within 3.8 A of one another), no two
    closer than 0.25 A, in a box wide enough that no image is within the cutoff."""
    rng = np.random.default_rng(seed)
    pts = []
    while len(pts) < k:
        p = rng.uniform(-1.9, 1.9, 3)
        if p @ p <= 1.9 ** 2 and all(((p - q) ** 2).sum() > 0.25 ** 2 for q in pts):
            pts.append(p)
    return np.array(pts) + 1.0, rng.integers(0, n_species, k).astype(np.int32)


@pytest.mark.parametrize("k", [1, 2, 3, 4, 32, 33, 34, 35, 64, 65, 66, 97])
def test_angular_blocks(gpu_mod, k):
    """k - 1 angular neighbours per atom: none, odd and even rings, the last ring
    of one block (32), two blocks (33, ...), three and four."""
    m = inputs.make_model("water")
    pos, types = _cluster(k, 2, seed=k)
    _compare(gpu_mod.AenetGPU(m, "fp32"), m, pos, types, np.full(3, 13.0))


@pytest.mark.parametrize("family,hidden,orders", [("water", (15, 15), (7, 5)), ("water", (32, 32), (12, 10)),
                                                  ("water", (20,), (22, 6)), ("water", (9, 8, 7), None),
                                                  ("amorphous", (16, 3), None), ("amorphous", (30, 30), None),
                                                  ("amorphous", (12, 12), (9, 5))])
def test_kernel_forms(gpu_mod, family, hidden, orders):
    """Every form of the basis and both width bounds: one dense box (more than
    32 angular neighbours with the solid's cutoff) and one small one."""
    m = inputs.make_model(family, hidden=hidden, orders=orders)
    g = gpu_mod.AenetGPU(m, "fp32")
    for st in (inputs.water(37, None, 5), inputs.water(8, 6.6, 2)) if family == "water" else \
            (inputs.amorphous(200, seed=3), inputs.amorphous(32, seed=4)):
        _compare(g, m, st.pos, st.types, st.box)


@pytest.mark.parametrize("family,n,box", [("water", 1, 5.0), ("water", 2, 4.0), ("water", 9, 40.0),
                                          ("amorphous", 1, 4.5), ("amorphous", 5, 5.0), ("amorphous", 1, 90.0)])
def test_few_atoms(gpu_mod, family, n, box):
    """Fewer atoms than a warp has lanes or a CTA warps; boxes shorter than the
    cutoff, whose atoms see themselves in up to 11^3 images (several chunks)."""
    m = inputs.make_model(family)
    rng = np.random.default_rng(n)
    pos = np.array([[0.3, 0.1, 0.2], [1.7, 0.4, 0.0], [0.0, 1.9, 1.1], [2.0, 2.1, 0.3], [0.4, 0.2, 2.4]] * 2)[:n]
    pos = pos + 0.01 * np.arange(n)[:, None] + (3.0 * (np.arange(n) // 5))[:, None]
    _compare(gpu_mod.AenetGPU(m, "fp32"), m, pos, rng.integers(0, m.n_species, n).astype(np.int32), np.full(3, box))


def test_rows_in_slices(gpu_mod):
    """663,552 atoms: their rows exceed one slice (1 GiB), so the second slice's
    forces add to atoms of the first; forces of atoms of the cells around the
    slice boundary and of both ends against the oracle."""
    st = inputs.water(221184, None, 9)
    m = inputs.make_model("water")
    g = gpu_mod.AenetGPU(m, "fp32")
    out = g.compute(st.pos, st.types, st.box)
    L = st.box[2]
    z = st.pos[:, 2] % L
    # sorted by cell with z slowest: a boundary between slices lies in a z-layer of cells
    centres = np.concatenate([np.flatnonzero(np.abs(z - f * L) < 0.3)[:24] for f in np.linspace(0.02, 0.98, 33)])
    F, _ = O.forces_subset(m, st.pos, st.types, st.box, centres)
    assert np.sqrt(((out["forces"][centres] - F) ** 2).mean()) <= 1e-4
    assert np.abs(out["forces"].sum(axis=0)).max() <= 5e-3 * np.sqrt(st.n)
