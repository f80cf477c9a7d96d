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


def _one_path_params(m, w2, b2):
    """Parameters whose only path is x1[0] = tanh(20) = 1, z2[0] = w2 x1[0] + b2, E = 2^20 tanh(z2[0])."""
    D, H1, H2, _ = m.widths
    W1, b1, W2, B2, w3 = np.zeros((H1, D)), np.zeros(H1), np.zeros((H2, H1)), np.zeros(H2), np.zeros(H2)
    b1[0], W2[0, 0], B2[0], w3[0] = 20.0, w2, b2, 2.0 ** 20
    p = np.concatenate([W1.ravel(), b1, W2.ravel(), B2, w3, [0.0]])
    return np.tile(p, (m.n_species, 1))


@pytest.mark.parametrize("precision", ["bf16", "bf16x3"])
@pytest.mark.parametrize("orders,fused", [(None, False), ((7, 5), True)])
def test_three_kernel_bias_is_added_in_fp32(gpu_mod, precision, orders, fused):
    """The three-kernel path, by the option or by the basis: 0.5 plus 3/4 of its last
    place rounds up. Summed by the tensor cores, which cut off, it would stay 0.5."""
    st = inputs.water(32, None, 3)
    m = inputs.make_model("water", hidden=(15, 15), orders=orders)
    g = gpu_mod.AenetGPU(m, precision)
    g.fuse_network(fused)

    def e_atom(w2, b2):
        g.set_params(_one_path_params(m, w2, b2))
        return g.compute(st.pos, st.types, st.box)["e_atom"]

    up = e_atom(0.0, 0.5 + 2.0 ** -24)
    assert not np.array_equal(up, e_atom(0.0, 0.5))
    assert np.array_equal(e_atom(0.75 * 2.0 ** -24, 0.5), up)


@pytest.mark.parametrize("precision", ["fp32", "bf16x3"])
def test_host_parameters_are_in_place_on_return(gpu_mod, precision):
    """set_params from a host array, then another stream: nothing may be left running
    on the stream before."""
    m = inputs.make_model("water", hidden=(32, 32))
    a, b = torch.cuda.Stream(), torch.cuda.Stream()
    with torch.cuda.stream(a):
        g = gpu_mod.AenetGPU(m, precision)
    assert a.query()
    for k in range(100):
        g.set_stream(a.cuda_stream if k % 2 else b.cuda_stream)
        g.set_params(m.params)
        assert (a if k % 2 else b).query()


@pytest.mark.parametrize("n", [60, 120, 162])
def test_lists_that_leave_room_for_few_warps(gpu_mod, n):
    """The solid's basis in a 6 A box: lists so long that a CTA of the list kernel holds
    five, two and one of them (descriptors: six, three, two); its tables are then filled
    by as few warps.

    Coefficients: sums of N products in FP32, N / 32 + 8 roundings deep at most, and
    |b| of T_a's Legendre series sums up to less than 3, twice (A^2) that in the angular
    ones: 6 (N / 32 + 8) units of the a = 0 coefficient. Forces: from coefficients good to
    some 300 units, and sums that cancel to the root of their N terms: 1e-3."""
    rng = np.random.default_rng(n)
    box = np.full(3, 6.0)
    pts = []
    while len(pts) < n:
        p = rng.uniform(0, 6.0, 3)
        if all((((p - q + 3.0) % 6.0 - 3.0) ** 2).sum() > 0.3 ** 2 for q in pts):
            pts.append(p)
    pos, types = np.array(pts), rng.integers(0, 4, n).astype(np.int32)
    m = inputs.make_model("amorphous")
    G = O.compute(m, pos, types, box, want_G=True)["G"]
    m.in_shift[:], m.in_scale[:] = G.mean(0), 1.0 / np.maximum(G.std(0), 1e-2 * np.abs(G).max(0))
    ref = O.compute(m, pos, types, box)
    g = gpu_mod.AenetGPU(m, "fp32")
    Kr, Ka, smax = m.order_rad + 1, m.order_ang + 1, float(np.abs(m.type_weights).max())
    unit = np.concatenate([np.full((n, Kr), 1.0) * G[:, [0]], np.full((n, Ka), 1.0) * G[:, [Kr]]], 1)
    unit = np.concatenate([unit, np.concatenate([smax * unit[:, :Kr], smax ** 2 * unit[:, Kr:]], 1)], 1)
    N = n / 216.0 * 4.18879 * 8.0 ** 3
    assert (np.abs(g.descriptors(pos, types, box) - G) <= 6 * (N / 32 + 8) * 2.0 ** -24 * unit + 1e-6).all()
    out = g.compute(pos, types, box)
    rms = np.sqrt((ref["forces"] ** 2).mean())
    assert rms > 1e-4
    assert np.sqrt(((out["forces"] - ref["forces"]) ** 2).mean()) <= 1e-3 * rms
    assert np.abs(out["e_atom"] - ref["e_atom"]).max() <= 1e-3 * max(1.0, np.abs(ref["e_atom"]).max())


@pytest.mark.parametrize("precision,hidden", [("fp32", (15, 15)), ("bf16x3", (15, 15)), ("fp32", (48, 48))])
def test_slices_of_rows_give_what_one_slice_gives(gpu_mod, precision, hidden):
    """24,000 atoms after a structure so dense (two atoms in 0.73 A^3) that the lists it
    sizes fill a slice of rows with some 20,500 atoms, against a context that never saw it:
    the fused, the three-kernel and the wide FP32 path, descriptors and a batch. Sums in
    another order, in FP32: a few units of 2^-24 of an atom's terms, 5e-6 of the RMS;
    through the split-BF16 network, whose products drop 2^-16 of a factor, 1e-4."""
    m = inputs.make_model("water", hidden=hidden)
    st, half = inputs.water(8000, None, 5), inputs.water(4000, None, 6)
    dense = np.array([[0.1, 0.2, 0.3], [0.55, 0.65, 0.75]]), np.array([0, 1], np.int32), np.full(3, 0.9)
    off = np.array([0, 12000, 24000])
    both = np.concatenate([half.pos, half.pos + 0.3]), np.tile(half.types, 2), np.stack([half.box] * 2)

    def results(after):
        g = gpu_mod.AenetGPU(m, precision)
        if after:
            g.fuse_network(False)  # (few atoms otherwise take the fused kernel, which has no room for such lists)
            g.compute(*dense)
            g.fuse_network(True)
        r = dict(g.compute(st.pos, st.types, st.box), stats=np.array(g.neighbor_stats()))
        r["G"] = g.descriptors(st.pos, st.types, st.box)
        r["G_stats"] = np.array(g.neighbor_stats())
        b = g.compute_batch(off, both[0], both[1], both[2])
        r.update({"b_" + k: v for k, v in b.items()}, b_stats=np.array(g.neighbor_stats()))
        return r

    one, many = results(False), results(True)
    tol = 5e-6 if precision == "fp32" else 1e-4
    for k, x in one.items():
        if k.endswith("stats"):
            assert x.min() > 0 and np.array_equal(x, many[k]), k
        else:
            x, y = np.asarray(x, dtype=np.float64), np.asarray(many[k], dtype=np.float64)
            assert np.sqrt(((x - y) ** 2).mean()) <= (5e-6 if k == "G" else tol) * np.sqrt((x ** 2).mean()), k


@pytest.mark.parametrize("mode", ["off", "on", "auto"])
@pytest.mark.parametrize("steps", [1, 3])
def test_continued_md_records_the_frame_it_starts_from(gpu_mod, mode, steps):
    """The third of three MD calls of the same shape (the second replays the first's
    captured step) continues the second: its frame 0 is the second's last one. Two
    reductions of the same FP32 numbers, so equal in every bit."""
    st = inputs.water(64, None, 4)
    m = inputs.make_model("water")
    g = gpu_mod.AenetGPU(m, "fp32")
    g.md_list(mode)
    pos = torch.as_tensor(st.pos, device="cuda")
    vel = torch.as_tensor(inputs.maxwell_boltzmann(m.masses[st.types], 300.0, seed=2), device="cuda")
    types = torch.as_tensor(st.types, device="cuda")
    e = [np.zeros(steps + 1) for _ in range(3)]
    for k in range(3):
        g.md_nve(pos, vel, types, st.box, 2.5e-4, steps, e[k], None, gpu_mod.AENET_MD_CONTINUE if k == 2 else 0)
    assert abs(e[1][0] - e[1][-1]) > 1e-6
    assert e[2][0] == e[1][-1]


@pytest.mark.parametrize("skin", [0.0, 0.5])
def test_md_after_descriptors_starts_from_its_forces(gpu_mod, skin):
    """Descriptors between two MD calls, the second, of one step, with AENET_MD_CONTINUE:
    x1 = x0 + dt v0 + dt^2 / 2 F(x0) c / m, so the step shows the forces it started from.
    They are those of a separate evaluation up to the order of FP32 sums: 5e-6 of the RMS."""
    st = inputs.water(64, None, 4)
    m = inputs.make_model("water")
    g = gpu_mod.AenetGPU(m, "fp32")
    g.set_skin(skin)
    dt, mass = 2.5e-4, m.masses[st.types][:, None]
    pos, vel = st.pos.copy(), inputs.maxwell_boltzmann(m.masses[st.types], 300.0, seed=2)
    g.md_nve(pos, vel, st.types, st.box, dt, 4)
    x0, v0 = pos.copy(), vel.copy()
    g.descriptors(st.pos[::-1].copy(), st.types[::-1].copy(), st.box)
    g.md_nve(pos, vel, st.types, st.box, dt, 1, flags=gpu_mod.AENET_MD_CONTINUE)
    F = 2.0 * (pos - x0 - dt * v0) / dt ** 2 * mass / inputs.EV_PER_AMU
    ref = gpu_mod.AenetGPU(m, "fp32").compute(x0, st.types, st.box)["forces"]
    rms = np.sqrt((ref ** 2).mean())
    assert rms > 0.1
    assert np.sqrt(((F - ref) ** 2).mean()) <= 5e-6 * rms


def test_path_flags_follow_the_last_captured_step(gpu_mod):
    """Pipelined, then not, then over a Verlet list with the pipelined frame 0."""
    st, m = inputs.water_192(), inputs.make_model("water")
    vel = inputs.maxwell_boltzmann(m.masses[st.types], 300.0, seed=2)
    g = gpu_mod.AenetGPU(m, "fp32")
    got = []
    for pipeline, skin in ((True, 0.0), (False, 0.0), (True, 0.5), (True, 0.5)):
        g.pipeline(pipeline)
        g.set_skin(skin)
        g.md_nve(st.pos.copy(), vel.copy(), st.types, st.box, 5e-4, 2, flags=gpu_mod.AENET_MD_TIMING)
        got.append(g.md_path_flags() & (gpu_mod.AENET_PATH_PIPELINED | gpu_mod.AENET_PATH_ROWS))
    assert got == [gpu_mod.AENET_PATH_PIPELINED, gpu_mod.AENET_PATH_ROWS, 0, 0]


def _shell(n, radius):
    """n atoms spread over a sphere (a golden spiral): all within its diameter of one another."""
    k = np.arange(n) + 0.5
    z, a = 1.0 - 2.0 * k / n, np.pi * (1.0 + 5.0 ** 0.5) * k
    s = np.sqrt(1.0 - z * z)
    return radius * np.stack([s * np.cos(a), s * np.sin(a), z], 1)


@pytest.mark.parametrize("skin", [0.0, 0.5])
def test_an_atom_may_have_as_many_neighbours_as_its_list(gpu_mod, skin):
    """65 atoms with exactly 64 neighbours each, the capacity that a sparse system's first
    call sets: an asynchronous evaluation, which cannot regrow it, and MD."""
    pos, box = _shell(65, 2.98) + 20.0, np.full(3, 40.0)
    r = np.linalg.norm(pos[:, None] - pos[None], axis=2)
    assert r.max() < 6.0 and ((r < 4.0).sum(1) - 1).max() <= 32
    types = (np.arange(65) % 3 > 0).astype(np.int32)
    m = inputs.make_model("water")
    ref = O.compute(m, pos, types, box)
    g = gpu_mod.AenetGPU(m, "fp32")
    g.compute(pos[:2], types[:2], box)
    p, t = torch.as_tensor(pos, device="cuda"), torch.as_tensor(types, device="cuda")
    F = torch.zeros((65, 3), dtype=torch.float64, device="cuda")
    g.compute_async(p, t, box, forces=F)
    g.check()
    rms = np.sqrt((ref["forces"] ** 2).mean())
    assert np.sqrt(((F.cpu().numpy() - ref["forces"]) ** 2).mean()) <= max(1e-4, 2e-5 * rms)
    g.set_skin(skin)
    g.md_nve(p, torch.zeros_like(p), t, box, 1e-6, 2)


@pytest.mark.parametrize("n", [4096, 4097])
def test_host_and_device_arrays_mixed(gpu_mod, n):
    """Both sides of the size up to which host arrays go through mapped memory, every
    array in turn on the host and on the device, against the call with all of them on the
    device: the same sums in FP32 in another order, 5e-6 of the RMS."""
    st = inputs.amorphous(n, seed=11)
    g = gpu_mod.AenetGPU(inputs.make_model("amorphous"), "fp32")
    shapes = {"energy": (1,), "forces": (n, 3), "virial": (3, 3), "e_atom": (n,)}

    def arrays(host):
        given = [torch.as_tensor(st.pos), torch.as_tensor(st.types)]
        given = [x.numpy() if k in host else x.cuda() for k, x in zip(("pos", "types"), given)]
        out = {k: np.zeros(s) if k in host else torch.zeros(s, dtype=torch.float64, device="cuda")
               for k, s in shapes.items()}
        g.compute(*given, st.box, **out)
        return {k: np.array(v) if k in host else v.cpu().numpy() for k, v in out.items()}

    ref = arrays(())
    for host in (("pos",), ("types",), ("forces",), ("e_atom", "energy"), ("virial",), ("pos", "types", "e_atom"),
                 ("pos", "types", "energy", "forces", "virial", "e_atom")):
        for k, x in arrays(host).items():
            assert np.sqrt(((x - ref[k]) ** 2).mean()) <= 5e-6 * np.sqrt((ref[k] ** 2).mean()), (host, k)


@pytest.mark.parametrize("family,n", [("water", 4095), ("water", 4098), ("amorphous", 1024), ("amorphous", 1025)])
def test_split_bf16_on_both_sides_of_the_fused_sizes(gpu_mod, family, n):
    """Energies, forces and the weight gradient where the fused tensor-core kernel gives way
    to the three kernels, against the FP32 form. The split drops 2^-16 of a factor: 1e-4
    of the RMS (E_i, forces); 1e-3 of the largest gradient, a sum over all atoms whose
    terms partly cancel."""
    st = inputs.water(n // 3, None, 7) if family == "water" else inputs.amorphous(n, seed=7)
    m = inputs.make_model(family)
    res = {}
    for precision in ("fp32", "bf16x3"):
        g = gpu_mod.AenetGPU(m, precision)
        g.keep_activations(True)
        res[precision] = dict(g.compute(st.pos, st.types, st.box), dEdW=g.grad_weights())
    a, b = res["fp32"], res["bf16x3"]
    for k in ("e_atom", "forces"):
        assert np.sqrt(((a[k] - b[k]) ** 2).mean()) <= 1e-4 * np.sqrt((a[k] ** 2).mean()), k
    assert np.abs(a["dEdW"] - b["dEdW"]).max() <= 1e-3 * np.abs(a["dEdW"]).max()


@pytest.mark.parametrize("box", [None, 70.0])
def test_md_turn_equals_single_steps(gpu_mod, box):
    """Four steps in one call (one kernel between two potentials) against four calls of one
    step, on a grid that the turn scans itself and on one of 1,331 cells that it leaves to
    the scan kernel. The FP64 steps are the same; the forces differ by the order of their
    FP32 sums, 5e-6 of the largest: positions by that acceleration over four steps."""
    st = inputs.water(512, box, 8)
    m = inputs.make_model("water")
    dt, mass = 2.5e-4, m.masses[st.types][:, None]
    v0 = inputs.maxwell_boltzmann(m.masses[st.types], 300.0, seed=2)
    g = gpu_mod.AenetGPU(m, "fp32")
    a = np.abs(g.compute(st.pos, st.types, st.box)["forces"] / mass).max() * inputs.EV_PER_AMU
    many, e = (st.pos.copy(), v0.copy()), (np.zeros(5), np.zeros(5))
    g.md_nve(*many, st.types, st.box, dt, 4, *e)
    one, e_pot, e_kin = (st.pos.copy(), v0.copy()), [], []
    for k in range(4):
        ep, ek = np.zeros(2), np.zeros(2)
        g.md_nve(*one, st.types, st.box, dt, 1, ep, ek, gpu_mod.AENET_MD_CONTINUE if k else 0)
        e_pot += list(ep if k == 0 else ep[1:])
        e_kin += list(ek if k == 0 else ek[1:])
    assert np.abs(many[0] - one[0]).max() <= 5e-6 * a * (4 * dt) ** 2
    assert np.abs(many[1] - one[1]).max() <= 5e-6 * a * 4 * dt
    np.testing.assert_allclose(e[0], e_pot, atol=2e-6 * st.n)
    np.testing.assert_allclose(e[1], e_kin, rtol=1e-5)


def test_verlet_lists_without_room_are_a_capacity_error(gpu_mod):
    """Five atoms in 1 A^3: one warp's lists fit a CTA, with the 3,375 image offsets of the
    Verlet list's grid beside them they do not."""
    m = inputs.make_model("water")
    g = gpu_mod.AenetGPU(m, "fp32")
    pos = np.array([[0.1, 0.1, 0.1], [0.6, 0.6, 0.1], [0.6, 0.1, 0.6], [0.1, 0.6, 0.6], [0.35, 0.35, 0.35]])
    types, box = np.array([0, 1, 1, 0, 1], np.int32), np.full(3, 1.0)
    g.set_skin(0.5)
    with pytest.raises(gpu_mod.AenetError) as e:
        g.md_nve(pos.copy(), np.zeros((5, 3)), types, box, 1e-6, 2)
    assert e.value.code == -3
    g.set_skin(0.0)
    g.md_nve(pos.copy(), np.zeros((5, 3)), types, box, 1e-6, 2)
