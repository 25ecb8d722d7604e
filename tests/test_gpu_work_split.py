"""The step's kernels at the edges of their work splits (needs a GB300), against the oracle.

The oracle evaluates every node of every pair in FP64 in its own order; the
tolerances are those of the parity tests (tests/parity.py).
"""
import numpy as np
import pytest

import oracle
from paper_2401_10878_gb300 import workloads as W
from tests.helpers import cube_planes, quat_axis_angle, state
from tests.parity import compare, gpu_step
from tests.test_gpu_box_pipeline import boxed
from tests.test_gpu_box_pipeline import run as run_box

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _parity(st, precision, **kw):
    from paper_2401_10878_gb300.contact import Contact
    m = Contact.from_state(st, precision=precision, **kw)
    g = gpu_step(m, st)
    r = oracle.contact_step(st)
    rep = compare(st, g, r, fp64=precision == 1, smooth=st.indicator == 1)
    m.close()
    return rep, r


# half extents across the lines of the pair box: 100, 121, 128 (one tile exactly), 144 and 20^2 lines (four tiles)
@pytest.mark.parametrize("across", [(5.0, 5.0), (5.5, 5.5), (8.0, 4.0), (6.0, 6.0), (10.0, 10.0)])
@pytest.mark.parametrize("indicator", [0, 1])
@pytest.mark.parametrize("kind", ["cuboid", "polytope"])
def test_fp64_form_at_tile_edges(across, indicator, kind):
    """Two slightly turned boxes pressed together over a whole face: hundreds
    of nodes on lines filling one tile or several."""
    h = (5.0, across[0], across[1])
    q = [quat_axis_angle([0.3, 1.0, 0.2], 0.02), quat_axis_angle([1.0, 0.1, 0.4], 0.03)]
    t, planes = (W.CUBOID, None) if kind == "cuboid" else (W.POLYTOPE, [cube_planes(h)] * 2)
    st = state([t] * 2, [h, h], [[30.23, 31.31, 32.17], [38.11, 31.12, 31.94]], quat=q, n=96, planes=planes,
               indicator=indicator)
    rep, ref = _parity(st, 1)
    assert ref.n_pairs == 1 and ref.pair_out[0, 0] > 100.0


def _crowd(n_small):
    """A ball and n_small small ones around it: the first row holds n_small partners."""
    k = np.arange(n_small) + 0.5
    th, ph = np.arccos(1.0 - 2.0 * k / n_small), np.pi * (1.0 + 5.0 ** 0.5) * k
    u = np.stack([np.sin(th) * np.cos(ph), np.sin(th) * np.sin(ph), np.cos(th)], 1)
    c = np.array([31.13, 32.21, 30.87])
    return state([W.SPHERE] * (n_small + 1), [[9.0, 0, 0]] + [[1.6, 0, 0]] * n_small,
                 np.concatenate([c[None], c + u * 9.5]), n=64)


# partners of one row: at and around the eight fetched ahead, and more than one warp round of pairs
@pytest.mark.parametrize("n_small", [1, 7, 8, 9, 31, 33, 60])
def test_pair_builder_rows(n_small):
    st = _crowd(n_small)
    rep, ref = _parity(st, 0)
    assert np.sum(ref.pair_ij[:, 0] == 0) == n_small


# partners of one particle around the eight read at a time, overlapping ones among them around the two
@pytest.mark.parametrize("n_small", [1, 2, 3, 7, 8, 9, 16, 17, 60])
@pytest.mark.parametrize("every", [1, 2, 5])
@pytest.mark.parametrize("last", [False, True])
def test_particle_sums_of_overlapping_pairs(n_small, every, last):
    """The forces are the pairs' forces added in FP64 in partner order, bit for
    bit: the ball first (partners above it) or last (below it), one partner in
    `every` pressed into it and the others near."""
    from paper_2401_10878_gb300.contact import Contact
    st = _crowd(n_small)
    st.shape_param[1:, 0] = np.where(np.arange(n_small) % every == 0, 1.6, 0.4)
    if last:
        st.shape_param[:] = st.shape_param[::-1].copy()
        st.pos[:] = st.pos[::-1].copy()
    m = Contact.from_state(st)
    g = gpu_step(m, st)
    m.close()
    want = np.zeros((n_small + 1, 3))
    for lower in (True, False):   # as j, by i; then as i, by j
        for (i, j), row in zip(g["pair_ij"], g["pair_out"]):
            if lower:
                want[j] = want[j] + row[8:11]
            else:
                want[i] = want[i] - row[8:11]
    assert np.array_equal(g["force"], want)
    assert np.count_nonzero(g["pair_out"][:, 0]) >= (n_small + every - 1) // every


# node ranges whose length the ten bits of a bin entry hold, and ones they do not
@pytest.mark.parametrize("half", [505.3, 511.3, 530.3])
@pytest.mark.parametrize("gap", [7.1, 8.1])
def test_broad_phase_long_ranges(half, gap):
    """Axis-aligned rods across the periodic boundary, overlapping (7.1) or with ranges one node apart (8.1)."""
    n = int(4 * half) + 60
    st = state([W.CUBOID] * 3, [[half, 4.3, 4.2]] * 3,
               [[5.2, 20.3, 40.4], [n - 300.3, 20.3 + gap, 41.7], [n / 2 + 3.3, 90.0, 40.1]], n=n)
    rep, ref = _parity(st, 0)
    assert ref.n_pairs == (1 if gap < 8.0 else 0) and np.all(ref.pair_out[:, 0] > 0)


# candidates of one particle: at and around the 96 listed at a time, then the
# most particles of one warp each and the fewest of half a warp each (odd and even)
@pytest.mark.parametrize("n", [94, 95, 96, 97, 191, 192, 193, 215, 4864, 4865, 4866])
@pytest.mark.parametrize("corner", [30.3, -9.6])
def test_broad_phase_crowded_bins(n, corner):
    """Small spheres on a jittered lattice around a larger one that sets the
    bins' width, inside the box and across its corner; more of them spread over
    the box for the larger counts."""
    rng = np.random.default_rng(n)
    box = 160 if n > 215 else 64
    a = np.stack(np.meshgrid(*[np.arange(6)] * 3, indexing="ij"), -1).reshape(-1, 3)
    x = corner + 3.4 * a + rng.uniform(-0.4, 0.4, (216, 3))
    if n > 215:
        g = np.stack(np.meshgrid(*[np.arange(18)] * 3, indexing="ij"), -1).reshape(-1, 3)
        f = 8.8 * g + 4.0 + rng.uniform(-0.4, 0.4, g.shape)
        near = np.all(np.abs(f - (corner + 8.5) - box * np.round((f - (corner + 8.5)) / box)) < 14.0, axis=1)
        x = np.concatenate([x, f[~near]])
    order = rng.permutation(n)
    x = np.mod(x[:n][order], box)
    r = np.where(order == 61, 4.4, 2.1)
    st = state([W.SPHERE] * n, np.stack([r, 0 * r, 0 * r], 1), x, n=box)
    rep, ref = _parity(st, 0)
    assert ref.n_pairs > 60


# one line and sample per direction up to the most, around the 32 lanes of a warp
@pytest.mark.parametrize("nc", [1, 2, 5, 6, 7, 33])
@pytest.mark.parametrize("kinds", ["grid", "cubes_walls", "polytopes"])
def test_box_pipeline_line_grids(nc, kinds):
    """Spheres with cubes, cubes with walls (every line of a wall's face ties)
    and polytopes, each kernel variant of the box pipeline."""
    if kinds == "grid":
        st = W.mixed_grid_27()
    elif kinds == "cubes_walls":
        st = W.floor_and_ceiling(state([W.CUBOID] * 3, [[6.0, 6.0, 6.0]] * 3,
                                       [[20.3, 20.6, 20.2], [31.1, 20.9, 21.3], [44.4, 44.1, 43.7]],
                                       quat=[[1.0, 0.0, 0.0, 0.0], quat_axis_angle([0.2, 1.0, 0.1], 0.3),
                                             quat_axis_angle([1.0, 0.3, 0.5], 0.7)]), gap=4.0)
    else:
        rng = np.random.default_rng(5)
        pl = [W.random_polytope(rng, 14, 9.0)[0] for _ in range(2)]
        st = state([W.POLYTOPE] * 2, [[0, 0, 0]] * 2, [[25.2, 26.1, 25.7], [30.9, 27.8, 26.6]], n=64, planes=pl,
                   quat=W.random_quaternions(rng, 2))
    rep, ref = run_box(boxed(st, nc))
    assert ref.n_pairs > 0


# faces of a polytope, one per lane in the box correction: few, and up to a lane each
@pytest.mark.parametrize("faces", [5, 12, 31, 32])
@pytest.mark.parametrize("other", ["sphere", "polytope", "wall"])
def test_box_pipeline_polytope_faces(faces, other):
    k = np.arange(faces) + 0.5
    th, ph = np.arccos(1.0 - 2.0 * k / faces), np.pi * (1.0 + 5.0 ** 0.5) * k
    n = np.stack([np.sin(th) * np.cos(ph), np.sin(th) * np.sin(ph), np.cos(th)], 1)
    pl = np.concatenate([n, np.full((faces, 1), 5.0)], 1)
    c = np.array([25.2, 26.1, 25.7])
    q = [quat_axis_angle([0.3, 1.0, 0.2], 0.4), quat_axis_angle([1.0, 0.1, 0.4], 0.9)]
    if other == "wall":
        st = W.with_walls(state([W.POLYTOPE], [[0, 0, 0]], [c], quat=q[:1], n=96, planes=[pl]), [[1.0, 0, 0, c[0] + 3.3]])
    else:
        kinds = [W.POLYTOPE, W.POLYTOPE if other == "polytope" else W.SPHERE]
        st = state(kinds, [[0, 0, 0], [5.0 * (other == "sphere"), 0, 0]], [c, c + [6.3, 1.2, -0.9]], quat=q, n=96,
                   planes=[pl, pl if other == "polytope" else None])
    rep, ref = run_box(boxed(st, 8))
    assert ref.pair_out[0, 0] > 0.0


# clipped nodes per tile: about one per line (at the limit above which a block shares a tile), several, many
@pytest.mark.parametrize("pen", [0.6, 1.1, 1.6, 3.2, 9.0])
@pytest.mark.parametrize("indicator", [0, 1])
@pytest.mark.parametrize("half", [5.6, 5.9, 12.0])
def test_shared_tiles_of_cubes(pen, indicator, half):
    """Cubes pressed together over a whole face, alone and with a third one
    aside: few tiles of many node passes."""
    q = [quat_axis_angle([0.3, 1.0, 0.2], 0.004), quat_axis_angle([1.0, 0.1, 0.4], 0.006), quat_axis_angle([1, 1, 0], 0.9)]
    c = np.array([40.23, 41.31, 42.17])
    st = state([W.CUBOID] * 3, [[half] * 3] * 3, [c, c + [2 * half - pen, 0.21, -0.17], c + [0.3, 1.9 * half, 7.7]],
               quat=q, n=128, indicator=indicator)
    rep, ref = _parity(st, 0)
    assert ref.pair_out[0, 0] > 0.0


# the same for the other kinds: tiles of about 128 clipped nodes (the limit of sharing) and of many node passes
@pytest.mark.parametrize("pen", [0.6, 1.1, 2.2, 7.0])
@pytest.mark.parametrize("indicator", [0, 1])
@pytest.mark.parametrize("kinds", ["sphere-sphere", "cuboid-sphere", "cuboid-cuboid", "cube-cuboid", "polytope-polytope",
                                   "polytope-sphere", "cuboid-polytope", "cube-wall", "polytope-wall"])
def test_shared_tiles_of_other_kinds(pen, indicator, kinds):
    """Two particles pressed together along x (a face on a face where they have
    one), or one pressed on a wall."""
    h = {"sphere": (14.0, 0, 0), "cuboid": (5.0, 9.0, 7.3), "cube": (6.0,) * 3, "polytope": (5.2, 8.1, 7.7)}
    code = {"sphere": W.SPHERE, "cuboid": W.CUBOID, "cube": W.CUBOID, "polytope": W.POLYTOPE}
    a, b = kinds.split("-")
    ks = [a] if b == "wall" else [a, b]
    c = np.array([40.23, 41.31, 42.17])
    pos = [c] if b == "wall" else [c, c + [h[a][0] + h[b][0] - pen, 0.21, -0.17]]
    q = [quat_axis_angle([0.3, 1.0, 0.2], 0.004), quat_axis_angle([1.0, 0.1, 0.4], 0.006)][:len(ks)]
    st = state([code[k] for k in ks], [h[k] for k in ks], pos, quat=q, n=128, indicator=indicator,
               planes=[cube_planes(h[k]) if k == "polytope" else None for k in ks])
    if b == "wall":
        st = W.with_walls(st, [[1.0, 0.0, 0.0, c[0] + h[a][0] - pen]])
    rep, ref = _parity(st, 0)
    assert ref.pair_out[0, 0] > 0.0


@pytest.mark.parametrize("max_pairs", [None, 8])
def test_pair_count_of_the_last_step(max_pairs):
    """contact_pair_count is the step's n_pairs, also beyond the capacity (0 before the first step)."""
    import ctypes

    from paper_2401_10878_gb300.contact import ECAPACITY, Contact, ContactError
    st = W.mixed_grid_27()
    m = Contact.from_state(st, max_pairs=max_pairs)
    n = ctypes.c_int32(-1)
    assert m.lib.contact_pair_count(m.ctx, ctypes.byref(n)) == 0 and n.value == 0
    pos, quat = torch.tensor(st.pos, device="cuda"), torch.tensor(st.quat, device="cuda")
    if max_pairs is None:
        assert m.step(pos, quat)["n_pairs"] == int(m.n_pairs.item())
    else:
        assert m.step(pos, quat, check=False)["n_pairs"] == max_pairs
        with pytest.raises(ContactError) as e:
            m.step(pos, quat)
        assert e.value.code == ECAPACITY
    assert m.lib.contact_pair_count(m.ctx, ctypes.byref(n)) == 0 and n.value == int(m.n_pairs.item()) > 8
    m.close()


def _lattice_state(n, indicator=0):
    """n small spheres, cubes and tetrahedra-like polytopes on a jittered grid, most touching a neighbour."""
    rng = np.random.default_rng(n)
    k = int(np.ceil(n ** (1.0 / 3.0)))
    g = np.stack(np.meshgrid(*[np.arange(k)] * 3, indexing="ij"), -1).reshape(-1, 3)[:n]
    step = 6.0
    pos = (g + 0.5) * step + rng.uniform(-0.6, 0.6, size=(n, 3))
    pl = W.random_polytope(rng, 12, 4.0)[0]
    t = np.array([W.SPHERE, W.CUBOID, W.POLYTOPE])[np.arange(n) % 3]
    params = np.where(t[:, None] == W.SPHERE, [[3.0, 0.0, 0.0]], [[2.5, 2.5, 2.5]])
    return state(t, params, pos, quat=W.random_quaternions(rng, n), n=int(k * step),
                 planes=[pl if x == W.POLYTOPE else None for x in t], indicator=indicator)


# around the sizes where the pair kernels gather by blocks (4096) and a pose warp takes 32 particles (6080)
@pytest.mark.parametrize("n", [4095, 4096, 4097, 6080, 6081, 6097])
@pytest.mark.parametrize("precision", [0, 1])
def test_larger_steps(n, precision):
    rep, ref = _parity(_lattice_state(n), precision)
    assert np.count_nonzero(ref.pair_out[:, 0]) > n // 4


@pytest.mark.parametrize("law", [False, True])
def test_larger_step_and_adjoint_equal_the_smaller(law):
    """One more particle, alone in the box, takes the step from single chunks to
    gathered blocks: the other 4096 keep their outputs and gradients bit for bit."""
    from paper_2401_10878_gb300.contact import Contact
    st = _lattice_state(4097, indicator=1)
    st.pos[4096] = np.array([15.5, 8.5, 8.5]) * 6.0
    rng = np.random.default_rng(1)
    vel = torch.tensor(rng.normal(size=(4097, 6)) * 0.02, device="cuda") if law else None
    kw = dict(friction=True, mu_s=0.3, mu_k=0.2, u_k=0.01, damping_c=0.4) if law else {}
    gf, gt = (torch.tensor(w, device="cuda") for w in W.loss_weights(4097))
    outs = []
    for n in (4097, 4096):
        s = st.subset(np.arange(n))
        m = Contact.from_state(s, **kw)
        o = m.step(torch.tensor(s.pos, device="cuda"), torch.tensor(s.quat, device="cuda"), None if vel is None else vel[:n].contiguous())
        gp, gq = m.backward(gf[:n].contiguous(), gt[:n].contiguous())
        outs.append([o["pair_ij"].clone(), o["pair_out"].clone(), o["force"][:4096].clone(), o["torque"][:4096].clone(),
                     gp[:4096], gq[:4096]])
        assert m.stats()["overlapping"] > 1000
        m.close()
    for a, b in zip(*outs):
        assert torch.equal(a, b)


# turned so that the far corner's coordinates (tens of thousands of cells) cancel in every face value
@pytest.mark.parametrize("seed", [13, 16, 201, 229])
@pytest.mark.parametrize("kind", ["cuboid", "polytope"])
def test_fp64_form_far_from_the_centres(seed, kind):
    """Two long rods end to end, smoothed over a fiftieth of a cell: FP32 rounds
    the ends' distances by a thousandth of a cell, and the all-FP64 form still
    takes every node of the band."""
    rng = np.random.default_rng(seed)
    axis, angle = rng.normal(size=3), rng.uniform(0.3, 1.2)
    q = [quat_axis_angle(axis, angle), quat_axis_angle(axis, angle + 1e-5)]
    h, n = (32000.0, 30.0, 30.0), 128200
    along = oracle.rotation(q[0])[:, 0]
    a = np.full(3, 40000.0) + rng.random(3)
    b = a + along * (2 * h[0] - 2.0) + 0.3 * rng.random(3)
    t, planes = (W.CUBOID, None) if kind == "cuboid" else (W.POLYTOPE, [cube_planes(h)] * 2)
    st = state([t] * 2, [h, h], np.mod([a, b], n), quat=q, n=n, planes=planes, indicator=1, w=0.02)
    rep, ref = _parity(st, 1)
    assert ref.n_pairs == 1 and ref.pair_out[0, 0] > 6000.0


# small steps and ones whose overlapping pairs are gathered
@pytest.mark.parametrize("n", [27, 4097])
def test_adjoint_of_friction_at_any_speed(n):
    """Velocities and u_K scaled by the same power of two leave the friction law,
    and so forces and gradients, unchanged, also where |u_t|^2 is beyond 1e60.
    (The adjoint's node seeds are FP32: an ulp of theirs is 6e-8.)"""
    from paper_2401_10878_gb300.contact import Contact
    st = W.mixed_grid_27() if n == 27 else _lattice_state(n)
    st.indicator = 1
    vel = np.random.default_rng(3).normal(size=(n, 6)) * 0.02
    gf, gt = (torch.tensor(w, device="cuda") for w in W.loss_weights(n))
    outs = []
    for scale in (1.0, 2.0 ** 110):
        m = Contact.from_state(st, friction=True, mu_s=0.3, mu_k=0.2, u_k=0.01 * scale)
        o = m.step(torch.tensor(st.pos, device="cuda"), torch.tensor(st.quat, device="cuda"),
                   torch.tensor(vel * scale, device="cuda"))
        gp, gq = m.backward(gf, gt)
        outs.append([o["force"].clone(), o["torque"].clone(), gp, gq])
        m.close()
    for (a, b), tol in zip(zip(*outs), (1e-12, 1e-12, 1e-6, 1e-6)):
        assert float((a - b).abs().max()) <= tol * float(a.abs().max())


def test_cell_list_memory():
    """The cell list keeps to its 2^26 entries of 20 bytes (five in each of 235^3 bins here)."""
    from paper_2401_10878_gb300.contact import Contact
    n, box = 16, 940
    x = np.random.default_rng(0).random((n, 3)) * 900.0
    st = state([W.SPHERE] * n, [[1.0, 0, 0]] * n, x, n=box)
    torch.cuda.synchronize()
    before = torch.cuda.mem_get_info()[0]
    m = Contact.from_state(st)
    used = before - torch.cuda.mem_get_info()[0]
    assert m.stats()["bins_x"] == 235
    m.close()
    entries, counts, rest = 2 ** 26 * 20, 4 * 235 ** 3, 64 << 20
    assert 235 ** 3 * 5 * 20 <= used <= entries + counts + rest


# most tiles of many node passes, several in every block (256 particles) and more than there are warps (1296):
# every pair of kinds with the wall's, polytopes among them, and each kind alone
@pytest.mark.parametrize("k", [16, 36])
@pytest.mark.parametrize("kinds", [[0, 1, 3], [0, 1, 2], [0, 0, 0], [1, 1, 1], [3, 3, 3]])
@pytest.mark.parametrize("indicator", [0, 1])
def test_deep_tiles_on_single_warps(k, kinds, indicator):
    """A layer of spheres, cuboids and cubes (or polytopes) pressed into one
    another, a floor and a ceiling."""
    from paper_2401_10878_gb300.contact import Contact
    rng = np.random.default_rng(7)
    edge = 16.0
    n = k * k
    g = np.stack(np.meshgrid(np.arange(k), np.arange(k), indexing="ij"), -1).reshape(-1, 2)
    pos = np.concatenate([(g + 0.5) * edge, np.full((n, 1), 40.0)], 1) + rng.uniform(-0.4, 0.4, (n, 3))
    code = np.array(kinds)[rng.integers(0, 3, n)]
    half = np.where(code[:, None] == 0, [[9.6, 0, 0]], np.where(code[:, None] == 1, [[9.4, 8.1, 7.3]], [[7.9] * 3]))
    pl = W.random_polytope(rng, 14, 10.0)[0]
    st = state(np.where(code == 3, W.CUBOID, code), half, pos, quat=W.random_quaternions(rng, n), n=(16 * k, 16 * k, 96),
               planes=[pl if c == 2 else None for c in code], indicator=indicator)
    st = W.floor_and_ceiling(st, gap=5.0)
    rep, ref = _parity(st, 0)
    m = Contact.from_state(st)
    gpu_step(m, st)
    s = m.stats()
    m.close()
    assert (s["tiles"] > 8 * s["narrow_grid"]) == (k == 36) and s["tiles"] > 2 * s["narrow_grid"]
    assert s["overlapping"] > 2 * n


# one tile a pair: around the counts up to which eight, four and two warps share one (on 304 blocks of eight)
@pytest.mark.parametrize("pairs", [1, 303, 304, 305, 608, 609, 1216, 1217, 2500])
@pytest.mark.parametrize("indicator", [0, 1])
def test_fp64_form_shared_tiles(pairs, indicator):
    """Pairs pressed together over a face, each alone, tiles of some twenty node
    passes: the first ones' outputs are the same bit for bit whatever number of
    warps shares a tile, and every pair agrees with the oracle."""
    from paper_2401_10878_gb300.contact import Contact
    rng = np.random.default_rng(2)
    g = np.stack(np.meshgrid(np.arange(14), np.arange(14), np.arange(14), indexing="ij"), -1).reshape(-1, 3)[:2500]
    at = g * [37.0, 27.0, 27.0] + 14.0 + rng.uniform(-1.0, 1.0, (2500, 3))
    q = [quat_axis_angle(a, 0.03) for a in rng.normal(size=(5000, 3))]
    h = np.array([6.5, 7.0, 7.0])
    sub = np.arange(2500)[:pairs]
    pos = np.stack([at[sub], at[sub] + [2 * h[0] - 2.6, 0.3, -0.2]], 1).reshape(-1, 3)
    st = state([W.CUBOID] * (2 * pairs), [h] * (2 * pairs), pos, quat=q[:2 * pairs], n=(14 * 37, 14 * 27, 14 * 27),
               indicator=indicator)
    rep, ref = _parity(st, 1)
    assert ref.n_pairs == pairs and ref.pair_out[:, 0].min() > 300.0
    outs = []
    for s in (st, st.subset(np.arange(2))):
        m = Contact.from_state(s, precision=1)
        outs.append(gpu_step(m, s)["pair_out"][0])
        assert m.stats()["tiles"] == s.n // 2
        m.close()
    assert np.array_equal(outs[0], outs[1])


# rows of particles per block of the pair builder: up to four, then eight; in the box pipeline two, then four
@pytest.mark.parametrize("n", [9727, 9728, 9735])
def test_pair_builder_rows_of_larger_steps(n):
    rep, ref = _parity(_lattice_state(n), 0)
    assert np.count_nonzero(ref.pair_out[:, 0]) > n // 4


@pytest.mark.parametrize("n", [4863, 4864, 4867])
def test_pair_builder_rows_of_larger_box_steps(n):
    rep, ref = run_box(boxed(_lattice_state(n), 3))
    assert np.count_nonzero(ref.pair_out[:, 0]) > n // 4


def _packed_block(kinds):
    """1728 small particles in 55^3, about a dozen candidate partners each; positions are multiples of 2^-20."""
    rng = np.random.default_rng(17)
    g = np.stack(np.meshgrid(*[np.arange(12)] * 3, indexing="ij"), -1).reshape(-1, 3)
    pos = (g + 0.5) * (55.0 / 12) + rng.uniform(-0.5, 0.5, g.shape)
    pos = np.mod(np.round(pos * 2.0 ** 20) / 2.0 ** 20, 55.0)
    pl = cube_planes([1.5, 1.3, 1.2])
    t = np.array(kinds)[np.arange(len(g)) % len(kinds)]
    params = np.where(t[:, None] == W.SPHERE, [[2.5, 0.0, 0.0]], [[2.0, 2.0, 2.0]])
    return state(t, params, pos, quat=W.random_quaternions(rng, len(g)), n=55,
                 planes=[pl if x == W.POLYTOPE else None for x in t], indicator=1)


def _repeated(st, m):
    """m^3 copies of the periodic state side by side (copy-major particle numbers)."""
    off = np.stack(np.meshgrid(*[np.arange(m)] * 3, indexing="ij"), -1).reshape(-1, 3) * st.box
    c = len(off)
    big = st.subset(np.tile(np.arange(st.n), c))
    big.pos = (st.pos[None] + off[:, None]).reshape(-1, 3)
    big.n_cells = tuple(int(v) * m for v in st.n_cells)
    return big


def _copies_agree(small, big, tol):
    """Every copy's rows equal the block's: the sums add in another order, and a pair across copies may name its
    particles the other way round, so FP32 sums of some thirty nodes differ by a few ulps of their terms."""
    for a, b in zip(small, big):
        assert float((b.reshape(-1, *a.shape) - a).abs().max()) <= tol * float(a.abs().max())


# more than 1024 candidate pairs for every block that gathers them, tiles enough for the adjoint's queue
@pytest.mark.parametrize("kinds", [[W.SPHERE], [W.CUBOID], [W.SPHERE, W.CUBOID, W.POLYTOPE]])
@pytest.mark.parametrize("law", [False, True])
def test_many_pairs_step_and_adjoint(kinds, law):
    from paper_2401_10878_gb300.contact import Contact
    st = _packed_block(kinds)
    vel = np.random.default_rng(2).normal(size=(st.n, 6)) * 0.02
    kw = dict(friction=True, mu_s=0.3, mu_k=0.2, u_k=0.01, damping_c=0.4) if law else {}
    gw = W.loss_weights(st.n)
    outs = []
    for m in (1, 3):
        s = st if m == 1 else _repeated(st, m)
        model = Contact.from_state(s, **kw)
        rep = lambda x: torch.tensor(np.tile(x, (m ** 3, 1)), device="cuda")  # noqa: E731
        o = model.step(torch.tensor(s.pos, device="cuda"), torch.tensor(s.quat, device="cuda"), rep(vel) if law else None)
        gp, gq = model.backward(rep(gw[0]), rep(gw[1]))
        outs.append([o["force"].clone(), o["torque"].clone(), gp, gq])
        pairs, tiles = o["n_pairs"], model.stats()["tiles"]
        model.close()
        if m == 1:
            block = pairs
            assert tiles < 4 * 8 * (2 if W.POLYTOPE in kinds else 3) * 152
    assert pairs == 27 * block > 2 * 152 * 1024 and tiles > 4 * 8 * 3 * 152
    _copies_agree(outs[0], outs[1], 1e-5)


def test_many_pairs_of_the_box_pipeline():
    from paper_2401_10878_gb300.contact import Contact
    st = _packed_block([W.SPHERE, W.CUBOID, W.POLYTOPE])
    outs = []
    for m in (1, 3):
        s = st if m == 1 else _repeated(st, m)
        model = Contact.from_state(s, box_mode=1, contact_resolution=3)
        o = model.step(torch.tensor(s.pos, device="cuda"), torch.tensor(s.quat, device="cuda"))
        outs.append([o["force"].clone(), o["torque"].clone()])
        model.close()
    _copies_agree(outs[0], outs[1], 1e-5)
