"""GPU tests of the pass kernels' variants: a variant chosen by a rule gives,
bit for bit, what the general form gives on the same state."""
import numpy as np
import pytest

from paper_1701_06658_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def L():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    from paper_1701_06658_gb300 import lsgg
    lsgg.lib()
    return lsgg


def lattice_seeds(n, k):
    """k^3 seeds on a cubic lattice: neighbouring functions are equal, to the bit, on the mid-planes."""
    a = (np.arange(k) + 0.5) * n / k
    return np.stack(np.meshgrid(a, a, a, indexing="ij"), -1).reshape(-1, 3)


def same_state(a, b):
    pa, pb = a.phi(), b.phi()
    assert (a.boxes() == b.boxes()).all()
    assert all(np.array_equal(pa[g], pb[g]) for g in pa) and pa.keys() == pb.keys()


@pytest.mark.parametrize("dims,seeds", [
    ((64, 64, 64), I.voronoi_seeds(5, 60, (64, 64, 64))),
    ((41, 27, 53), I.voronoi_seeds(6, 20, (41, 27, 53))),        # ragged tiles, boxes across full axes
    ((48, 48, 48), lattice_seeds(48, 3)),                        # exact ties
])
def test_field_pass_without_grains_equals_the_one_with(L, dims, seeds):
    G = len(seeds)
    with L.Microstructure(*dims, G, seeds=seeds) as a, L.Microstructure(*dims, G, seeds=seeds) as b:
        L.keep_field(b.ctx, True)                                # the variant that tracks the top two's grains
        for m in (a, b):
            m.step(3, 1.0)
            m.sync()
        same_state(a, b)


def test_group_with_a_member_that_keeps_the_field(L):
    kw = [((40, 40, 40), 12, 3), ((48, 32, 40), 14, 4)]
    ms = [L.Microstructure(*d, g, seeds=I.voronoi_seeds(s, g, d)) for d, g, s in kw]
    alone = [L.Microstructure(*d, g, seeds=I.voronoi_seeds(s, g, d)) for d, g, s in kw]
    L.keep_field(ms[1].ctx, True)
    L.keep_field(alone[1].ctx, True)
    with L.Group(ms) as grp:
        grp.step(3, 1.0)
        for m in ms:
            m.sync()
        for m in alone:
            m.step(3, 1.0)
            m.sync()
        for a, b in zip(ms, alone):
            same_state(a, b)
        assert L.grain_neighbours(ms[1].ctx, kw[1][1]) == L.grain_neighbours(alone[1].ctx, kw[1][1])
    for m in ms + alone:
        m.close()


@pytest.mark.parametrize("dims,G,big", [
    ((72, 72, 72), 250, 0.0),        # boxes small against the domain: one image per neighbour
    ((41, 27, 53), 20, 0.0),         # ragged tiles, several images
    ((16, 16, 16), 1500, 0.0),       # more seeds than a tile's list holds
    ((40, 40, 48), 90, 300.0),       # power diagram with one grain over most of the domain
    ((70, 45, 1), 60, 0.0),          # 2D tiles
])
def test_start_from_seeds_against_the_oracle(L, dims, G, big):
    """Boxes equal, functions the FP32 rounding of the oracle's FP64 ones (whose own rounding, about 1e-13 of
    values up to 7, can move a value across a rounding boundary: one unit in the last place)."""
    from oracle import lsgg_oracle as O
    seeds = I.voronoi_seeds(17, G, dims)
    w = None
    if big:
        w = np.zeros(G)
        w[3] = big
    ref = O.tessellate((dims[2], dims[1], dims[0]), seeds, w)
    with L.Microstructure(*dims, G, seeds=seeds, weights=w) as ms:
        boxes, phi = ms.boxes(), ms.phi()
    for g, r in enumerate(ref.grains):
        assert bool(boxes[g, 0]) == r.alive
        if not r.alive:
            continue
        assert tuple(boxes[g, 1:4][::-1]) == r.origin and tuple(boxes[g, 4:7][::-1]) == r.dims
        want = r.phi.astype(np.float32)
        assert (np.abs(phi[g] - want) <= np.spacing(np.abs(want))).all()


def test_field_pass_with_overflowing_tile_lists(L):
    """More boxes on a tile than its list holds: the tile takes every box in batches.  The ID-field is the
    oracle's argmax of the step's own phi_p, m its value (copies of FP32 numbers: equal)."""
    from oracle import lsgg_oracle as O
    dims, G = (20, 22, 24), 300
    quats = I.random_quaternions(8, G)
    with L.Microstructure(*dims, G, seeds=I.voronoi_seeds(8, G, dims), quats=quats,
                          physics=L.PHYSICS_READ_SHOCKLEY) as ms:
        boxes, (phip, m, idm, phic, _) = ms.debug_step(1.0)
    grains, pp = [], {}
    for g in range(G):
        if g not in phip:
            grains.append(O.Grain(g, (0, 0, 0), np.full((1, 1, 1), -7.0), alive=False))
            continue
        b = boxes[g]
        pp[g] = phip[g].astype(np.float64)
        grains.append(O.Grain(g, (int(b[3]), int(b[2]), int(b[1])), pp[g]))
    assert len(pp) > 128
    for g in pp:
        rm, rid = O.neighbour_max(g, grains, pp, (dims[2], dims[1], dims[0]), 7.0)
        assert np.array_equal(m[g], rm.astype(np.float32)) and np.array_equal(idm[g], rid)
        assert np.array_equal(phic[g], np.float32(0.5) * (phip[g] - m[g]))


def test_wide_field_tiles_equal_the_others(L):
    """A domain above the size from which physics takes 32-column tiles, made of two copies of one below it along
    x (seed coordinates of 20 binary places, so that every displacement is the same number in both): each copy's
    grains have the boxes and volumes of the single one's, bit for bit."""
    nx, ny, nz, steps = 512, 320, 320, 3
    G = nx * ny * nz // 6000
    one = np.round(I.voronoi_seeds(9, G, (nx, ny, nz)) * 2.0 ** 20) / 2.0 ** 20
    e = 4e-3 * I.u01(9, 7, np.arange(G))
    res = []
    for k in (1, 2):
        seeds = np.concatenate([one + [nx * c, 0.0, 0.0] for c in range(k)])
        with L.Microstructure(k * nx, ny, nz, k * G, seeds=seeds, energy=np.tile(e, k), physics=L.PHYSICS_MAGNETIC) as ms:
            ms.step(steps, 1.0)
            res.append((ms.grain_volumes(), ms.boxes()))
    (v1, b1), (v2, b2) = res
    for c in (0, 1):
        s = slice(c * G, (c + 1) * G)
        assert np.array_equal(v2[s], v1)
        assert np.array_equal(b2[s][:, [0, 2, 3, 4, 5, 6]], b1[:, [0, 2, 3, 4, 5, 6]])
        assert np.array_equal((b2[s][:, 1] - nx * c) % (2 * nx) % nx, b1[:, 1] % nx)


@pytest.mark.parametrize("kind", ["read_shockley", "magnetic"])
@pytest.mark.parametrize("dims,G,bf16", [
    ((36, 36, 160), 6, False),       # columns of up to a hundred cells beside short ones
    ((44, 40, 52), 40, False),       # column lengths on both sides of a batch of eight
    ((44, 40, 52), 40, True),        # previous phi in BF16
    ((24, 24, 24), 6, False),        # periodic columns: the general form
])
def test_physics_z_pass_against_the_oracle(L, kind, dims, G, bf16):
    """phi_p of the second step (previous boxes and ID-field of the first) within the FP32 tolerance of the
    parity tests, 3e-5."""
    from oracle import lsgg_oracle as O
    from tests.parity import oracle_from_gpu
    quats, e = I.random_quaternions(12, G), 4e-2 * I.u01(12, 7, np.arange(G))
    kw = {"quats": quats, "physics": L.PHYSICS_READ_SHOCKLEY} if kind == "read_shockley" else \
        {"energy": e, "physics": L.PHYSICS_MAGNETIC}
    ph = O.read_shockley_physics(quats) if kind == "read_shockley" else O.isotropic_physics(e)
    shape = (dims[2], dims[1], dims[0])
    with L.Microstructure(*dims, G, seeds=I.voronoi_seeds(12, G, dims), storage=L.STORAGE_BF16 if bf16 else
                          L.STORAGE_FP32, **kw) as ms:
        old, (_, _, idm, _, _) = ms.debug_step(1.0)
        boxes, phi = ms.boxes(), ms.phi()
        ref = oracle_from_gpu(shape, boxes, phi, None, ph)
        for g in phi:                                # the first step's ID-field on the boxes after it
            was = O.Grain(g, (int(old[g, 3]), int(old[g, 2]), int(old[g, 1])), idm[g].astype(np.float64))
            ref.grains[g].idf = O.sample(was, O.box_positions(ref.grains[g], shape), shape, -1)[0].astype(np.int64)
        _, (phip, *_rest) = ms.debug_step(1.0)
    taps = O.heat_kernel_taps(1.0, 5)
    for g in phip:
        want = O.predict(ref.grains[g], shape, taps, 7.0, ph, 1.0)
        assert np.max(np.abs(phip[g] - want)) <= 3e-5, g


@pytest.mark.parametrize("bf16", [False, True])
@pytest.mark.parametrize("dims,G", [
    ((96, 90, 84), 20),              # sides over 40 and over 48: the larger plane grids
    ((33, 70, 41), 12),              # odd numbers of planes, boxes across full axes of odd length
    ((24, 24, 24), 30),              # small boxes
])
def test_ideal_convolution_against_the_oracle(L, dims, G, bf16):
    """phi_p of the third step (boxes moved since the state was stored) within the parity tests' 2e-5."""
    from oracle import lsgg_oracle as O
    from tests.parity import oracle_from_gpu
    shape = (dims[2], dims[1], dims[0])
    with L.Microstructure(*dims, G, seeds=I.voronoi_seeds(21, G, dims),
                          storage=L.STORAGE_BF16 if bf16 else L.STORAGE_FP32) as ms:
        ms.step(2, 1.0)
        ms.sync()
        ref = oracle_from_gpu(shape, ms.boxes(), ms.phi())
        _, (phip, *_rest) = ms.debug_step(1.0)
    taps = O.heat_kernel_taps(1.0, 5)
    for g in phip:
        assert np.max(np.abs(phip[g] - O.predict(ref.grains[g], shape, taps, 7.0))) <= 2e-5, g


@pytest.mark.parametrize("bf16", [False, True])
@pytest.mark.parametrize("dims,G", [
    ((26, 28, 140), 9),              # columns of every length up to a hundred, long ones past the register form
    ((60, 58, 62), 45),
    ((24, 25, 23), 4),               # periodic on every axis
    ((130, 20, 22), 5),              # boxes wider than the shared-memory plane grids
])
def test_reinitialisation_of_the_step_s_own_phi_c(L, dims, G, bf16):
    """phi after the step against the oracle's re-initialisation of the step's phi_c: the same FP32 inputs, at most
    six roundings of values up to 7 and the reciprocal square root of the distance (2 ulp): 1e-5; in BF16 the
    stored value's rounding, 2^-8 of it, on top."""
    from oracle import lsgg_oracle as O
    shape = (dims[2], dims[1], dims[0])
    with L.Microstructure(*dims, G, seeds=I.voronoi_seeds(23, G, dims),
                          storage=L.STORAGE_BF16 if bf16 else L.STORAGE_FP32) as ms:
        ms.step(1, 1.0)
        ms.sync()
        boxes, (_, _, _, phic, phin) = ms.debug_step(1.0)
        phi = ms.phi()
        new = ms.boxes()
    for g in phin:
        b = boxes[g]
        full = tuple(int(b[6 - a]) == shape[a] for a in range(3))
        want = O.redistance(phic[g].astype(np.float64), full, 7.0, (0, 1, 2))
        assert np.array_equal(phin[g] > 0, phic[g] > 0)
        assert np.max(np.abs(phin[g] - want)) <= 1e-5, g
        if new[g, 0]:                                # the stored state: the same values on the new box
            was = O.Grain(g, (int(b[3]), int(b[2]), int(b[1])), phin[g].astype(np.float64))
            box = O.Grain(g, tuple(int(v) for v in new[g, 3:0:-1]), np.zeros(tuple(int(v) for v in new[g, 6:3:-1])))
            kept = O.sample(was, O.box_positions(box, shape), shape, -7.0)[0]
            assert np.all(np.abs(phi[g] - kept) <= (2.0 ** -8 * np.abs(kept) if bf16 else 0.0)), g


@pytest.mark.parametrize("dims,G", [((24, 26, 28), 1), ((40, 40, 40), 256), ((40, 44, 40), 257), ((64, 64, 70), 900)])
def test_box_update_over_one_and_several_chunks(L, dims, G):
    """The counts that the box update adds up over its chunks of boxes, against the boxes themselves (whole numbers:
    equal), and the state of a context stepped alone (one launch closes the update) and in a group (two)."""
    def make():
        return L.Microstructure(*dims, G, seeds=I.voronoi_seeds(31, G, dims))

    with make() as ms, make() as other:
        done = 0
        for _ in range(3):
            b = ms.boxes().astype(np.int64)
            done += int((b[:, 0] * b[:, 4] * b[:, 5] * b[:, 6]).sum())
            ms.step(1, 1.0)
            ms.sync()
            b = ms.boxes().astype(np.int64)
            cells = b[:, 0] * b[:, 4] * b[:, 5] * b[:, 6]
            st = ms.stats()
            assert st.cell_updates == done
            assert st.alive == int(b[:, 0].sum()) and st.box_cells == int(cells.sum())
            assert sum(st.pass_cells) == int(cells.sum())
            side = np.maximum(b[:, 4], b[:, 5])
            for t, (lo, hi) in enumerate(((0, 32), (32, 40), (40, 48), (48, 64), (64, 1 << 30))):
                assert st.pass_cells[t] == int(cells[(side > lo) & (side <= hi)].sum())
        with L.Group([other]) as g:
            g.step(3, 1.0)
        other.sync()
        assert other.stats().cell_updates == done
        assert np.array_equal(ms.boxes(), other.boxes())
        assert np.array_equal(L.get_phi(ms.ctx), L.get_phi(other.ctx))


@pytest.mark.parametrize("dims,G", [((24, 24, 24), 4), ((64, 60, 64), 110), ((96, 90, 100), 300)])
def test_slab_depth_follows_the_box_planes(L, dims, G):
    """The depth that the context starts with, and the same bits as with the depths that a tuning tries."""
    import torch
    seeds = I.voronoi_seeds(37, G, dims)
    with L.Microstructure(*dims, G, seeds=seeds) as ms, L.Microstructure(*dims, G, seeds=seeds) as tuned:
        slab = 8
        planes = int(ms.boxes()[:, 6].sum())
        while slab > 2 and planes < 4 * torch.cuda.get_device_properties(0).multi_processor_count * slab:
            slab //= 2
        assert L.pass_tuning(ms.ctx)["slab"] == slab
        ms.step(6, 1.0)
        ms.sync()
        L.autotune(tuned.ctx, 1, 1.0)                    # four steps
        assert L.pass_tuning(tuned.ctx)["slab"] in (4, 8, 16)
        tuned.step(2, 1.0)
        tuned.sync()
        assert np.array_equal(ms.boxes(), tuned.boxes())
        assert np.array_equal(L.get_phi(ms.ctx), L.get_phi(tuned.ctx))


@pytest.mark.parametrize("side", [32, 33, 40, 41, 48, 49, 64, 65])
def test_steps_leave_out_only_tiers_without_boxes(L, side):
    """Replayed steps launch the tiers that the domain's boxes can be in; profiled steps launch every tier.  The same
    bits for boxes that span the domain's longer side, alone and in a group with a smaller domain."""
    dims, G = (side, 24, 20), 2
    seeds = np.array([[0.0, 6.0, 3.0], [0.0, 18.0, 13.0]])       # both grains span x
    small = I.voronoi_seeds(42, 4, (24, 24, 24))
    with L.Microstructure(*dims, G, seeds=seeds) as ms, L.Microstructure(*dims, G, seeds=seeds) as every, \
            L.Microstructure(*dims, G, seeds=seeds) as member, L.Microstructure(24, 24, 24, 4, seeds=small) as other:
        L.profile(every.ctx, True)
        ms.step(4, 1.0)
        every.step(4, 1.0)
        with L.Group([other, member]) as g:
            g.step(4, 1.0)
        for m in (ms, every, member):
            m.sync()
        assert int(every.boxes()[:, 4].max()) == side
        for m in (ms, member):
            assert np.array_equal(m.boxes(), every.boxes())
            assert np.array_equal(L.get_phi(m.ctx), L.get_phi(every.ctx))


@pytest.mark.parametrize("dims,G", [((128, 126, 140), 2600)])
def test_deep_slabs_for_many_planes(L, dims, G):
    import torch
    seeds = I.voronoi_seeds(43, G, dims)
    with L.Microstructure(*dims, G, seeds=seeds) as ms, L.Microstructure(*dims, G, seeds=seeds) as tuned:
        n_sm = torch.cuda.get_device_properties(0).multi_processor_count
        assert (L.pass_tuning(ms.ctx)["slab"] == 16) == (int(ms.boxes()[:, 6].sum()) >= 16 * 16 * n_sm)
        ms.step(5, 1.0)
        ms.sync()
        L.autotune(tuned.ctx, 1, 1.0)                # four steps with 8, 8, 4 and 16 planes
        tuned.step(1, 1.0)
        tuned.sync()
        assert np.array_equal(ms.boxes(), tuned.boxes())
        assert np.array_equal(L.get_phi(ms.ctx), L.get_phi(tuned.ctx))


@pytest.mark.parametrize("kind", ["ideal", "magnetic"])
def test_field_pass_over_tiles_without_boxes(L, kind):
    """A state that covers one corner of the domain: the other tiles list no box, many CTAs' first tile among them.
    The grains around the boxes' cells are the oracle's, those of the empty tiles none."""
    from oracle import lsgg_oracle as O
    n = 96
    dims = (n, n, n)
    kw = {"physics": L.PHYSICS_MAGNETIC, "energy": np.zeros(2)} if kind == "magnetic" else {}
    boxes = np.zeros((2, 7), np.int32)
    boxes[0] = (1, 4, 4, 4, 22, 20, 24)
    boxes[1] = (1, 12, 4, 4, 22, 20, 24)
    z, y, x = np.meshgrid(np.arange(24), np.arange(20), np.arange(22), indexing="ij")
    ball = np.clip(6.0 - np.sqrt((x - 11.0) ** 2 + (y - 10.0) ** 2 + (z - 12.0) ** 2), -7.0, 7.0).astype(np.float32)
    phi = {0: ball, 1: ball.copy()}
    idf = {g: np.full(ball.shape, 1 - g, np.int32) for g in phi}
    with L.Microstructure(*dims, 2, seeds=np.array([[15.0, 14.0, 16.0], [23.0, 14.0, 16.0]]), **kw) as ms:
        ms.set_state(boxes, phi, idf)
        L.keep_field(ms.ctx, True)
        was, (phip, m, idm, phic, _) = ms.debug_step(1.0)
        near = L.grain_neighbours(ms.ctx, 2)
    grains = [O.Grain(g, (4, 4, int(was[g, 1])), phip[g].astype(np.float64)) for g in (0, 1)]
    pp = {g: phip[g].astype(np.float64) for g in (0, 1)}
    for g in (0, 1):
        rm, rid = O.neighbour_max(g, grains, pp, dims, 7.0)
        assert np.array_equal(m[g], rm.astype(np.float32)) and np.array_equal(idm[g], rid)
        assert np.array_equal(phic[g], np.float32(0.5) * (phip[g] - m[g]))
        assert list(near[g]) == [1 - g]


def test_neighbour_collection_of_many_boxes(L):
    """More boxes than take eight CTAs each: phi_p of the second step, whose pairs' weights come from the lists that
    two CTAs a box collect from the first step's ID-field, within the parity tests' 3e-5."""
    from oracle import lsgg_oracle as O
    from tests.parity import oracle_from_gpu
    dims, G = (72, 68, 70), 2100
    quats = I.random_quaternions(14, G)
    ph = O.read_shockley_physics(quats)
    shape = (dims[2], dims[1], dims[0])
    with L.Microstructure(*dims, G, seeds=I.voronoi_seeds(14, G, dims), quats=quats,
                          physics=L.PHYSICS_READ_SHOCKLEY) as ms:
        old, (_, _, idm, _, _) = ms.debug_step(1.0)
        boxes, phi = ms.boxes(), ms.phi()
        _, (phip, *_rest) = ms.debug_step(1.0)
    ref = oracle_from_gpu(shape, boxes, phi, None, ph)
    taps = O.heat_kernel_taps(1.0, 5)
    seen = 0
    for g in list(phip)[::9]:
        was = O.Grain(g, (int(old[g, 3]), int(old[g, 2]), int(old[g, 1])), idm[g].astype(np.float64))
        ref.grains[g].idf = O.sample(was, O.box_positions(ref.grains[g], shape), shape, -1)[0].astype(np.int64)
        seen = max(seen, len(np.unique(ref.grains[g].idf)))
        want = O.predict(ref.grains[g], shape, taps, 7.0, ph, 1.0)
        assert np.max(np.abs(phip[g] - want)) <= 3e-5, g
    assert seen > 16                                 # lists of some length


@pytest.mark.parametrize("with_weights", [False, True])
def test_start_in_a_wide_domain(L, with_weights):
    """Two equal halves of 4096 columns (seed coordinates of 12 binary places, so that every displacement is the same
    FP64 number in both), where a seed's rounding to FP32 is far above that of the values and differs between the
    halves: the second half's grains have the first's boxes and, bit for bit, their functions."""
    nx, ny, nz = 4096, 80, 80
    G = nx * ny * nz // 1728
    seeds = np.round(I.voronoi_seeds(19, G, (nx, ny, nz)) * 2.0 ** 12) / 2.0 ** 12
    w = np.tile(20.0 * I.u01(19, 6, np.arange(G)), 2) if with_weights else None
    both = np.concatenate([seeds, seeds + [float(nx), 0.0, 0.0]])
    with L.Microstructure(2 * nx, ny, nz, 2 * G, seeds=both, weights=w) as ms:
        boxes, phi = ms.boxes(), ms.phi()
    assert np.array_equal(boxes[:G, [0, 2, 3, 4, 5, 6]], boxes[G:, [0, 2, 3, 4, 5, 6]])
    alive = boxes[:G, 0] != 0
    assert alive.sum() > G // 2
    assert np.array_equal((boxes[G:][alive, 1] - nx) % (2 * nx), boxes[:G][alive, 1])
    different = [g for g in np.flatnonzero(alive) if not np.array_equal(phi[g], phi[g + G])]
    assert not different, (len(different), max(np.max(np.abs(phi[g] - phi[g + G])) for g in different))


@pytest.mark.parametrize("dims,G,own", [((32, 32, 32), 20, 2), ((64, 64, 64), 50, 2), ((64, 64, 64), 95, 4)])
def test_tuning_keeps_the_depth_of_few_planes(L, dims, G, own):
    """A small microstructure's slab items hold few planes; a tuning leaves it at that depth, whatever depth it chose
    for more planes."""
    with L.Microstructure(*dims, G, seeds=I.voronoi_seeds(1, G, dims)) as ms:
        assert L.debug_slab_depth(ms.ctx) == own
        L.autotune(ms.ctx, 2, 1.0)
        assert L.debug_slab_depth(ms.ctx) == own


def test_coarsening_takes_the_depth_of_the_coarse_boxes(L):
    dims, G = (64, 64, 64), 95
    with L.Microstructure(*dims, G, seeds=I.voronoi_seeds(1, G, dims)) as ms:
        assert L.debug_slab_depth(ms.ctx) == 4
        L.coarsen(ms.ctx, 32, 32, 32)
        assert L.debug_slab_depth(ms.ctx) == 2
