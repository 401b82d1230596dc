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
