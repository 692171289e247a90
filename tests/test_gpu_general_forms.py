"""The forms that large batches take, on the layouts that the small ones test.

Batches of up to 12,288 atoms take one warp an atom, lists of up to 57,344 atoms
eight lanes an atom, and structures of up to 14,000 atoms one CTA each, so the
comparisons here put the structures beside enough others that k_build, the
six-launch preparation, the FP32 pair cache and several work items for each
persistent CTA run.  All are exact."""

import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu
RC = (6.0, 4.0)


@pytest.fixture(scope="module")
def tn():
    from paper_2312_05233_gb300 import tnep
    return tnep


def water(n_mol, rng, drop=0):
    p, t, b = synth.water_box(n_mol, rng)
    keep = len(t) - drop
    return synth.Structure(np.mod(p, b)[:keep].astype(np.float32), t[:keep], b.astype(np.float32))


def random_box(rng, box, extent, n=200):
    pos = (rng.uniform(0, 1, (n, 3)) * extent).astype(np.float32)
    return synth.Structure(pos, np.zeros(n, np.int32), np.asarray(box, np.float32))


@pytest.fixture(scope="module")
def layouts():
    """Structures of every cell layout with their float32 brute-force lists: boxes
    of few cells (rint per pair), windows that wrap, slabs, rods, open clusters,
    unwrapped coordinates."""
    rng = np.random.default_rng(5)
    frames, types, box = synth.water_small(1)
    structs = [synth.Structure(frames[0], types, box),
               synth.Structure((frames[0] + box * rng.integers(-1, 2, size=frames[0].shape)).astype(np.float32), types,
                               box), water(300, rng, 1)]
    for n in (1, 7, 40):
        p, t, b = synth.water_cluster(n, rng)
        structs.append(synth.Structure(p.astype(np.float32), t, b.astype(np.float32)))
    structs += [random_box(rng, (12.1, 19.0, 19.0), (12.1, 19.0, 19.0)),
                random_box(rng, (15.1, 19.0, 19.0), (15.1, 19.0, 19.0)),
                random_box(rng, (20.0, 19.0, 0.0), (20.0, 19.0, 15.0)),
                random_box(rng, (0.0, 18.5, 18.5), (30.0, 18.5, 18.5))]
    refs = [[oracle.neighbours_fp32(s.pos, s.box, rc) for rc in RC] for s in structs]
    return structs, refs, water(19500, rng)


@pytest.mark.parametrize("n_types", [2, 3])
@pytest.mark.parametrize("cell_div,x_div", [(1, 1), (2, 1), (3, 1), (1, 2), (1, 3), (1, 4), (2, 4)])
def test_lists_of_every_layout_beside_a_large_box(tn, layouts, n_types, cell_div, x_div):
    structs, refs, filler = layouts
    order = structs[:4] + [filler] + structs[4:]  # the large box in between
    bt = synth.concat_structures(order)
    assert bt.offsets[-1] > 57344 and len(filler.types) > 14000
    hp = synth.HyperParams(n_types=n_types, rank=1)
    model = tn.Model.from_hyper(hp, synth.model_params(hp, np.random.default_rng(1)), synth.default_q_scaler(hp))
    with tn.tnep_create([model], n_types, RC) as ctx:
        tn.tnep_set_option(ctx, tn.TNEP_OPT_CELL_DIV, cell_div)
        tn.tnep_set_option(ctx, tn.TNEP_OPT_CELL_XDIV, x_div)
        cR, cA, lR, lA = tn.tnep_neighbors(ctx, bt.offsets, bt.pos, bt.box, cap_R=256, cap_A=128)
    for k, ref in enumerate(refs):
        a0 = bt.offsets[k if k < 4 else k + 1]
        for a, (rR, rA) in enumerate(zip(*ref)):
            g = a0 + a
            assert cR[g] == len(rR) and cA[g] == len(rA)
            assert np.array_equal(np.sort(lR[g, :cR[g]]) - a0, rR)
            assert np.array_equal(np.sort(lA[g, :cA[g]]) - a0, rA)


# (atoms beyond 12,288 for the FP32 network, beyond two 128-atom blocks on every
# SM for the tensor-core one; the last block is partly filled)
@pytest.mark.parametrize("mode,n_mol,drop", [(0, 4400, 1), (1, 13500, 5), (2, 13500, 5)])
@pytest.mark.parametrize("small,n_types", [(False, 2), (True, 3)])
def test_pair_cache_and_cta_sizes_of_large_batches(tn, mode, n_mol, drop, small, n_types):
    """The backward walk reads the cache (a column for each resident thread with
    the tensor-core network, overwritten by its next item) or recomputes the
    pairs, and the FP32 form takes 64 or 128 atoms a CTA: the same bits."""
    rng = np.random.default_rng(7)
    structs = [water(n_mol, rng, drop), water(64, rng)]
    for n in (1, 20):
        p, t, b = synth.water_cluster(n, rng)
        structs.append(synth.Structure(p.astype(np.float32), t, b.astype(np.float32)))
    for s in structs:
        s.types = (np.arange(len(s.types)) * 3 % 7 % n_types).astype(np.int32)
    bt = synth.concat_structures(structs)
    sizes = dict(n_max_R=3, n_max_A=2, basis_R=6, basis_A=5, l_max=3) if small else {}
    models = []
    for rank in (1, 2):
        hp = synth.HyperParams(n_types=n_types, rank=rank, **sizes)
        models.append(tn.Model.from_hyper(hp, synth.model_params(hp, rng), synth.default_q_scaler(hp)[:hp.dim],
                                          mlp_precision=mode))
    forms = [(1, 128), (0, 128)] + ([(1, 64), (0, 64)] if mode == 0 else [])
    outs = []
    with tn.tnep_create(models, n_types, RC) as ctx:
        for cache, block in forms:
            tn.tnep_set_option(ctx, tn.TNEP_OPT_PAIR_CACHE, cache)
            tn.tnep_set_option(ctx, tn.TNEP_OPT_BLOCK_ATOMS, block)
            outs.append(tn.tnep_eval_batch(ctx, bt.offsets, bt.pos, bt.box, bt.types, per_atom=True))
    for form, (tensors, atoms) in zip(forms[1:], outs[1:]):
        for m in range(2):
            assert np.array_equal(tensors[m], outs[0][0][m]), (form, m)
            assert np.array_equal(atoms[m], outs[0][1][m]), (form, m)


@pytest.mark.parametrize("edges", [(6e9, 6e9, 6e9), (3e9, 5e9, 7e10), (1e12, 20.0, 1e12), (1e30, 1e30, 1e30)])
def test_huge_boxes_have_the_pairs_of_open_axes(tn, layouts, edges):
    """More cells along an axis than an int holds: the plan keeps to 2 n + 8 cells
    in both preparations."""
    rng = np.random.default_rng(9)
    pos = rng.uniform(0.0, 18.0, (300, 3)).astype(np.float32)
    box = np.float32(edges)
    short = np.where(box < 100.0, box, 0.0).astype(np.float32)  # the axis that does wrap
    want = [oracle.neighbours_fp32(pos, short, rc) for rc in RC]
    hp = synth.HyperParams(n_types=2, rank=1)
    model = tn.Model.from_hyper(hp, synth.model_params(hp, rng), synth.default_q_scaler(hp))
    for beside in ([], [layouts[2]]):
        bt = synth.concat_structures([synth.Structure(pos, np.zeros(300, np.int32), box)] + beside)
        with tn.tnep_create([model], 2, RC) as ctx:
            cR, cA, lR, lA = tn.tnep_neighbors(ctx, bt.offsets, bt.pos, bt.box, cap_R=256, cap_A=128)
        for a in range(300):
            assert np.array_equal(np.sort(lR[a, :cR[a]]), want[0][a])
            assert np.array_equal(np.sort(lA[a, :cA[a]]), want[1][a])
