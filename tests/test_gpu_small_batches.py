"""Routes that are chosen by the sizes of a batch give the same bits.

Structures of at most 14000 atoms are prepared by one CTA each, batches with a
larger one by the general pipeline; atom order, lists and sums are defined to
be the same, so a structure's tensors and per-atom contributions must not
depend on what else is in the batch (exact comparison, no tolerance).  Batches
of at most 12288 atoms take one warp per atom for the FP32 network (and for the
lists and moments of the tensor-core one), larger ones a thread."""

import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def tn():
    from paper_2312_05233_gb300 import tnep
    return tnep


def water(n_mol, rng, drop=0):
    p, t, b = synth.water_box(n_mol, rng)
    p = np.mod(p, b)
    keep = len(t) - drop
    return synth.Structure(p[:keep].astype(np.float32), t[:keep], b.astype(np.float32))


def context(tn, n_types, precision, seed=3):
    rng = np.random.default_rng(seed)
    models = []
    for rank in (1, 2):
        hp = synth.HyperParams(n_types=n_types, rank=rank)
        models.append(tn.Model.from_hyper(hp, synth.model_params(hp, rng), synth.default_q_scaler(hp),
                                          mlp_precision=precision))
    return tn.tnep_create(models, n_types, (6.0, 4.0))


@pytest.mark.parametrize("n_types", [2, 3])
@pytest.mark.parametrize("precision", [0, 2])
def test_a_structure_alone_and_beside_a_large_one(tn, n_types, precision):
    rng = np.random.default_rng(11)
    structs = [water(4667, rng), water(4667, rng, 1), water(345, rng, 11), water(342, rng, 2), water(65, rng, 1)]  # 14001, 14000, 1024, 1024, 194 atoms
    p, t, b = synth.water_cluster(7, rng)
    structs.append(synth.Structure(p.astype(np.float32), t, b.astype(np.float32)))
    structs.append(synth.Structure(np.zeros((0, 3), np.float32), np.zeros(0, np.int32), np.zeros(3, np.float32)))
    structs.append(synth.Structure(np.float32([[1, 2, 3]]), np.int32([1]), np.zeros(3, np.float32)))
    wide = water(343, rng)  # coordinates outside the box
    wide.pos[::5] += wide.box[0]
    structs.append(wide)
    if n_types == 3:
        for s in structs:
            s.types = np.where(np.arange(len(s.types)) % 7 == 0, 2, s.types).astype(np.int32)
    bt = synth.concat_structures(structs)
    with context(tn, n_types, precision) as ctx:
        all_out, all_pa = tn.tnep_eval_batch(ctx, bt.offsets, bt.pos, bt.box, bt.types, per_atom=True)
        for k, s in enumerate(structs):
            if len(s.types) == 0:
                continue
            out, pa = tn.tnep_eval_batch(ctx, [0, len(s.types)], s.pos, s.box[None], s.types, per_atom=True)
            for m in range(2):
                assert np.array_equal(out[m][0], all_out[m][k]), (k, m)
                assert np.array_equal(pa[m], all_pa[m][bt.offsets[k]:bt.offsets[k + 1]]), (k, m)


VARIANTS = {"std": {}, "small": dict(n_max_R=3, n_max_A=2, basis_R=6, basis_A=5, l_max=3)}


@pytest.mark.parametrize("n_types", [1, 2, 3, 6])
@pytest.mark.parametrize("variant", ["std", "small"])
def test_warp_per_atom_equals_thread_per_atom(tn, n_types, variant):
    """Small batches against the same structures beside 13,000 other atoms; no
    neighbours, one, more than 32 and more than 64 angular ones (two and three
    chunks of pairs), types absent from a neighbourhood, n_hidden above 32."""
    rng = np.random.default_rng(17)
    structs = [water(64, rng), water(81, rng, 1)]
    for n in (1, 2, 33):
        p, t, b = synth.water_cluster(n, rng)
        structs.append(synth.Structure(p.astype(np.float32), t, b.astype(np.float32)))
    structs.append(synth.Structure(np.float32([[0, 0, 0]]), np.int32([0]), np.zeros(3, np.float32)))
    for n in (40, 90):  # dense balls: every atom sees n - 1 others within the angular cutoff
        v = rng.standard_normal((n, 3))
        v *= (1.9 * rng.uniform(0.2, 1.0, (n, 1)) ** (1 / 3)) / np.linalg.norm(v, axis=1, keepdims=True)
        structs.append(synth.Structure(v.astype(np.float32), np.zeros(n, np.int32), np.zeros(3, np.float32)))
    for s in structs:
        s.types = (np.arange(len(s.types)) * 7 % 11 % n_types).astype(np.int32)
    filler = water(4400, rng)
    filler.types = (np.arange(len(filler.types)) % n_types).astype(np.int32)
    models = []
    for rank, hidden in ((1, 30), (2, 30), (2, 40), (1, 5), (1, 64)):
        hp = synth.HyperParams(n_types=n_types, rank=rank, n_hidden=hidden, **VARIANTS[variant])
        models.append(tn.Model.from_hyper(hp, synth.model_params(hp, rng), synth.default_q_scaler(hp)[:hp.dim]))
    with tn.tnep_create(models, n_types, (6.0, 4.0)) as ctx:
        small, big = synth.concat_structures(structs), synth.concat_structures(structs + [filler])
        o1, p1 = tn.tnep_eval_batch(ctx, small.offsets, small.pos, small.box, small.types, per_atom=True)
        o2, p2 = tn.tnep_eval_batch(ctx, big.offsets, big.pos, big.box, big.types, per_atom=True)
        for m in range(len(models)):
            assert np.array_equal(p1[m], p2[m][:small.offsets[-1]]), m
            assert np.array_equal(o1[m], o2[m][:len(structs)]), m


def test_small_batch_regrows_its_lists(tn):
    """More neighbours than the lists hold at first: both routes repeat the
    batch with larger ones, and refuse above the hard cap."""
    rng = np.random.default_rng(23)
    v = rng.standard_normal((300, 3))
    v *= (2.5 * rng.uniform(0.3, 1.0, (300, 1)) ** (1 / 3)) / np.linalg.norm(v, axis=1, keepdims=True)
    dense = synth.Structure(v.astype(np.float32), np.arange(300, dtype=np.int32) % 2, np.zeros(3, np.float32))
    filler = water(4400, rng)
    outs = []
    for structs in ([dense], [dense, filler]):
        bt = synth.concat_structures(structs)
        with context(tn, 2, 0) as ctx:
            outs.append(tn.tnep_eval_batch(ctx, bt.offsets, bt.pos, bt.box, bt.types)[0])
        with context(tn, 2, 0) as ctx:
            tn.tnep_set_option(ctx, tn.TNEP_OPT_MAX_NEIGHBORS, 200)
            with pytest.raises(tn.TnepError) as e:
                tn.tnep_eval_batch(ctx, bt.offsets, bt.pos, bt.box, bt.types)
            assert e.value.status == 4
    for a, b in zip(*outs):
        assert np.array_equal(a[0], b[0])


@pytest.mark.parametrize("n_types", [1, 2, 3, 4, 5])
def test_lists_of_large_batches(tn, n_types):
    """Beside 60,300 other atoms the lists are built by a thread per atom; the
    same bits as alone, for lists with types missing and with few entries, and
    the same neighbours."""
    rng = np.random.default_rng(31)
    structs = [water(64, rng), water(100, rng, 2)]
    for n in (1, 2, 9):
        p, t, b = synth.water_cluster(n, rng)
        structs.append(synth.Structure(p.astype(np.float32), t, b.astype(np.float32)))
    for k, s in enumerate(structs):
        s.types = ((np.arange(len(s.types)) * 5 % 13 + k) % n_types).astype(np.int32)
    structs[1].types[:] = n_types - 1
    filler = water(20100, rng)
    filler.types = (np.arange(len(filler.types)) % n_types).astype(np.int32)
    models = []
    for rank in (1, 2):
        hp = synth.HyperParams(n_types=n_types, rank=rank)
        models.append(tn.Model.from_hyper(hp, synth.model_params(hp, rng), synth.default_q_scaler(hp)))
    small, big = synth.concat_structures(structs), synth.concat_structures(structs + [filler])
    N = small.offsets[-1]
    with tn.tnep_create(models, n_types, (6.0, 4.0)) as ctx:
        o1, p1 = tn.tnep_eval_batch(ctx, small.offsets, small.pos, small.box, small.types, per_atom=True)
        o2, p2 = tn.tnep_eval_batch(ctx, big.offsets, big.pos, big.box, big.types, per_atom=True)
        n1 = tn.tnep_neighbors(ctx, small.offsets, small.pos, small.box)
        n2 = tn.tnep_neighbors(ctx, big.offsets, big.pos, big.box)
    for m in range(2):
        assert np.array_equal(p1[m], p2[m][:N]), m
        assert np.array_equal(o1[m], o2[m][:len(structs)]), m
    assert np.array_equal(n1[0], n2[0][:N]) and np.array_equal(n1[1], n2[1][:N])
    for a, b in zip(n1[2:], n2[2:]):
        assert np.array_equal(np.sort(a, 1), np.sort(b[:N], 1))


def test_uneven_batches_are_not_prepared_at_the_largest_size(tn):
    """Thousands of small structures beside a larger one leave the preparation by
    one CTA each (six launches more), with the same bits as alone."""
    rng = np.random.default_rng(37)
    structs = [water(400, rng)]
    for k in range(5000):
        n = 1 + k % 3
        p = 1.5 * np.arange(3 * n).reshape(n, 3) * rng.uniform(0.5, 1, (n, 3))
        structs.append(synth.Structure(p.astype(np.float32), (np.arange(n) % 2).astype(np.int32),
                                       np.zeros(3, np.float32)))
    few, all_ = synth.concat_structures(structs[:50]), synth.concat_structures(structs)
    with context(tn, 2, 0) as ctx:
        launches, outs = [], []
        for bt in (few, all_):
            n0 = tn.tnep_get_option(ctx, tn.TNEP_OPT_KERNEL_LAUNCHES_TOTAL)
            outs.append(tn.tnep_eval_batch(ctx, bt.offsets, bt.pos, bt.box, bt.types, per_atom=True))
            launches.append(tn.tnep_get_option(ctx, tn.TNEP_OPT_KERNEL_LAUNCHES_TOTAL) - n0)
    for m in range(2):
        assert np.array_equal(outs[0][0][m], outs[1][0][m][:50])
        assert np.array_equal(outs[0][1][m], outs[1][1][m][:few.offsets[-1]])
    assert launches[1] == launches[0] + 5


@pytest.mark.parametrize("n_mol,precisions,frames,launches",
                         [(64, (0, 0), 1, 1), (64, (0,) * 5, 1, 2), (64, (2, 2), 1, 2), (64, (0, 2), 1, 2),
                          (4400, (0, 0), 1, 2), (64, (0, 0), 3, 3), (4400, (0, 2), 3, 6)])
def test_model_launches_are_counted(tn, n_mol, precisions, frames, launches):
    """TNEP_OPT_LAST_KERNEL_LAUNCHES: one launch takes up to four FP32 models of a
    small batch, otherwise each model has its own; three passes of one frame."""
    rng = np.random.default_rng(41)
    s = water(n_mol, rng)
    models = []
    for k, precision in enumerate(precisions):
        hp = synth.HyperParams(n_types=2, rank=1 + k % 2)
        models.append(tn.Model.from_hyper(hp, synth.model_params(hp, rng), synth.default_q_scaler(hp),
                                          mlp_precision=precision))
    with tn.tnep_create(models, 2, (6.0, 4.0)) as ctx:
        tn.tnep_set_option(ctx, tn.TNEP_OPT_FRAMES_PER_BATCH, 1)
        tn.tnep_eval(ctx, np.repeat(s.pos[None], frames, 0), s.box, s.types)
        assert tn.tnep_get_option(ctx, tn.TNEP_OPT_LAST_KERNEL_LAUNCHES) == launches
