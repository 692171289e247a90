"""Routes that are chosen by the sizes of a batch give the same bits.

Structures of at most 4095 atoms are prepared by one CTA each, batches with a
larger one by the general pipeline; atom order, lists and sums are defined to
be the same, so a structure's tensors and per-atom contributions must not
depend on what else is in the batch (exact comparison, no tolerance)."""

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
    structs = [water(1366, rng, 2), water(1366, rng, 3), water(64, rng), water(65, rng, 1)]  # 4096, 4095, 192, 194 atoms
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
