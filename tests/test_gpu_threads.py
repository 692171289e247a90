"""Contexts used by several host threads at once, one context per thread."""

import threading

import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def tn():
    from paper_2312_05233_gb300 import tnep
    return tnep


def batch(n_types, n_mol, rng):
    p, t, b = synth.water_box(n_mol, rng)
    types = (np.arange(len(t)) % n_types).astype(np.int32)
    return np.mod(p, b).astype(np.float32), types, b.astype(np.float32)


def ball(n, rng):
    """An open ball of n atoms that all see each other."""
    v = rng.standard_normal((n, 3))
    return (v * (2.5 * rng.uniform(0.3, 1.0, (n, 1)) ** (1 / 3)) / np.linalg.norm(v, axis=1, keepdims=True))


# one warp per atom, and a thread per atom
@pytest.mark.parametrize("n_mol,calls", [(64, 4000), (4400, 1500)])
def test_contexts_of_different_sizes_in_two_threads(tn, n_mol, calls):
    """The kernels' shared memory differs with the number of types and the list
    capacities (grown for the balls of the second context); every call is
    answered, with the bits it has alone."""
    errors, barrier = [], threading.Barrier(2)

    def work(n_types, dense):
        try:
            rng = np.random.default_rng(n_types)
            pos, types, box = batch(n_types, n_mol, rng)
            if dense:
                pos = np.concatenate([pos, ball(dense, rng).astype(np.float32)])
                types = np.concatenate([types, (np.arange(dense) % n_types).astype(np.int32)])
            offsets = [0, 3 * n_mol] + ([len(types)] if dense else [])
            boxes = np.stack([box, np.zeros(3, np.float32)])[:len(offsets) - 1]
            hp = synth.HyperParams(n_types=n_types, rank=1)
            model = tn.Model.from_hyper(hp, synth.model_params(hp, rng), synth.default_q_scaler(hp))
            with tn.tnep_create([model], n_types, (6.0, 4.0)) as ctx:
                first = tn.tnep_eval_batch(ctx, offsets, pos, boxes, types)[0][0]
                barrier.wait(60)
                for _ in range(calls):
                    assert np.array_equal(first, tn.tnep_eval_batch(ctx, offsets, pos, boxes, types)[0][0])
        except Exception as e:
            errors.append((n_types, repr(e)))
            barrier.abort()

    threads = [threading.Thread(target=work, args=a) for a in ((1, 0), (8, 300))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors
