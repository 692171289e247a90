"""Device memory: models on two streams, scratch kept between calls."""

import os
import subprocess
import sys

import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
N_MOL = 40000
# What one atom of a two-type batch takes with lists of 128 and 64 entries: lists
# with a scratch copy, moments, one pair cache of 64 x 64 bytes, outputs of two
# models, cells and orders; buffers are allocated a quarter larger.
ATOM_BYTES = (2 * 128 + 64) * 4 + 2 * 9 * 10 * 4 + 64 * 64 + 2 * 9 * 4 + 128
ONE_CACHE = int(1.25 * 3 * N_MOL * ATOM_BYTES)
SECOND_CACHE = int(1.25 * 3 * N_MOL * 64 * 64)
SLACK = 128 << 20  # roundings of the allocator, code


@pytest.fixture(scope="module")
def tn():
    from paper_2312_05233_gb300 import tnep
    return tnep


@pytest.fixture(scope="module")
def structure():
    rng = np.random.default_rng(41)
    p, t, b = synth.water_box(N_MOL, rng)
    return np.mod(p, b).astype(np.float32), t.astype(np.int32), b.astype(np.float32)


def context(tn):
    rng = np.random.default_rng(42)
    models = []
    for rank in (1, 2):
        hp = synth.HyperParams(n_types=2, rank=rank)
        models.append(tn.Model.from_hyper(hp, synth.model_params(hp, rng), synth.default_q_scaler(hp)))
    return tn.tnep_create(models, 2, (6.0, 4.0))


def test_served_batches_stay_within_their_estimate(tn, structure):
    """120,000 atoms through the server take the memory of one pair cache, which
    is what the admission counts, and give the bits of the plain call."""
    import torch
    pos, types, box = structure
    with context(tn) as ctx:
        tn.tnep_eval(ctx, pos[None, :192], np.float32([30, 30, 30]), types[:192])  # loads the kernels
        torch.cuda.synchronize()
        before = torch.cuda.mem_get_info()[0]
        with tn.tnep_server_start(ctx, mem_budget_bytes=4 << 30, max_batch_atoms=len(types), n_pipelines=1) as srv:
            ticket = srv.submit(pos, types, box)
            counted = srv.stats()["bytes_in_use"]
            out, _ = srv.wait(ticket)
            used = before - torch.cuda.mem_get_info()[0]
        plain = tn.tnep_eval(ctx, pos[None], box, types)
    assert np.array_equal(out, np.concatenate([plain[0][0], plain[1][0]]))
    assert used <= ONE_CACHE + SLACK < ONE_CACHE + SECOND_CACHE
    assert counted == 0 or counted >= 0.9 * 3 * N_MOL * ATOM_BYTES


def test_a_second_pair_cache_that_does_not_fit_is_left_out(tn, structure):
    """With room for one pair cache only, the models run one after the other:
    the same bits as with room for two."""
    import torch
    pos, types, box = structure
    with context(tn) as ctx:
        ref = tn.tnep_eval(ctx, pos[None], box, types)
    torch.cuda.empty_cache()
    with context(tn) as ctx:
        room = ONE_CACHE + SLACK + SECOND_CACHE // 4
        hold = torch.empty(torch.cuda.mem_get_info()[0] - room, dtype=torch.uint8, device="cuda")
        try:
            got = tn.tnep_eval(ctx, pos[None], box, types)
        finally:
            del hold
            torch.cuda.empty_cache()
    for a, b in zip(ref, got):
        assert np.array_equal(a, b)


KEPT = """
import numpy as np, torch, synth
from paper_2312_05233_gb300 import tnep as tn
series = np.random.default_rng(43).standard_normal((250_000, 9))  # about 105 MB of scratch
hp = synth.HyperParams(n_types=2, rank=1)
model = tn.Model.from_hyper(hp, synth.model_params(hp, np.random.default_rng(1)), synth.default_q_scaler(hp))

def spectrum():
    tn.tnep_spectrum(series, 0.5, tn.TNEP_SPECTRUM_RAMAN_ANISO, 10_000)

def held():
    return free - torch.cuda.mem_get_info()[0]

free = 0
spectrum()
tn.lib().tnep_destroy(None)
free = torch.cuda.mem_get_info()[0]
spectrum()
assert 64 << 20 < held() <= 256 << 20, held()
tn.lib().tnep_destroy(None)
assert held() <= 4 << 20, held()
with tn.tnep_create([model], 2, (6.0, 4.0)):  # with a context it stays until the last one goes
    spectrum()
    tn.lib().tnep_destroy(None)
    assert held() >= 64 << 20, held()
assert held() <= 4 << 20, held()
"""


def test_kept_scratch_is_given_back_without_a_context():
    """A program that only computes spectra has no context whose end gives the
    kept scratch back (in a process of its own: no context of another test)."""
    r = subprocess.run([sys.executable, "-c", KEPT], cwd=ROOT, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stderr[-2000:]
