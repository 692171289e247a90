"""A trajectory whose second pass fails leaves nothing running.

The allocation for the second pass's positions is made to fail on the host
(TNEP_FAULT=oom@N, read when the library loads, so in a child process) while the
first pass still runs on the device: once the call has returned, nothing writes
the caller's output any more, and a call of one pass gives its own results."""

import json
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CHILD = """
import json, sys
import numpy as np, torch, synth
from paper_2312_05233_gb300 import tnep as tn
rng = np.random.default_rng(3)
pos, types, box = synth.water_box(5000, rng)
pos = np.mod(pos, box).astype(np.float32)
models = []
for rank in (1, 2) * 6:  # tens of milliseconds a pass
    hp = synth.HyperParams(n_types=2, rank=rank)
    models.append(tn.Model.from_hyper(hp, synth.model_params(hp, rng), synth.default_q_scaler(hp)))
ctx = tn.tnep_create(models, 2, (6.0, 4.0))
one = [x[0].tolist() for x in tn.tnep_eval(ctx, pos[None, :192], box, types[:192])]
tn.tnep_set_option(ctx, tn.TNEP_OPT_FRAMES_PER_BATCH, 60)
frames = np.repeat(pos[None], 120, 0)
out = torch.full((120 * 72,), -7.0, dtype=torch.float64, device="cuda")
side = torch.cuda.Stream()
with torch.cuda.stream(side):
    now = out.clone()  # loads what the copy below needs
torch.cuda.synchronize()
status = 0
try:
    tn.tnep_eval(ctx, frames, box, types, out=out)
except tn.TnepError as e:
    status = e.status
with torch.cuda.stream(side):
    now = out.clone()
side.synchronize()
allocs = tn.tnep_get_option(ctx, tn.TNEP_OPT_ALLOC_COUNT)
again = [x[0].tolist() for x in tn.tnep_eval(ctx, pos[None, :192], box, types[:192])]
torch.cuda.synchronize()
print(json.dumps(dict(status=status, allocs=int(allocs), still=bool(torch.equal(now, out)), same=one == again)))
"""


def run(fault=None):
    env = {k: v for k, v in os.environ.items() if k != "TNEP_FAULT"}
    if fault:
        env["TNEP_FAULT"] = fault
    r = subprocess.run([sys.executable, "-c", CHILD], cwd=ROOT, capture_output=True, text=True, env=env, timeout=300)
    assert r.returncode == 0, r.stderr[-2000:]
    return json.loads(r.stdout.strip().splitlines()[-1])


def test_failed_second_pass_leaves_nothing_running():
    ref = run()
    assert ref["status"] == 0 and ref["still"] and ref["same"]
    got = run(f"oom@{ref['allocs']}")  # the last one: the second pass's positions
    assert got["status"] == 2
    assert got["still"] and got["same"]
