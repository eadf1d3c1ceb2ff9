"""The autotuner's file (STG_TUNE_CACHE): a choice timed for the half-pass and
one timed for A are kept apart, also in the next process; lines of older files,
which do not say what they were timed for, serve both.

Each case runs in a process of its own, since a process reads the file once.
"""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
KEY = "4 4 4 8 1 12 4"  # lattice, FP32, 12-real, 4 systems

PROGRAM = """
import sys
sys.path.insert(0, %r)
import numpy as np
import torch
import gen
import paper_1111_0125_gb300 as stg
dims = (4, 4, 4, 8)
with stg.Gauge(dims, gen.gauge_field(dims, "haar", seed=1), sloppy=stg.STG_FP32, recon=12) as g:
    f = torch.cat([g.pack(torch.from_numpy(b).cuda(), stg.STG_FP32) for b in gen.source(dims, seed=2, nrhs=4)])
    out = torch.empty_like(f)
    stg.stg_dslash_mrhs(g.handle, 0, 4, f, out, stg.STG_FP32)
    stg.stg_apply_A_mrhs(g.handle, 4, np.full(4, 0.1), f, out, stg.STG_FP32)
    torch.cuda.synchronize()
    print("shape", *stg.stg_mrhs_tuning(g.handle, stg.STG_FP32, 4))
""" % ROOT


def _run(path):
    env = {k: v for k, v in os.environ.items() if not k.startswith("STG_")}
    r = subprocess.run([sys.executable, "-c", PROGRAM], env={**env, "STG_TUNE_CACHE": str(path)}, capture_output=True,
                       text=True, timeout=300)
    assert r.returncode == 0, r.stderr[-2000:]
    return tuple(int(v) for v in r.stdout.split("shape")[1].split()), path.read_text().splitlines()


def test_choices_keep_their_use(tmp_path):
    path = tmp_path / "tune"
    path.write_text("")
    _, lines = _run(path)
    assert sorted(ln.rsplit(" ", 1)[1] for ln in lines) == ["0", "1"]
    assert all(ln.startswith(KEY + " ") and len(ln.split()) == 9 for ln in lines)


@pytest.mark.parametrize("lines, want", [
    # half-pass: register-fed shape 0; A: staged on (re, im) pairs, NB = 2
    ([f"{KEY} 0 0", f"{KEY} 14 1"], (2, -2)),
    ([f"{KEY} 14 1", f"{KEY} 0 0"], (2, -2)),
    ([f"{KEY} 0", f"{KEY} 14 1", f"{KEY} 0 0"], (2, -2)),
    # an older file
    ([f"{KEY} 15"], (4, -2)),
])
def test_choices_of_a_file_are_used(tmp_path, lines, want):
    path = tmp_path / "tune"
    path.write_text("".join(ln + "\n" for ln in lines))
    shape, after = _run(path)
    assert shape == want
    assert after == lines  # nothing was timed again
