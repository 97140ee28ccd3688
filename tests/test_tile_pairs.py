"""CTA pairs of the tensor-core streaming form: no load is multicast over a
cluster (the library also runs as one rank per GPU of several), and shapes
asked for or kept under the code of an earlier multicast form run as pair MMAs."""

import glob
import json
import os
import re
import subprocess
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

CHILD = """
import json, math, sys
import numpy as np
import synth
from paper_2312_05837_gb300 import api
ctx = api.Context(0)
inst = synth.sk_dense(300, 51, 1 / math.sqrt(300), np.float32, h_std=0.3)
s = api.Session(ctx, inst, restarts=500, steps=40, seed=6, streaming=True)
if len(sys.argv) > 1:
    s.set_tiles(224, int(sys.argv[1]))
s.run(40)
s.finish()
r = s.result()
s.close()
print(json.dumps({k: r[k] for k in ("tile_restarts", "tile_pair", "best_energy", "best_step")}))
"""


def test_no_load_is_multicast():
    for f in glob.glob(os.path.join(ROOT, "paper_2312_05837_gb300", "csrc", "*")):
        if not f.endswith((".cu", ".cuh")):
            continue
        src = re.sub(r'"\s*\n\s*"', "", open(f).read())  # (asm strings over several lines)
        assert not re.search(r"cp\.async\.bulk[^;]*multicast", src), f


def _child(env, *args):
    out = subprocess.run([sys.executable, "-c", CHILD, *args], cwd=ROOT, capture_output=True, text=True,
                         env={**os.environ, "PYTHONPATH": ROOT, **env}, timeout=300)
    assert out.returncode == 0, out.stderr
    return json.loads(out.stdout.strip().splitlines()[-1])


@pytest.mark.gpu
def test_earlier_codes_run_as_pair_mmas(tmp_path):
    single, asked = _child({}, "0"), _child({}, "1")
    assert (single["tile_restarts"], single["tile_pair"]) == (224, 0)
    assert (asked["tile_restarts"], asked["tile_pair"]) == (224, 2)
    cache = tmp_path / "tune"
    first = _child({"ISING_TUNE_CACHE": str(cache)})
    key = cache.read_text().strip().splitlines()[-1].rsplit("|", 1)[0]
    cache.write_text(f"{key}|{224 | 1 << 16}\n")  # kept by the multicast form
    kept = _child({"ISING_TUNE_CACHE": str(cache)})
    assert (kept["tile_restarts"], kept["tile_pair"]) == (224, 2)
    for r in (asked, first, kept):
        assert (r["best_energy"], r["best_step"]) == (single["best_energy"], single["best_step"])
