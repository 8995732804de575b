"""Records of the fused restriction pass that another revision of the library
wrote are not used: the pass is timed again and recorded under the present key,
while a record under that key is used as it stands."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

CHILD = r"""
import torch
import workloads as w
import paper_2502_05279_gb300 as bmg
kind, planes, f = w.binary_contrast_problem(2047, 16, seed_k=2, seed_f=3)
h = bmg.Hierarchy(kind, torch.from_numpy(planes).cuda(), precision="fp32", arith="fused")
assert h.tuned_pair(0) >= 0
print(h.launch_count)
"""


def run_child(cache):
    env = dict(os.environ, BMG_TUNE_CACHE=str(cache))
    r = subprocess.run([sys.executable, "-c", CHILD], cwd=ROOT, env=env, capture_output=True, text=True, timeout=600)
    assert r.returncode == 0, r.stderr[-2000:]
    return int(r.stdout.split()[-1])


def test_records_of_another_revision_are_timed_again(tmp_path):
    cache = tmp_path / "tune.txt"
    run_child(cache)
    lines = cache.read_text().splitlines()
    mine = [ln for ln in lines if " pair_restrict:" in ln]
    assert mine
    warm = run_child(cache)                                    # everything found: nothing timed
    assert cache.read_text().splitlines() == lines
    for revision in ("", ":1"):                                # no revision in the key, and an older one
        old = []
        for ln in lines:
            dev, key, *rest = ln.split()
            old.append(" ".join([dev, key.rsplit(":", 1)[0] + revision if ln in mine else key] + rest))
        cache.write_text("\n".join(old) + "\n")
        assert run_child(cache) > warm
        fresh = cache.read_text().splitlines()[len(old):]
        assert [ln.split()[:3] for ln in fresh] == [ln.split()[:3] for ln in mine]
