"""Decisions in a DSRG_TUNE_CACHE file belong to a revision of the kernels: a
file of an earlier one (its lines carry none) is timed anew, not followed."""
import json
import os
import re
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CHILD = r"""
import json, sys
sys.path.insert(0, %r)
import synth, paper_1701_02011_gb300 as g
h = g.Dsrg(synth.make_instance(2, 4, 4, 30, 120, 0.5, seed=5), precision=g.DSRG_PREC_SPLIT, slices=6, tune=True)
print(json.dumps(h.pt3()))
h.close()
""" % ROOT


@pytest.fixture(scope="module")
def lib():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1701_02011_gb300 import build
    build.build()


def _run(path):
    env = dict(os.environ, DSRG_TUNE_CACHE=path)
    out = subprocess.run([sys.executable, "-c", CHILD], env=env, capture_output=True, text=True, timeout=600)
    assert out.returncode == 0, out.stderr
    return json.loads(out.stdout.strip().splitlines()[-1])


def test_file_of_an_earlier_revision_is_timed_anew(lib, tmp_path):
    path = str(tmp_path / "tune.txt")
    _run(path)
    new = open(path).read().splitlines()
    old = [re.sub(r"/r\d+ ", " ", line) for line in new]
    with open(path, "w") as f:
        f.write("\n".join(old) + "\n")
    _run(path)
    lines = open(path).read().splitlines()
    assert lines[: len(old)] == old
    key = lambda line: line.split()[:6]  # noqa: E731
    assert sorted(map(key, lines[len(old):])) == sorted(map(key, new))
