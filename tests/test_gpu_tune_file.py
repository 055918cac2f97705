"""The autotuner's file: choices written by a library with other kernels are
timed again, a line out of range is ignored, and one that fits is applied."""
import json
import os
import subprocess
import sys
import textwrap

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CHILD = textwrap.dedent("""
    import json, os, sys
    sys.path.insert(0, os.environ["ROOT"])
    from paper_1411_2087_gb300 import stag, synth
    dims = (6, 6, 4, 8)
    U = synth.su3_field(dims, 0.3, 7).numpy()
    with stag.Lattice(dims) as lat:
        lat.upload_gauge(U, None, precisions=("f32",))
        res, cached = lat.autotune_all("f32")
    print(json.dumps({"cached": cached, "chosen": [(r["kernel"], r["block"], r["regs"], r["group"])
                                                   for r in res if r["chosen"]]}))
""")


def run(path):
    env = dict(os.environ, ROOT=ROOT, STAG_TUNE_CACHE=str(path))
    p = subprocess.run([sys.executable, "-c", CHILD], env=env, capture_output=True, text=True, timeout=300)
    assert p.returncode == 0, p.stderr
    return json.loads(p.stdout.strip().splitlines()[-1])


def test_lines_of_other_kernels_are_timed_again(tmp_path):
    path = tmp_path / "tune.txt"
    assert not run(path)["cached"]
    words = path.read_text().split()
    key, kset = " ".join(words[1:8]), words[14]
    assert len(words) == 15
    for line in (f"stag-tune2 {key} 64 1 512 2 256 4",              # no kernel set
                 f"stag-tune2 {key} 64 1 512 2 256 4 {int(kset) - 1}",
                 f"stag-tune2 {key} 1000 0 128 0 128 8 {kset}",     # no 1000-thread Dslash
                 f"stag-tune2 {key} 128 0 128 7 128 8 {kset}",      # no register variant 7
                 f"stag-tune2 {key} 128 0 128 0 128 64 {kset}"):    # a group beyond the kernels' arrays
        path.write_text(line + "\n")
        assert not run(path)["cached"], line
        assert len(path.read_text().splitlines()) == 2
    path.write_text(f"stag-tune2 {key} 64 1 512 2 256 4 {kset}\n")
    out = run(path)
    assert out["cached"]
    assert [tuple(c) for c in out["chosen"]] == [("dslash", 64, 1, 0), ("M", 512, 2, 0), ("batch", 256, 0, 4)]
