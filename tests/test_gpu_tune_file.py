"""A kept file of plans (RIFT_ILE_TUNE_CACHE) written for other kernels: its lines carry no version
(or another) and are not taken; those of this version are."""
import json
import os
import subprocess
import sys

import pytest

import ile_synth as S

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

# one detector, 5 modes, 334 bins, 9000 samples: a class of this test's own
RUN = """
import json, sys
import ile_synth as S, paper_2505_11655_gb300 as G
G.load(build_if_missing=True)
p = S.make_problem(("L1",), 5, 4096.0, n_t=334, snr=15.0, seed=S.config_seed(3, 9101))
with G.ILE(p, precision=G.RIFT_FP32, max_samples=9000) as s:
    s.adapt(1, 9000)
    print(json.dumps(s.plan()))
"""


def plan(path):
    # (the file is read once a process)
    env = dict(os.environ, RIFT_ILE_TUNE_CACHE=str(path), PYTHONPATH=ROOT)
    env.pop("RIFT_ILE_TC", None)
    out = subprocess.run([sys.executable, "-c", RUN], cwd=ROOT, env=env, capture_output=True, text=True, timeout=300)
    assert out.returncode == 0, out.stderr
    return json.loads(out.stdout.strip().splitlines()[-1])


def test_lines_of_other_versions(tmp_path):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    p = S.make_problem(("L1",), 5, 4096.0, n_t=334, snr=15.0, seed=S.config_seed(3, 9101))
    path = tmp_path / "plans.txt"
    unnamed = f"K1_kp1_nt334_nq{p.n_q}_n4^6"
    path.write_text(f"{unnamed} 0 64 0\n{unnamed}_v1 0 64 0\n")   # a fill that no candidate has
    assert plan(path)[1] in (2, 4, 8)
    lines = [x.split() for x in path.read_text().splitlines()]
    assert len(lines) == 3 and lines[2][0].startswith(unnamed + "_v")
    path.write_text(f"{lines[2][0]} 0 64 0\n")
    assert plan(path)[1] == 64
