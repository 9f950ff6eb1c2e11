"""The autotuner's file cache: picks timed on another build of the kernels
are not taken over; the same build's are."""
import json
import os
import subprocess
import sys

import pytest

from paper_2303_13403_gb300 import pqmc  # noqa: F401

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CODE = """
import json, torch
torch.cuda.set_device(0)
from paper_2303_13403_gb300 import pqmc, workloads
t = pqmc.autotune([workloads.honeycomb(2, two_theta=2.0, g=0.6, M_N=0.21)], prec=pqmc.FP32, n_stab=2)
print(json.dumps([bool(t["from_cache"]), t["delay_k"], t["cta_threads"]]))
"""


def tune(path):
    env = dict(os.environ, PQMC_AUTOTUNE_CACHE=str(path), PYTHONPATH=ROOT)
    r = subprocess.run([sys.executable, "-c", CODE], env=env, cwd=ROOT, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stderr
    return json.loads(r.stdout.strip().splitlines()[-1])


def test_picks_of_another_build_are_timed_again(tmp_path):
    path = tmp_path / "tune.json"
    path.write_text("{}")
    first = tune(path)
    assert first[0] is False
    assert tune(path) == [True] + first[1:]
    # the same entry as another build would have written it
    (key, entry), = json.loads(path.read_text()).items()
    path.write_text(json.dumps({key: dict(entry, delay_k=64, cta_threads=64, build="0123456789ab")}))
    assert tune(path)[0] is False
    assert json.loads(path.read_text())[key]["build"] == entry["build"]
    # and as a user pins it
    path.write_text(json.dumps({key: {"delay_k": 64, "cta_threads": 64, "ms_per_sweep": 1.0}}))
    assert tune(path) == [True, 64, 64]
