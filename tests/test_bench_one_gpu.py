"""bench.py runs the library on one GPU only: its contraction kernel loads with TMA
multicast, which stays out of calls on several GPUs.  A launch with several ranks,
or --gpus above 1, prints one line from rank 0 and touches no GPU (there is none
where this runs: anything else would fail)."""
import json
import os
import subprocess
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.mark.parametrize("env,gpus,lines", [({"RANK": "0", "WORLD_SIZE": "2", "LOCAL_RANK": "0"}, 2, 1),
                                            ({"RANK": "1", "WORLD_SIZE": "2", "LOCAL_RANK": "1"}, 2, 0),
                                            ({}, 4, 1)])
def test_several_gpus_are_refused(env, gpus, lines):
    r = subprocess.run([sys.executable, os.path.join(ROOT, "bench.py"), "--gpus", str(gpus), "--steps", "1",
                        "--warmup", "0"], env=dict(os.environ, CUDA_VISIBLE_DEVICES="", **env),
                       capture_output=True, text=True, timeout=120)
    out = r.stdout.strip().splitlines()
    assert r.returncode == 0 and len(out) == lines, r.stderr
    if lines:
        assert json.loads(out[0])["n_gpus"] == gpus and "one GPU" in json.loads(out[0])["unavailable"]
