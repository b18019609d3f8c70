"""The status of a batched plan when a product of a pair on a stream gives up waiting for the
tensor cores: the plan reports the timeout, whichever product it was, and the device word of the
single calls stays clear of it. The waits are made to run out at once by a limit of zero polls, in
a process of its own."""
import json
import os
import subprocess
import sys

import pytest

torch = pytest.importorskip("torch")

pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA GPU")]

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_timeout_of_a_stream_pair_is_the_plans_status():
    from paper_2410_04385_gb300 import binding, build
    if not os.path.exists(binding.LIB_PATH):
        build.build()
    p = subprocess.run([sys.executable, os.path.join(ROOT, "tests", "mma_timeout_check.py")], capture_output=True,
                       text=True, env=dict(os.environ, HATT_MMA_WAITS="0", HATT_BATCH_FORM="lanes"), timeout=600,
                       cwd=ROOT)
    assert p.returncode == 0, p.stderr[-3000:]
    r = json.loads(p.stdout.strip().splitlines()[-1])
    batches = [k for k in r if k.endswith(("first", "again"))]
    assert len(batches) == 8 and all(r[k] == binding.TT_ERR_TIMEOUT for k in batches), r
    assert r["device_after_batches"] == binding.TT_OK
    assert r["device_after_fp64"] == r["device_after_tf32"] == binding.TT_ERR_TIMEOUT
    assert r["device_after_small"] == binding.TT_OK and r["small_rel"] <= 1e-12
