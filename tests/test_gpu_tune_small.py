"""SHA3GB_TUNE=full and batches that take the single launch of one warp per message: there is nothing to tune for a size
class all of whose batches do.  The library reads the variable once per process, so each case runs in a child."""
import json
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

REPO = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CHILD = r"""
import hashlib, json, sys
import torch
from paper_1902_05320_gb300 import binding as kb
n = eval(sys.argv[1], {"sms": torch.cuda.get_device_properties(0).multi_processor_count})
data = [bytes([i % 251]) * (i % 300) for i in range(n)]
assert kb.hash_many(data) == [hashlib.sha3_256(d).digest() for d in data]
print(json.dumps(n))
"""


@pytest.mark.parametrize("n,tuned", [("200", False), ("20 * sms // 4", False), ("20 * sms + 1", True)])
def test_full_tunes_only_size_classes_that_use_it(tmp_path, n, tuned):
    cache = tmp_path / "tune.jsonl"
    env = dict(os.environ, SHA3GB_TUNE="full", SHA3GB_TUNE_CACHE=str(cache))
    r = subprocess.run([sys.executable, "-c", CHILD, n], cwd=REPO, env=env, capture_output=True, text=True, timeout=600)
    assert r.returncode == 0, r.stderr[-2000:]
    rows = [json.loads(line) for line in cache.read_text().splitlines()] if cache.exists() else []
    assert [row["size_class"] for row in rows] == ([json.loads(r.stdout).bit_length() - 1] if tuned else [])
