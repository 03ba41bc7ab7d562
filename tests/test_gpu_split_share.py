"""The tuned split of a length is kept per share of kept outputs: a plan of another share is tuned for its own."""
import json
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
RUN = """
import json, sys, time
import torch
import paper_1809_07592_gb300 as pa
L = 131072
torch.zeros(1, device="cuda")

def made(m):
    torch.cuda.synchronize()
    t = time.perf_counter()
    pa.Plan(L + 1 - m, m, int(sys.argv[1])).close()
    return time.perf_counter() - t

made(L // 3)  # tunes, and loads the kernels
known = max(made(L // 3 + i) for i in range(3))
print(json.dumps([known] + [made(m) for m in (L // 16, L // 16 + 1, L // 5, L // 5 + 1)]))
"""


def plan_times(dtype):
    r = subprocess.run([sys.executable, "-c", RUN, str(dtype)], cwd=ROOT, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stderr
    return json.loads(r.stdout.strip().split("\n")[-1])


def test_each_share_is_tuned_once():
    """Tuning runs six batches of 32 key pairs for each of five splits, tens of times a plan whose split is known."""
    known, eighth, again8, quarter, again4 = plan_times(0)  # FP64
    assert eighth > 5 * known and quarter > 5 * known
    assert again8 < eighth / 5 and again4 < quarter / 5


def test_exact_transform_has_one_share():
    known, *others = plan_times(2)  # NTT64: no pruned butterflies
    assert max(others) < 5 * known
