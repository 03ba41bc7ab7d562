"""A split file with an entry the planner does not offer: the entry is ignored, the batch is tuned and exact."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
RUN = """
import numpy as np, torch
import paper_1809_07592_gb300 as pa
from oracle import oracle
from paper_1809_07592_gb300 import inputs
from tests.gpu_util import to_dev
n, m = 60000, 20000  # length 81920 = 5 * 2^14
key, seed = inputs.block_inputs(n, m, base_seed=1)
out = torch.zeros((m + 127) // 128 * 2, dtype=torch.int64, device="cuda")
h = pa.pa_uneven_create([(n, m, to_dev(key)[0], to_dev(seed)[0], out)], pa.PA_FP32_GUARD, use_graph=True)
pa.pa_uneven_run(h, 1)
torch.cuda.synchronize()
assert np.array_equal(out.cpu().numpy().view(np.uint64)[: (m + 63) // 64], oracle.toeplitz_hash(n, m, seed, key))
(c,) = pa.pa_uneven_classes(h)
assert c[0] == 81920 and c[1] >= 64, c
pa.pa_uneven_destroy(h)
print("exact")
"""


def test_entry_outside_the_planner_is_ignored(tmp_path):
    cache = tmp_path / "splits"
    cache.write_text("81920 1 2 0 5 12\n")  # length, mode, log2 of a first pass of 4, no middle, innermost 5 * 2^12
    r = subprocess.run([sys.executable, "-c", RUN], cwd=ROOT, capture_output=True, text=True, timeout=300,
                       env={**os.environ, "PA_TUNE_CACHE": str(cache)})
    assert r.returncode == 0 and "exact" in r.stdout, r.stderr
    lines = cache.read_text().split("\n")
    assert len(lines) > 2 and lines[1].startswith("81920 1 ")  # the tuned split was added
