"""The last pass's pruned last stage at both sides of its thresholds, on first passes that have it: a full-radix stage 0,
length 256 in single precision, 64 and 512 in double. And the 64-bit prime's passes on every split of its shortest length."""
import os
import subprocess
import sys

import numpy as np
import pytest
import torch

import paper_1809_07592_gb300 as pa
from oracle import oracle
from paper_1809_07592_gb300 import inputs
from tests.gpu_util import to_dev, to_host

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
LENGTH = 1 << 17
SHARES = [LENGTH // 8, LENGTH // 8 + 1, LENGTH // 4, LENGTH // 4 + 1]


def check(plan, m, seed, keys):
    plan.set_seed(to_dev(seed)[0])
    got = to_host(plan.hash(to_dev(keys)), (m + 63) // 64)
    torch.cuda.synchronize()
    plan.close()
    for k in range(keys.shape[0]):
        np.testing.assert_array_equal(got[k], oracle.toeplitz_hash(plan.n, m, seed, keys[k]), err_msg=f"key {k}")


@pytest.mark.parametrize("m", SHARES)
@pytest.mark.parametrize("dtype,split", [(pa.PA_FP32_GUARD, (256, 512, 1)), (pa.PA_FP64, (64, 2048, 1)),
                                         (pa.PA_FP64, (512, 256, 1))], ids=["fp32-256", "fp64-64", "fp64-512"])
def test_pair(m, dtype, split):
    n = LENGTH + 1 - m
    plan = pa.Plan(n, m, dtype, split=split)
    assert plan.shape() == (LENGTH,) + split
    check(plan, m, inputs.bernoulli_bits(m, 1, LENGTH), inputs.batch_keys(n, 2, base_seed=m))


# a lone key's split cannot be forced: untuned, a half length of 2^20 takes 256 * 4096 (single), one of 2^17 64 * 2048
@pytest.mark.parametrize("dtype,half", [(pa.PA_FP32_GUARD, 1 << 20), (pa.PA_FP64, 1 << 17)], ids=["fp32", "fp64"])
@pytest.mark.parametrize("eighths,more", [(1, 0), (1, 1), (2, 0), (2, 1)])
def test_lone_key(dtype, half, eighths, more, monkeypatch):
    monkeypatch.setenv("PA_PLAN_TUNE", "0")
    m = 2 * (eighths * half // 8 + more)  # two output bits per element
    n = 2 * half + 1 - m
    check(pa.Plan(n, m, dtype), m, inputs.bernoulli_bits(m, 1, n + m - 1), inputs.batch_keys(n, 1, base_seed=m))


UNEVEN = """
import sys
import numpy as np, torch
import paper_1809_07592_gb300 as pa
from oracle import oracle
from paper_1809_07592_gb300 import inputs
from tests.gpu_util import to_dev
L, dtype, first = 131072, int(sys.argv[1]), int(sys.argv[2])
for ms in ((L // 8, L // 8 + 1), (L // 4 + 1, L // 8), (1, L // 4), (L // 4,)):  # pruned by the longer of a pair
    data = [inputs.block_inputs(L + 1 - m, m, base_seed=m) for m in ms]
    blocks = [(L + 1 - m, m, to_dev(k)[0], to_dev(s)[0], torch.zeros((m + 127) // 128 * 2, dtype=torch.int64, device="cuda"))
              for m, (k, s) in zip(ms, data)]
    h = pa.pa_uneven_create(blocks, dtype, use_graph=False)
    assert pa.pa_uneven_classes(h)[0][:2] == (L, first)
    pa.pa_uneven_run(h, len(blocks))
    torch.cuda.synchronize()
    for (n, m, _, _, out), (k, s) in zip(blocks, data):
        assert np.array_equal(out.cpu().numpy().view(np.uint64)[: (m + 63) // 64], oracle.toeplitz_hash(n, m, s, k)), m
    pa.pa_uneven_destroy(h)
print("exact")
"""


@pytest.mark.parametrize("dtype,lg", [(pa.PA_FP32_GUARD, 8), (pa.PA_FP64, 6), (pa.PA_FP64, 9)])
def test_uneven_pair(dtype, lg, tmp_path):
    cache = tmp_path / "splits"
    cache.write_text(f"{LENGTH} {dtype} {lg} 0 1 {17 - lg}\n")
    r = subprocess.run([sys.executable, "-c", UNEVEN, str(dtype), str(1 << lg)], cwd=ROOT, capture_output=True, text=True,
                       timeout=300, env={**os.environ, "PA_TUNE_CACHE": str(cache)})
    assert r.returncode == 0 and "exact" in r.stdout, r.stderr


def test_every_split_of_the_64_bit_prime():
    m = (1 << 19) + 7
    n = (1 << 26) + (1 << 20) + 1  # length 2^27, the first that the word-sized prime has no roots for
    g = torch.Generator(device="cuda").manual_seed(1)
    words = lambda *s: torch.randint(-(1 << 63), (1 << 63) - 1, s, generator=g, device="cuda", dtype=torch.int64)
    keys, seed = words(2, (n + 127) // 128 * 2), words((n + m + 126) // 128 * 2)

    def hashed(dtype, split=None):
        plan = pa.Plan(n, m, dtype, split=split)
        plan.set_seed(seed)
        out = torch.zeros((2, (m + 127) // 128 * 2), dtype=torch.int64, device="cuda")
        plan.hash(keys, out)
        torch.cuda.synchronize()
        plan.close()
        return out

    want = hashed(pa.PA_FP64)
    splits = pa.pa_plan_splits(n, m, pa.PA_NTT64)
    assert len(splits) > 5 and all(a * b * c == 1 << 27 for a, b, c in splits)
    for split in splits:
        assert torch.equal(hashed(pa.PA_NTT64, split), want), split
