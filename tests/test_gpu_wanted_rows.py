"""The last pass forms only the outputs a batch keeps: shares of the transform at and just past each of its
thresholds (an eighth and a quarter of the length), for a lone key (half-length form) and an odd batch."""
import numpy as np
import pytest
import torch

import paper_1809_07592_gb300 as pa
from oracle import oracle
from paper_1809_07592_gb300 import inputs
from tests.gpu_util import to_dev, to_host

pytestmark = pytest.mark.gpu

LENGTH = 1 << 17  # n + m - 1: a length the planner takes as it is


@pytest.mark.parametrize("nkeys", [1, 3])
@pytest.mark.parametrize("dtype", [pa.PA_FP32_GUARD, pa.PA_FP64, pa.PA_NTT64], ids=["fp32g", "fp64", "ntt64"])
@pytest.mark.parametrize("m", [1, LENGTH // 8, LENGTH // 8 + 1, LENGTH // 4, LENGTH // 4 + 1])
def test_kept_share_of_the_outputs(m, dtype, nkeys):
    n = LENGTH + 1 - m
    seed = inputs.bernoulli_bits(m, 1, LENGTH)
    keys = inputs.batch_keys(n, nkeys, base_seed=m)
    plan = pa.Plan(n, m, dtype)
    assert plan.shape()[0] == LENGTH
    plan.set_seed(to_dev(seed)[0])
    out, (marg, mode, esc) = plan.hash(to_dev(keys), info=True)
    torch.cuda.synchronize()
    got = to_host(out, (m + 63) // 64)
    plan.close()
    for k in range(nkeys):
        np.testing.assert_array_equal(got[k], oracle.toeplitz_hash(n, m, seed, keys[k]), err_msg=f"key {k}")
    assert esc == 0 and all(v == dtype for v in mode)
