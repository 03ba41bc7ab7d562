"""Admission to the byte: a served block counts one and a half slots, its 48-byte descriptor and two counters."""
import numpy as np
import pytest
import torch

import paper_1809_07592_gb300 as pa
from oracle import oracle
from paper_1809_07592_gb300 import inputs
from tests.gpu_util import to_dev

pytestmark = pytest.mark.gpu

N, M, LENGTH = 60000, 20000, 81920  # 5 * 2^14


@pytest.mark.parametrize("dtype,value", [(pa.PA_FP32_GUARD, 8), (pa.PA_FP64, 16)], ids=["fp32g", "fp64"])
def test_cap_of_one_block(dtype, value):
    key, seed = inputs.block_inputs(N, M, base_seed=9)
    kd, sd = to_dev(key)[0], to_dev(seed)[0]
    out = torch.zeros((M + 127) // 128 * 2, dtype=torch.int64, device="cuda")
    need = LENGTH * value * 3 // 2 + 48 + 8
    srv = pa.pa_server_create(hbm_cap_bytes=need, dtype=dtype)
    res = pa.pa_wait(srv, pa.pa_submit(srv, N, M, kd, sd, out), 60000)
    torch.cuda.synchronize()
    assert res.status == pa.PA_OK and pa.pa_server_stats(srv)["peak_inflight_bytes"] == need
    np.testing.assert_array_equal(out.cpu().numpy().view(np.uint64)[: (M + 63) // 64], oracle.toeplitz_hash(N, M, seed, key))
    pa.pa_server_destroy(srv)
    srv = pa.pa_server_create(hbm_cap_bytes=need - 1, dtype=dtype)
    with pytest.raises(pa.PAError) as e:
        pa.pa_submit(srv, N, M, kd, sd, out)
    assert e.value.code == pa.PA_EINVAL
    pa.pa_server_destroy(srv)
