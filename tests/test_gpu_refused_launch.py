"""A launch that the runtime refuses fails its own call only: the next call on another plan runs."""
import ctypes

import numpy as np
import pytest
import torch

import paper_1809_07592_gb300 as pa
from oracle import oracle
from paper_1809_07592_gb300 import inputs
from tests.gpu_util import to_dev, to_host

pytestmark = pytest.mark.gpu


def test_refused_launch_is_reported_once():
    n, m, count = 100, 37, 65536  # one class of more blocks than a grid has rows
    key, seed = inputs.block_inputs(n, m, base_seed=5)
    kd, sd = to_dev(key)[0], to_dev(seed)[0]
    out = torch.zeros(2, dtype=torch.int64, device="cuda")
    one = pa.BlockDesc(n, m, kd.data_ptr(), sd.data_ptr(), out.data_ptr())
    blocks = (pa.BlockDesc * count)(*([one] * count))
    plan = pa.Plan(n, m, pa.PA_FP32_GUARD)
    h = ctypes.c_void_p()
    assert pa.lib().pa_uneven_create(blocks, count, pa.PA_FP32_GUARD, 0, ctypes.byref(h)) == pa.PA_OK
    with pytest.raises(pa.PAError) as e:
        pa.pa_uneven_run(h, count)
    assert e.value.code == pa.PA_ECUDA
    plan.set_seed(sd)  # its first launch is an ordinary one, which asks for the runtime's last error
    got = to_host(plan.hash(kd.view(1, -1)), 1)
    np.testing.assert_array_equal(got[0], oracle.toeplitz_hash(n, m, seed, key))
    plan.close()
    pa.pa_uneven_destroy(h)
