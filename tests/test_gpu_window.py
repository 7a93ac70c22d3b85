"""Parity of the window unroll's forms and of the epilogue's branches against the CPU oracle, at the sizes where
they can go wrong.  All sums are exact integers, so every comparison is element by element."""
import numpy as np
import pytest
import torch

import oracle
import paper_2104_04731_b200 as b2c
from paper_2104_04731_b200.synth import int8_uniform

from gpu_util import check_against_oracle, to_dev

pytestmark = pytest.mark.gpu


# ---- per-channel bias: whole runs of channels with one load per four values, ragged runs one by one ----------
@pytest.mark.parametrize("K,groups", [(64, 1), (48, 1), (33, 1), (20, 1), (24, 4), (128, 2)])   # 24 / 4 = 6: bias not on 16 bytes
def test_bias_vector_and_scalar_loads(lib, K, groups):
    N, C, H, W = 2, 32, 9, 8
    x = int8_uniform((N, C, H, W), 1011)
    w = int8_uniform((K, C // groups, 3, 3), 1012)
    bias = int8_uniform((K,), 1013).astype(np.int32) * 701
    want = oracle.conv2d_int8(x, w, 1, 1, 1, 6, bias=bias, relu=True, groups=groups)
    d = lib.make_desc(N, C, H, W, K, 3, 3, 1, 1, 1, 6, out_mode=3)
    for e in [None] if groups > 1 else lib.enumerate_embeddings(d):
        plan = lib.Plan(d, groups=groups) if groups > 1 else lib.Plan(d, e.id)
        plan.set_weights(to_dev(w))
        plan.set_activation(to_dev(bias), True)
        y32 = torch.full((N, K, H, W), -7777777, dtype=torch.int32, device="cuda")
        y8 = torch.full((N, K, H, W), 77, dtype=torch.int8, device="cuda")
        ws = torch.zeros(max(16, plan.workspace_bytes()), dtype=torch.uint8, device="cuda")
        plan.run(to_dev(x), y32, y8, ws)
        torch.cuda.synchronize()
        assert plan.device_status() == b2c.OK
        assert np.array_equal(y32.cpu().numpy(), want[0]) and np.array_equal(y8.cpu().numpy(), want[1])
        plan.destroy()
