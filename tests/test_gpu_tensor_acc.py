"""Tensor accumulation over more contributors than one unreduced sum takes (255 per batch): an epoch whose
user batch meets several hundred groups in one launch set equals the same epoch in launch sets of 100."""
import numpy as np
import pytest

from paper_2509_03024_gb300 import capi
from paper_2509_03024_gb300 import workloads as W
from tests.gpu_common import gpu_ctx, torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("preset", ["t11a2", "t10"])
def test_long_accumulations(preset):
    csr = W.uniform_ratings(100, 700, 0.05, 4)
    k = 2
    ctx = gpu_ctx(preset, 41)
    ctx.add_rotation_keys(ctx.mf_rotation_steps(k))
    rng = np.random.default_rng(5)
    U, V = rng.normal(0, 0.1, (csr.n, k)), rng.normal(0, 0.1, (csr.m, k))
    out = []
    for chunk in (None, 100):
        plan = capi.MfPlan(ctx, csr.n, csr.m, k, csr.row_ptr, csr.col_idx, csr.vals)
        assert plan.n_ub == 1 and plan.info.n_groups > 511
        if chunk:
            plan.set_chunk(chunk)
        UD, VD = ctx.empty_ct(plan.n_ub), ctx.empty_ct(plan.n_vb)
        plan.encrypt_factors(0, U, UD)
        plan.encrypt_factors(1, V, VD)
        plan.sgd_epoch(UD, VD, ctx.top, 0.01, 0.02)
        out.append((UD, VD))
    torch.cuda.synchronize()
    assert torch.equal(out[0][0], out[1][0]) and torch.equal(out[0][1], out[1][1])
