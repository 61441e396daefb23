"""Observation scores over the fit-row counts that change how the passes share
their rows: one to twelve pairs of 16-row blocks (an odd block at the end,
blocks that are not full, more than eight blocks, so that partial sums take
several), and context lengths beside a half tile and a tile.  Bound: the
protocol's 1e-4 relative error against the oracle."""
import numpy as np
import pytest
import torch

import oracle as orc
from paper_2607_29591_gb300 import build as B
from paper_2607_29591_gb300 import reskv as R

from helpers import bf16_to_f64

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def lib():
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    B.build()
    return R.load_library()


@pytest.mark.parametrize("group,n_fit", [(1, 1), (1, 16), (1, 17), (2, 24), (4, 16), (1, 65), (4, 24), (1, 113),
                                         (4, 32), (2, 72), (1, 161), (4, 50), (4, 96)])
@pytest.mark.parametrize("s", [190, 193, 640])
def test_scores(group, n_fit, s):
    g = torch.Generator().manual_seed(100 * n_fit + s)
    K = (2 * torch.randn(1, 2, s, 128, generator=g)).to(torch.bfloat16)
    Q = torch.randn(1, 2 * group, n_fit, 128, generator=g).to(torch.bfloat16)
    cfg = R.reskv_config_default(batch=1, n_layers=1, n_kv_heads=2, group=group, seq_len=s, budget=100, n_obs=n_fit,
                                 n_fit=n_fit, n_val=0, residual_override=np.zeros(2, np.int32), keep_debug=1)
    cache = R.reskv_build_cache(cfg, [K.cuda()], [K.cuda()], [Q.cuda()])
    R.reskv_check_status(cache)
    got = R.reskv_export_debug(cache, R.RESKV_DEBUG_SCORES).reshape(2, s)
    cache.free()
    for h in range(2):
        ref = orc.scores_obs_pool(bf16_to_f64(K[0, h]), bf16_to_f64(Q[0, h * group:(h + 1) * group]), cfg.pool_kernel)
        np.testing.assert_allclose(got[h], ref, rtol=1e-4, atol=0)
