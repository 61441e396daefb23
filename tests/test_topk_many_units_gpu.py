"""Ranking with more units than SMs (two blocks per SM), at n_top on both sides of
one and two keys per thread: the GPU's own scores, highest first, ties to the
lower position."""
import numpy as np
import pytest
import torch

import oracle as orc
from paper_2607_29591_gb300 import build as B
from paper_2607_29591_gb300 import reskv as R

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def lib():
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    B.build()
    return R.load_library()


@pytest.mark.parametrize("b", [65, 1088, 1089, 2112, 2113])
def test_ranking(b):
    units, s = 200, 2300
    g = torch.Generator(device="cuda").manual_seed(b)
    K = torch.randn(1, units, s, 128, generator=g, device="cuda").to(torch.bfloat16)
    K[:, :, 100:140] = K[:, :, 200:240]                  # equal scores
    cfg = R.reskv_config_default(batch=1, n_layers=1, n_kv_heads=units, group=1, seq_len=s, budget=b, n_obs=0, n_fit=0,
                                 n_val=0, score_mode=R.RESKV_SCORE_KEYNORM,
                                 residual_override=np.zeros(units, np.int32), keep_debug=1)
    cache = R.reskv_build_cache(cfg, [K], [K], None)
    R.reskv_check_status(cache)
    scores = R.reskv_export_debug(cache, R.RESKV_DEBUG_SCORES).reshape(units, s)
    top = R.reskv_export_debug(cache, R.RESKV_DEBUG_RANKED).reshape(units, -1)
    cache.free()
    for u in range(0, units, 13):
        assert np.array_equal(orc.rank_evictable(scores[u], 64)[:b - 64], top[u][:b - 64]), u
