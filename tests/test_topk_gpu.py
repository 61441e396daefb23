"""The ranking of the evictable tokens (Eq. main_selection) over the shapes of
its cluster kernel: unit counts that give clusters of 8 to 1 CTAs, ranked
widths around the sort's sizes (1024, 2048, 4096), few tokens, and many equal
scores.  Key-norm scores, so the ranking is known exactly."""
import numpy as np
import pytest
import torch

from paper_2607_29591_gb300 import build as B
from paper_2607_29591_gb300 import reskv as R

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def lib():
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    B.build()
    return R.load_library()


@pytest.mark.parametrize("units,s,budget,P", [(1, 70, 66, 64), (1, 9000, 1088, 64), (3, 2500, 1089, 64),
                                              (16, 1200, 500, 10), (40, 700, 300, 0), (160, 300, 100, 64),
                                              (2, 6001, 2112, 64), (1, 6001, 2113, 64), (1, 9001, 4161, 64),
                                              (1, 20011, 8256, 64)])
@pytest.mark.parametrize("values", ["spread", "ties"])
def test_ranking_is_exact(units, s, budget, P, values):
    g = torch.Generator().manual_seed(s + units)
    K = torch.zeros(1, units, s, 128, dtype=torch.bfloat16)
    if values == "spread":
        K[..., :2] = torch.randn((1, units, s, 2), generator=g).to(torch.bfloat16)
    else:                                 # five distinct norms
        K[..., 0] = torch.randint(0, 5, (1, units, s), generator=g).to(torch.bfloat16)
    cfg = R.reskv_config_default(batch=1, n_layers=1, n_kv_heads=units, group=1, seq_len=s, budget=budget,
                                 recent_window=P, n_obs=0, n_fit=0, n_val=0,
                                 score_mode=R.RESKV_SCORE_KEYNORM, keep_debug=1,
                                 residual_override=np.zeros(units, np.int32))
    Kd = K.cuda()
    cache = R.reskv_build_cache(cfg, [Kd], [Kd], None)
    R.reskv_check_status(cache)
    top = R.reskv_export_debug(cache, R.RESKV_DEBUG_RANKED)
    pos = R.reskv_export_cache(cache)["slot_pos"]
    cache.free()
    score = K[0].double().square().sum(-1).numpy()[:, :s - P]
    for u in range(units):
        order = np.argsort(-score[u], kind="stable")[:budget - P]      # ties: lower position
        assert np.array_equal(top[u], order), u
        assert np.array_equal(pos[u, :budget], np.sort(np.concatenate([order, np.arange(s - P, s)]))), u
