"""Member lists on both sides of the rule that gives a thread four tokens (two
blocks of 4096 tokens per SM), with context lengths beside a multiple of 1024
and 4096.  Entries and counts against the oracle's Lloyd."""
import numpy as np
import pytest
import torch

from paper_2607_29591_gb300 import build as B
from paper_2607_29591_gb300 import reskv as R

from helpers import bf16_to_f64, unit_from_layout
from parity import check_entries

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def lib():
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    B.build()
    return R.load_library()


@pytest.mark.parametrize("units,s", [(320, 1025), (160, 4097), (106, 8193), (100, 8192), (310, 500)])
def test_lists(units, s):
    g = torch.Generator(device="cuda").manual_seed(s)
    K = torch.randn(1, units, s, 128, generator=g, device="cuda").to(torch.bfloat16)
    V = torch.randn(1, units, s, 128, generator=g, device="cuda").to(torch.bfloat16)
    r = np.array([(7 * u) % 24 for u in range(units)], np.int32)
    cfg = R.reskv_config_default(batch=1, n_layers=1, n_kv_heads=units, group=1, seq_len=s, budget=128, n_obs=0,
                                 n_fit=0, n_val=0, score_mode=R.RESKV_SCORE_KEYNORM, residual_override=r, keep_debug=1)
    cache = R.reskv_build_cache(cfg, [K], [V], None)
    R.reskv_check_status(cache)
    lay = R.reskv_export_cache(cache)
    top = R.reskv_export_debug(cache, R.RESKV_DEBUG_RANKED)
    cache.free()
    for u in (1, units // 2, units - 1):
        check_entries(unit_from_layout(lay, u), bf16_to_f64(K[0, u]), bf16_to_f64(V[0, u]), top[u], 64, s, 128, 4)
