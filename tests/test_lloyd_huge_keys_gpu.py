"""Lloyd assignment (Sec. 5.3) where a unit holds keys whose squared norm or dot
products leave the fp32 range (the norm past 2^63.5): such a token still belongs
to the centre beside it.  Counts and entries against the oracle's Lloyd on the
GPU's evicted set."""
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


@pytest.mark.parametrize("norm", [1e18, 1.5e19, 6e19, 1e30])
@pytest.mark.parametrize("r,finite", [(3, 1), (3, 2), (40, 30), (300, 299)])
def test_keys_past_the_fp32_range(norm, r, finite):
    """`finite` of the r first centres have ordinary norms."""
    s, P = 1200, 64
    g = torch.Generator().manual_seed(r)
    b = r + P + 50
    n_huge = 50 + r - finite              # the largest fill the main cache, the others come first
    K = torch.randn(1, 1, s, 128, generator=g)
    V = torch.randn(1, 1, s, 128, generator=g).to(torch.bfloat16)
    at = torch.randperm(s - P, generator=g)[:n_huge]
    way = torch.randn(3, 128, generator=g)
    way = way / way.norm(dim=1, keepdim=True)
    size = norm * (1 + 0.2 * torch.rand(n_huge, 1, generator=g))
    K[0, 0, at] = size * (way[torch.arange(n_huge) % 3] + 0.001 * torch.randn(n_huge, 128, generator=g))
    K = K.to(torch.bfloat16)
    cfg = R.reskv_config_default(batch=1, n_layers=1, n_kv_heads=1, group=1, seq_len=s, budget=b,
                                 recent_window=P, n_obs=0, n_fit=0, n_val=0,
                                 score_mode=R.RESKV_SCORE_KEYNORM,
                                 residual_override=np.array([r], np.int32), keep_debug=1)
    cache = R.reskv_build_cache(cfg, [K.cuda()], [V.cuda()], None)
    torch.cuda.synchronize()
    R.reskv_check_status(cache)
    lay = R.reskv_export_cache(cache)
    top = R.reskv_export_debug(cache, R.RESKV_DEBUG_RANKED)
    cache.free()
    check_entries(unit_from_layout(lay, 0), bf16_to_f64(K[0, 0]), bf16_to_f64(V[0, 0]), top[0], P, s, b, 4)
