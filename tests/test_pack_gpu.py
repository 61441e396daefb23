"""Packing over clusters of one to eight blocks per unit: lists and rows of the
main cache against the exported ranking, at context lengths beside a warp's and
a block's run of positions and beyond the 32 steps whose bits a warp keeps."""
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


@pytest.mark.parametrize("units,s,b", [(1, 100, 90), (2, 1023, 200), (3, 8193, 500), (1, 270000, 300), (30, 4097, 80),
                                       (80, 33000, 128), (160, 129, 128), (2, 600, 640)])
def test_main_slots(units, s, b):
    g = torch.Generator(device="cuda").manual_seed(s)
    K = torch.randn(1, units, s, 128, generator=g, device="cuda").to(torch.bfloat16)
    V = torch.randn(1, units, s, 128, generator=g, device="cuda").to(torch.bfloat16)
    cfg = R.reskv_config_default(batch=1, n_layers=1, n_kv_heads=units, group=1, seq_len=s, budget=b, n_obs=0,
                                 n_fit=0, n_val=0, score_mode=R.RESKV_SCORE_KEYNORM,
                                 residual_override=np.zeros(units, np.int32), keep_debug=1)
    cache = R.reskv_build_cache(cfg, [K], [V], None)
    R.reskv_check_status(cache)
    lay = R.reskv_export_cache(cache)
    top = R.reskv_export_debug(cache, R.RESKV_DEBUG_RANKED)
    cache.free()
    P, m = 64, min(b, s)
    for u in {0, units // 2, units - 1}:
        want = np.sort(np.concatenate([top[u][:m - P], np.arange(s - P, s)]))
        assert lay["n_main"][u] == m and lay["n_res"][u] == 0
        assert np.array_equal(lay["slot_pos"][u][:m], want)
        for slots, src in (("kslots", K), ("vslots", V)):
            rows = src[0, u, torch.from_numpy(want.astype(np.int64)).cuda()].view(torch.int16).cpu().numpy()
            assert np.array_equal(lay[slots][u][:m].view(np.int16), rows)
        assert not lay["logc"][u][:m].any() and not lay["counts"][u][:m].any()
