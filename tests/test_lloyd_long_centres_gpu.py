"""Centres of more than 2^15 members whose values all leave something below the
grid of the float pairs that hold the member sums, with one sign: the exact sum
of what is left needs more bits the more members there are.  Entries against
the oracle's Lloyd (one centre: the mean of every evicted token)."""
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


@pytest.mark.parametrize("s", [33200, 66000])
@pytest.mark.parametrize("value", [2.0 ** -28, -(2.0 ** -21) * (1 + 2.0 ** -7), 255 * 2.0 ** -36, 2.0 ** -60],
                         ids=["2^-28", "two_bits", "255", "2^-60"])
def test_one_sign_over_many_members(s, value):
    b, P, r = 128, 64, 1
    g = torch.Generator().manual_seed(s)
    K = torch.randn(1, 1, s, 128, generator=g).to(torch.bfloat16)
    V = torch.randn(1, 1, s, 128, generator=g).to(torch.bfloat16)
    for X in (K, V):
        X[..., 11] = value
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
    u = unit_from_layout(lay, 0)
    assert u.kbar[0, 11] == u.vbar[0, 11] == float(K[0, 0, 0, 11])
    check_entries(u, bf16_to_f64(K[0, 0]), bf16_to_f64(V[0, 0]), top[0], P, s, b, 4)


def test_large_sums_with_dropped_bits():
    """Sums past 2^21 of which one member's low bits are dropped: more bits than
    a float64 holds, so the total is rounded from 128 bits."""
    s, b, P, r = 33200, 128, 64, 1
    g = torch.Generator().manual_seed(5)
    K = torch.randn(1, 1, s, 128, generator=g).to(torch.bfloat16)
    V = torch.randn(1, 1, s, 128, generator=g).to(torch.bfloat16)
    for X, sign in ((K, 1.0), (V, -1.0)):
        X[..., 11] = 100.0 * sign
        X[..., 700, 11] = 173 * 2.0 ** -36 * sign
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
