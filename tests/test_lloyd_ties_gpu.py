"""Lloyd assignment (Sec. 5.3) where distances are zero, or so small that their
squares underflow fp32: evicted keys that are all zero (a zero-padded sequence
whose tokens all fit the main cache), and keys scaled by 2^-60 .. 2^-80.  Exact
ties go to the lower centre; the status stays clear.  Counts and entries against
the oracle's Lloyd on the GPU's evicted set."""
import numpy as np
import pytest
import torch

from paper_2607_29591_gb300 import build as B
from paper_2607_29591_gb300 import reskv as R
from paper_2607_29591_gb300 import workloads as wl

from helpers import bf16_to_f64, unit_from_layout
from parity import check_entries

pytestmark = pytest.mark.gpu
S, P = 1500, 64


@pytest.fixture(scope="module", autouse=True)
def lib():
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    B.build()
    return R.load_library()


def check(K, V, b, r):
    cfg = R.reskv_config_default(batch=1, n_layers=1, n_kv_heads=2, group=1, seq_len=S, budget=b,
                                 recent_window=P, n_obs=0, n_fit=0, n_val=0,
                                 score_mode=R.RESKV_SCORE_KEYNORM,
                                 residual_override=np.full(2, r, np.int32), keep_debug=1)
    cache = R.reskv_build_cache(cfg, [K.cuda()], [V.cuda()], None)
    torch.cuda.synchronize()
    R.reskv_check_status(cache)
    lay = R.reskv_export_cache(cache)
    top = R.reskv_export_debug(cache, R.RESKV_DEBUG_RANKED)
    cache.free()
    for h in range(2):
        check_entries(unit_from_layout(lay, h), bf16_to_f64(K[0, h]), bf16_to_f64(V[0, h]), top[h],
                      P, S, b, 4)


def inputs(r):
    w = wl.scaled(wl.WORKLOADS["small_budget_b64"], seq_len=S, budget=r + P + 140, batch=1, n_layers=1,
                  n_kv_heads=2, recent_window=P)
    K, V, _, _ = wl.layer_inputs(w, 0, "cpu")
    return K, V, w.budget


@pytest.mark.parametrize("r", [1, 2, 8, 300])
def test_zero_keys(r):
    K, V, b = inputs(r)
    K[0, 0, 100:] = 0                     # 100 tokens, then padding; the other head is full
    check(K, V, b, r)


@pytest.mark.parametrize("r", [1, 2, 8, 300])
@pytest.mark.parametrize("e", [-60, -70, -80])
def test_tiny_keys(e, r):
    K, V, b = inputs(r)
    check((K.float() * 2.0 ** e).to(torch.bfloat16), V, b, r)
