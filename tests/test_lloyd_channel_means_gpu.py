"""Member sums of keys and values with a large mean in one dimension, as key
biases give: rows below 128 keep the exact pair of floats, larger ones are summed
in fp64.  Entries against the oracle's Lloyd, and the time of the first kind
beside that of centred keys."""
import numpy as np
import pytest
import torch

from paper_2607_29591_gb300 import build as B
from paper_2607_29591_gb300 import reskv as R

from helpers import bf16_to_f64, unit_from_layout
from parity import check_entries

pytestmark = pytest.mark.gpu
P = 64


@pytest.fixture(scope="module", autouse=True)
def lib():
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    B.build()
    return R.load_library()


def inputs(U, s, mean):
    g = torch.Generator().manual_seed(s)
    X = torch.randn(2, 1, U, s, 128, generator=g)
    X[..., 7] = (X[..., 7] + mean).clamp(-127.5 if mean < 128 else -1000, 127.5 if mean < 128 else 1000)
    return X.to(torch.bfloat16)


def build(K, V, b, r):
    _, U, s, _ = K.shape
    cfg = R.reskv_config_default(batch=1, n_layers=1, n_kv_heads=U, group=1, seq_len=s, budget=b,
                                 recent_window=P, n_obs=0, n_fit=0, n_val=0,
                                 score_mode=R.RESKV_SCORE_KEYNORM,
                                 residual_override=np.full(U, r, np.int32), keep_debug=1)
    cache = R.reskv_build_cache(cfg, [K], [V], None)
    torch.cuda.synchronize()
    R.reskv_check_status(cache)
    return cache


@pytest.mark.parametrize("mean", [-63.0, 65.0, 127.5, 130.0, -300.0])
@pytest.mark.parametrize("r", [1, 9])
def test_entries(r, mean):
    s, b = 3001, 200
    K, V = inputs(2, s, mean)
    cache = build(K.cuda(), V.cuda(), b, r)
    lay = R.reskv_export_cache(cache)
    top = R.reskv_export_debug(cache, R.RESKV_DEBUG_RANKED)
    cache.free()
    for h in range(2):
        check_entries(unit_from_layout(lay, h), bf16_to_f64(K[0, h]), bf16_to_f64(V[0, h]), top[h], P, s, b, 4)


def test_rows_below_128_take_the_time_of_centred_rows():
    """Two centres of 16K tokens: an fp64 sum over their members takes about a
    hundred times the rest (42.8 ms beside 0.3)."""
    ms = []
    for mean in (0.0, 100.0):
        K, V = (x.cuda() for x in inputs(8, 32768, mean))
        runs = []
        for _ in range(4):
            cache = build(K, V, 512, 2)
            runs.append(R.reskv_get_info(cache)["build_ms"][3])
            cache.free()
        ms.append(min(runs))
    assert ms[1] < 5 * ms[0], ms
