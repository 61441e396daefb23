"""Pooled scores bit for bit: a width of 1 exports the sums A themselves, and any
width must give the fp64 sums of A in ascending order, divided and rounded once.
Context lengths beside a multiple of the four positions a thread takes."""
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


def scores(K, Q, pool):
    _, H, s, _ = K.shape
    cfg = R.reskv_config_default(batch=1, n_layers=1, n_kv_heads=H, group=1, seq_len=s, budget=70, n_obs=Q.shape[2],
                                 n_fit=Q.shape[2], n_val=0, pool_kernel=pool, residual_override=np.zeros(H, np.int32),
                                 keep_debug=1)
    cache = R.reskv_build_cache(cfg, [K], [K], [Q])
    R.reskv_check_status(cache)
    out = R.reskv_export_debug(cache, R.RESKV_DEBUG_SCORES).reshape(H, s).copy()
    cache.free()
    return out


@pytest.mark.parametrize("s", [76, 193, 1022, 2051])
def test_pooled_scores(s):
    g = torch.Generator(device="cuda").manual_seed(s)
    K = (3 * torch.randn(1, 3, s, 128, generator=g, device="cuda")).to(torch.bfloat16)
    Q = torch.randn(1, 3, 20, 128, generator=g, device="cuda").to(torch.bfloat16)
    A = scores(K, Q, 1)
    for pool in (3, 5, 7, 9, 31, 49):
        half = pool // 2
        pad = np.pad(A, ((0, 0), (half, half)))
        acc = np.zeros_like(A)
        for j in range(pool):
            acc += pad[:, j:j + s]
        assert np.array_equal(scores(K, Q, pool), acc / pool), pool
