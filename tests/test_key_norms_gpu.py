"""Key-norm scores at the edges of the 64-bit form: values 19 to 22 binades apart,
the lowest exponents at which it applies, every value at the top of its binade
(the largest sum), zeros and infinities between common rows, and row counts that
are no multiple of a warp's 32.  Bit for bit with the correctly rounded sum."""
import math

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


def rows(s):
    g = torch.Generator().manual_seed(s)
    K = torch.randn(s, 128, generator=g)
    top = 1.9921875                                    # 255 / 128
    for i in range(0, s, 3):
        e = (i % 24) * 10 - 120                        # the row's largest exponent
        span = 18 + (i // 3) % 6
        K[i] = top * 2.0 ** e
        K[i, 1::2] *= -1
        K[i, i % 128] = 2.0 ** max(e - span, -133)
    K[1] = 0
    K[4, 3] = math.inf
    for j, e in enumerate((-107, -106, -105, -126, 127)):   # around the lowest usable exponent
        K[7 + 3 * j] = top * 2.0 ** e
        K[7 + 3 * j, 5] = 2.0 ** max(e - 20, -133)
    return K.to(torch.bfloat16)


@pytest.mark.parametrize("s", [97, 255, 416])
@pytest.mark.parametrize("r", [0, 6])
def test_scores(s, r):
    K = rows(s)[None, None]
    if r:
        K = torch.where(K.isinf(), torch.zeros_like(K), K)  # (no infinities for the residual entries)
        K[K.float().abs() > 2.0 ** 60] = 1.5
    V = torch.zeros_like(K)
    cfg = R.reskv_config_default(batch=1, n_layers=1, n_kv_heads=1, group=4, seq_len=s, budget=80, n_obs=0, n_fit=0,
                                 n_val=0, score_mode=R.RESKV_SCORE_KEYNORM,
                                 residual_override=np.array([r], np.int32), keep_debug=1)
    cache = R.reskv_build_cache(cfg, [K.cuda()], [V.cuda()], None)
    R.reskv_check_status(cache)
    got = R.reskv_export_debug(cache, R.RESKV_DEBUG_SCORES).ravel()
    cache.free()
    Kd = K[0, 0].double().numpy()
    ref = np.array([math.inf if np.isinf(x).any() else math.fsum(x * x) for x in Kd])
    assert np.array_equal(got, ref), np.nonzero(got != ref)[0][:5]


@pytest.mark.parametrize("span", [11, 12, 13, 14])
@pytest.mark.parametrize("top", [-120, -112, -111, 0, 123, 124, 125])
def test_scores_of_narrow_rows(span, top):
    """Every row spans `span` binades (13 is the last that float additions take),
    at the largest exponents on both sides of that form's range; one row in 40
    spans more, so that its neighbours leave the form too."""
    s = 164
    g = torch.Generator().manual_seed(span)
    e = torch.randint(-span, 1, (s, 128), generator=g)
    K = (1 + torch.randint(0, 128, (s, 128), generator=g) / 128) * torch.exp2(e.float()) * 2.0 ** top
    K[:, 3], K[:, 77] = 1.9921875 * 2.0 ** top, 1.0078125 * 2.0 ** max(top - span, -126)
    K[::40, 5] = 2.0 ** max(top - 18, -133)
    K[:, 1::2] *= -1
    K[:, 9] = 0
    K = K.to(torch.bfloat16)[None, None]
    cfg = R.reskv_config_default(batch=1, n_layers=1, n_kv_heads=1, group=4, seq_len=s, budget=80, n_obs=0, n_fit=0,
                                 n_val=0, score_mode=R.RESKV_SCORE_KEYNORM,
                                 residual_override=np.zeros(1, np.int32), keep_debug=1)
    cache = R.reskv_build_cache(cfg, [K.cuda()], [K.cuda()], None)
    R.reskv_check_status(cache)
    got = R.reskv_export_debug(cache, R.RESKV_DEBUG_SCORES).ravel()
    cache.free()
    ref = np.array([math.fsum(x * x) for x in K[0, 0].double().numpy()])
    assert np.array_equal(got, ref), np.nonzero(got != ref)[0][:5]
