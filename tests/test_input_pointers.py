"""Construction refuses inputs on a smaller boundary than its kernels read
(include/reskv.h), before any CUDA call: the pointers here are never followed
and no GPU is needed."""
import ctypes

import numpy as np
import pytest

from paper_2607_29591_gb300 import build as B
from paper_2607_29591_gb300 import reskv as R

BASE = 1 << 20


@pytest.fixture(scope="module")
def lib():
    B.build()
    return R.load_library()


def build(lib, k=0, v=0, q=0, layers=1, s=1024, budget=96, **cfg):
    c = R.reskv_config_default(batch=1, n_layers=layers, n_kv_heads=2, group=4, seq_len=s, budget=budget,
                               **cfg)
    ptrs = [(ctypes.c_void_p * layers)(*[BASE + (off if l == layers - 1 else 0) for l in range(layers)])
            for off in (k, v, q)]
    out = ctypes.c_void_p()
    st = lib.reskv_build_cache(ctypes.byref(c), ptrs[0], ptrs[1], ptrs[2], None, ctypes.byref(out))
    assert not out.value
    return st, lib.reskv_last_error().decode()


KEYNORM = dict(score_mode=R.RESKV_SCORE_KEYNORM, n_obs=0, n_fit=0, n_val=0)
OBS = dict(n_obs=128, n_fit=96, n_val=32)


def fixed(r, layers=1):
    return np.full(2 * layers, r, np.int32)


@pytest.mark.parametrize("what,cfg", [
    (dict(k=8), OBS), (dict(v=8), OBS), (dict(q=2), OBS),                              # the validation proxy
    (dict(k=8), dict(OBS, residual_override=fixed(8))),                                # observation scores
    (dict(q=2), dict(OBS, residual_override=fixed(8))),
    (dict(v=4), dict(OBS, residual_override=fixed(8))),
    (dict(k=8), dict(KEYNORM, residual_override=fixed(8))),                            # residual entries
    (dict(k=4), dict(KEYNORM, residual_override=fixed(0))),                            # rows are copied
    (dict(v=4), dict(KEYNORM, residual_override=fixed(0))),
    (dict(k=4), dict(KEYNORM, residual_override=fixed(8), s=60, budget=32, recent_window=16)),   # fewer keys than a tile
    (dict(k=8, layers=3), dict(KEYNORM, residual_override=fixed(8, 3))),               # any layer
])
def test_misaligned_inputs_are_refused(lib, what, cfg):
    st, msg = build(lib, **what, **cfg)
    assert st == R.RESKV_ERR_INVALID_ARG, (st, msg)
    assert "aligned" in msg
