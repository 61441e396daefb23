"""Inputs that lie on an 8-byte boundary only (views into a larger buffer) where
no stage needs more: values of a build with given residual budgets, and keys of
a query-free build without residual entries.  The result is that of aligned
copies, bit for bit: the kernels differ in how they load, not in what."""
import numpy as np
import pytest
import torch

from paper_2607_29591_gb300 import build as B
from paper_2607_29591_gb300 import reskv as R
from paper_2607_29591_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def lib():
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    B.build()
    return R.load_library()


def shifted(t):
    """A copy of t that starts 8 bytes after a 16-byte boundary."""
    flat = torch.empty(t.numel() + 4, dtype=t.dtype, device=t.device)
    out = flat[4:].view(t.shape)
    out.copy_(t)
    assert out.is_contiguous() and out.data_ptr() % 16 == 8
    return out


def export(K, V, r, s):
    cfg = R.reskv_config_default(batch=1, n_layers=1, n_kv_heads=2, group=4, seq_len=s, budget=200,
                                 n_obs=0, n_fit=0, n_val=0, score_mode=R.RESKV_SCORE_KEYNORM,
                                 residual_override=np.array(r, np.int32))
    cache = R.reskv_build_cache(cfg, [K], [V], None)
    R.reskv_check_status(cache)
    lay = R.reskv_export_cache(cache)
    cache.free()
    return lay


@pytest.mark.parametrize("s", [700, 2049])
@pytest.mark.parametrize("r,shift_keys", [((40, 7), False), ((0, 0), True), ((0, 0), False)])
def test_shifted_inputs(s, r, shift_keys):
    w = wl.scaled(wl.WORKLOADS["small_budget_b64"], seq_len=s, budget=200, batch=1, n_layers=1, n_kv_heads=2)
    K, V, _, _ = wl.layer_inputs(w, 0, "cuda")
    ref = export(K, V, r, s)
    out = export(shifted(K) if shift_keys else K, shifted(V), r, s)
    assert ref.keys() == out.keys()
    for k in ref:
        assert np.array_equal(np.asarray(ref[k]), np.asarray(out[k])), k
