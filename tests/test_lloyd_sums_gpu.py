"""Centre means (Eq. summary) where the member sums leave their exact pair of
floats: values whose low bits it drops (added as a second integer), values
below that as well, and running sums that leave the binade (both summed in
fp64).  Counts and bf16 entries against the oracle's Lloyd on the GPU's
evicted set."""
import numpy as np
import pytest
import torch

from paper_2607_29591_gb300 import build as B
from paper_2607_29591_gb300 import reskv as R
from paper_2607_29591_gb300 import workloads as wl

from helpers import bf16_to_f64, unit_from_layout
from parity import check_entries

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def lib():
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    B.build()
    return R.load_library()


@pytest.mark.parametrize("r", [1, 8, 40])
@pytest.mark.parametrize("case", ["one_tail", "all_tails", "below_tails", "one_sign", "large"])
def test_member_sums_outside_the_float_pair(case, r):
    s, b, P = 1500, 256, 64
    w = wl.scaled(wl.WORKLOADS["small_budget_b64"], seq_len=s, budget=b, batch=1, n_layers=1,
                  n_kv_heads=2)
    K, V, _, _ = wl.layer_inputs(w, 0, "cpu")
    g = np.random.default_rng(r)
    m = torch.from_numpy(g.integers(128, 256, size=(2, s)) * g.choice([-1.0, 1.0], size=(2, s)))
    for X in (K, V):
        if case == "one_tail":           # one value below 2^-20 in the whole unit
            X[0, :, 700, 3] = float(2.0 ** -31 * 173)
        elif case == "all_tails":
            X[0, :, :, 11] = (m * 2.0 ** -35).to(torch.bfloat16)
        elif case == "below_tails":      # bits below 2^-76
            X[0, :, :, 11] = (m * 2.0 ** -79).to(torch.bfloat16)
        elif case == "one_sign":         # 64 rows of one sign sum past 2^12
            X[0, :, :, 11] = (m.abs() * 0.5).to(torch.bfloat16)
        else:
            X[0, :, ::50, 11] = (m[:, ::50] * 2.0 ** 8).to(torch.bfloat16)
    cfg = R.reskv_config_default(batch=1, n_layers=1, n_kv_heads=2, group=w.group, seq_len=s,
                                 budget=b, recent_window=P, n_obs=0, n_fit=0, n_val=0,
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
                      P, s, b, 4)
