"""Lloyd assignment (Sec. 5.3, Eq. residual_partition) at the edges of its
kernel: one to four 16-column blocks per warp, one to three segments of 256
centres, units without centres between, a layer with fewer keys than a tile,
and repeated keys (exact ties: the lower centre).  Counts and entries against
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


@pytest.fixture(scope="module", autouse=True)
def lib():
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    B.build()
    return R.load_library()


def run(s, b, P, ovr, repeat=1):
    U = len(ovr)
    w = wl.scaled(wl.WORKLOADS["small_budget_b64"], seq_len=s, budget=b, batch=1, n_layers=1,
                  n_kv_heads=U, recent_window=P)
    K, V, _, _ = wl.layer_inputs(w, 0, "cpu")
    if repeat > 1:                        # every key `repeat` times
        K = K[:, :, torch.arange(s) // repeat].contiguous()
    cfg = R.reskv_config_default(batch=1, n_layers=1, n_kv_heads=U, group=w.group, seq_len=s,
                                 budget=b, recent_window=P, n_obs=0, n_fit=0, n_val=0,
                                 score_mode=R.RESKV_SCORE_KEYNORM,
                                 residual_override=np.array(ovr, np.int32), keep_debug=1)
    cache = R.reskv_build_cache(cfg, [K.cuda()], [V.cuda()], None)
    torch.cuda.synchronize()
    R.reskv_check_status(cache)
    lay = R.reskv_export_cache(cache)
    top = R.reskv_export_debug(cache, R.RESKV_DEBUG_RANKED)
    cache.free()
    for h in range(U):
        gu = unit_from_layout(lay, h)
        assert gu.r == ovr[h]
        check_entries(gu, bf16_to_f64(K[0, h]), bf16_to_f64(V[0, h]), top[h], P, s, b, 4)


@pytest.mark.parametrize("ovr", [[64, 0, 3, 16], [128, 1, 65, 0, 17], [0, 192, 129, 48],
                                 [256, 193, 0, 5], [257, 64, 320, 0, 512], [513, 1, 300, 600]])
def test_assignment_over_centre_counts(ovr):
    run(1700, 700, 64, ovr)


@pytest.mark.parametrize("s", [100, 127, 128, 129])
def test_assignment_of_few_keys(s):
    run(s, 48, 16, [9])


@pytest.mark.parametrize("r", [20, 100, 300])
def test_repeated_keys_go_to_the_lower_centre(r):
    run(1500, 420, 64, [r, 0, 7], repeat=3)
