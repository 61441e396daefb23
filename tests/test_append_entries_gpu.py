"""The residual entry that takes the oldest appended token (the nearest-centre
rule of Eq. residual_partition), at the edges of the append kernel's two steps:
entry counts around its groups of 8 entries, its candidate list (64) and its
chunk of distances (1024), more equal entries than the list holds, distances
that overflow fp32, and values that are not finite.  The reference is the
oracle's exact nearest_entry, and fold_into_entry bit for bit."""
import numpy as np
import pytest
import torch

import oracle as orc
from paper_2607_29591_gb300 import build as B
from paper_2607_29591_gb300 import reskv as R

from helpers import bf16_bits

pytestmark = pytest.mark.gpu
MAIN = 4


@pytest.fixture(scope="module", autouse=True)
def lib():
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    B.build()
    return R.load_library()


def fold(entries, k):
    """One unit with these residual entries (count 3 each): k is appended into
    its one ring slot and pushed out again.  Returns the status error and the
    unit's exported entries."""
    r, b = len(entries), MAIN + len(entries)
    S = b + 1
    E = torch.from_numpy(np.asarray(entries, np.float32)).to(torch.bfloat16)
    kt = torch.from_numpy(np.asarray(k, np.float32)).to(torch.bfloat16)
    slots = torch.zeros(1, S, 128, dtype=torch.bfloat16)
    slots[0, MAIN:b] = E
    counts = np.zeros((1, S), np.int32)
    counts[0, MAIN:b] = 3
    cfg = R.reskv_config_default(batch=1, n_layers=1, n_kv_heads=1, group=1, seq_len=8 * b,
                                 budget=b, append_capacity=1)
    h = R.reskv_import_cache(cfg, np.array([MAIN]), np.array([r]), bf16_bits(slots), bf16_bits(slots),
                             np.log(np.maximum(counts, 1)).astype(np.float32), counts=counts)
    x = kt.reshape(1, 1, 128).cuda()
    R.reskv_append(h, 0, x, x)
    R.reskv_append(h, 0, x * 0, x * 0)
    torch.cuda.synchronize()
    err = None
    try:
        R.reskv_check_status(h)
    except R.ReskvError as e:
        err = e
    ex = R.reskv_export_cache(h)
    h.free()
    return err, ex, E.double().numpy(), kt.double().numpy()


def check(entries, k):
    err, ex, E, kd = fold(entries, k)
    assert err is None, err
    want = orc.nearest_entry(kd, E)
    counts = ex["counts"][0, MAIN:MAIN + len(E)]
    assert np.flatnonzero(counts != 3).tolist() == [want] and counts[want] == 4
    kb, vb, _, logc = orc.fold_into_entry(E[want], E[want], 3, kd, kd, 1.0)
    assert np.array_equal(orc.bf16_bits_to_f64(ex["kslots"][0, MAIN + want]), kb)
    assert np.array_equal(orc.bf16_bits_to_f64(ex["vslots"][0, MAIN + want]), vb)
    assert abs(ex["logc"][0, MAIN + want] - logc) <= 3e-7 * logc


@pytest.mark.parametrize("r", [1, 7, 8, 9, 63, 64, 65, 511, 1023, 1024, 1025, 1100])
@pytest.mark.parametrize("near", ["spread", "last"])
def test_nearest_entry_over_entry_counts(r, near):
    g = np.random.RandomState(r)
    E, k = g.randn(r, 128), g.randn(128)
    if near == "last":                    # the nearest entry is the last one
        E[-1] = k + 0.01 * g.randn(128)
    check(E, k)


@pytest.mark.parametrize("r", [3, 64, 70, 1030])
def test_equal_entries_go_to_the_lowest(r):
    """All entries equal but the first: more candidates than the list holds."""
    g = np.random.RandomState(r)
    E = np.repeat(g.randn(1, 128), r, 0)
    E[0] += 5.0
    check(E, E[1] + 0.25)


@pytest.mark.parametrize("scale", [2.0 ** 100, 2.0 ** -70, 2.0 ** -100])
def test_distances_outside_fp32(scale):
    """Squares that overflow fp32, and squares that underflow."""
    g = np.random.RandomState(5)
    check(scale * g.randn(40, 128), scale * g.randn(128))


@pytest.mark.parametrize("where", ["entry", "token"])
def test_values_that_are_not_finite_drop_the_token(where):
    g = np.random.RandomState(6)
    E, k = g.randn(20, 128), g.randn(128)
    (E[13] if where == "entry" else k)[5] = np.inf if where == "entry" else np.nan
    err, ex, _, _ = fold(E, k)
    assert err is not None and err.status == R.RESKV_ERR_DEVICE_STATUS
    assert (ex["counts"][0, MAIN:MAIN + 20] == 3).all()
