"""A ring fold with a value that is not finite drops the token and raises the
status, wherever among the entries the value lies: each warp of the append
kernel finds out for its own groups of 8 entries, and none may be missed.  Many
units per launch, so that the warps of a CTA meet in many orders."""
import numpy as np
import pytest
import torch

from paper_2607_29591_gb300 import build as B
from paper_2607_29591_gb300 import reskv as R

from helpers import bf16_bits

pytestmark = pytest.mark.gpu
MAIN, UNITS = 4, 512


@pytest.fixture(scope="module", autouse=True)
def lib():
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    B.build()
    return R.load_library()


@pytest.mark.parametrize("r,at", [(9, 8), (64, 63), (65, 8), (200, 57), (1030, 1025)])
@pytest.mark.parametrize("value", [float("inf"), float("-inf"), float("nan")])
def test_one_value_anywhere_drops_the_token(r, at, value):
    b, U = MAIN + r, UNITS if r <= 200 else 64
    g = torch.Generator().manual_seed(r)
    slots = torch.zeros(U, b + 1, 128)
    slots[:, MAIN:b] = torch.randn(U, r, 128, generator=g)
    slots[:, MAIN + at, 77] = value
    bits = bf16_bits(slots.to(torch.bfloat16))
    counts = np.zeros((U, b + 1), np.int32)
    counts[:, MAIN:b] = 3
    cfg = R.reskv_config_default(batch=U, n_layers=1, n_kv_heads=1, group=1, seq_len=8 * b, budget=b,
                                 append_capacity=1)
    h = R.reskv_import_cache(cfg, np.full(U, MAIN), np.full(U, r), bits, bits,
                             np.log(np.maximum(counts, 1)).astype(np.float32), counts=counts)
    x = torch.randn(U, 128, generator=g).to(torch.bfloat16).cuda()
    for _ in range(4):                    # the first fills the ring, the others push a token out
        R.reskv_append(h, 0, x, x)
    torch.cuda.synchronize()
    with pytest.raises(R.ReskvError) as e:
        R.reskv_check_status(h)
    assert e.value.status == R.RESKV_ERR_DEVICE_STATUS
    ex = R.reskv_export_cache(h)
    h.free()
    assert (ex["counts"][:, MAIN:b] == 3).all()
    assert np.array_equal(ex["kslots"][:, MAIN:b], bits.reshape(U, b + 1, 128)[:, MAIN:b])
    assert np.array_equal(ex["vslots"][:, MAIN:b], bits.reshape(U, b + 1, 128)[:, MAIN:b])
