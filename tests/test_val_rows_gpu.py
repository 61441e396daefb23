"""Validation targets and losses (Eqs. valloss, valproxy) over the row counts that
change how their kernels share the work: one, two, four and eight groups of 16
rows per CTA, groups that are not full, a second row block (more than 128 rows),
and context lengths beside a tile of 128 tokens.  The protocol and its bounds
are those of the other build tests (losses within 2e-3 of the oracle's)."""
import pytest

from paper_2607_29591_gb300 import workloads as wl

from test_build_gpu import lib, run_case  # noqa: F401  (lib: the module's fixture)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("group,n_val,s", [
    (1, 16, 2048), (1, 20, 2047), (4, 8, 2049), (2, 24, 1921), (4, 16, 2048), (1, 80, 2175),
    (4, 32, 2177), (4, 33, 2048), (4, 40, 2111)])
def test_rows_per_unit(group, n_val, s):
    w = wl.scaled(wl.WORKLOADS["llama8b_layer_32k"], seq_len=s, budget=256, batch=1, n_kv_heads=2,
                  group=group, n_obs=n_val + 24, n_fit=24, n_val=n_val)
    run_case(w)
