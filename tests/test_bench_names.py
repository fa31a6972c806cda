"""The kernel names that bench.py reports, against the library's launch rules."""
import re

import pytest

import bench

FORWARD = (bench.ROOT / "paper_2202_11770_gb300" / "csrc" / "hlb_forward.cu").read_text()


@pytest.mark.parametrize("n", [1001, 449_999, 450_000, 20_000_864, 20_000_865])
@pytest.mark.parametrize("precision", ["fp32", "bf16", "fp16", "fp64"])
def test_names_on_the_row_form(precision, n):
    pull, odd = bench.kernel_names(n, "rows", precision=precision)
    assert pull == ("k_step" if precision == "fp64" else "k_step2")
    two = precision == "fp32" or (precision in ("bf16", "fp16") and n >= 450_000)
    assert odd == ("k_aa_odd2" if two else "k_aa_odd")
    for name in (pull, odd):
        assert re.search(rf"\b{name}\(", FORWARD)


def test_size_limits_are_the_librarys():
    assert f"kOddPairSites = {bench.ODD_PAIR_SITES};" in FORWARD
    assert str(bench.AA_IN_GRID_SITES) in FORWARD


def test_form_stats_names_what_runs():
    import types
    lat = types.SimpleNamespace(n=1_000_000)
    durs = [0.5] * 10
    for precision in ("fp32", "bf16", "fp64"):
        for scheme, k in (("ab", 0), ("aa", 1)):
            d = bench.form_stats(lat, precision, scheme, sum(durs), durs, 0, 10, 6796.9, "rows")
            assert bench.kernel_names(lat.n, "rows", precision=precision)[k] in d["kernels"]
