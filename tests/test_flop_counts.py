"""Work counts behind the rooflines: fixed substeps do without the third
stage's solve and the error norm, and the forms with S_h2 algebraic without
products that are always zero."""
import os
import sys

import pytest

from paper_2311_08927_gb300 import chad as CH
from paper_2311_08927_gb300 import inputs as I

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
NS = I.NS


@pytest.fixture(scope="module")
def pattern():
    sys.path.insert(0, os.path.join(ROOT, "paper_2311_08927_gb300", "csrc"))
    import gen_sparse as G
    return G.jacobian_pattern()


def test_entries_of_the_second_sherman_morrison_level(pattern):
    """dS_h2/dy: the S_h2 row of the Jacobian and the states of Eq. 7; p2:
    every state that a rate moves (the ions only dilute)."""
    h2 = I.SIDX["S_h2"]
    eq7 = {I.SIDX[n] for n in ("S_va", "S_bu", "S_pro", "S_ac", "S_IC", "S_IN", "S_cat", "S_an")}
    F = CH.flop_counts()
    direct = {j for j in range(NS) if pattern[h2, j]}
    assert F["h2_reads"] >= len((direct | eq7) - {h2})  # fill of the LU may add some
    assert F["h2_reads"] < NS - 1
    assert F["h2_moves"] == NS - 3


def test_products_with_structural_zeros_are_counted_apart():
    F, a = CH.flop_counts(), CH.attempt_flops(CH.PREC_FP64, True)
    executed = a["fp64"] - a["fp64_zero"]
    nr, nm = F["h2_reads"], F["h2_moves"]
    # 59 = 2 x 29 + 1, 117 = 2 x 29 + 1 + 2 x 29, 58 = 2 x 29 of the full products
    full = 59 + 3 * 117 + 2 * 58
    left = (2 * nr + 1) + 3 * (2 * nr + 1 + 2 * nm) + 2 * 2 * nr
    assert a["fp64"] - executed == full - left > 0
    # form 4: two level-2 updates and one S_h2 direction per stage, one dot product
    stage = 2 * (2 * nr + 1 + 2 * nm) + 13 * nr + 8 * 13 + 33 * NS
    assert F["mx_stage"] == stage
    assert F["mx_fp32_extra"] == 83 + NS + 2 * nr + 3 + 3 * stage + NS + 19 * NS + 62 * NS


@pytest.mark.parametrize("h2", [False, True])
def test_fixed_substeps_of_the_fp64_forms(h2):
    F = CH.flop_counts()
    a, b = CH.attempt_flops(CH.PREC_FP64, h2), CH.attempt_flops(CH.PREC_FP64, h2, True)
    done = lambda c: c["fp64"] - c.get("fp64_zero", 0)
    left = F["solve_h2a"] if h2 else F["solve"]
    left += F["sm_update"]
    left += 2 * F["h2_reads"] + 1 + 2 * F["h2_moves"] if h2 else 0
    left += 5 * NS + 7 * NS  # right-hand side; error, scale and ratio
    assert done(a) - done(b) == left
    assert CH.attempt_flops(CH.PREC_MIXED) == CH.attempt_flops(CH.PREC_MIXED, False, True)


def test_fixed_substeps_of_the_mixed_form_with_h2_algebraic():
    F = CH.flop_counts()
    a, b = CH.attempt_flops_h2_mixed(), CH.attempt_flops_h2_mixed(True)
    left = (F["rates_f"] - F["factors"]) + 2 * (F["solve_h2a"] + F["sm_update"]) + F["mx_stage"]
    left += F["jx_twofloat"] + F["rates_partials"] + 62 * NS
    assert a["fp32"] - b["fp32"] == left and a["fp64"] == b["fp64"]
    assert 0 < F["factors"] < F["rates_f"]
