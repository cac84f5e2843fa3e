"""The Eq. 7 root from every kind of start: Newton ended by the third-order
step, and the bracket that takes over where Newton leaves (0, inf) or its
residual grows.  The library's host build of the kernels' routine against the
oracle's own solver (plain bisection and Newton)."""
import numpy as np
import pytest

import oracle as O
from paper_2311_08927_gb300 import chad as CH
from paper_2311_08927_gb300 import inputs as I

# E(S) is a sum of ~10 terms of up to 0.3 kmol/m^3, each rounded to 1.1e-16
# relative: |dS| <= 10 * 0.3 * 1.1e-16 / E'(S).  The third-order step leaves
# 2 (2^-18)^3 = 1.1e-16 relative on top.
TERMS = 10


def _slope(p, T, y, S):
    """E'(S) >= 1 of Eq. 7 (numpy)."""
    P = dict(zip(I.PARAM_NAMES, p))
    hoff = lambda dH: np.exp(dH / P["R_J"] * (1 / P["T_base"] - 1 / T))
    kw = 10.0 ** -P["pK_w"] * hoff(P["dH_K_w"])
    d = 1.0 + kw / S ** 2
    K = 10.0 ** -P["pK_a_IN"] * hoff(P["dH_K_a_IN"])
    d += K * y[I.SIDX["S_IN"]] / (K + S) ** 2
    for s, K, w in (("S_IC", 10.0 ** -P["pK_a_co2"] * hoff(P["dH_K_a_co2"]), 1.0),
                    ("S_ac", 10.0 ** -P["pK_a_ac"], 64.0), ("S_pro", 10.0 ** -P["pK_a_pro"], 112.0),
                    ("S_bu", 10.0 ** -P["pK_a_bu"], 160.0), ("S_va", 10.0 ** -P["pK_a_va"], 208.0)):
        d += K * y[I.SIDX[s]] / (K + S) ** 2 / w
    return d


def _states():
    rng = np.random.default_rng(5)
    base = I.x_ss()
    yield base
    for _ in range(6):
        yield base * np.exp(0.5 * rng.standard_normal(I.NS))
    acid = base.copy()
    acid[I.SIDX["S_ac"]] = 20.0       # acidified: pH below 5
    yield acid
    water = np.zeros(I.NS)            # no buffer at all: pH of water
    yield water
    salt = water.copy()
    salt[I.SIDX["S_cat"]] = 0.05      # strong base, pH above 12
    yield salt


@pytest.mark.parametrize("guess", [1e-14, 1e-9, 1e-7, 1e-3, 1.0, float("nan"), -1.0, None])
def test_root_from_any_start_is_the_oracles(guess):
    p = I.default_params()
    for y in _states():
        for T in (303.15, 313.15):
            ref = O.charge_solve(p, T, y)[0]
            start = ref * (1.0 + 1e-4) if guess is None else guess
            SH = CH.eval_model(p, T, y, SH_guess=start)[2]
            scale = max(np.max(np.abs(y[[I.SIDX[s] for s in ("S_cat", "S_an", "S_IN", "S_IC")]])), ref,
                        y[I.SIDX["S_ac"]] / 64.0)
            tol = 2 * (TERMS * scale * 1.1e-16 / _slope(p, T, y, ref) + 2e-16 * ref) + 1e-15 * ref
            # the oracle stops at |E| <= 1e-15 or |dS| <= 1e-14 S
            tol += 1e-15 / _slope(p, T, y, ref) + 1e-14 * ref
            assert abs(SH - ref) <= tol, (guess, T, SH, ref)
