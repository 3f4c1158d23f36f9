"""The interpolation coefficients of csrc/series_coef.cuh against their
definition: every function of the band (|omega| <= pi / 2 per sample) is
reproduced between its samples to the errors that series_fit.py states."""
import os
import re

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_1903_06555_gb300", "csrc")


def coefficients(name, terms, half):
    src = open(os.path.join(CSRC, "series_coef.cuh")).read()
    body = src.split(name)[1].split("};")[0].split("=", 1)[1]
    v = [float(t) for t in re.findall(r"[-+]?\d[\d.]*(?:e[-+]?\d+)?(?=f?[,}\s])", body)]
    if name == "c_series_f":
        assert v[0::2] == v[1::2]
        v = v[0::2]
    return np.array(v).reshape(terms, half)


@pytest.mark.parametrize("name,terms,half,edge,inner", [("c_series_f", 8, 10, 6.5e-8, 6e-9),
                                                       ("c_series_d", 14, 20, 4e-15, 4e-15)])
def test_band_is_reproduced(name, terms, half, edge, inner):
    C = coefficients(name, terms, half)
    om = np.linspace(0.0, np.pi / 2, 65)[:, None]
    t = np.linspace(-1.0, 1.0, 101)
    d = np.arange(half)
    for phase in (0.0, 0.5 * np.pi):        # cos and sin about the interval's middle
        f = lambda x: np.cos(om * (x - 0.5) - phase)
        s = np.array([f(1.0 + d) + (-1.0) ** m * f(-1.0 * d) for m in range(terms)])
        got = np.einsum("md,mod,mt->ot", C, s, t[None, :] ** np.arange(terms)[:, None])
        err = np.abs(got - f(0.5 * (t + 1.0)))
        assert err.max() < edge and err[:33].max() < inner
