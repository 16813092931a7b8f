"""The normal distribution function of the products' epilogues (Abramowitz and Stegun 7.1.26), with the constants of the source:
what its comment says of its error, in fp32 and for results stored as bf16."""
import os
import re

import numpy as np
from scipy.special import erf, erfc

from spa_workloads import bf16_round

SRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2410_23608_b200", "csrc", "spa_common.cuh")
F = np.float32


def formula(u):
    """cdf, pdf of the source in the precision of u."""
    body = re.search(r"void normal_cdf_pdf\(.*?\n}", open(SRC).read(), re.S).group(0)
    p, a = re.search(r"fmaf\(([\d.]+)f, x, 1\.f\)", body), re.findall(r"(-?\d\.\d{9})f", body)
    T = u.dtype.type
    a5, a4, a3, a2, a1 = (T(v) for v in a)
    x = np.abs(u) * T(0.70710678118654752)
    e = np.exp(-x * x)
    t = T(1) / (T(p.group(1)) * x + T(1))
    tail = T(0.5) * t * ((((a5 * t + a4) * t + a3) * t + a2) * t + a1) * e
    return np.where(u < 0, tail, T(1) - tail), T(0.3989422804014327) * e


def test_error_of_the_formula():
    u = np.linspace(-9, 9, 360001)
    exact = 0.5 * erfc(-u / np.sqrt(2))
    assert np.abs(formula(u)[0] - exact).max() < 7.5e-8
    assert np.abs(formula(u.astype(F))[0] - 0.5 * erfc(-u.astype(F).astype(float) / np.sqrt(2))).max() < 4e-7
    for at, rel in ((-3.0, 6e-5), (-4.0, 6e-4), (-6.0, 5e-3), (-8.0, 2e-2)):
        v = np.array([at])
        assert abs(formula(v)[0][0] / (0.5 * erfc(-at / np.sqrt(2))) - 1) < rel


def test_results_stored_as_bf16_are_as_good_as_by_erf():
    u = (np.arange(65536, dtype=np.uint32) << 16).view(F)
    u = u[np.isfinite(u) & (np.abs(u) < 12) & (np.abs(u) > 1e-3)]
    d, (cdf, pdf) = u.astype(float), formula(u)
    one_plus_erf = F(1) + erf((u * F(0.70710678118654752)).astype(float)).astype(F)
    pdf_erf = F(0.3989422804014327) * np.exp((F(-0.5) * u * u).astype(float)).astype(F)
    phi, Phi = np.exp(-d * d / 2) / np.sqrt(2 * np.pi), 0.5 * erfc(-d / np.sqrt(2))
    near = np.abs(u) < 4
    for new, old, exact in ((u * cdf, F(0.5) * u * one_plus_erf, d * Phi), (u * pdf + cdf, F(0.5) * one_plus_erf + u * pdf_erf, Phi + d * phi)):
        n, o = bf16_round(new.astype(float)), bf16_round(old.astype(float))
        assert (n != o)[near].sum() <= 4
        rms = lambda v: np.sqrt(((v - exact) ** 2).mean())
        assert rms(n) <= rms(o) * 1.00001
        beyond = lambda v: (np.abs(v - exact) > 2.0 ** -8 * np.abs(exact)).sum()   # values off by more than a rounding
        assert beyond(n) <= beyond(o)
