"""The table build at the edges of its ranges against the oracle's tables: the smallest grids, odd sizes, rows whose
spectrum the panels' Legendre series does not resolve (large chi), r down to the end of the logit grid."""
import numpy as np
import pytest

import oracle as O
from paper_2511_08929_gb300 import binding as B
from paper_2511_08929_gb300 import buffers as Q

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("chi_min,chi_max,n_chi,n_r,y_lo,y_hi", [
    (1e-4, 1e3, 2, 4, -20.0, 20.0),     # the smallest grid
    (1e-3, 1e2, 3, 257, -20.0, 16.0),   # more entries than threads, odd
    (0.5, 1e3, 7, 33, -25.0, 12.0),     # large chi: entries finished on the quadrature
    (1e-6, 2e-4, 5, 65, -12.0, 12.0),   # small chi: 8/(3 chi) beyond the Bessel table
])
def test_table_edges_match_oracle(chi_min, chi_max, n_chi, n_r, y_lo, y_hi):
    d = (chi_min, chi_max, n_chi, n_r, y_lo, y_hi)
    g = Q.Tables(*d)
    e = g.export()
    amm = B.qed_tables_export_amm(g.handle, g.desc)
    g.close()
    o = O.tables(*d)
    # rates: the quadrature's rounding, and that of exp(-x)'s exponents
    np.testing.assert_allclose(e["nlc_rate"], o.nlc_rate, rtol=0, atol=1e-12)
    np.testing.assert_allclose(e["nbw_rate"], o.nbw_rate, rtol=0, atol=1e-11)
    # ICDFs: 2e-11 as on the standard grid, and one rounding unit of the target and of the CDF sum (4.4e-16
    # together) over the tail 1 - r that is left there
    y = y_lo + (y_hi - y_lo) * np.arange(n_r) / (n_r - 1)
    tol = 2e-11 + 4.4e-16 * (1.0 + np.exp(y))
    for k in ("nlc_icdf", "nbw_icdf"):
        assert np.all(np.isfinite(e[k]))
        assert np.all(np.abs(e[k] - getattr(o, k)) <= tol), (k, np.abs(e[k] - getattr(o, k)).max(axis=(0, 1)))
    np.testing.assert_allclose(amm, o.ensure_amm().amm, rtol=0, atol=1e-12)


@pytest.mark.parametrize("n_r", [64, 65, 129, 1000])
def test_rows_do_not_depend_on_how_many_there_are(n_r):
    """The NLC rows take blocks of 128 threads where every row has an SM, else of 64: the entries of a grid's end rows
    are the same in a grid of two rows and in one that has them among many."""
    lo, hi = 1e-3, 1e2
    few = Q.Tables(lo, hi, 2, n_r)
    many = Q.Tables(lo, hi, 201, n_r)
    a, b = few.export(), many.export()
    few.close()
    many.close()
    for k in ("nlc_rate", "nbw_rate"):
        np.testing.assert_allclose(a[k], b[k][:, [0, -1]], rtol=0, atol=1e-13)  # (chi_max = chi_min e^(n d) to rounding)
    for k in ("nlc_icdf", "nbw_icdf"):
        assert np.array_equal(a[k][:, 0], b[k][:, 0]), k


@pytest.mark.parametrize("chi_min,chi_max", [(1e4, 3e5), (1e5, 1e7), (1e6, 1e10)])
def test_rows_of_very_large_chi_invert_their_quadrature(chi_min, chi_max):
    """Rows whose spectrum the panels' nodes do not resolve (chi above 1e5) still invert the CDF of their 12-point
    quadrature: the oracle's tables under the same rule, each row rising.  1e-5: where that CDF is nearly flat an entry
    hangs on its rounding."""
    d = (chi_min, chi_max, 9, 65, -20.0, 20.0)
    g = Q.Tables(*d)
    e = g.export()
    g.close()
    O.set_quadrature(12, 1.0 / 16.0)
    try:
        o = O.tables(*d)
        want = {k: np.array(getattr(o, k)) for k in ("nbw_rate", "nbw_icdf")}
    finally:
        O.set_quadrature(10, 1.0 / 16.0)
    np.testing.assert_allclose(e["nbw_rate"], want["nbw_rate"], rtol=0, atol=1e-11)
    assert np.all(np.diff(e["nbw_icdf"], axis=2) > 0)
    assert np.abs(e["nbw_icdf"] - want["nbw_icdf"]).max() <= 1e-5
