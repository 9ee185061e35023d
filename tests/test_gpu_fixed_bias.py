"""Sums over many sites of the fixed-point products (csrc/fixed.cuh): roundings that leaned to one side would add up
where random ones cancel.  S and Q of the double-precision forms against the same sums in long double, averaged over
fields.

Bounds.  A record is rounded to U = 2^-53 and its sums add a few U at random, so that the mean relative error of S over
eight fields stays within U; half as much again is allowed.  Q is a sum of densities of size amp^4: its absolute
error, per unit of 1, stays far below U, a quarter of which is allowed.
"""
import numpy as np
import pytest

from oracle import tgf_oracle as O
from paper_2107_03747_gb300 import inputs as I

pytestmark = pytest.mark.gpu

U = 2.0 ** -53
TW = I.default_twist(1)


@pytest.mark.parametrize("N", [None, 2, 3, 4])  # None: the SU(3) kernels
def test_observables_are_unbiased(tgf, N, monkeypatch):
    monkeypatch.setattr(O, "float", lambda x: x, raising=False)  # the oracle's sums stay in long double
    n = N or 3
    L = (4, 4, 8, 8)
    s, q = [], []
    for seed in range(8):
        u = I.random_links(L, 40 + seed, 0.12, N=n)
        b = tgf.FlowBatch([L], "fp64", any_extents=True) if N is None else tgf.SunBatch(N, [L], any_extents=True)
        b.set_links([u])
        g = b.measure()[0].tolist()
        o = O.measure(u.astype(np.clongdouble), TW)
        assert isinstance(o["S"], np.longdouble)
        s.append(float((np.longdouble(g[4]) - o["S"]) / o["S"]))
        q.append(float(np.longdouble(g[2]) - o["Q"]))
    assert abs(np.mean(s)) <= 1.5 * U
    assert abs(np.mean(q)) <= 0.25 * U
