"""The fixed-point matrix products of the double-precision kernels (csrc/fixed.cuh) against the oracle at
the edges of their range, where a thread goes over to FP64 arithmetic: links larger than 1, products T
and staple sums out of bounds, entries that are exactly 0, -0, +-1 or far below 2^-58, and fields in
which only some links are of that kind, so that both paths run in one warp.

Tolerances, relative to the size of what is compared: FP64 arithmetic carries about 100 roundings of 2^-53
along a link (six staples, Omega, the exponential, the update), 1.1e-14 in the worst case; the
fixed-point products are held to the same bound, scaled by the size of the staple sum that enters.
"""
import numpy as np
import pytest

from oracle import tgf_mc_oracle as M
from oracle import tgf_oracle as O
from paper_2107_03747_gb300 import inputs as I

pytestmark = pytest.mark.gpu

TW = I.default_twist(1)
L = (3, 2, 5, 4)  # 120 sites: a partly filled last block of 32
U = 2.0 ** -53


def edge_field(kind, N=3, L=L, amp=0.7):
    u = I.random_links(L, 5, amp, N=N)
    rng = np.random.default_rng(7)
    hit = rng.random(u.shape[:5]) < 0.1
    if kind == "su":
        return u
    if kind == "unit":  # exact 0, 1 and -0 entries
        u = np.zeros_like(u)
        u[..., range(N), range(N)] = 1.0
        u[hit] = -0.0 * u[hit] + np.where(np.eye(N) > 0, 1.0, -0.0)
        return u
    if kind == "tiny":  # off-diagonal entries down to denormals
        s = 10.0 ** -rng.uniform(0, 320, u.shape)
        d = np.zeros_like(u)
        d[..., range(N), range(N)] = 1.0
        return d + u * s * (1 - np.eye(N))
    if kind == "some_large":  # entries above 1 + 2^-10 in a tenth of the links
        u[hit] *= 1.7
        return u
    if kind == "all_large":
        return 3.0 * u
    if kind == "wide":  # links of one direction far from unitary, every entry and staple sum within its bound, W not
        v = np.zeros_like(u)
        v[..., range(N), range(N)] = 1.0
        v[:, :, :, :, 0] = rng.choice([-1.0, 1.0], (N, N)) + 1j * rng.choice([-1.0, 1.0], (N, N))
        return v
    if kind == "just_in":  # at the bound of a link entry
        v = np.zeros_like(u)
        v[..., range(N), range(N)] = 1.0 + 2.0 ** -11
        return v
    if kind == "not_unitary":  # every entry within the bound, T = V B^+ far beyond 2
        return np.sign(u.real) + 1j * np.sign(u.imag)
    raise ValueError(kind)


KINDS = ["su", "unit", "tiny", "some_large", "all_large", "just_in", "not_unitary"]


@pytest.mark.parametrize("kind", KINDS)
def test_stage_matches_the_oracle_at_the_edges_of_the_range(tgf, kind):
    u = edge_field(kind)
    b = tgf.FlowBatch([L], "fp64", any_extents=True)
    b.set_links([u])
    scale = max(1.0, np.abs(u).max()) ** 4
    h = 0.02 / scale
    b.stage(1, h)
    ref = np.matmul(O.expm(0.25 * h * O.force(u, TW)), u)
    assert np.abs(b.get_links()[0] - ref).max() <= 100 * U * np.abs(u).max()


@pytest.mark.parametrize("kind", KINDS)
def test_measure_matches_the_oracle_at_the_edges_of_the_range(tgf, kind):
    u = edge_field(kind)
    b = tgf.FlowBatch([L], "fp64", any_extents=True)
    b.set_links([u])
    g = b.measure()[0]
    o = O.measure(u, TW)
    # plaquette deviations (up to 3 + 9 m^4 a plaquette) and clovers (entries up to 9 m^4): absolute bounds
    m = np.abs(u).max()
    big = 9.0 * (1.0 if kind in ("su", "unit", "tiny", "just_in") else m ** 4 * 9)
    V = u[..., 0, 0, 0].size
    assert abs(g[4] - o["S"]) <= 100 * U * 6 * V * big
    assert abs(g[1] - o["E"]) <= 100 * U * 6 * 9 * big * big
    assert abs(g[2] - o["Q"]) <= 100 * U * V * 9 * big * big


def test_one_bad_link_stays_local(tgf):
    """A NaN link makes the links whose staples contain it NaN, and no others."""
    u = edge_field("su")
    u[1, 2, 1, 0, 2] = np.nan
    b = tgf.FlowBatch([L], "fp64", any_extents=True)
    b.set_links([u])
    b.stage(1, 0.02)
    got = b.get_links()[0]
    with np.errstate(invalid="ignore"):
        bad = np.isnan(O.force(u, TW)).any((-1, -2))
    assert np.array_equal(np.isnan(got).any((-1, -2)), bad)
    clean = u.copy()
    clean[1, 2, 1, 0, 2] = np.eye(3)
    ref = np.matmul(O.expm(0.005 * O.force(clean, TW)), clean)
    assert np.abs(got - ref)[~bad].max() <= 100 * U


@pytest.mark.parametrize("kind", ["su", "unit", "some_large", "all_large", "wide"])
@pytest.mark.parametrize("n_or", [0, 2])
def test_monte_carlo_matches_the_oracle_at_the_edges_of_the_range(tgf, kind, n_or):
    # bar of the Monte Carlo parity tests: rounding amplified by the division by k, 1e-10 on the links
    Lm = (4, 2, 2, 6)
    u = edge_field(kind, L=Lm, amp=0.4)
    b = tgf.FlowBatch([Lm], "fp64", any_extents=True)
    b.set_links([u])
    tgf.tgf_mc_sweeps(b.prec, b.lat, b.links, 6.0, 1, n_or, 3, 1)
    ref = M.hybrid(u, TW, 6.0, n_or, 3, 0, 1)
    assert np.abs(b.get_links()[0] - ref).max() <= 1e-10 * max(1.0, np.abs(u).max())


def test_monte_carlo_keeps_links_unitary(tgf):
    """Rounding drift off SU(3) of 50 sweeps of reflections, a random walk of about 40 roundings of 2^-53
    per link and sweep: sqrt(50 x 40) 2^-53 = 5e-15 on an entry of U U^+, ten times that over all links."""
    Lm = (4, 4, 12, 12)
    b = tgf.FlowBatch([Lm], "fp64")
    b.set_links([I.random_links(Lm, 3, 0.2)])
    tgf.tgf_mc_sweeps(b.prec, b.lat, b.links, 20.0, 1, 49, 3, 0)
    g = b.get_links()[0]
    assert np.abs(g @ np.conj(np.swapaxes(g, -1, -2)) - np.eye(3)).max() <= 5e-14


@pytest.mark.parametrize("N", [2, 3, 4])
@pytest.mark.parametrize("kind", KINDS)
def test_sun_stage_matches_the_oracle_at_the_edges_of_the_range(tgf, N, kind):
    u = edge_field(kind, N=N)
    b = tgf.SunBatch(N, [L], any_extents=True)
    b.set_links([u])
    scale = max(1.0, np.abs(u).max()) ** 4
    h = 0.02 / scale
    b.stage(1, h)
    ref = np.matmul(O.expm(0.25 * h * O.force(u, TW)), u)
    assert np.abs(b.get_links()[0] - ref).max() <= 100 * U * np.abs(u).max()


@pytest.mark.parametrize("N", [2, 3, 4])
@pytest.mark.parametrize("kind", KINDS)
def test_sun_measure_matches_the_oracle_at_the_edges_of_the_range(tgf, N, kind):
    u = edge_field(kind, N=N)
    b = tgf.SunBatch(N, [L], any_extents=True)
    b.set_links([u])
    g = b.measure()[0]
    o = O.measure(u, TW)
    m = np.abs(u).max()
    big = 9.0 * (1.0 if kind in ("su", "unit", "tiny", "just_in") else m ** 4 * N * N)
    V = u[..., 0, 0, 0].size
    assert abs(g[4] - o["S"]) <= 100 * U * 6 * V * big
    assert abs(g[1] - o["E"]) <= 100 * U * 6 * N * N * big * big
    assert abs(g[2] - o["Q"]) <= 100 * U * V * N * N * big * big
