"""Fields on which the fixed-point products of the double-precision kernels (csrc/fixed.cuh) must give way to FP64
arithmetic or widen their sums, against the oracle: links whose entries add up in phase, so that T = V B^+, the
staples, Omega and the traces come out far beyond those of unitary matrices, and weak fields, whose small entries FP64
holds to 53 bits.

Tolerances.  FP64 arithmetic carries about 6N + 6 roundings of U = 2^-53 along a link: 100 U of the size of the terms
covers them in the worst case; as random numbers of rms U / sqrt(3) each they add up to 2.8 U for N = 3, bar 4 U.
"""
import numpy as np
import pytest

from oracle import tgf_oracle as O
from paper_2107_03747_gb300 import inputs as I

pytestmark = pytest.mark.gpu

U = 2.0 ** -53
L = (4, 2, 6, 4)  # 192 sites
TW = I.default_twist(1)
FLAT = [[0] * 4 for _ in range(4)]


def in_phase(kind, N):
    J = np.ones((N, N))
    shape = (L[3], L[2], L[1], L[0], 4, N, N)
    x3, x2, x1, x0 = np.meshgrid(*(np.arange(L[d]) for d in (3, 2, 1, 0)), indexing="ij")
    x = (x0, x1, x2, x3)
    u = np.empty(shape, complex)
    if kind == "all":  # T = 2N
        u[...] = (1 + 1j) * J
    elif kind == "nine_tenths":  # T = 1.62 N
        u[...] = 0.9 * (1 + 1j) * J
    elif kind == "phases":  # T = 2N times a fourth root of 1
        ph = 1j ** np.random.default_rng(3).integers(0, 4, shape[:5])
        u[...] = ph[..., None, None] * (1 + 1j) * J
    elif kind == "below_six":  # T just inside 6 for N = 3
        u[...] = 0.9999 * (1 + 1j) * J
    elif kind == "omega":  # |T| < 2 and staple sums of 7.5 (1 +- i), but Im Tr Omega = 15 N^2
        a = np.sqrt(7.5 / (6 * N * N))
        u[..., 0, :, :] = (1 + 1j) * J
        for nu in (1, 2, 3):
            ph = np.exp(0.5j * np.pi * x0 * (-1.0) ** x[nu])
            u[..., nu, :, :] = a * ph[..., None, None] * J
    elif kind == "trace":  # staples of 1.9 (1 - i) in the planes of direction 0: Re Tr(U F) = 3.8 N^2
        u[...] = np.sqrt(1.9) / N * J
        u[..., 0, :, :] = (1 + 1j) * J
    return u


IN_PHASE = ["all", "nine_tenths", "phases", "below_six", "omega", "trace"]


def batch(tgf, N, tw=None):
    if N is None:
        return tgf.FlowBatch([L], "fp64", tw, any_extents=True)
    return tgf.SunBatch(N, [L], tw, any_extents=True)


@pytest.mark.parametrize("N", [None, 2, 3, 4])  # None: the SU(3) kernels
@pytest.mark.parametrize("kind", IN_PHASE)
def test_stage_of_links_in_phase(tgf, kind, N):
    n = N or 3
    u = in_phase(kind, n)
    b = batch(tgf, N)
    b.set_links([u])
    h = 0.02 / (6 * n ** 3 * np.abs(u).max() ** 4)  # X stays small whatever the force
    b.stage(1, h)
    ref = np.matmul(O.expm(0.25 * h * O.force(u, TW)), u)
    assert np.abs(b.get_links()[0] - ref).max() <= 100 * U * np.abs(u).max()


@pytest.mark.parametrize("N", [None, 2, 3, 4])
@pytest.mark.parametrize("kind", IN_PHASE)
def test_measure_of_links_in_phase(tgf, kind, N):
    n = N or 3
    u = in_phase(kind, n)
    b = batch(tgf, N)
    b.set_links([u])
    g = b.measure()[0].tolist()
    o = O.measure(u, TW)
    V = u[..., 0, 0, 0].size
    size = n ** 3 * np.abs(u).max() ** 4  # of a leaf's entry
    assert abs(g[4] - o["S"]) <= 100 * U * 6 * V * n * size
    assert abs(g[1] - o["E"]) <= 100 * U * 6 * n * n * size ** 2
    assert abs(g[2] - o["Q"]) <= 100 * U * V * n * n * size ** 2


@pytest.mark.parametrize("kind", IN_PHASE)
def test_measured_flow_step_of_links_in_phase(tgf, kind):
    """The clover halves of a measured stage are those of the measurement alone."""
    u = in_phase(kind, 3)
    b = batch(tgf, None)
    b.set_links([u])
    ref = b.measure()[0].tolist()
    obs, _ = b.flow(1e-6, 1e-6)
    got = obs.cpu().numpy()[0, 0]
    size = 27 * np.abs(u).max() ** 4
    V = u[..., 0, 0, 0].size
    assert abs(got[4] - ref[4]) <= 100 * U * 6 * V * 3 * size
    assert abs(got[1] - ref[1]) <= 100 * U * 54 * size ** 2


AMPS = [1e-2, 1e-3, 1e-4, 1e-6, 1e-8]


def weak_field(amp, N, kind="unit"):
    """Links near the unit matrix, or (kind "signed") near matrices of one entry +-1, +-i in each row and column."""
    u = I.random_links(L, 11, amp, N=N)
    if kind == "signed":
        rng = np.random.default_rng(2)
        g = np.zeros(u.shape[:4] + (N, N), complex)
        for at in np.ndindex(*u.shape[:4]):
            g[at][np.arange(N), rng.permutation(N)] = 1j ** rng.integers(0, 4, N)
        for mu in range(4):
            f = np.roll(g, -1, axis=3 - mu)
            u[..., mu, :, :] = g @ u[..., mu, :, :] @ np.conj(np.swapaxes(f, -1, -2))
    return u


def exp_m1(x):
    r = t = x
    for k in range(2, 30):
        t = np.matmul(t, x) / k
        r = r + t
    return r


@pytest.mark.parametrize("N", [None, 2, 3, 4])
@pytest.mark.parametrize("amp", AMPS)
@pytest.mark.parametrize("kind", ["unit", "signed"])
def test_weak_field_force_keeps_its_relative_precision(tgf, kind, amp, N):
    """One stage with eps/4 = 1: W' - W is of the size of the force, whose entries are compared one by one."""
    n = N or 3
    u = weak_field(amp, n, kind)
    b = batch(tgf, N, [(0,) * 6])
    b.set_links([u])
    b.stage(1, 4.0)
    got = b.get_links()[0].astype(np.clongdouble)
    w = u.astype(np.clongdouble)
    z = O.force(w, FLAT)
    assert z.dtype == np.clongdouble
    ref = w + np.matmul(exp_m1(z), w)
    d = got - ref
    small = np.stack([np.abs(w.real) < 0.5, np.abs(w.imag) < 0.5])  # the others round by 2^-54 of 1
    err = np.where(small, np.stack([d.real, d.imag]), 0) / np.abs(z).max((-1, -2))[..., None, None]
    rms = float(np.sqrt((err ** 2).sum() / small.sum()))
    assert rms <= 4 * U


@pytest.mark.parametrize("N", [None, 2, 3, 4])
@pytest.mark.parametrize("amp", AMPS)
def test_weak_field_observables_keep_their_relative_precision(tgf, amp, N):
    n = N or 3
    u = weak_field(amp, n)
    b = batch(tgf, N, [(0,) * 6])
    b.set_links([u])
    g = b.measure()[0].tolist()
    o = O.measure(u, FLAT)
    V = u[..., 0, 0, 0].size
    assert abs(g[1] / o["E"] - 1) <= 100 * U
    assert abs(g[2] - o["Q"]) <= 100 * U * V * o["E"]
    assert abs(g[4] - o["S"]) <= 100 * U * 6 * V * n


def test_weak_and_strong_links_in_one_warp(tgf):
    """Sites with strong links among weak ones: each link keeps the precision of its own force, and a measured flow
    step records what the measurement alone does, to the bit."""
    u = weak_field(1e-5, 3)
    strong = I.random_links(L, 12, 0.5)
    hit = np.random.default_rng(1).random(u.shape[:4]) < 0.02
    u[hit] = strong[hit]
    b = batch(tgf, None, [(0,) * 6])
    b.set_links([u])
    ref = b.measure()[0].tolist()
    obs, _ = b.flow(0.01, 0.01)
    assert obs.cpu().numpy()[0, 0, 1:].tolist() == ref[1:]
    b.set_links([u])
    b.stage(1, 4.0)
    w = u.astype(np.clongdouble)
    z = O.force(w, FLAT)
    far = np.abs(z).max((-1, -2)) < 1e-3  # links with no strong one in their staples
    assert far.sum() > 100
    d = (b.get_links()[0].astype(np.clongdouble) - (w + np.matmul(exp_m1(z), w)))[far]
    off = ~np.eye(3, dtype=bool)
    err = (d / np.abs(z[far]).max((-1, -2))[..., None, None])[..., off]
    assert float(np.sqrt((np.abs(err) ** 2).mean() / 2)) <= 4 * U


def test_weak_sites_do_not_depend_on_the_launch(tgf):
    """A launch of 26 configurations (156 blocks, one thread per link) and of one (6 blocks, three threads per link)
    take the same sites through FP64, to the bit."""
    u = weak_field(0.03, 3)
    strong = I.random_links(L, 12, 0.5)
    hit = np.random.default_rng(1).random(u.shape[:4]) < 0.1
    u[hit] = strong[hit]
    one = batch(tgf, None)
    one.set_links([u])
    rec = one.measure()[0].tolist()
    one.stage(1, 0.01)
    many = tgf.FlowBatch([L] * 26, "fp64", any_extents=True)
    many.set_links([u] * 26)
    assert all(r.tolist() == rec for r in many.measure())
    many.stage(1, 0.01)
    ref = one.get_links()[0]
    assert all(np.array_equal(g, ref) for g in many.get_links())


def test_su4_exponential_keeps_small_entries(tgf):
    """Links of large diagonal phases and off-diagonal entries of 1e-6, one stage with eps/4 = 1e-4: the force is within
    4 U of its size (below 6) and enters with 1e-4, 2.7e-19 = 2^-61.7 off the diagonal; exp(X) - 1 is scaled to X, so that it adds no
    2^-58 of its own.  Bar 2^-60."""
    rng = np.random.default_rng(4)
    ph = rng.uniform(-1, 1, (L[3], L[2], L[1], L[0], 4, 4))
    ph -= ph.mean(-1, keepdims=True)
    u = np.exp(1j * ph)[..., None] * I.random_links(L, 5, 1e-6, N=4)
    b = batch(tgf, 4, [(0,) * 6])
    b.set_links([u])
    b.stage(1, 4e-4)
    w = u.astype(np.clongdouble)
    z = O.force(w, FLAT)
    assert np.abs(z).max() < 6
    d = b.get_links()[0].astype(np.clongdouble) - (w + np.matmul(exp_m1(1e-4 * z), w))
    off = d[..., ~np.eye(4, dtype=bool)]
    assert float(np.sqrt((np.abs(off) ** 2).mean() / 2)) <= 2.0 ** -60
