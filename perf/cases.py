"""The work that users of this framework have it do, as cases that can be timed one by one.

A case is a dict of plain values.  ``prepare`` makes what a program holds before the call (seeded
link fields in canonical FP64 layout on the GPU and the batch with its device buffers), ``run`` is
one pass through the public Python entry points, ``exact`` the same numbers from plain torch in
64 bits.  Kinds of work:

* ``flow``     pack the canonical field, flow every configuration with RK3 (eps = 0.01) recording
               E, Q, P, S, and unpack the flowed field: what a measurement program runs for each
               configuration of an ensemble
* ``measure``  one measurement of a batch at a given flow time
* ``slices``   the time-slice charge q(x0, t) of a batch along a long direction
* ``mc``       hybrid Monte Carlo sweeps (1 heat-bath + n_or over-relaxation sweeps) of a set of
               chains, and their links unpacked: ensemble generation
* ``sun``      RK3 steps and a measurement of SU(N) configurations, N = 2, 3, 4

Results of the FP32 forms are returned as float32 (that is the precision they are computed in; the
library widens records and unpacked links to double), those of FP64 as float64.
"""
import math

import numpy as np
import torch

from paper_2107_03747_gb300 import binding as tgf

EPS = 0.01
DEV = "cuda"


# ---------------------------------------------------------------------------------------------
# the cases
# ---------------------------------------------------------------------------------------------

def flow(name, l, n, prec, steps, every=1, reunit=0, tile=0, amp=0.3, k=1):
    """``steps`` RK3 steps (a fraction: a last short step) of ``n`` boxes l x l x 3l x 3l; ``l`` as a
    text "4,6,8" is a mixed batch, whose members flow steps * (l / largest l)^2 steps each (the flow
    time of the scheme goes with l^2)."""
    return {"name": name, "kind": "flow", "l": str(l), "n": n, "prec": prec, "steps": float(steps), "every": every,
            "reunit": reunit, "tile": tile, "amp": amp, "k": k}


def listed():
    return [
        # the smallest lattice of the scheme, alone, over its whole flow to t = c^2 l^2 / 8 = 0.18:
        # a new program's first run, and a single configuration looked at by hand (launch latency)
        flow("flow_fp32_l4", 4, 1, "fp32", 18, reunit=20),
        # the same in FP64, a few steps: the check that an installation works
        flow("flow_fp64_l4", 4, 1, "fp64", 3),
        # one measurement round of an ensemble: chains of the smallest box flowed to the coupling's
        # own scale sqrt(8t) = 0.3 * 12, t = 1.62, with the observables wanted at the end only
        flow("flow_fp32_ensemble_l4x32", 4, 32, "fp32", 162, every=1 << 20, amp=0.2),
        # an ensemble of mixed box sizes in one batch, each to its own flow time (a step-scaling run)
        flow("flow_fp32_mixed_l4_6_8", "4,6,8", 96, "fp32", 8, reunit=20, amp=0.4),
        # the large production batch, 4 x 16x16x48x48, with the launch setting that the tuner picks there
        flow("flow_fp32_l16x4", 16, 4, "fp32", 6, reunit=20, tile=3, amp=0.4),
        # the memory-saving 12-real form on the middle box, observables every second step
        flow("flow_fp32_r12_l12x2", 12, 2, "fp32_r12", 8, every=2, reunit=20, amp=0.5),
        # double precision flow: the form that accuracy statements are made against
        flow("flow_fp64_l8x4", 8, 4, "fp64", 4),
        # one measurement in double precision of boxes whose site count is no multiple of a warp (7x7x21x21)
        {"name": "measure_fp64_l7x4", "kind": "measure", "l": "7", "n": 4, "prec": "fp64", "traceless": False, "amp": 0.3, "k": 1},
        # the time-slice charge density along x3 at some flow time, in the working precision of the flow
        {"name": "slices_fp32_l12x2", "kind": "slices", "l": "12", "n": 2, "prec": "fp32", "dir": 3, "amp": 0.3, "k": 1},
        # ensemble generation: one hybrid sweep (1 heat-bath + L~ = 12 over-relaxation) of 256 chains at 18 b = 20
        {"name": "mc_l4x256", "kind": "mc", "l": 4, "n": 256, "beta": 20.0, "hybrid": 1, "n_or": 12, "amp": 0.2, "k": 1},
        # the other gauge groups of the scheme, one RK3 step and a measurement
        {"name": "sun2_l8x8", "kind": "sun", "N": 2, "l": 8, "n": 8, "steps": 2, "amp": 0.3, "k": 1},
        {"name": "sun4_l6x4", "kind": "sun", "N": 4, "l": 6, "n": 4, "steps": 1, "amp": 0.3, "k": 1},
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    """One more case of the same ranges: box sizes l = 3..16 (odd ones too), site counts spread over
    their logarithm, every precision, interval and group, at most the work of the largest listed one."""
    kind = rng.choice(["flow", "flow", "flow", "flow", "measure", "slices", "mc", "sun"])
    amp = round(rng.uniform(0.15, 0.5), 3)
    k = rng.choice([1, 1, 2])

    def boxes(lo, hi, N=3, even=False, lmax=16):
        total = _log(rng, lo, hi)
        top = max(3, min(lmax, int((total / (N * N)) ** 0.25)))
        ls = [l for l in range(2 if N > 2 else 4, top + 1) if l >= 3 and not (even and l % 2)] or [4]
        l = rng.choice(ls)
        return l, max(1, min(256, round(total / (N * N * l ** 4))))

    if kind == "flow":
        prec = rng.choice(["fp32", "fp32", "fp32_r12", "fp64"])
        fp64 = prec == "fp64"
        l, n = boxes(729, 1.5e5 if fp64 else 2.3e6)
        sites = 9 * l ** 4 * n
        most = max(1.0, min(60.0, (6e5 if fp64 else 1.2e7) / sites))
        steps = round(_log(rng, 1.0, most + 0.001), 1)
        every = rng.choice([1, 1, 2, 5, 1 << 20])
        reunit = 0 if fp64 else rng.choice([0, 20])
        tile = 0 if fp64 else rng.choice([0, 0, 3, 4])
        if rng.random() < 0.2 and n >= 3:
            l = "%d,%d,%d" % (max(3, l - 2), max(3, l - 1), l)
        c = flow("", l, n, prec, steps, every, reunit, tile, amp, k)
        del c["name"]
        return c
    if kind in ("measure", "slices"):
        prec = rng.choice(["fp32", "fp32_r12", "fp64"])
        l, n = boxes(729, 4e5 if prec == "fp64" else 1.2e6)
        c = {"kind": kind, "l": str(l), "n": n, "prec": prec, "amp": amp, "k": k}
        if kind == "measure":
            c["traceless"] = rng.random() < 0.3
        else:
            c["dir"] = rng.choice([2, 3])
        return c
    if kind == "mc":
        l, n = boxes(2304, 5.9e5, even=True, lmax=8)
        n_or = rng.randint(2, 12)
        return {"kind": "mc", "l": l, "n": n, "beta": round(rng.uniform(8.0, 40.0), 2), "hybrid": 1, "n_or": n_or,
                "amp": round(rng.uniform(0.15, 0.3), 3), "k": k}
    N = rng.choice([2, 3, 4])
    l, n = boxes(1000, {2: 6e5, 3: 2e5, 4: 8e4}[N], N=N, lmax=10)
    return {"kind": "sun", "N": N, "l": l, "n": n, "steps": rng.randint(1, 2), "amp": amp, "k": k}


# ---------------------------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------------------------

def _members(c):
    """Box extents of every configuration and its number of steps."""
    ls = [int(x) for x in str(c["l"]).split(",")]
    N = c.get("N", 3)
    out = []
    for i in range(c["n"]):
        l = ls[i % len(ls)]
        st = c.get("steps", 0)
        if len(ls) > 1:
            st = round(st * (l / max(ls)) ** 2, 1)
        out.append(((l, l, N * l, N * l), st))
    return out


def _mm(a, b):
    """Batched product of small matrices, summed over the inner index in order."""
    r = a[..., :, 0:1] * b[..., 0:1, :]
    for q in range(1, a.shape[-1]):
        r = r + a[..., :, q:q + 1] * b[..., q:q + 1, :]
    return r


def _dag(a):
    return a.mH


def _exp(x, deg):
    """Taylor polynomial of degree ``deg`` by Horner's scheme."""
    eye = torch.eye(x.shape[-1], dtype=x.dtype, device=x.device)
    r = eye + x / deg
    for j in range(deg - 1, 0, -1):
        r = eye + _mm(x, r) / j
    return r


def _generators(N):
    g = []
    for j in range(N):
        for q in range(j + 1, N):
            a = np.zeros((N, N), complex)
            a[j, q] = a[q, j] = 0.5
            b = np.zeros((N, N), complex)
            b[j, q], b[q, j] = -0.5j, 0.5j
            g += [a, b]
    for m in range(1, N):
        d = np.zeros((N, N), complex)
        d[np.arange(m), np.arange(m)] = 1
        d[m, m] = -m
        g.append(d / math.sqrt(2.0 * m * (m + 1)))
    return torch.tensor(np.array(g), dtype=torch.complex128, device=DEV)


def _random_links(L, gen, amp, N, cold=False, k=1):
    """Links exp(i amp omega_a T_a), omega ~ N(0, 1), as [x3, x2, x1, x0, mu, N, N]; ``cold`` puts the
    fluctuations on the field of zero twisted action (clock and shift matrices at the corner rows),
    the neighbourhood in which Monte Carlo chains live at weak coupling."""
    L0, L1, L2, L3 = L
    V = L0 * L1 * L2 * L3
    T = _generators(N)
    om = torch.randn(V * 4, N * N - 1, dtype=torch.float64, device=DEV, generator=gen)
    x = (1j * amp) * torch.einsum("na,aij->nij", om.to(torch.complex128), T)
    u = _exp(x, 24)
    # unitary to the last bits: Gram-Schmidt by rows
    rows = []
    for i in range(N):
        r = u[:, i]
        for p in rows:
            r = r - (p.conj() * r).sum(-1, keepdim=True) * p
        rows.append(r / r.abs().square().sum(-1, keepdim=True).sqrt())
    u = torch.stack(rows, 1).reshape(L3, L2, L1, L0, 4, N, N)
    if cold:
        w = np.exp(2j * math.pi * k / 3)
        g1 = torch.tensor(np.diag([1, w, w * w]), dtype=torch.complex128, device=DEV)
        g2 = torch.zeros(3, 3, dtype=torch.complex128, device=DEV)
        for j in range(3):
            g2[(j + 1) % 3, j] = 1
        u[:, :, :, 0, 0] = _mm(u[:, :, :, 0, 0], g1)
        u[:, :, 0, :, 1] = _mm(u[:, :, 0, :, 1], g2)
    return u.contiguous()


def _fields(c, seed):
    gen = torch.Generator(DEV).manual_seed(seed)
    return [_random_links(L, gen, c["amp"], c.get("N", 3), cold=c["kind"] == "mc", k=c["k"]) for L, _ in _members(c)]


def _flat(fields):
    return torch.cat([torch.view_as_real(f).reshape(-1) for f in fields])


def prepare(case, seed):
    c = case
    mem = _members(c)
    Ls = [L for L, _ in mem]
    tw = [(c["k"], 0, 0, 0, 0, 0)] * len(Ls)
    canon = _flat(_fields(c, seed))
    if c["kind"] == "sun":
        b = tgf.SunBatch(c["N"], Ls, tw)
        return {"case": c, "batch": b, "canon": canon, "out": torch.empty_like(canon)}
    b = tgf.FlowBatch(Ls, c.get("prec", "fp64"), tw)
    s = {"case": c, "batch": b, "canon": canon, "out": torch.empty_like(canon)}
    if c["kind"] == "flow":
        s["t_end"] = [st * EPS for _, st in mem]
        cap = max(tgf.tgf_flow_records(EPS, t, c["every"]) for t in s["t_end"])
        s["obs"] = torch.zeros(len(Ls) * cap * 5, dtype=torch.float64, device=DEV)
    elif c["kind"] == "measure":
        s["obs"] = torch.zeros(len(Ls) * 5, dtype=torch.float64, device=DEV)
        b.set_links_device(canon)
    elif c["kind"] == "slices":
        T = max(L[c["dir"]] for L in Ls)
        s["T"] = T
        s["q"] = torch.zeros(len(Ls) * T, dtype=torch.float64, device=DEV)
        b.set_links_device(canon)
    return s


# ---------------------------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------------------------

def run(state):
    c, b = state["case"], state["batch"]
    kind = c["kind"]
    if kind == "flow":
        b.set_links_device(state["canon"])
        obs, _ = b.flow(EPS, state["t_end"], measure_every=c["every"], reunit_every=c["reunit"], flags=c["tile"] << 13,
                        obs=state["obs"])
        tgf.tgf_unpack(b.prec, b.lat, b.links, state["out"])
        if c["prec"] == "fp64":
            return {"records": obs, "links": state["out"]}
        return {"records": obs.float(), "links": state["out"].float()}
    if kind == "measure":
        tgf.tgf_measure(b.prec, b.lat, b.links, b.scratch, state["obs"], 1, 0, 0.1,
                        tgf.TGF_CLOVER_TRACELESS if c["traceless"] else 0)
        return state["obs"] if c["prec"] == "fp64" else state["obs"].float()
    if kind == "slices":
        tgf.tgf_measure_slices(b.prec, b.lat, b.links, b.scratch, c["dir"], state["q"], state["T"])
        return state["q"] if c["prec"] == "fp64" else state["q"].float()
    if kind == "mc":
        b.set_links_device(state["canon"])
        tgf.tgf_mc_sweeps(b.prec, b.lat, b.links, c["beta"], c["hybrid"], c["n_or"], 2107, 50)
        tgf.tgf_unpack(b.prec, b.lat, b.links, state["out"])
        return state["out"]
    # fields that stay on the device go in and out by the C entry points (SunBatch's own set_links and
    # get_links take and give host arrays)
    N, lat, st = c["N"], b.lat, torch.cuda.current_stream().cuda_stream
    _ok(tgf._lib.tgf_sun_pack(N, lat, len(lat), state["canon"].data_ptr(), b.links.data_ptr(), st))
    for _ in range(c["steps"]):
        b.step(EPS)
    m = b.measure(c["steps"] * EPS)
    _ok(tgf._lib.tgf_sun_unpack(N, lat, len(lat), b.links.data_ptr(), state["out"].data_ptr(), st))
    return {"records": m, "links": state["out"]}


def _ok(status):
    if status != tgf.TGF_OK:
        raise RuntimeError(tgf.status_string(status))


def work(case):
    """Bytes: the canonical field in and out once (and the few records); a measurement reads its links
    in their stored form.  Flops: 3x3 complex products at 198 (NxN: N^2 (8N - 2)), 64 of them and
    about 760 scalar operations per site and RK3 stage, 15.1 kflop per measured site."""
    c = case
    N = c.get("N", 3)
    prod = N * N * (8 * N - 2)
    stage, meas = 64 * prod + 760 * (N / 3) ** 2, 72 * prod + 850 * (N / 3) ** 2
    byt = fl = 0.0
    for L, st in _members(c):
        V = L[0] * L[1] * L[2] * L[3]
        field = V * 4 * N * N * 16
        if c["kind"] in ("measure", "slices"):
            byt += V * 4 * {"fp64": 144, "fp32": 72, "fp32_r12": 48}[c["prec"]]
            fl += V * meas
        elif c["kind"] == "mc":
            # 13 products and the three SU(2) subgroup updates (about 600 flops) of every link and sweep
            byt += 2 * field
            fl += V * 4 * c["hybrid"] * (1 + c["n_or"]) * (13 * prod + 600)
        else:
            ns = math.ceil(st - 1e-9)
            nm = -(-ns // c.get("every", 1 << 20)) + 1 if c["kind"] == "flow" else 1
            out = field if c.get("prec", "fp64") == "fp64" else field / 2
            byt += field + out + nm * 40
            fl += V * (3 * ns * stage + nm * meas)
    return {"bytes": byt, "flops": fl}


# ---------------------------------------------------------------------------------------------
# the same in plain torch, 64 bits
# ---------------------------------------------------------------------------------------------

def _sh(a, d, step):
    """The field at n + step d (x_d sits on axis 3 - d of [.., x3, x2, x1, x0] counted from the front,
    after one leading batch axis)."""
    return torch.roll(a, -step, dims=4 - d)


def _phase(W, mu, nu, k, N):
    """Z_{mu nu}(n): exp(2 pi i k / N) on plaquettes with corner x_0 = x_1 = 0 of the plane (0, 1)."""
    if {mu, nu} != {0, 1} or k % N == 0:
        return None
    z = torch.ones(W.shape[1:5], dtype=torch.complex128, device=W.device)
    z[:, :, 0, 0] = np.exp(2j * math.pi * (k if mu == 0 else -k) / N)
    return z[None, ..., None, None]


def _staples(W, mu, k):
    N = W.shape[-1]
    U = [W[..., d, :, :] for d in range(4)]
    sig = torch.zeros_like(U[mu])
    for nu in range(4):
        if nu == mu:
            continue
        f = _mm(_mm(_sh(U[nu], mu, 1), _dag(_sh(U[mu], nu, 1))), _dag(U[nu]))
        b = _mm(_dag(_mm(U[mu], _sh(U[nu], mu, 1))), U[nu])
        z = _phase(W, mu, nu, k, N)
        if z is not None:
            f, b = z.conj() * f, z * b
        sig = sig + f + _sh(b, nu, -1)
    return sig


def _force(W, k):
    N = W.shape[-1]
    out = torch.empty_like(W)
    for mu in range(4):
        m = _mm(W[..., mu, :, :], _staples(W, mu, k))
        a = (m - _dag(m)) / 2
        tr = torch.diagonal(a, dim1=-2, dim2=-1).sum(-1) / N
        out[..., mu, :, :] = -(a - tr[..., None, None] * torch.eye(N, dtype=a.dtype, device=a.device))
    return out


def _step(W, eps, k):
    x = 0.25 * eps * _force(W, k)
    W = W + _mm(_exp(x, 13) - torch.eye(W.shape[-1], device=W.device), W)
    x = (8 / 9) * eps * _force(W, k) - (17 / 9) * x
    W = W + _mm(_exp(x, 13) - torch.eye(W.shape[-1], device=W.device), W)
    x = 0.75 * eps * _force(W, k) - x
    return W + _mm(_exp(x, 13) - torch.eye(W.shape[-1], device=W.device), W)


def _clover(W, k, traceless):
    N = W.shape[-1]
    U = [W[..., d, :, :] for d in range(4)]
    G, s = {}, 0.0
    for mu in range(4):
        for nu in range(mu + 1, 4):
            P = _mm(_mm(U[mu], _sh(U[nu], mu, 1)), _dag(_mm(U[nu], _sh(U[mu], nu, 1))))
            z = _phase(W, mu, nu, k, N)
            if z is not None:
                P = z.conj() * P
            s = s + N - torch.diagonal(P, dim1=-2, dim2=-1).sum(-1).real
            # the plaquettes with corners n, n - nu, n - mu, n - mu - nu, each carried to n
            H = P + _sh(_mm(_mm(_dag(U[nu]), P), U[nu]), nu, -1)
            C = H + _sh(_mm(_mm(_dag(U[mu]), H), U[mu]), mu, -1)
            g = -0.125j * (C - _dag(C))
            if traceless:
                g = g - torch.diagonal(g, dim1=-2, dim2=-1).sum(-1)[..., None, None] / N * torch.eye(N, dtype=g.dtype, device=g.device)
            G[mu, nu] = g

    def tr(a, b):
        return (a * b.transpose(-1, -2)).sum((-2, -1)).real

    e = sum(tr(g, g) for g in G.values())
    q = (tr(G[0, 1], G[2, 3]) - tr(G[0, 2], G[1, 3]) + tr(G[0, 3], G[1, 2])) / (4 * math.pi ** 2)
    return e, q, s


def _record(W, t, k, traceless=False):
    N = W.shape[-1]
    V = W[0, ..., 0, 0, 0].numel()
    e, q, s = (x.flatten(1).sum(1) for x in _clover(W, k, traceless))
    return torch.stack([torch.full_like(e, t), e / V, q, 1 - s / (6 * N * V), s], -1)


def _exact_flow(c, fields):
    mem = _members(c)
    cap = max(-(-math.ceil(st - 1e-9) // c["every"]) + 1 for _, st in mem)
    rec = torch.zeros(len(mem), cap, 5, dtype=torch.float64, device=DEV)
    links = [None] * len(mem)
    groups = {}
    for i, m in enumerate(mem):
        groups.setdefault(m, []).append(i)
    for (L, st), idx in groups.items():
        per = max(1, int(6e5 // (L[0] * L[1] * L[2] * L[3])))
        for lo in range(0, len(idx), per):
            part = idx[lo:lo + per]
            W = torch.stack([fields[i] for i in part])
            n, r, t = math.ceil(st - 1e-9), 0, 0.0
            for j in range(n):
                if j % c["every"] == 0:
                    rec[part, r] = _record(W, j * EPS, c["k"])
                    r += 1
                W = _step(W, min(EPS, (st - j) * EPS), c["k"])
            rec[part, r] = _record(W, st * EPS, c["k"])
            for q, i in enumerate(part):
                links[i] = W[q]
    out = {"records": rec, "links": _flat(links)}
    return out if c["prec"] == "fp64" else {k: v.float() for k, v in out.items()}


def _srl(z, n):
    return (z >> n) & ((1 << (64 - n)) - 1)


def _i64(v):
    return v - (1 << 64) if v >= 1 << 63 else v


GOLDEN = 0x9E3779B97F4A7C15


def _hash(key, counter):
    """SplitMix64's output function of key + (counter + 1) * golden, on int64 tensors that wrap."""
    z = key + (counter + 1) * _i64(GOLDEN)
    z = (z ^ _srl(z, 30)) * _i64(0xBF58476D1CE4E5B9)
    z = (z ^ _srl(z, 27)) * _i64(0x94D049BB133111EB)
    return z ^ _srl(z, 31)


def _draw(key, counter):
    return (_srl(_hash(key, counter), 11).double() + 1.0) * 2.0 ** -53


def _qmul(a, b):
    a0, a1, a2, a3 = a
    b0, b1, b2, b3 = b
    return (a0 * b0 - (a1 * b1 + a2 * b2 + a3 * b3), a0 * b1 + b0 * a1 - (a2 * b3 - a3 * b2),
            a0 * b2 + b0 * a2 - (a3 * b1 - a1 * b3), a0 * b3 + b0 * a3 - (a1 * b2 - a2 * b1))


def _heat_x0(alpha, key, c0):
    """X0 ~ sqrt(1 - X0^2) exp(alpha X0) by rejection: Kennedy-Pendleton above alpha = 2, Creutz below."""
    x0 = torch.zeros_like(alpha)
    done = torch.zeros_like(alpha, dtype=torch.bool)
    e2a = torch.exp(-2.0 * alpha)
    for a in range(64):
        r1, r2, r3, r4 = (_draw(key, c0 + 4 * a + j) for j in range(4))
        cs = torch.cos(2 * math.pi * r2)
        lam2 = -(torch.log(r1) + cs * cs * torch.log(r3)) / (2 * alpha)
        kp = alpha > 2.0
        xc = torch.where(alpha < 1e-8, 2 * r1 - 1, 1 + torch.log(e2a + (1 - e2a) * r1) / alpha)
        ok = torch.where(kp, r4 * r4 <= 1 - lam2, r2 * r2 <= 1 - xc * xc) & ~done
        x0 = torch.where(ok, torch.where(kp, 1 - 2 * lam2, xc), x0)
        done |= ok
        if bool(done.all()):
            break
    return x0, done


def _exact_mc(c, fields):
    W = torch.stack(fields)
    n, L3, L2, L1, L0 = W.shape[:5]
    V = L0 * L1 * L2 * L3
    x = torch.meshgrid(*(torch.arange(v, device=DEV) for v in (L3, L2, L1, L0)), indexing="ij")
    par = ((x[0] + x[1] + x[2] + x[3]) % 2)[None].expand(n, -1, -1, -1, -1)
    site = (((x[0] * L2 + x[1]) * L1 + x[2]) * L0 + x[3])[None]
    key = _hash(torch.tensor(2107, device=DEV), torch.arange(n, device=DEV)).view(n, 1, 1, 1, 1)
    for h in range(c["hybrid"]):
        for o in range(-1, c["n_or"]):
            for mu in range(4):
                for p in range(2):
                    U = W[..., mu, :, :]
                    M = _mm(U, _staples(W, mu, c["k"]))
                    for g, (i, j) in enumerate(((0, 1), (0, 2), (1, 2))):
                        q = (0.5 * (M[..., i, i].real + M[..., j, j].real), 0.5 * (M[..., i, j].imag + M[..., j, i].imag),
                             0.5 * (M[..., i, j].real - M[..., j, i].real), 0.5 * (M[..., i, i].imag - M[..., j, j].imag))
                        kk = torch.sqrt(q[0] ** 2 + q[1] ** 2 + q[2] ** 2 + q[3] ** 2)
                        vc = (q[0] / kk, -q[1] / kk, -q[2] / kk, -q[3] / kk)
                        if o >= 0:
                            R = _qmul(vc, vc)
                        else:
                            c0 = ((((50 + h) * 4 + mu) * V + site) * 3 + g) * 260
                            x0, ok = _heat_x0(2 * c["beta"] * kk / 3, key, c0)
                            ct = 2 * _draw(key, c0 + 256) - 1
                            ph = 2 * math.pi * _draw(key, c0 + 257)
                            sn = torch.sqrt(torch.clamp(1 - ct * ct, min=0))
                            rr = torch.sqrt(torch.clamp(1 - x0 * x0, min=0))
                            X = (x0, rr * sn * torch.cos(ph), rr * sn * torch.sin(ph), rr * ct)
                            R = _qmul(X, vc)
                            R = tuple(torch.where(ok, r, torch.full_like(r, float(m == 0))) for m, r in enumerate(R))
                        r00, r01 = torch.complex(R[0], R[3])[..., None], torch.complex(R[2], R[1])[..., None]
                        r10, r11 = torch.complex(-R[2], R[1])[..., None], torch.complex(R[0], -R[3])[..., None]

                        def rot(m):
                            m = m.clone()
                            a, b = m[..., i, :].clone(), m[..., j, :].clone()
                            m[..., i, :], m[..., j, :] = r00 * a + r01 * b, r10 * a + r11 * b
                            return m

                        U, M = rot(U), rot(M)
                    W = W.clone()
                    W[..., mu, :, :] = torch.where((par == p)[..., None, None], U, W[..., mu, :, :])
    return _flat([W])


def exact(case, seed):
    c = case
    fields = _fields(c, seed)
    mem = _members(c)
    if c["kind"] == "flow":
        if sum(L[0] * L[1] * L[2] * L[3] * st for L, st in mem) > 1.6e7:
            return None  # minutes of plain torch; the smaller flows of the same form have their values
        return _exact_flow(c, fields)
    if c["kind"] == "measure":
        r = torch.cat([_record(f[None], 0.1, c["k"], c["traceless"]) for f in fields]).reshape(-1)
        return r if c["prec"] == "fp64" else r.float()
    if c["kind"] == "slices":
        ax = 3 - c["dir"]
        out = []
        for f in fields:
            q = _clover(f[None], c["k"], False)[1][0]
            out.append(q.sum([a for a in range(4) if a != ax]))
        q = torch.cat(out)
        return q if c["prec"] == "fp64" else q.float()
    if c["kind"] == "mc":
        return _exact_mc(c, fields)
    W = torch.stack(fields)
    for _ in range(c["steps"]):
        W = _step(W, EPS, c["k"])
    return {"records": _record(W, c["steps"] * EPS, c["k"]), "links": _flat([W])}
