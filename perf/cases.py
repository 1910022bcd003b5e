"""Workloads of the library as its users run them, for timing and for comparing two
versions of it: H.v on one sector, Lanczos chains of one sector, whole FTLM jobs,
batches of clusters, general-spin sectors and the request loop.

A case is a dict of plain values.  listed() gives the fixed ones, draw(rng) another
of the same ranges, prepare(case, seed) the state a program holds before the call
(sector tables, workspaces, plans, inputs), run(state) one pass through the public
entry points, work(case) the bytes and operations of a pass, and exact(case, seed)
the outputs in 64 bits, computed with plain torch.
"""
import math

import numpy as np
import torch

from paper_2605_26261_gb300 import ftlm, inputs, serve

DTYPES = {"f32": torch.float32, "f64": torch.float64}
BYTES = {"f32": 4, "f64": 8}


def listed():
    return [
        # The smallest call: H.v on the N = 16 ring, one double vector.
        dict(name="hv f64 ring16", kind="hv", graph="ring", N=16, two_sz=0, B=1, dtype="f64"),
        # A block H.v of a mid-sized random cluster (lookup-table rank).
        dict(name="hv f32 block8 random22", kind="hv", graph="random", N=22, two_sz=0, B=8, dtype="f32"),
        # Double blocks on an odd cluster off the largest sector (combinatorial rank).
        dict(name="hv f64 block4 random23", kind="hv", graph="random", N=23, two_sz=3, B=4, dtype="f64"),
        # A whole small job in double: every sector of the N = 16 ring, R = 20, M = 100.
        dict(name="job f64 ring16", kind="job", graph="ring", N=16, R=20, M=100, dist="gauss", dtype="f64", h=0.0),
        # One sector of a small ladder: the launch-bound end of the Lanczos path.
        dict(name="lanczos f32 ladder18", kind="lanczos", graph="ladder", N=18, two_sz=0, R=8, M=100, dist="gauss",
             dtype="f32"),
        # The S^z = 0 sector of the 4 x 6 J1-J2 lattice (2.7 M rows), float vectors.
        dict(name="lanczos f32 j1j2", kind="lanczos", graph="j1j2", N=24, two_sz=0, R=8, M=100, dist="rademacher",
             dtype="f32"),
        # The same sector with double vectors (the precision comparison's other leg).
        dict(name="lanczos f64 j1j2", kind="lanczos", graph="j1j2", N=24, two_sz=0, R=4, M=20, dist="rademacher",
             dtype="f64"),
        # The icosidodecahedron's S^z = 0 sector (155 M rows), 8 chains: the benchmark's
        # sector and block with fewer steps.
        dict(name="lanczos f32 icosidodecahedron", kind="lanczos", graph="icosidodecahedron", N=30, two_sz=0, R=8,
             M=16, dist="rademacher", dtype="f32"),
        # Spin-2 icosahedron, S^z = 0 (19.6 M rows): general spin, one large sector.
        dict(name="spin2 f32 icosahedron", kind="spin", N=12, two_s=4, two_sz=0, R=8, M=20, dtype="f32"),
        # Spin-1 icosahedron, every sector in one batch (13 sectors, 24 chains each).
        dict(name="spin1 f32 batch", kind="batch", graph="icosahedron", sizes="12", two_s=2, R=24, M=100, dtype="f32"),
        # A few random clusters of the many-cluster workload, every sector in one batch.
        dict(name="clusters f32 batch", kind="batch", graph="random", sizes="18,20,22,20", two_s=1, R=16, M=100,
             dtype="f32"),
        # Requests (rings and ladders with a field) through the request loop.
        dict(name="serving f32", kind="serving", sizes="16,22,18,20,24,20", R=8, M=80, dtype="f32"),
    ]


def _pick(rng, lo, hi):
    """A whole number of [lo, hi], spread over its logarithm."""
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    """Another case: every kind, rank mode, width and type of the listed ones, over
    sector sizes from about 10^3 rows to a few 10^6 (listed: 10^4 to 1.6 10^8)."""
    kind = rng.choice(["hv", "hv", "lanczos", "lanczos", "lanczos", "spin", "job", "batch"])
    dtype = rng.choice(["f32", "f64"])
    dist = rng.choice(["gauss", "rademacher"])
    if kind == "hv":
        N = rng.randint(13, 25)
        tz = N % 2 + 2 * rng.randint(0, 2)
        return dict(kind="hv", graph=rng.choice(["ring", "random"]), N=N, two_sz=rng.choice([-1, 1]) * tz,
                    B=rng.choice([1, 4, 8, 16]), dtype=dtype)
    if kind == "lanczos":
        N = rng.randint(16, 24)
        if dtype == "f64":  # few steps: later ones depend on the last bit
            M, R = rng.randint(6, 20), _pick(rng, 1, 9)
        else:
            M, R = rng.randint(20, 110), _pick(rng, 1, 17)
        if N >= 22:
            M, R = min(M, 40), min(R, 9)
        return dict(kind="lanczos", graph=rng.choice(["ring", "random"]), N=N, two_sz=N % 2 + 2 * rng.randint(0, 1),
                    R=R, M=M, dist=dist, dtype=dtype)
    if kind == "spin":
        two_s = rng.choice([2, 3, 4])
        N = rng.randint(8, {2: 12, 3: 11, 4: 9}[two_s])
        return dict(kind="spin", N=N, two_s=two_s, two_sz=(N * two_s) % 2 + 2 * rng.randint(0, 1), R=_pick(rng, 1, 17),
                    M=rng.randint(8, 20), dtype=dtype)
    if kind == "job":
        return dict(kind="job", graph=rng.choice(["ring", "random"]), N=rng.randint(10, 16), R=_pick(rng, 2, 21),
                    M=_pick(rng, 20, 110), dist=dist, dtype=dtype, h=rng.choice([0.0, round(rng.uniform(0.1, 2.0), 3)]))
    sizes = ",".join(str(rng.randint(14, 19)) for _ in range(rng.randint(2, 5)))
    return dict(kind="batch", graph="random", sizes=sizes, two_s=1, R=_pick(rng, 2, 17), M=_pick(rng, 20, 110),
                dtype="f32")


# ------------------------------------------------------------------ inputs
def _bonds(graph, N, seed):
    if graph == "ring":
        return inputs.ring(N)
    if graph == "ladder":
        return inputs.ladder(N, J_rung=0.6, J_leg=1.0)
    if graph == "j1j2":
        return inputs.square_j1j2()
    if graph == "icosidodecahedron":
        return inputs.icosidodecahedron()
    if graph == "icosahedron":
        return inputs.icosahedron()
    return inputs.random_graph(N, seed=100_003 + seed)


def _spin_bonds(N):
    return inputs.icosahedron() if N == 12 else inputs.ring(N)


def _dist(case):
    return {"gauss": ftlm.GAUSS, "rademacher": ftlm.RADEMACHER}[case.get("dist", "rademacher")]


def _clusters(case, seed):
    return [(int(n), _bonds(case["graph"], int(n), 7 * seed + c)) for c, n in enumerate(case["sizes"].split(","))]


def _requests(case, seed):
    """Rings and two-leg ladders with couplings U[0.2, 1.5] and a field U[0, 2]."""
    rng = np.random.default_rng(seed)
    out = []
    for k, n in enumerate(case["sizes"].split(",")):
        n = int(n)
        bonds = (inputs.ring(n, J=float(rng.uniform(0.2, 1.5))) if k % 2 == 0 else
                 inputs.ladder(n, J_rung=float(rng.uniform(0.2, 1.5)), J_leg=float(rng.uniform(0.2, 1.5))))
        out.append(dict(N=n, bonds=bonds, h=float(rng.uniform(0.0, 2.0)), seed=1000 * seed + k))
    return out


def _vector(case, seed):
    D = math.comb(case["N"], (case["N"] + case["two_sz"]) // 2)
    g = torch.Generator(device="cuda").manual_seed(seed)
    shape = (D,) if case["B"] == 1 else (D, case["B"])
    x = torch.randn(shape, generator=g, device="cuda", dtype=torch.float64)
    return x.to(DTYPES[case["dtype"]])


def prepare(case, seed):
    st = dict(case=case, seed=seed)
    dev = torch.device("cuda", torch.cuda.current_device())
    kind, dt = case["kind"], DTYPES[case["dtype"]]
    if kind == "hv":
        st["basis"] = ftlm.Basis(case["N"], case["two_sz"], _bonds(case["graph"], case["N"], seed))
        st["x"] = _vector(case, seed)
        st["y"] = torch.empty_like(st["x"])
    elif kind in ("lanczos", "spin"):
        if kind == "spin":
            b = ftlm.Basis(case["N"], case["two_sz"], _spin_bonds(case["N"]), two_s=case["two_s"])
        else:
            b = ftlm.Basis(case["N"], case["two_sz"], _bonds(case["graph"], case["N"], seed))
        nbytes = ftlm.ftlm_lanczos_workspace_bytes(b.handle, case["R"], case["M"], dt)
        st["basis"], st["work"] = b, torch.empty((nbytes + 255) // 256 * 256, dtype=torch.uint8, device=dev)
    elif kind == "job":
        st["bonds"] = _bonds(case["graph"], case["N"], seed)
        st["T"] = torch.as_tensor(inputs.log_t_grid(200), device=dev)
    elif kind == "batch":
        st["T"] = torch.as_tensor(inputs.log_t_grid(200), device=dev)
        st["bases"], entries, st["span"] = [], [], []
        for c, (N, bonds) in enumerate(_clusters(case, seed)):
            bs = ftlm.Basis.sectors(N, ftlm.computed_two_sz(N, case["two_s"]), bonds, two_s=case["two_s"])
            st["span"].append((len(entries), len(entries) + len(bs)))
            entries += [(b, case["R"], seed + c, 0) for b in bs]
            st["bases"] += bs
        st["batch"] = ftlm.Batch(entries, case["M"], ftlm.RADEMACHER, dt)
    else:
        st["requests"] = _requests(case, seed)
        st["engine"] = serve.Engine(R=case["R"], M=case["M"], dtype=dt, T=inputs.log_t_grid(200),
                                    memory_budget=4 << 30)
    return st


def _observables(obs, h):
    # without a field <S^z> is zero by symmetry: its computed value is rounding noise
    return {k: obs[k] for k in (("E", "C", "chi") if h == 0.0 else ("E", "C", "chi", "mag"))}


def run(st):
    case, kind = st["case"], st["case"]["kind"]
    if kind == "hv":
        if case["B"] == 1:
            ftlm.ftlm_hv(st["basis"].handle, st["x"], st["y"])
        else:
            ftlm.ftlm_hv_block(st["basis"].handle, case["B"], st["x"], st["y"])
        return st["y"]
    dt = DTYPES[case["dtype"]]
    if kind in ("lanczos", "spin"):
        return ftlm.lanczos(st["basis"], case["R"], case["M"], seed=st["seed"], dist=_dist(case), dtype=dt,
                            work=st["work"], keep_coeffs=True)
    if kind == "job":
        obs = ftlm.run_ftlm(case["N"], st["bonds"], case["R"], case["M"], st["T"], seed=st["seed"], dist=_dist(case),
                            dtype=dt, h=case["h"])
        return _observables(obs, case["h"])
    if kind == "batch":
        res = st["batch"].run()
        out = []
        for a, b in st["span"]:
            secs = [(st["bases"][k].two_sz, st["bases"][k].dim, res[k]) for k in range(a, b)]
            out.append(_observables(ftlm.thermo(secs, st["T"], case["R"], case["M"]), 0.0))
        return out
    eng = st["engine"]
    eng.finished.clear()
    jobs = [serve.Job(job_id=k, N=r["N"], bonds=r["bonds"], h=r["h"], seed=r["seed"])
            for k, r in enumerate(st["requests"])]
    done = sorted(eng.run(jobs), key=lambda j: j.job_id)
    return [j.result for j in done]  # (4, nT) each: E, C, chi, <S^z>


# ------------------------------------------------------------------ work
def _levels(N, two_s):
    """Number of states of N spins by digit sum."""
    c = [1]
    for _ in range(N):
        n = [0] * (len(c) + two_s)
        for a, v in enumerate(c):
            for q in range(two_s + 1):
                n[a + q] += v
        c = n
    return c


def _sector(N, two_s, two_sz, nb):
    """(rows, matrix elements of one H.v): the diagonal and every ladder term."""
    A = (N * two_s + two_sz) // 2
    D, rest = _levels(N, two_s)[A], _levels(N - 2, two_s)
    off = sum(rest[A - a - b] for a in range(two_s) for b in range(1, two_s + 1) if 0 <= A - a - b < len(rest))
    return D, D + 2 * nb * off


def work(case):
    """Bytes and operations of one pass.  H.v reads x and writes y once; a Lanczos step
    reads q_j and q_{j-1} and writes q_{j+1} once; two operations per matrix element,
    and six per row of a step for the recurrence and its two dot products."""
    s, kind = BYTES[case["dtype"]], case["kind"]

    def chains(D, upd, R, M):
        m = min(M, D)
        return 3.0 * D * R * s * m, (2.0 * upd + 6.0 * D) * R * m

    if kind == "hv":
        D, upd = _sector(case["N"], 1, case["two_sz"], len(_bonds(case["graph"], case["N"], 0)[0]))
        return {"bytes": 2.0 * D * case["B"] * s, "flops": 2.0 * upd * case["B"]}
    if kind == "lanczos":
        nb = len(_bonds(case["graph"], case["N"], 0)[0])
        parts = [chains(*_sector(case["N"], 1, case["two_sz"], nb), case["R"], case["M"])]
    elif kind == "spin":
        nb = len(_spin_bonds(case["N"])[0])
        parts = [chains(*_sector(case["N"], case["two_s"], case["two_sz"], nb), case["R"], case["M"])]
    else:
        if kind == "job":
            cl = [(case["N"], _bonds(case["graph"], case["N"], 0))]
        elif kind == "batch":
            cl = _clusters(case, 0)
        else:
            cl = [(r["N"], r["bonds"]) for r in _requests(case, 0)]
        two_s = case.get("two_s", 1)
        parts = [chains(*_sector(N, two_s, tz, len(b[0])), case["R"], case["M"])
                 for N, b in cl for tz in ftlm.computed_two_sz(N, two_s)]
    return {"bytes": sum(p[0] for p in parts), "flops": sum(p[1] for p in parts)}


# ------------------------------------------------------------------ exact
class _Operator:
    """H on one sector in double with torch: labels with base-d digits in increasing
    order, sources found in the sorted labels."""

    def __init__(self, N, two_s, two_sz, bonds):
        dev = torch.device("cuda" if torch.cuda.is_available() else "cpu")
        d, A = two_s + 1, (N * two_s + two_sz) // 2
        parts, step = [], 1 << 26
        for a in range(0, d ** N, step):
            n = torch.arange(a, min(d ** N, a + step), device=dev)
            t, m = torch.zeros_like(n), n.clone()
            for _ in range(N):
                t += m % d
                m //= d
            parts.append(n[t == A])
        lab = torch.cat(parts)
        self.D, self.N, self.A, self.two_s = len(lab), N, A, two_s
        s = 0.5 * two_s
        self.diag = torch.zeros(self.D, dtype=torch.float64, device=dev)
        up = [math.sqrt(s * (s + 1) - (a - s) * (a - s + 1)) if a < two_s else 0.0 for a in range(d)]
        up = torch.tensor(up, dtype=torch.float64, device=dev)
        self.terms = []  # (source rows, coefficient: a number or one per row)
        self.jsum = float(np.abs(bonds[2]).sum())
        pad = torch.tensor(self.D, device=dev)
        for i, j, J in zip(*bonds):
            i, j, J = int(i), int(j), float(J)
            ai, aj = lab // d ** i % d, lab // d ** j % d
            self.diag += J * (ai.to(torch.float64) - s) * (aj.to(torch.float64) - s)
            if two_s == 1:
                src = lab + torch.where(ai > aj, d ** j - d ** i, d ** i - d ** j)
                pos = torch.searchsorted(lab, src).clamp_(max=self.D - 1)
                self.terms.append((torch.where(ai != aj, pos, pad).to(torch.int32), 0.5 * J))
                continue
            for p, q, ap, aq in ((i, j, ai, aj), (j, i, aj, ai)):  # s_p^+ s_q^-
                ok = (ap >= 1) & (aq < two_s)
                pos = torch.searchsorted(lab, lab - d ** p + d ** q).clamp_(max=self.D - 1)
                c = 0.5 * J * up[(ap - 1).clamp(min=0)] * up[aq]
                self.terms.append((torch.where(ok, pos, pad).to(torch.int32), torch.where(ok, c, 0.0)))

    def __call__(self, x):  # x: (D, R)
        xp = torch.cat([x, torch.zeros_like(x[:1])])
        y = self.diag[:, None] * x
        for src, c in self.terms:
            for a in range(0, self.D, 1 << 25):
                e = min(self.D, a + (1 << 25))
                g = xp.index_select(0, src[a:e])
                if isinstance(c, float):
                    y[a:e].add_(g, alpha=c)
                else:
                    y[a:e].addcmul_(g, c[a:e, None])
        return y


_MASK = (1 << 64) - 1
_GAMMA = 0x9E3779B97F4A7C15


def _mix_int(z):
    z = ((z ^ (z >> 30)) * 0xBF58476D1CE4E5B9) & _MASK
    z = ((z ^ (z >> 27)) * 0x94D049BB133111EB) & _MASK
    return z ^ (z >> 31)


def _signed(v):
    v &= _MASK
    return v - (1 << 64) if v >> 63 else v


def _shift(z, k):
    return (z >> k) & ((1 << (64 - k)) - 1)


def _mix(z):  # int64 tensors wrap around like unsigned ones
    z = (z ^ _shift(z, 30)) * _signed(0xBF58476D1CE4E5B9)
    z = (z ^ _shift(z, 27)) * _signed(0x94D049BB133111EB)
    return z ^ _shift(z, 31)


def _start(op, R, seed, dist):
    key_n = op.N | (op.two_s << 8 if op.two_s > 1 else 0)
    x = torch.empty((op.D, R), dtype=torch.float64, device=op.diag.device)
    t = torch.arange(op.D, device=op.diag.device)
    for r in range(R):
        tag = key_n << 48 | op.A << 32 | r
        key = _mix_int((_mix_int((seed + _GAMMA) & _MASK) + tag + _GAMMA) & _MASK)
        u = lambda c: _mix(_signed(key) + (c + 1) * _signed(_GAMMA))
        if dist == ftlm.RADEMACHER:
            x[:, r] = torch.where(u(t) < 0, -1.0, 1.0)
        else:
            u1 = (_shift(u(2 * t), 11).to(torch.float64) + 1.0) * 2.0 ** -53
            u2 = _shift(u(2 * t + 1), 11).to(torch.float64) * 2.0 ** -53
            x[:, r] = torch.sqrt(-2.0 * torch.log(u1)) * torch.cos(2.0 * math.pi * u2)
    return x


def _chains(op, R, M, seed, dist, dtype):
    """Lanczos coefficients (R x M), chain lengths, and the Ritz values and weights."""
    s = 0.5 * op.two_s
    tau = 100.0 * (2.0 ** -24 if dtype == "f32" else 2.0 ** -53) * s * (s + 1.0) * op.jsum
    q = _start(op, R, seed, dist)
    q /= torch.linalg.vector_norm(q, dim=0)
    prev, b = torch.zeros_like(q), torch.zeros(R, dtype=torch.float64, device=q.device)
    m_max = min(M, op.D)
    alpha = torch.zeros((R, M), dtype=torch.float64, device=q.device)
    beta = torch.zeros_like(alpha)
    m = torch.full((R,), m_max, dtype=torch.int64, device=q.device)
    live = torch.ones(R, dtype=torch.bool, device=q.device)
    for j in range(m_max):
        y = op(q)
        y.addcmul_(prev, -b)
        a = (q * y).sum(0)
        y.addcmul_(q, -a)
        b = torch.linalg.vector_norm(y, dim=0)
        alpha[:, j] = torch.where(live, a, 0.0)
        if j + 1 == m_max:
            break
        ends = live & (b <= tau)
        m = torch.where(ends, torch.full_like(m, j + 1), m)
        live = live & ~ends
        b = torch.where(live, b, 0.0)
        beta[:, j] = b
        prev, q = q, torch.where(live, y / torch.where(live, b, 1.0), 0.0)
    theta, weight = torch.zeros_like(alpha), torch.zeros_like(alpha)
    ah, bh = alpha.cpu().numpy(), beta.cpu().numpy()
    for r in range(R):
        k = int(m[r])
        ev, S = np.linalg.eigh(np.diag(ah[r, :k]) + np.diag(bh[r, :k - 1], 1) + np.diag(bh[r, :k - 1], -1))
        theta[r, :k] = torch.as_tensor(ev)
        weight[r, :k] = torch.as_tensor(S[0] ** 2)
    return dict(theta=theta, weight=weight, m_eff=m.to(torch.int32), alpha=alpha, beta=beta)


def _sums(sectors, R, h, g=2.0):
    """E, C, chi and <S^z> of (two_sz, D, chains) on the temperature grid; sectors with
    S^z > 0 stand for both signs."""
    e, w, sz = [], [], []
    for tz, D, c in sectors:
        for sign in (1.0, -1.0) if tz > 0 else (1.0,):
            m = sign * 0.5 * tz
            keep = torch.arange(c["theta"].shape[1], device=c["theta"].device)[None, :] < c["m_eff"][:, None]
            e.append(c["theta"][keep] - h * m)
            w.append(c["weight"][keep] * (D / R))
            sz.append(torch.full_like(e[-1], m))
    e, w, sz = torch.cat(e), torch.cat(w), torch.cat(sz)
    T = torch.as_tensor(inputs.log_t_grid(200), device=e.device)
    e0 = e.min()
    out = {"E": [], "C": [], "chi": [], "mag": []}
    for beta in (1.0 / T).tolist():
        p = w * torch.exp(-beta * (e - e0))
        p /= p.sum()
        mean, mag = (p * (e - e0)).sum(), (p * sz).sum()
        out["E"].append(e0 + mean)
        out["C"].append(beta * beta * (p * (e - e0 - mean) ** 2).sum())
        var = (p * sz * sz).sum() if h == 0.0 else (p * (sz - mag) ** 2).sum()
        out["chi"].append(g * g * beta * var)
        out["mag"].append(mag)
    return {k: torch.stack(v) for k, v in out.items()}


def _job(N, two_s, bonds, R, M, seed, dist, dtype, h):
    secs = []
    for tz in range((N * two_s) % 2, N * two_s + 1, 2):
        op = _Operator(N, two_s, tz, bonds)
        secs.append((tz, op.D, _chains(op, R, M, seed, dist, dtype)))
    return _sums(secs, R, h)


def exact(case, seed):
    kind = case["kind"]
    if kind == "hv":
        op = _Operator(case["N"], 1, case["two_sz"], _bonds(case["graph"], case["N"], seed))
        x = _vector(case, seed)
        return op(x.to(torch.float64).reshape(op.D, -1)).reshape(x.shape)
    if kind in ("lanczos", "spin"):
        two_s = case.get("two_s", 1)
        bonds = _spin_bonds(case["N"]) if kind == "spin" else _bonds(case["graph"], case["N"], seed)
        if case["dtype"] == "f32" and case["M"] > 24:
            # after the first Ritz value has converged, which step of the recurrence
            # meets it again depends on the rounding of the vectors: no exact values
            return None
        op = _Operator(case["N"], two_s, case["two_sz"], bonds)
        return _chains(op, case["R"], case["M"], seed, _dist(case), case["dtype"])
    if kind == "job":
        obs = _job(case["N"], 1, _bonds(case["graph"], case["N"], seed), case["R"], case["M"], seed, _dist(case),
                   case["dtype"], case["h"])
        return _observables(obs, case["h"])
    if kind == "batch":
        return [_observables(_job(N, case["two_s"], bonds, case["R"], case["M"], seed + c, ftlm.RADEMACHER,
                                  case["dtype"], 0.0), 0.0) for c, (N, bonds) in enumerate(_clusters(case, seed))]
    out = []
    for r in _requests(case, seed):
        obs = _job(r["N"], 1, r["bonds"], case["R"], case["M"], r["seed"], ftlm.GAUSS, case["dtype"], r["h"])
        out.append(torch.stack([obs[k] for k in ("E", "C", "chi", "mag")]))
    return out
