"""Thermodynamic sums on the GPU against numpy in the forms the kernel's variants take:
few pairs (one CTA per temperature), clusters of 4 and 8 CTAs with the weights kept in
shared memory, more pairs than fit, 64 sectors, chains and sectors without pairs, a
field, no mirror images, and Ritz values that are not numbers.

Tolerance (relative to the largest value of an observable): the sums have positive
terms, so each is within a few (number of pairs)^(1/2) 2^-53 and the rounding of the
exponents beta E (below 10^3 x 2^-53 where a weight matters): 1e-12.
"""
import numpy as np
import pytest
import torch

from paper_2605_26261_gb300 import ftlm

pytestmark = pytest.mark.gpu


def sectors(ns, R, M, seed, empty=()):
    rng = np.random.default_rng(seed)
    out = []
    for s in range(ns):
        m = rng.integers(0 if ns > 1 else 1, M + 1, size=R).astype(np.int32)
        if s in empty:
            m[:] = 0
        th, w = np.zeros((R, M)), np.zeros((R, M))
        for r in range(R):
            th[r, :m[r]] = np.sort(rng.uniform(-6.0, 4.0, size=m[r]))
            x = rng.random(m[r])
            w[r, :m[r]] = x / x.sum() if m[r] else x
        out.append((2 * s, int(rng.integers(1, 10**6)), th, w, m))
    return out


def reference(secs, T, R, g, h, mirror):
    e, b0, sz = [], [], []
    for tz, D, th, w, m in secs:
        for sign in ((1, -1) if mirror and tz > 0 else (1,)):
            mz = 0.5 * sign * tz
            for r in range(R):
                e.append(th[r, :m[r]] - h * mz)
                b0.append(w[r, :m[r]] * D / R)
                sz.append(np.full(m[r], mz))
    e, b0, sz = (np.concatenate(v).astype(np.longdouble) for v in (e, b0, sz))
    e0, out = e.min(), {k: [] for k in ("E", "C", "chi", "mag", "Z")}
    for t in T:
        beta = np.longdouble(1.0) / np.longdouble(t)
        b = b0 * np.exp(-beta * (e - e0))
        Z = b.sum()
        e1, m1 = (b * (e - e0)).sum() / Z, (b * sz).sum() / Z
        out["Z"].append(Z)
        out["E"].append(e0 + e1)
        out["C"].append(beta ** 2 * (b * (e - e0 - e1) ** 2).sum() / Z)
        out["chi"].append(g * g * beta * ((b * sz * sz).sum() / Z if h == 0 else (b * (sz - m1) ** 2).sum() / Z))
        out["mag"].append(m1)
    return {k: np.array(v, dtype=float) for k, v in out.items()}


@pytest.mark.parametrize("ns,R,M,empty", [(1, 1, 1, ()), (1, 1, 7, ()), (3, 5, 30, (1,)),  # one CTA
                                          (2, 32, 33, ()), (11, 16, 100, (0, 5)),          # clusters of 4
                                          (64, 7, 20, (0, 63)),
                                          (13, 40, 100, ()),                               # of 8
                                          (20, 64, 100, (3,))])                            # weights computed twice
@pytest.mark.parametrize("h,mirror", [(0.0, True), (0.7, True), (0.3, False)])
def test_sums_match_numpy(cuda_dev, ns, R, M, empty, h, mirror):
    secs = sectors(ns, R, M, 1000 * ns + R, empty)
    T = np.logspace(-2, 1, 23)
    dev = [(tz, D, {"theta": torch.as_tensor(th, device=cuda_dev), "weight": torch.as_tensor(w, device=cuda_dev),
                    "m_eff": torch.as_tensor(m, device=cuda_dev)}) for tz, D, th, w, m in secs]
    Td = torch.as_tensor(T, device=cuda_dev)
    got = ftlm.thermo(dev, Td, R, M, g=2.0, h=h, mirror=mirror)
    Z, E0 = torch.empty_like(Td), torch.empty_like(Td)
    ftlm.ftlm_partition([s[0] for s in dev], [s[1] for s in dev], R, M, [s[2]["theta"] for s in dev],
                        [s[2]["weight"] for s in dev], [s[2]["m_eff"] for s in dev], mirror, h, Td, Z, E0)
    ref = reference(secs, T, R, 2.0, h, mirror)
    for k in ("E", "C", "chi", "mag"):
        scale = max(np.abs(ref[k]).max(), 1e-3)
        assert np.abs(got[k].cpu().numpy() - ref[k]).max() <= 1e-12 * scale, k
    assert np.abs(Z.cpu().numpy() / ref["Z"] - 1).max() <= 1e-11
    again = ftlm.thermo(dev, Td, R, M, g=2.0, h=h, mirror=mirror)
    for k in ("E", "C", "chi", "mag"):
        assert torch.equal(got[k], again[k])


@pytest.mark.parametrize("whole_sector", [False, True])
def test_an_unconverged_chain_shows_in_every_observable(cuda_dev, whole_sector):
    secs = sectors(4, 6, 20, 3)
    for tz, D, th, w, m in secs:
        m[:] = 20
    bad = slice(None) if whole_sector else 2
    secs[1][2][bad] = np.nan
    secs[1][3][bad] = np.nan
    dev = [(tz, D, {"theta": torch.as_tensor(th, device=cuda_dev), "weight": torch.as_tensor(w, device=cuda_dev),
                    "m_eff": torch.as_tensor(m, device=cuda_dev)}) for tz, D, th, w, m in secs]
    got = ftlm.thermo(dev, torch.tensor([0.1, 1.0], device=cuda_dev, dtype=torch.float64), 6, 20)
    for k in ("E", "C", "chi"):
        assert torch.isnan(got[k]).all()


def test_as_many_pairs_as_are_accepted(cuda_dev):
    # 2^31 - 2 pairs: the index of a thread's last step passes 2^31.  Two chains have pairs, the
    # first and the last.
    M, R = 1023, 2099202
    rng = np.random.default_rng(1)
    th, w = (torch.zeros((R, M), dtype=torch.float64, device=cuda_dev) for _ in range(2))
    m = torch.zeros(R, dtype=torch.int32, device=cuda_dev)
    secs = []
    for r in (0, R - 1):
        t, x = np.sort(rng.uniform(-6.0, 4.0, size=(1, M))), rng.random((1, M))
        th[r], w[r], m[r] = torch.as_tensor(t[0]), torch.as_tensor(x[0]), M
        secs.append((0, R, t, x, np.array([M])))
    T = np.array([0.3, 2.0])
    got = ftlm.thermo([(0, R, {"theta": th, "weight": w, "m_eff": m})], torch.as_tensor(T, device=cuda_dev), R, M)
    ref = reference(secs, T, 1, 2.0, 0.0, True)
    for k in ("E", "C"):
        assert np.abs(got[k].cpu().numpy() - ref[k]).max() <= 1e-12 * np.abs(ref[k]).max(), k
