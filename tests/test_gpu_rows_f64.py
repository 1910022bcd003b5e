"""H.v of doubles (per-lane bond lists) against the definition, over the forms a bond
list can take: more bonds than one list word (64), none, zero and negative couplings,
labels beyond 32 bits, sectors smaller than a warp and off the tile size, both rank
modes and every block width.

Tolerance: a row has at most nb + 1 terms of size |J| max|x| / 2, each rounded once:
(nb + 2) 2^-53 sum_b |J_b| / 2 max|x|, times 2 for the diagonal.
"""
import itertools

import numpy as np
import pytest
import torch

from paper_2605_26261_gb300 import ftlm, inputs

pytestmark = pytest.mark.gpu


def reference(N, K, bonds, x):
    """y = H x by the definition, labels by enumeration of the K up sites."""
    labels = sorted(sum(1 << s for s in up) for up in itertools.combinations(range(N), K))
    pos = {n: t for t, n in enumerate(labels)}
    y = np.zeros_like(x)
    for i, j, J in zip(*bonds):
        m = (1 << int(i)) | (1 << int(j))
        for t, n in enumerate(labels):
            if (n & m) in (0, m):
                y[t] += 0.25 * J * x[t]
            else:
                y[t] += -0.25 * J * x[t] + 0.5 * J * x[pos[n ^ m]]
    return y


def complete(N, seed, zero=False):
    rng = np.random.default_rng(seed)
    p = list(itertools.combinations(range(N), 2))
    J = rng.normal(size=len(p))
    if zero:
        J[::3] = 0.0
    return (np.array([a for a, _ in p], dtype=np.int32), np.array([b for _, b in p], dtype=np.int32), J)


EMPTY = (np.zeros(0, dtype=np.int32), np.zeros(0, dtype=np.int32), np.zeros(0))
CASES = [(12, 6, complete(12, 1)),         # 66 bonds: two words
         (16, 3, complete(16, 2, True)),   # 120 bonds, some of coupling zero
         (17, 2, complete(17, 3)),         # 136 bonds: three words
         (9, 4, inputs.ring(9)),
         (5, 1, inputs.ring(5)),           # 5 rows
         (10, 10, inputs.ring(10)),        # one row
         (11, 5, EMPTY),
         (34, 2, inputs.ring(34)),         # labels beyond 32 bits (no lookup table)
         (33, 32, complete(20, 4))]


@pytest.mark.parametrize("mode", [ftlm.RANK_CLT, ftlm.RANK_CR])
@pytest.mark.parametrize("case", range(len(CASES)))
def test_rows_of_doubles_match_the_definition(cuda_dev, case, mode):
    N, K, bonds = CASES[case]
    if mode == ftlm.RANK_CLT and N > 32:
        pytest.skip("no lookup table beyond 32 sites")
    with ftlm.Basis(N, 2 * K - N, bonds, mode) as b:
        x = np.random.default_rng(case).normal(size=(b.dim, 16))
        want = np.stack([reference(N, K, bonds, np.ascontiguousarray(x[:, r])) for r in range(2)], axis=1)
        tol = 2 * (len(bonds[2]) + 2) * 2.0 ** -53 * np.abs(bonds[2]).sum() * np.abs(x).max()
        xd = torch.as_tensor(x, device=cuda_dev)
        cols = []
        for r in range(16):
            xr = xd[:, r].clone()
            y = torch.empty_like(xr)
            ftlm.ftlm_hv(b.handle, xr, y)
            cols.append(y)
        for r in range(2):
            assert np.abs(cols[r].cpu().numpy() - want[:, r]).max() <= tol
        for B in (4, 8, 16):
            xb = xd[:, :B].clone(memory_format=torch.contiguous_format)
            y = torch.empty_like(xb)
            ftlm.ftlm_hv_block(b.handle, B, xb, y)
            for r in range(B):
                assert torch.equal(y[:, r], cols[r])


@pytest.mark.parametrize("scale", [1e-200, 1e200])
def test_couplings_far_from_one(cuda_dev, scale):
    N = 12
    bi, bj, J = inputs.random_graph(N, seed=8)
    root = np.sqrt(scale)  # the norms of a chain are squares: only |J| below 1e154 has them
    with ftlm.Basis(N, 0, (bi, bj, J)) as b, ftlm.Basis(N, 0, (bi, bj, J * scale)) as c:
        x = torch.randn(b.dim, device=cuda_dev, dtype=torch.float64)
        y, z = torch.empty_like(x), torch.empty_like(x)
        ftlm.ftlm_hv(b.handle, x, y)
        ftlm.ftlm_hv(c.handle, x, z)
        assert torch.abs(z / scale - y).max().item() <= 1e-13 * torch.abs(y).max().item()
        ref = ftlm.lanczos(b, 4, 8, seed=2, dtype=torch.float64, keep_coeffs=True)["alpha"]
        for mode in (ftlm.RANK_CLT, ftlm.RANK_CR):
            with ftlm.Basis(N, 0, (bi, bj, J * root), mode) as d:
                a = ftlm.lanczos(d, 4, 8, seed=2, dtype=torch.float64, keep_coeffs=True)["alpha"] / root
                assert torch.abs(a - ref).max().item() <= 1e-10 * torch.abs(ref).max().item()


@pytest.mark.parametrize("mode", [ftlm.RANK_CLT, ftlm.RANK_CR])
def test_couplings_whose_sum_of_magnitudes_overflows(cuda_dev, mode):
    # sum |J| = 3.2e308 is out of range, H and its rows are not
    N, scale = 8, 4e307
    bi, bj, J = inputs.ring(N)
    J = J * np.linspace(0.5, 1.0, N)
    with ftlm.Basis(N, 0, (bi, bj, J), mode) as b, ftlm.Basis(N, 0, (bi, bj, J * scale * 4 / 3), mode) as c:
        x = torch.randn(b.dim, device=cuda_dev, dtype=torch.float64) / 16
        y, z = torch.empty_like(x), torch.empty_like(x)
        ftlm.ftlm_hv(b.handle, x, y)
        ftlm.ftlm_hv(c.handle, x, z)
        assert torch.isfinite(z).all()
        assert torch.abs(z / (scale * 4 / 3) - y).max().item() <= 1e-13 * torch.abs(y).max().item()
        ref = ftlm.lanczos(b, 4, 3, seed=2, dtype=torch.float64, keep_coeffs=True)
        got = ftlm.lanczos(c, 4, 3, seed=2, dtype=torch.float64, keep_coeffs=True)
        a, g = ref["alpha"][:, 0], got["alpha"][:, 0] / (scale * 4 / 3)
        assert torch.abs(g - a).max().item() <= 1e-12 * torch.abs(ref["alpha"]).max().item()


@pytest.mark.parametrize("mode", [ftlm.RANK_CLT, ftlm.RANK_CR])
@pytest.mark.parametrize("scale", [2.0 ** -930, 2.0 ** -960, 2.0 ** -990, 2.0 ** 1000])
def test_couplings_near_the_ends_of_the_range(cuda_dev, mode, scale):
    # the unit of the whole-number diagonal has no inverse in range below about 2^-960
    N = 12
    bi, bj, J = inputs.random_graph(N, seed=8)
    with ftlm.Basis(N, 0, (bi, bj, J), mode) as b, ftlm.Basis(N, 0, (bi, bj, J * scale), mode) as c:
        x = torch.randn(b.dim, device=cuda_dev, dtype=torch.float64)
        y, z = torch.empty_like(x), torch.empty_like(x)
        ftlm.ftlm_hv(b.handle, x, y)
        ftlm.ftlm_hv(c.handle, x, z)
        assert torch.abs(z / scale - y).max().item() <= 1e-13 * torch.abs(y).max().item()
