"""General-spin rows on every launch shape: sectors of few and of many rows, with and
without the lists of a tile's bonds, tiles of one and of several high labels, every block
width and type, against sampled rows of the oracle and against each other."""
import numpy as np
import pytest
import torch

from oracle import spin
from paper_2605_26261_gb300 import ftlm, inputs

pytestmark = pytest.mark.gpu


def complete(N):
    return np.array([(i, j, 0.3 + 0.1 * ((i + j) % 3)) for i in range(N) for j in range(i + 1, N)])


def as_bonds(a):
    return a[:, 0].astype(np.int32), a[:, 1].astype(np.int32), a[:, 2].copy()


CASES = [  # (N, two_s, two_sz, bonds)
    (3, 2, 0, inputs.ring(3)),                       # 7 rows, no high digits
    (9, 3, 1, inputs.random_graph(9, seed=6)),       # no lists: 39 000 rows
    (12, 2, 18, as_bonds(complete(12))),             # small groups of one high label, 66 bonds
    (9, 6, 0, as_bonds(complete(9))),                # lists, 3.1 M rows, d = 7, ten high-high bonds
    (14, 2, 2, inputs.random_graph(14, seed=8)),     # lists, blocks of few rows
    (16, 2, 14, as_bonds(complete(16))),             # lists, 64 cross bonds (two rounds of lanes)
]


@pytest.mark.parametrize("case", CASES, ids=lambda c: f"N{c[0]}_2s{c[1]}_2sz{c[2]}")
@pytest.mark.parametrize("dtype", [torch.float32, torch.float64])
def test_rows_of_every_launch_shape(cuda_dev, dtype, case):
    N, two_s, two_sz, bonds = case
    s = 0.5 * two_s
    norm = s * (s + 1) * float(np.abs(bonds[2]).sum())  # >= every row's sum of |H_ij|
    eps = 2.0**-24 if dtype == torch.float32 else 2.0**-53
    with ftlm.Basis(N, two_sz, bonds, two_s=two_s) as b:
        X = inputs.hashed_vector_torch(b.dim * 16, dtype, cuda_dev).view(b.dim, 16)
        Y = torch.empty_like(X)
        ftlm.ftlm_hv_block(b.handle, 16, X, Y)
        for B in (1, 4, 8):  # bitwise: the terms and their order are those of the row
            x = X[:, :B].contiguous()
            y = torch.empty_like(x)
            if B == 1:
                ftlm.ftlm_hv(b.handle, x.view(-1), y.view(-1))
            else:
                ftlm.ftlm_hv_block(b.handle, B, x, y)
            assert torch.equal(Y[:, :B], y), B
        # the oracle's rows: 2 nb + 2 roundings per row
        ref_b = spin.basis(N, two_s, spin.sector_A(N, two_s, two_sz))
        x0 = X[:, 0].double().cpu().numpy()
        y0 = Y[:, 0].double().cpu().numpy()
        tol = (2 * len(bonds[2]) + 8) * eps * norm * np.abs(x0).max()
        for t0 in np.linspace(0, max(0, b.dim - 512), 12).astype(np.int64):
            t1 = min(b.dim, int(t0) + 512)
            want = spin.hv_range(N, two_s, bonds, ref_b, x0, int(t0), t1)
            np.testing.assert_allclose(y0[t0:t1], want, rtol=0, atol=tol)
        # alpha_1 of the Lanczos launches = x . H x / x . x of the plain ones, up to the rounding of
        # the scaled entries; every chain of a block, and again to the same bits
        for B in (1, 4, 8):
            start = X[:, :B].double().t().contiguous()
            got = ftlm.lanczos(b, B, 2, dtype=dtype, start=start, keep_coeffs=True)
            again = ftlm.lanczos(b, B, 2, dtype=dtype, start=start, keep_coeffs=True)
            assert torch.equal(got["alpha"], again["alpha"]) and torch.equal(got["beta"], again["beta"])
            xd, yd = X[:, :B].double(), Y[:, :B].double()
            want = (xd * yd).sum(0) / (xd * xd).sum(0)
            assert (got["alpha"][:, 0] - want).abs().max().item() <= (2 * len(bonds[2]) + 8) * eps * norm
