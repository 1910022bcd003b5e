"""Lookup-table Lanczos launches of 8-wide FP32 blocks on both sides of the row count where the
bond chunk changes, with bond counts that leave every remainder: the first step against
the plain H.v, whose launches keep one chunk."""
import numpy as np
import pytest
import torch

from paper_2605_26261_gb300 import ftlm, inputs

pytestmark = pytest.mark.gpu


def bonds(N, n):
    e = []
    for i, j in [(i, (i + k) % N) for k in (1, 2, 3) for i in range(N)]:
        if (min(i, j), max(i, j)) not in e:  # a bond appears once
            e.append((min(i, j), max(i, j)))
    e, n = e[:n], min(n, len(e))
    return (np.array([p[0] for p in e], dtype=np.int32), np.array([p[1] for p in e], dtype=np.int32),
            0.5 + 0.01 * np.arange(n))


@pytest.mark.parametrize("N,R", [(6, 8), (16, 24), (19, 8), (18, 16), (21, 8)])
@pytest.mark.parametrize("n", [5, 8, 17])
def test_first_step_of_every_chunk(cuda_dev, N, R, n):
    bd = bonds(N, n)
    norm = 0.75 * float(bd[2].sum())
    with ftlm.Basis(N, N % 2, bd, ftlm.RANK_CLT) as b:
        n = len(bd[2])
        X = inputs.hashed_vector_torch(b.dim * R, torch.float32, cuda_dev).view(b.dim, R)
        got = ftlm.lanczos(b, R, 2, dtype=torch.float32, start=X.double().t().contiguous(), keep_coeffs=True)
        for r in range(0, R, 8):
            x = X[:, r:r + 8].contiguous()
            y = torch.empty_like(x)
            ftlm.ftlm_hv_block(b.handle, 8, x, y)
            xd, yd = x.double(), y.double()
            want = (xd * yd).sum(0) / (xd * xd).sum(0)
            # 2 n + 8 roundings per entry of either side, against ||H||
            assert (got["alpha"][r:r + 8, 0] - want).abs().max().item() <= (2 * n + 8) * 2.0**-23 * norm
