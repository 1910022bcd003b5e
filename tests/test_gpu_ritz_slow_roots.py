"""Merges with roots next to poles of tiny weight (converged Ritz values and their ghosts):
the Ritz values and spectral sums against numpy."""
import numpy as np
import pytest
import torch

from paper_2605_26261_gb300 import ftlm

pytestmark = pytest.mark.gpu


def lanczos_rows(D, m, seed):
    """Lanczos without reorthogonalization on a diagonal matrix: extreme Ritz values
    converge, their components in the last rows fall to rounding level, ghosts follow."""
    rng = np.random.default_rng(seed)
    d = np.concatenate([rng.uniform(-1, 1, D - 4), [-3.0, -2.5, 2.0, 3.5]])
    q, p, beta = rng.standard_normal(D), np.zeros(D), 0.0
    q /= np.linalg.norm(q)
    a, b = np.zeros(m), np.zeros(m)
    for j in range(m):
        w = d * q - beta * p
        a[j] = q @ w
        w -= a[j] * q
        beta = np.linalg.norm(w)
        b[j] = beta
        p, q = q, w / beta
    return a, b


@pytest.mark.parametrize("m", [17, 40, 65, 100, 160])
def test_roots_next_to_poles_of_tiny_weight(cuda_dev, m):
    rows = [lanczos_rows(400, m, s) for s in range(6)]
    a = torch.as_tensor(np.stack([r[0] for r in rows]), device=cuda_dev)
    b = torch.as_tensor(np.stack([r[1] for r in rows]), device=cuda_dev)
    me = torch.full((6,), m, dtype=torch.int32, device=cuda_dev)
    theta, weight = torch.empty_like(a), torch.empty_like(a)
    ftlm.ftlm_ritz(6, m, a, b, me, theta, weight)
    assert ftlm.ftlm_ritz_status() == 0
    for r, (ra, rb) in enumerate(rows):
        T = np.diag(ra) + np.diag(rb[:m - 1], 1) + np.diag(rb[:m - 1], -1)
        ev, S = np.linalg.eigh(T)
        th, w = theta[r].cpu().numpy(), weight[r].cpu().numpy()
        scale = np.abs(ev).max()
        # backward error of both solvers: a few eps m ||T||
        np.testing.assert_allclose(th, ev, rtol=0, atol=8 * 2.0**-53 * m * scale)
        for beta in (0.0, 0.5, 2.0, 8.0):  # the sums the weights enter
            f = np.exp(-beta * (ev - ev[0]))
            got, want = (w * np.exp(-beta * (th - ev[0]))).sum(), (S[0]**2 * f).sum()
            assert abs(got - want) <= 8 * 2.0**-53 * m * (1 + beta * scale)
