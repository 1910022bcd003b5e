"""Ritz step by divide and conquer on the GPU against LAPACK (numpy eigh): sizes around
the thread count and the powers of two of the merge tree, spectra that deflate, and
coefficients that are not finite.

Tolerances: the method is backward stable, so eigenvalues are within a modest multiple
of 2^-52 ||T|| (1e-13: 450 of them), and so are the smooth spectral sums
sum_k w_k g(theta_k) with |g|, |g'| ||T|| <= 8 (1e-12).  Weights inside a cluster of
close eigenvalues are defined only as a sum, hence the sums.
"""
import ctypes
import subprocess

import numpy as np
import pytest
import torch

from paper_2605_26261_gb300 import ftlm

pytestmark = pytest.mark.gpu


def problems(m, rng):
    """Coefficient rows (a, b) of length m."""
    a, b = rng.normal(size=m), np.abs(rng.normal(size=m)) + 0.1
    half = np.abs(np.arange(m) - m // 2).astype(float)
    cut = b.copy()
    cut[::3] = 0.0
    tiny = np.ones(m)
    tiny[::5] = 1e-13
    return [(a, b),
            (a, -b),                                     # couplings of either sign
            (a, cut),                                    # decoupled blocks
            (np.zeros(m), np.ones(m)),                   # Toeplitz
            (half, np.ones(m)),                          # Wilkinson: pairs close to rounding
            (np.tile(half[:m // 4 + 1], 4)[:m], tiny),   # glued copies of one block
            (np.ones(m), np.full(m, 1e-9)),              # nearly a multiple of the identity
            (np.zeros(m), np.zeros(m)),
            (10.0 ** (-12 * np.arange(m) / m), 10.0 ** (-12 * np.arange(m) / m - 0.3)),  # graded
            (1e180 * a, 1e180 * b),
            (1e-180 * a, 1e-180 * b)]


def ritz(a, b, m, dev):
    n, M = a.shape
    th = torch.full((n, M), 7.0, dtype=torch.float64, device=dev)
    w = th.clone()
    ftlm.ftlm_ritz(n, M, torch.as_tensor(a, device=dev), torch.as_tensor(b, device=dev),
                   torch.as_tensor(np.asarray(m, dtype=np.int32), device=dev), th, w)
    return th.cpu().numpy(), w.cpu().numpy()


@pytest.mark.parametrize("m", [1, 2, 3, 4, 31, 32, 33, 64, 65, 100, 127, 128, 129, 257, 1024])
def test_divide_and_conquer_matches_lapack(cuda_dev, m):
    rng = np.random.default_rng(m)
    probs = problems(m, rng)
    M = min(1024, m + 3)  # rows longer than the problems, where they may be
    a, b = np.zeros((len(probs), M)), np.zeros((len(probs), M))
    for c, (x, y) in enumerate(probs):
        a[c, :m], b[c, :m] = x, y
    ftlm.ftlm_ritz_status()
    th, w = ritz(a, b, [m] * len(probs), cuda_dev)
    assert ftlm.ftlm_ritz_status() == 0
    for c, (x, y) in enumerate(probs):
        scale = max(np.abs(x).max(), np.abs(y).max()) or 1.0
        T = np.diag(x / scale) + np.diag(y[:m - 1] / scale, 1) + np.diag(y[:m - 1] / scale, -1)
        ev, S = np.linalg.eigh(T)
        got = th[c, :m] / scale
        norm = max(np.abs(ev).max(), 1e-300)
        assert np.all(np.diff(got) >= 0)
        assert np.abs(got - ev).max() <= 1e-13 * norm, c
        for beta in (0.0, 1.0, 4.0):
            g = lambda e: np.exp(-beta * (e - ev[0]) / norm)
            assert abs((w[c, :m] * g(got)).sum() - (S[0] ** 2 * g(ev)).sum()) <= 1e-12, (c, beta)
        assert np.all(w[c, :m] >= 0) and np.all(th[c, m:] == 0) and np.all(w[c, m:] == 0)


def test_non_finite_coefficients_give_nan_rows(cuda_dev):
    rng = np.random.default_rng(1)
    M = 20
    a, b = rng.normal(size=(5, M)), np.abs(rng.normal(size=(5, M))) + 0.1
    a[0, 3], b[1, 4], a[2, 0] = np.nan, np.inf, -np.inf
    b[3, M - 1] = np.nan  # past the last coupling: not part of the problem
    ftlm.ftlm_ritz_status()
    th, w = ritz(a, b, [M] * 5, cuda_dev)
    with pytest.raises(ftlm.FtlmError) as e:
        ftlm.ftlm_ritz_status()
    assert e.value.status == ftlm.FTLM_ENOCONV and e.value.unconverged == 3
    assert np.all(np.isnan(th[:3])) and np.all(np.isnan(w[:3]))
    assert np.all(np.isfinite(th[3:])) and np.all(np.isfinite(w[3:]))


def test_a_chain_does_not_depend_on_the_others(cuda_dev):
    rng = np.random.default_rng(2)
    n, M = 40, 77
    a, b = rng.normal(size=(n, M)), np.abs(rng.normal(size=(n, M))) + 0.1
    m = rng.integers(1, M + 1, size=n)
    th, w = ritz(a, b, m, cuda_dev)
    for c in (0, 17, 39):
        t1, w1 = ritz(a[c:c + 1], b[c:c + 1], m[c:c + 1], cuda_dev)
        assert np.array_equal(t1[0], th[c]) and np.array_equal(w1[0], w[c])


@pytest.mark.parametrize("m", [4, 8, 33, 130])
@pytest.mark.parametrize("scale", [1e-60, 1e-119, 1e-122, 1e-150, 1e-200, 1e-300, 1e-309])
def test_blocks_of_scales_far_apart(cuda_dev, m, scale):
    # a block of coefficients near one and a block of much smaller ones, in either order and
    # in turn; the tolerances of the file's head
    rng = np.random.default_rng(m)
    a, b = rng.normal(size=m), np.abs(rng.normal(size=m)) + 0.1
    f = np.ones(m)
    f[m // 2:] = scale
    turn = np.where(np.arange(m) % 4 < 2, 1.0, scale)
    probs = [(a * f, b * f), (a * f[::-1], b * f[::-1]), (a * turn, b * turn), (0 * a, b * f), (f, b * f)]
    th, w = ritz(np.array([p[0] for p in probs]), np.array([p[1] for p in probs]), [m] * len(probs), cuda_dev)
    for c, (x, y) in enumerate(probs):
        ev, S = np.linalg.eigh(np.diag(x) + np.diag(y[:m - 1], 1) + np.diag(y[:m - 1], -1))
        norm = np.abs(ev).max()
        assert np.abs(th[c] - ev).max() <= 1e-13 * norm, c
        for beta in (0.0, 1.0, 4.0):
            g = lambda e: np.exp(-beta * (e - ev[0]) / norm)
            assert abs((w[c] * g(th[c])).sum() - (S[0] ** 2 * g(ev)).sum()) <= 1e-12, (c, beta)
    ftlm.ftlm_ritz_status()


RECIP = r"""
#include <cstring>
#include "tridiag_dc.cuh"
__global__ void recip_kernel(int n, const double *x, double *got, double *want)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) {
        got[i] = ftlm::dc::recip(x[i]);
        want[i] = __drcp_rn(x[i]);
    }
}
extern "C" int recip_all(int n, const double *x, double *got, double *want)
{
    recip_kernel<<<(n + 255) / 256, 256>>>(n, x, got, want);
    return (int)cudaDeviceSynchronize();
}
"""


def test_reciprocal_against_cuda(cuda_dev, tmp_path):
    """dc::recip against the correctly rounded reciprocal over its range: within one unit in the last
    place (the Newton step's own rounding is half of one; the error before it is 2^-80)."""
    from paper_2605_26261_gb300 import _build

    src, so = tmp_path / "recip.cu", tmp_path / "recip.so"
    src.write_text(RECIP)
    subprocess.run([_build._nvcc(), "-shared", "-Xcompiler", "-fPIC", "-std=c++17", *_build.ARCH, "-I", _build.CSRC,
                    str(src), "-o", str(so)], check=True)
    rng = np.random.default_rng(5)
    n = 1 << 20
    x = np.ldexp(1.0 + rng.random(n), rng.integers(-1021, 1021, size=n)) * rng.choice([-1.0, 1.0], size=n)
    x[:n // 2] = np.ldexp(1.0 + rng.random(n // 2), rng.integers(-60, 3, size=n // 2))
    edge = [np.ldexp(m, e) for e in (-1021, -1020, -400, -1, 0, 1, 400, 1019, 1020)
            for m in (1.0, 1.0 + 2.0**-52, 2.0 - 2.0**-52, 1.5, 1.0 + 2.0**-20, 1.0 + 2.0**-21, 2.0 - 2.0**-21)]
    x[-len(edge):] = edge
    xd = torch.as_tensor(x, device=cuda_dev)
    got, want = torch.empty_like(xd), torch.empty_like(xd)
    lib = ctypes.CDLL(str(so))
    p = ctypes.c_void_p
    assert lib.recip_all(n, p(xd.data_ptr()), p(got.data_ptr()), p(want.data_ptr())) == 0
    got, want = got.cpu().numpy(), want.cpu().numpy()
    assert np.all(np.abs(got - want) <= np.spacing(np.abs(want)))
