"""Blocks of chains that run side by side in one launch give the bits of blocks run
alone: every rank mode, type and width, with remainders (blocks of 8 / 4 / 1) and more
blocks than one launch takes."""
import pytest
import torch

from paper_2605_26261_gb300 import ftlm, inputs

pytestmark = pytest.mark.gpu


def basis(kind):
    if kind == "spin":
        return ftlm.Basis(7, 0, inputs.ring(7), two_s=2)  # 393 rows
    return ftlm.Basis(16, 2, inputs.random_graph(16, seed=4), ftlm.RANK_CLT if kind == "clt" else ftlm.RANK_CR)


@pytest.mark.parametrize("dtype", [torch.float32, torch.float64])
@pytest.mark.parametrize("kind", ["clt", "cr", "spin"])
def test_blocks_side_by_side_match_blocks_alone(cuda_dev, kind, dtype):
    R, M = 30, 9  # FP32: 8 8 8 4 1 1; FP64: seven blocks of 4, then two chains
    w = 8 if dtype == torch.float32 else 4
    with basis(kind) as b:
        g = torch.Generator(device=cuda_dev).manual_seed(3)
        start = torch.randn((R, b.dim), generator=g, device=cuda_dev, dtype=torch.float64)
        whole = ftlm.lanczos(b, R, M, dtype=dtype, start=start, keep_coeffs=True)
        r = 0
        while r < R:
            n = w if R - r >= w else (4 if R - r >= 4 else 1)
            part = ftlm.lanczos(b, n, M, dtype=dtype, start=start[r:r + n].contiguous(), keep_coeffs=True)
            for k in ("alpha", "beta", "theta", "weight", "m_eff"):
                assert torch.equal(whole[k][r:r + n], part[k]), (k, r)
            r += n
        seeded = ftlm.lanczos(b, R, M, seed=5, dtype=dtype, keep_coeffs=True)
        first = ftlm.lanczos(b, w, M, seed=5, dtype=dtype, keep_coeffs=True)
        assert torch.equal(seeded["alpha"][:w], first["alpha"])
        assert not torch.equal(seeded["alpha"][:w], seeded["alpha"][w:2 * w])  # later blocks have keys of their own


def test_workspace_keeps_the_scratch_free_limit(cuda_dev):
    # more blocks side by side never push a call past the static scratch
    for N, R in ((16, 64), (18, 40), (20, 9), (21, 3)):
        with ftlm.Basis(N, N % 2, inputs.ring(N)) as b:
            one = ftlm.ftlm_lanczos_workspace_bytes(b.handle, 1, 20, torch.float32)
            many = ftlm.ftlm_lanczos_workspace_bytes(b.handle, R, 20, torch.float32)
            assert many >= one
            assert many <= max(24 << 20, 10 * one)


@pytest.mark.parametrize("N,R", [(18, 16), (19, 16), (19, 24), (20, 16), (20, 24), (21, 24)])
def test_a_chain_does_not_depend_on_the_blocks_beside_it(cuda_dev, N, R):
    # around the row counts where the H.v launch changes its shape: 320, 608, 1215 and 2320 rows per
    # SM, with two and three blocks of 8 side by side, or two and then one, where they fit
    with ftlm.Basis(N, N % 2, inputs.random_graph(N, seed=4), ftlm.RANK_CLT) as b:
        g = torch.Generator(device=cuda_dev).manual_seed(3)
        start = torch.randn((R, b.dim), generator=g, device=cuda_dev, dtype=torch.float64)
        whole = ftlm.lanczos(b, R, 9, dtype=torch.float32, start=start, keep_coeffs=True)
        for r in range(0, R, 8):
            part = ftlm.lanczos(b, 8, 9, dtype=torch.float32, start=start[r:r + 8].contiguous(), keep_coeffs=True)
            for k in ("alpha", "beta", "theta", "weight", "m_eff"):
                assert torch.equal(whole[k][r:r + 8], part[k]), (k, r)


@pytest.mark.parametrize("mode", [ftlm.RANK_CLT, ftlm.RANK_CR])
@pytest.mark.parametrize("N,R,width", [(22, 8, 8), (23, 9, 8), (23, 1, 1), (24, 4, 4)])
def test_workspace_is_two_vector_blocks(cuda_dev, mode, N, R, width):
    with ftlm.Basis(N, N % 2, inputs.ring(N), mode) as b:
        for dtype, size in ((torch.float32, 4), (torch.float64, 8)):
            vectors = 2 * b.dim * min(width, 32 // size) * size  # blocks of 8 floats, 4 doubles
            got = ftlm.ftlm_lanczos_workspace_bytes(b.handle, R, 50, dtype)
            assert vectors <= got <= max(24 << 20, vectors + (1 << 18))
