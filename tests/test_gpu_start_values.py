"""FP32 Gaussian start vectors come from two-float arithmetic with a check of the rounding:
the stored floats are those of the FP64 definition."""
import math

import pytest
import torch

from paper_2605_26261_gb300 import ftlm, inputs

pytestmark = pytest.mark.gpu

MASK = (1 << 64) - 1
GAMMA = 0x9E3779B97F4A7C15


def signed(x):
    x &= MASK
    return x - (1 << 64) if x >> 63 else x


def shift(x, n):
    return (x >> n) & ((1 << (64 - n)) - 1)


def mix(z):
    z = (z ^ shift(z, 30)) * signed(0xBF58476D1CE4E5B9)
    z = (z ^ shift(z, 27)) * signed(0x94D049BB133111EB)
    return z ^ shift(z, 31)


def mix_int(z):
    z &= MASK
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9 & MASK
    z = (z ^ (z >> 27)) * 0x94D049BB133111EB & MASK
    return z ^ (z >> 31)


def definition(D, R, N, K, seed, dev):
    t = torch.arange(D, device=dev)
    rows = []
    for r in range(R):
        key = mix_int(mix_int(seed + GAMMA) + (N << 48 | K << 32 | r) + GAMMA)
        u1 = shift(mix(signed(key) + (2 * t + 1) * signed(GAMMA)), 11).to(torch.float64)
        u2 = shift(mix(signed(key) + (2 * t + 2) * signed(GAMMA)), 11).to(torch.float64)
        rows.append(torch.sqrt(-2.0 * torch.log((u1 + 1.0) * 2.0**-53)) * torch.cos(2.0 * math.pi * u2 * 2.0**-53))
    return torch.stack(rows)


# Bitwise: both roundings are of the same FP64 values; two FP64 libraries that differ by an
# ulp would move a float in one of 2^28 values, and the largest case here has 1.5 M.
@pytest.mark.parametrize("N,K,R", [(4, 3, 1), (9, 5, 3), (14, 8, 13), (18, 9, 8), (20, 10, 8)])
def test_fp32_start_values_are_the_rounded_definition(cuda_dev, N, K, R):
    with ftlm.Basis(N, 2 * K - N, inputs.random_graph(N, seed=N)) as b:
        want = definition(b.dim, R, N, K, 77, cuda_dev)
        got = ftlm.lanczos(b, R, 3, seed=77, keep_coeffs=True)
        ref = ftlm.lanczos(b, R, 3, start=want, keep_coeffs=True)
        assert torch.equal(got["alpha"], ref["alpha"])
        assert torch.equal(got["beta"], ref["beta"])
