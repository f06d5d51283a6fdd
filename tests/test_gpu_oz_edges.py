"""The slice GEMM (`csrc/oz.cu`) where it can go wrong: ragged tiles and K blocks, skinny
products, K splits, operands whose digits reach the bound that keeps the FP32 level sums
exact, and non-finite rows.

Bound of one complex part: every left-out digit product and every rounded digit tail is below
2^-55 of the row's and column's power of two (each at most twice the largest entry), 2 K terms,
about ten of them per term: |error| <= 32 K 2^-53 max|A_i.| max|B_.j| holds with room."""
from fractions import Fraction

import numpy as np
import pytest
import torch

from paper_1610_02244_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    from paper_1610_02244_gb300 import build as b
    b.build()
    from paper_1610_02244_gb300 import tnt
    return tnt.Context(0)


def dev(x):
    return torch.from_numpy(np.ascontiguousarray(x)).to("cuda:0")


@pytest.mark.parametrize("M,N,K", [(16, 16, 16 * 110), (17, 4100, 130), (127, 63, 257), (128, 64, 256), (129, 65, 258),
                                   (130, 1, 400), (255, 193, 31), (700, 130, 33), (64, 64, 8192), (127, 63, 513), (128, 64, 512),
                                   (129, 65, 514)])
@pytest.mark.parametrize("conj,order", [(False, "rr"), (True, "cc")])
def test_ragged_products(ctx, M, N, K, conj, order):
    g = synth.rng(M + 3 * N + 7 * K)
    A, B = synth.complex_gaussian(g, (M, K)), synth.complex_gaussian(g, (K, N))
    B *= 10.0 ** g.uniform(-150, 150, N)[None, :]
    A *= 10.0 ** g.uniform(-100, 100, M)[:, None]
    Ad = dev(A.T).T if order[0] == "c" else dev(A)
    Bd = dev(B.T).T if order[1] == "c" else dev(B)
    C = ctx.matmul(Ad, Bd, conj_a=conj, conj_b=conj).cpu().numpy()
    ld = np.longdouble
    s = -1 if conj else 1
    Ar, Ai, Br, Bi = A.real.astype(ld), s * A.imag.astype(ld), B.real.astype(ld), s * B.imag.astype(ld)
    bound = 32 * K * 2.0 ** -53 * np.abs(A).max(1)[:, None].astype(ld) * np.abs(B).max(0)[None, :]
    assert np.all(np.abs(C.real - (Ar @ Br - Ai @ Bi)) <= bound)
    assert np.all(np.abs(C.imag - (Ar @ Bi + Ai @ Br)) <= bound)


@pytest.mark.parametrize("digit", [63, -64])
def test_largest_digits(ctx, digit):
    """Every digit at the end of its range and every product of one sign: the level sums come
    within 3% of 2^24."""
    F = sum((63 if digit > 0 else (64 if p == 0 else -64)) * 128 ** (7 - p) for p in range(8))
    v = float(Fraction(F, 2 ** 55))
    F = int(Fraction(v) * 2 ** 55)  # what 53 bits keep of it
    K = 768
    A = np.full((160, K), v * (1 + 1j))
    B = np.full((K, 96), v * (1 - 1j))
    C = ctx.matmul(dev(A), dev(B)).cpu().numpy()
    want = Fraction(2 * K * F * F, 2 ** 110)
    assert np.all(C == C[0, 0]) and C[0, 0].imag == 0.0
    assert abs(Fraction(float(C[0, 0].real)) - want) <= Fraction(32 * K, 2 ** 53)


def test_value_does_not_depend_on_the_split(ctx):
    g = synth.rng(9)
    A, B = synth.complex_gaussian(g, (1100, 900)), synth.complex_gaussian(g, (900, 1300))
    whole = ctx.matmul(dev(A), dev(B))
    part = ctx.matmul(dev(A[:70]), dev(B[:, :90]))  # few tiles: K is split
    assert torch.equal(whole[:70, :90], part)


def test_non_finite_rows_stay_apart(ctx):
    g = synth.rng(10)
    A, B = synth.complex_gaussian(g, (200, 300)), synth.complex_gaussian(g, (300, 150))
    ref = ctx.matmul(dev(A), dev(B)).cpu().numpy()
    A[3, 17], A[100, 5], B[299, 149] = np.inf, complex(0.0, np.nan), complex(-np.inf, 1.0)
    C = ctx.matmul(dev(A), dev(B)).cpu().numpy()
    bad = np.zeros(C.shape, dtype=bool)
    bad[[3, 100], :], bad[:, 149] = True, True
    assert np.all(np.isnan(C[bad].real)) and np.all(np.isnan(C[bad].imag))
    assert np.array_equal(C[~bad], ref[~bad])
