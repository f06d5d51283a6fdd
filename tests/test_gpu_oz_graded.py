"""Products whose entries span decades along the summed index, at sizes from the line where the slice
products take over: what each of the two FP64 engines promises.

Slices (the default there): every entry is kept to 55 bits of its row's or column's largest one.
Per real term, 7.05 2^-56 of the two powers of two from the pairs left out and 2^-55 from the
digits' rounding, two terms per K and part: below 3 K 2^-53 sigma_i tau_j, and one rounding of the
result.  FP64 units (tnt_set_fp64_gemm): (2 K + 8) 2^-53 of the sum over absolute values, which
follows the entries however they are graded."""
import numpy as np
import pytest
import torch

from paper_1610_02244_gb300 import synth

pytestmark = pytest.mark.gpu
U = 2.0 ** -53


@pytest.fixture(scope="module")
def ctx():
    from paper_1610_02244_gb300 import build as b
    b.build()
    from paper_1610_02244_gb300 import tnt
    c = tnt.Context(0)
    yield c
    c.set_fp64_gemm(tnt.TNT_FP64_GEMM_TC)


def dev(x):
    return torch.from_numpy(np.ascontiguousarray(x)).to("cuda:0")


def above(x, axis):
    """The powers of two just above the largest real or imaginary part along the axis."""
    return 2.0 ** (np.floor(np.log2(np.maximum(np.abs(x.real), np.abs(x.imag)).max(axis))) + 1.0)


@pytest.mark.parametrize("M,N,K", [(16, 64, 400), (100, 100, 400), (128, 512, 128), (256, 1024, 64), (17, 4100, 130),
                                   (512, 2048, 24)])
@pytest.mark.parametrize("ga,gb", [(4, 0), (0, 8), (6, 6), (3, -3), (8, -8)])
def test_graded_along_k(ctx, M, N, K, ga, gb):
    g = synth.rng(M + 3 * N + 7 * K)
    x = g.permutation(np.linspace(0.0, 1.0, K))
    A = synth.complex_gaussian(g, (M, K)) * 10.0 ** (-ga * x)[None, :]
    B = synth.complex_gaussian(g, (K, N)) * 10.0 ** (-gb * x)[:, None]
    jj = np.sort(g.permutation(N)[:96])  # the reference's columns
    ld = np.longdouble
    Ar, Ai, Br, Bi = A.real.astype(ld), A.imag.astype(ld), B[:, jj].real.astype(ld), B[:, jj].imag.astype(ld)
    re, im = Ar @ Br - Ai @ Bi, Ar @ Bi + Ai @ Br
    sre, sim = abs(Ar) @ abs(Br) + abs(Ai) @ abs(Bi), abs(Ar) @ abs(Bi) + abs(Ai) @ abs(Br)
    for engine in (1, 0):
        ctx.set_fp64_gemm(engine)
        C = ctx.matmul(dev(A), dev(B)).cpu().numpy()[:, jj]
        for got, want, mag in ((C.real, re, sre), (C.imag, im, sim)):
            if engine:
                bound = 3 * K * U * above(A, 1)[:, None] * above(B[:, jj], 0)[None, :] + 1.01 * U * np.abs(want)
            else:
                bound = (2 * K + 8) * U * mag
            assert np.all(np.abs(got - want) <= bound)
