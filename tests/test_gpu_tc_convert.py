"""Operand conversion (turned in shared memory up to 256 rows, in chunks of
columns) and split-K sums of the tensor-core GEMM at their edges, against the
FP64 grouped GEMM."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    from paper_2609_09990_gb300 import build, gbdmrg
    build.build()
    return gbdmrg.Context(0)


# M, N, K, terms: one row and column; blocks of 17 x 119 and 120 (one chunk of
# columns and one more), 255 to 257 rows (the last that is turned, and not),
# chunks of a few columns; 1 to 17 slots of 512 columns, also 8, 9 and 16
@pytest.mark.parametrize("shape", [(1, 1, 1, 1), (17, 17, 119, 1), (17, 16, 120, 3), (255, 256, 40, 2), (257, 255, 33, 1),
                                   (256, 257, 7, 5), (200, 33, 512, 8), (31, 200, 513, 3), (129, 20, 512 * 9, 1),
                                   (20, 140, 512 * 16 + 1, 1)])
@pytest.mark.parametrize("flags", [0, 1, 2, 3])
@pytest.mark.parametrize("prec", [3, 4])
def test_conversion_and_sums(ctx, shape, flags, prec):
    M, N, K, nt = shape
    err, ref = ctx.gemm_tc_selftest(M, N, K, nt, flags, prec, seed=M + 3 * N + 5 * K + flags)
    # operands are hi + lo within 2^-21 (TF32x3) or 2^-16 (BF16x3) of each
    # element and lo * lo is left out (2^-22, 2^-16): at most three such terms
    # a product, independent over K * nt products of normal entries, six
    # standard deviations; FP32 accumulation adds 2e-6 of the scale per 512
    rel = 6 * 3 * (2.0 ** -21 if prec == 3 else 2.0 ** -16) + 2e-6
    scale = max(ref, (K * nt) ** 0.5)
    assert err <= rel * scale, (err, ref)
