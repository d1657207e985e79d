"""Operands of the split FP64 GEMM are rounded to nearest, whatever their sign.

Rows of 32 elements: one of magnitude 1, which fixes the row's last digit at
u = 2^-54, and 31 small ones with bits below it, all of one sign; B is ones, so
that every product keeps the digits of A.  A sum then has 31 rounding errors
uniform in +-u/2, one of the sum and one of FP64 uniform in +-2 u: standard
deviation 2.3 u, 0.29 u for the mean over 64 rows, if none is biased.
The bound is 2 u; a rounding that drops the half of one sign is off by 15 u."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("sign", [1.0, -1.0])
@pytest.mark.parametrize("flags", [4, 7])
def test_mean_error_of_one_signed_rows(sign, flags):
    from paper_2609_09990_gb300 import build, gbdmrg
    build.build()
    rng = np.random.default_rng(11)
    A = sign * rng.uniform(2.0 ** -9, 2.0 ** -8, (64, 32))
    A[:, 0] = sign
    B = np.ones((32, 64))
    ctx = gbdmrg.Context(0)
    got = ctx.gemm_f64((A.T if flags & 1 else A)[None], (B.T if flags & 2 else B)[None], flags)
    ctx.close()
    exact = A.astype(np.longdouble).sum(1)
    err = ((got[:, 0] - exact) * np.longdouble(2.0 ** 54)).astype(float)
    assert abs(err.mean()) <= 2.0, err.mean()
