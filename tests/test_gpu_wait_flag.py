"""A wait that ran out is reported by one call, and the context's next calls
run: the flags are raised as the kernels raise them, no wait runs out."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("sigma", [0, 1])
def test_context_survives_a_reported_timeout(sigma):
    from gbd_synth import make_integrals
    from paper_2609_09990_gb300 import build, gbdmrg
    build.build()
    ctx = gbdmrg.Context(0)
    rng = np.random.default_rng(2)
    A, B = rng.normal(size=(1, 80, 64)), rng.normal(size=(1, 64, 72))
    want = ctx.gemm_f64(A, B, 4)
    h, chol = make_integrals(6, 8, 1)
    solve = lambda: ctx.solve(h, chol, 6, 0, [64] * 2, [1e-8] * 2, seed=1, precision=2)["energy"]
    ctx.set_tc_min_two_site(0)
    energy = solve()
    for _ in range(2):
        with pytest.raises(gbdmrg.GbdError, match="GBD_ERR_TIMEOUT"):
            ctx.wait_flag_selftest(sigma)
        assert np.array_equal(ctx.gemm_f64(A, B, 4), want)
        assert solve() == energy
    ctx.close()


def test_other_values_are_refused():
    from paper_2609_09990_gb300 import build, gbdmrg
    build.build()
    ctx = gbdmrg.Context(0)
    with pytest.raises(gbdmrg.GbdError, match="GBD_ERR_ARG"):
        ctx.wait_flag_selftest(2)
    ctx.close()
