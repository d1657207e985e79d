"""Products of results where the device has no room for split operands: they run
on FMAs, as a plan that is not one of results, and every call still gives its
values.  The room is bounded by a limit on the plans' buffers."""
import numpy as np
import pytest

from gbd_synth import make_integrals

pytestmark = pytest.mark.gpu


@pytest.fixture()
def ctx():
    from paper_2609_09990_gb300 import build, gbdmrg
    build.build()
    c = gbdmrg.Context(0)
    yield c
    c.close()


@pytest.mark.parametrize("M,N,K,terms", [(64, 64, 32, 1), (130, 70, 1000, 1), (40, 50, 33, 9)])
def test_without_room_the_product_is_the_fma_one(ctx, M, N, K, terms):
    rng = np.random.default_rng(M)
    A, B, C0 = rng.normal(size=(terms, M, K)), rng.normal(size=(terms, K, N)), rng.normal(size=(M, N))
    fma, split = ctx.gemm_f64(A, B, 0, -0.7, C0), ctx.gemm_f64(A, B, 4, -0.7, C0)
    assert not np.array_equal(fma, split)
    for limit in (0, 1 << 12):
        ctx.set_split_limit(limit)
        assert np.array_equal(ctx.gemm_f64(A, B, 4, -0.7, C0), fma)
    ctx.set_split_limit(1 << 62)
    assert np.array_equal(ctx.gemm_f64(A, B, 4, -0.7, C0), split)


def test_calls_without_room(ctx):
    n = 10
    h, chol = make_integrals(n, 20, 4)
    ctx.solve(h, chol, n, 0, [96] * 2, [1e-6] * 2, seed=4)
    x = np.random.default_rng(1).normal(size=ctx.two_site_size(0))

    def values():
        g1, g2 = ctx.rdms(n)
        return [g1, g2, ctx.rdm3(n), ctx.orbital_entropies(n)[1], ctx.apply_heff(0, x), np.array(ctx.final_energy())]
    have = values()
    for limit in (0, 1 << 20):   # no plan, and none of the larger ones
        ctx.set_split_limit(limit)
        for a, b in zip(values(), have):
            assert np.abs(a - b).max() <= 1e-11 * max(1.0, np.abs(b).max())


def test_negative_limits_are_refused(ctx):
    from paper_2609_09990_gb300 import gbdmrg
    with pytest.raises(gbdmrg.GbdError, match="GBD_ERR_ARG"):
        ctx.set_split_limit(-1)
