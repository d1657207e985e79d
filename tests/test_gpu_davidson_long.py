"""The fused kernels of a Davidson iteration on long two-site vectors, against
the separate vector kernels bit for bit (a subspace limit above 32 takes the
latter): more than 256 reduction blocks, whose parts one thread adds in
several rounds, and lengths on either side of the longest that the fused
kernels take (608 x 1024; 853,776 is all of CAS(12,12))."""
import numpy as np
import pytest

from gbd_synth import make_integrals

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M,above,upto", [(760, 256, 608), (1024, 608, 1 << 20)])
def test_long_vectors_are_bit_identical(M, above, upto):
    from paper_2609_09990_gb300 import build, gbdmrg
    build.build()
    n = 12
    h, chol = make_integrals(n, 36, 5)
    ctx = gbdmrg.Context(0)
    got, sizes = [], set()
    for space in (20, 40):
        ctx.setup(h, chol, n, 0, [M], [1e-9], seed=3, precision=1, max_iter=3, max_subspace=space)
        ctx.init_state()
        sizes |= {ctx.two_site_size(k) for k in range(n - 1)}
        got.append(ctx.solve(h, chol, n, 0, [M], [1e-9], seed=3, precision=1, max_iter=3, max_subspace=space))
    ctx.close()
    assert any(above * 1024 < s <= upto * 1024 for s in sizes), sorted(sizes)
    assert got[0]["n_matvec"] == got[1]["n_matvec"]
    assert np.array_equal(got[0]["sweep_energies"], got[1]["sweep_energies"])
    assert got[0]["energy"] == got[1]["energy"]
