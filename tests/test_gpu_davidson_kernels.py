"""The fused kernels of a Davidson iteration against the separate vector
kernels: a subspace limit above 32 takes the latter, and with fewer
iterations than either limit both solves run the same arithmetic, so sweep
energies and RDMs agree bit for bit.  The two-site vectors run from 4 elements
at the chain ends over 65536 (64 reduction blocks, up to where the last CTA
adds the parts) to 88,000."""
import numpy as np
import pytest

from gbd_synth import make_integrals

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def G():
    from paper_2609_09990_gb300 import build, gbdmrg
    build.build()
    return gbdmrg


@pytest.mark.parametrize("n,ne,two_sz,M,precision,iters", [(2, 2, 0, 4, 0, 15), (5, 5, 1, 20, 0, 15),
                                                          (9, 9, 1, 100, 1, 15), (12, 12, 0, 256, 0, 6)])
def test_fused_iteration_is_bit_identical(G, n, ne, two_sz, M, precision, iters):
    h, chol = make_integrals(n, 3 * n, 5)
    ctx = G.Context(0)
    got = [ctx.solve(h, chol, ne, two_sz, [M], [1e-9], rdms=n < 6, seed=3, precision=precision, max_iter=iters,
                     max_subspace=space) for space in (20, 40)]
    ctx.close()
    assert got[0]["n_matvec"] == got[1]["n_matvec"]
    assert np.array_equal(got[0]["sweep_energies"], got[1]["sweep_energies"])
    assert got[0]["energy"] == got[1]["energy"]
    if n < 6:
        assert np.array_equal(got[0]["rdm2"], got[1]["rdm2"])
