"""States of a few modes from their covariance: one pivot block of the sweep (up to 8 modes) and just
beyond, where the launches around it are the cost."""
import numpy as np
import pytest

import gbs_inputs as gi
import oracle
import paper_1810_00900_gb300 as gbs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    from paper_1810_00900_gb300 import build
    build.build()
    c = gbs.Context(0)
    yield c
    c.close()


@pytest.mark.parametrize("M", [1, 2, 3, 7, 8, 9, 16, 17])
def test_state_from_covariance(ctx, M):
    p = gi.uniform_squeezed_state(M, 0.8, seed=M, eta=0.7)
    V = oracle.covariance(p.U, p.r, p.eta)
    gbs.state_from_V(ctx, V).free()
    before = ctx.launch_count
    st = gbs.state_from_V(ctx, V)
    # Sigma, the pivot block, the negated inverse, the determinant; panel and update per further block
    assert ctx.launch_count - before <= (4 if M <= 8 else 4 + 2 * ((2 * M + 15) // 16))
    S = oracle.sigma(V)
    assert abs(st.logdet_sigma - oracle.logdet_sigma(S)) <= 1e-13 * 2 * M
    modes = list(range(M))[:20]
    want = oracle.sigma_inv_block(S, modes)
    # sweep of a matrix with condition number below 10: some units per pivot
    assert np.abs(gbs.sigma_inv_block(ctx, st, modes) - want).max() <= 2 * M * 10 * 2.0 ** -52 * np.abs(want).max()
    st.free()


def test_bad_covariances_are_refused_whatever_their_size(ctx):
    for M in (1, 8, 9):
        V = np.eye(2 * M, dtype=complex)
        for bad, status in ((np.nan, 1), (np.inf, 1), (-0.6, 3)):
            W = V.copy()
            W[M, M] = bad
            with pytest.raises(gbs.GbsError) as e:
                gbs.state_from_V(ctx, W)
            assert e.value.status == status, (M, bad)
