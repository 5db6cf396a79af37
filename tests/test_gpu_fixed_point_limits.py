"""The fixed-point tree engine at the limits of what it takes: matrices with large entries (states
given by a covariance that promises Sigma > 0 only)."""
import numpy as np
import pytest

import oracle
import paper_1810_00900_gb300 as gbs
from helpers import frac3, oracle_tor

pytestmark = pytest.mark.gpu

GBS_EPRECISION = 4
# units of the error model |Tor - exact| <= 4 n u sum|terms|
U_OF = {"fxn": 2.0 ** -108, "fx": 2.0 ** -140, "fxw": 2.0 ** -158}


@pytest.fixture(scope="module")
def ctx():
    from paper_1810_00900_gb300 import build
    build.build()
    c = gbs.Context(0)
    yield c
    c.close()


def covariance_of_inverse(H):
    """The covariance V (block order) of a state with Sigma^-1 = H in the real x/p basis."""
    n = H.shape[0] // 2
    Q = np.kron(np.eye(n), np.array([[1, 1j], [1, -1j]]) / np.sqrt(2))
    S = Q @ np.linalg.inv(H) @ Q.conj().T
    order = np.concatenate([np.arange(0, 2 * n, 2), np.arange(1, 2 * n, 2)])
    V = S[np.ix_(order, order)] - 0.5 * np.eye(2 * n)
    return 0.5 * (V + V.conj().T)


def spiked(n, c, w, seed):
    """c I + w v v^T over the first two modes, whose 2 x 2 determinants are c^2 + c w / 2 from entries
    of order w / 4; the others well conditioned, with couplings of order 0.1 among them."""
    rng = np.random.default_rng(seed)
    H = np.diag(rng.uniform(0.8, 1.2, 2 * n))
    H += 0.1 * (lambda x: (x + x.T) / 2)(rng.uniform(-1, 1, (2 * n, 2 * n)))
    H[:4] = H[:, :4] = 0.0
    H[:4, :4] = c * np.eye(4)
    v = np.zeros(2 * n)
    v[:4] = 0.5, -0.5, 0.5, 0.5
    return H + w * np.outer(v, v)


@pytest.mark.parametrize("prec", ["fxn", "fx", "fxw"])
@pytest.mark.parametrize("n,c,w", [(2, 0.9, 1500.0), (3, 0.9, 1500.0), (2, 0.9, 3000.0), (6, 0.9, 3000.0),
                                   (12, 0.9, 3000.0), (18, 0.9, 3000.0), (2, 0.05, 6e4), (6, 0.05, 6e4)])
def test_entries_far_beyond_those_of_a_physical_state(ctx, prec, n, c, w):
    # entries of Sigma^-1 up to w / 4 in magnitude, of both signs, while every pivot's
    # determinant stays within the types' range
    st = gbs.state_from_V(ctx, covariance_of_inverse(spiked(n, c, w, n)))
    modes = list(range(n))
    G = gbs.sigma_inv_block(ctx, st, modes, "real")
    assert np.abs(G).max() > 0.2 * w and G.min() < -0.2 * w
    ref, ref_abs = oracle_tor(G)
    pr = gbs.torontonian(ctx, st, modes, prec)
    # entries are held to 2^-32F of one unit; a determinant is the difference of products of
    # order (w/4)^2, so the model's unit is scaled by that over the determinant (1 at least)
    scale = max(1.0, (w / 4) ** 2 / (c * c + c * w / 2))
    assert abs(float(frac3(pr.tor) - ref.to_fraction())) <= 8 * n * U_OF[prec] * scale * ref_abs
    st.free()


@pytest.mark.parametrize("prec", ["fxn", "fx", "fxw"])
@pytest.mark.parametrize("n,c", [(2, 0.01), (6, 0.01), (18, 0.2)])
def test_matrices_whose_determinants_would_wrap_are_refused(ctx, prec, n, c):
    # a mode's diagonal entries multiply to 2^33: the determinant cannot be checked
    st = gbs.state_from_V(ctx, covariance_of_inverse(spiked(n, c, 4 * 2.0 ** 16.5, n)))
    with pytest.raises(gbs.GbsError) as e:
        gbs.torontonian(ctx, st, list(range(n)), prec)
    assert e.value.status == GBS_EPRECISION
    st.free()
