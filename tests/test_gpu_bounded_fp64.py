"""FP64 trees in 64-bit fixed point at the limits of what the engine takes: states with sigma_max just
below 16 (and just beyond, where the floating-point engine takes over), n log2(1 + sigma_max) on both
sides of 92, and sampler trees with sigma_max near 64."""
import math

import numpy as np
import pytest

import gbs_inputs as gi
import paper_1810_00900_gb300 as gbs
from helpers import frac3

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    from paper_1810_00900_gb300 import build
    build.build()
    c = gbs.Context(0)
    yield c
    c.close()


def bright(ctx, M, sigma_max, seed):
    """A pure state with the given largest eigenvalue (e^2r + 1) / 2 of Sigma."""
    return gbs.build_state(ctx, gi.haar_unitary(M, seed), np.full(M, 0.5 * math.log(2 * sigma_max - 1)), 1.0)


def launches(ctx, f):
    before = ctx.launch_count
    r = f()
    return r, ctx.launch_count - before


def check(ctx, st, modes):
    n = len(modes)
    # triple-double on the same block, u = 2^-152: exact for this purpose
    ref = gbs.torontonian(ctx, st, modes, "td", "real")
    exact = frac3(ref.tor)
    got = gbs.torontonian(ctx, st, modes, "fp64", "real")
    err = abs(float(frac3(got.tor) - exact))
    assert err <= (4 * n + 24) * 2.0 ** -53 * ref.abs_sum  # what err_bound promises
    assert abs(got.abs_sum - ref.abs_sum) <= 1e-12 * ref.abs_sum
    assert got.err_bound <= (4 * n + 24) * 2.0 ** -53 * ref.abs_sum * math.exp(-0.5 * st.logdet_sigma) * (1 + 1e-9)
    # and no further off than the floating-point engine's tree over the same block, or 2^-53 a term
    _, _, tor, _ = gbs.subset_sum(ctx, gbs.sigma_inv_block(ctx, st, modes, "real"), "real", "fp64")
    assert err <= max(abs(float(frac3(tor) - exact)), 2.0 ** -53 * ref.abs_sum)
    return got


@pytest.mark.parametrize("n", [4, 9, 12, 17, 18, 20, 22])
@pytest.mark.parametrize("extra", [0, 2])
def test_sigma_max_just_below_16(ctx, n, extra):
    st = bright(ctx, n + extra, 15.99, 7 * n)
    check(ctx, st, gi.random_modes(n + extra, n, n))
    st.free()


@pytest.mark.parametrize("n", [6, 14, 18])
def test_either_side_of_sigma_max_16(ctx, n):
    # the same unitary and pattern just below and just beyond: two engines (by their launches),
    # values that continue one another
    below, beyond = bright(ctx, n + 1, 15.9999, n), bright(ctx, n + 1, 16.0001, n)
    modes = gi.random_modes(n + 1, n, n)
    a, la = launches(ctx, lambda: gbs.torontonian(ctx, below, modes, "fp64", "real"))
    b, lb = launches(ctx, lambda: gbs.torontonian(ctx, beyond, modes, "fp64", "real"))
    assert la != lb
    check(ctx, below, modes)
    check(ctx, beyond, modes)
    # d log p / d sigma_max is of order n
    assert abs(math.log(a.p / b.p)) <= 2e-4 * 4 * n
    below.free()
    beyond.free()


@pytest.mark.parametrize("sigma_max,bounded", [(14.99, True), (15.02, False)])
def test_either_side_of_the_sums_range(ctx, sigma_max, bounded):
    # 23 log2(1 + sigma_max) = 91.98 and 92.04: s and the sums have 95 integer bits
    n = 23
    assert (n * math.log2(1 + sigma_max) < 92) == bounded
    st = bright(ctx, n, sigma_max, 5)
    got = gbs.torontonian(ctx, st, list(range(n)), "fp64", "real")
    ref = gbs.torontonian(ctx, st, list(range(n)), "td", "real")
    err = abs(float(frac3(got.tor) - frac3(ref.tor)))
    assert err <= (4 * n + 24) * 2.0 ** -53 * ref.abs_sum
    assert abs(got.abs_sum - ref.abs_sum) <= 1e-12 * ref.abs_sum
    st.free()


@pytest.mark.parametrize("sigma_max", [40.0, 63.9, 64.1])
def test_sampler_near_sigma_max_64(ctx, sigma_max):
    # forced clicks, so that FP64 trees of up to 10 modes of the brightest admitted state are
    # formed; certified steps are within 5e-10 of the exact p0, as triple-double's are
    M = 14
    st = bright(ctx, M, sigma_max, 3)
    clicks = [sorted(gi.random_modes(M, 9, s)) for s in range(4)]
    out = {p: gbs.sample(ctx, st, 4, 9, 9, 1, forced_clicks=clicks, prec=p, want_p0=True) for p in ("auto", "fp64", "td")}
    for p in ("auto", "td"):
        assert out[p][2]["uncertified"] == 0
    assert np.abs(out["auto"][1] - out["td"][1]).max() <= 1e-9
    # FP64 by itself: its steps are certified or counted
    if out["fp64"][2]["uncertified"] == 0:
        assert np.abs(out["fp64"][1] - out["td"][1]).max() <= 1e-9
    st.free()
