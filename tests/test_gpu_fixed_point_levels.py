"""The fixed-point engine's top, level and leaf kernels under every shape they take: trees too large
for one launch, and smaller ones among so many that they go by levels.  (Alone, trees of up to 17 modes
take one launch, on which a shape does not act.)  Sums are exact: the same bits whatever the shape."""
import numpy as np
import pytest

import gbs_inputs as gi
import paper_1810_00900_gb300 as gbs
from helpers import frac3, oracle_tor

pytestmark = pytest.mark.gpu

# precision -> (name of its launch shape, unit of the error model |Tor - exact| <= 4 n u sum|terms|)
TYPES = {"fp64": ("fp64_fixed", 2.0 ** -53), "fxn": ("fxn", 2.0 ** -108), "fx": ("fx", 2.0 ** -140),
         "fxw": ("fxw", 2.0 ** -158)}
SHAPES = [(d_top, q_drop) for d_top in (0, 6, 7, 10) for q_drop in (0, 1, 2)]


@pytest.fixture(scope="module")
def ctx():
    from paper_1810_00900_gb300 import build
    build.build()
    c = gbs.Context(0)
    yield c
    c.close()


@pytest.fixture(scope="module")
def state(ctx):
    p = gi.uniform_squeezed_state(60, 0.7, seed=3, eta=0.8)
    return gbs.build_state(ctx, p.U, p.r, p.eta)


def bits(r):
    return r.tor, r.abs_sum, r.p


@pytest.mark.parametrize("prec", TYPES)
@pytest.mark.parametrize("n", [18, 19])
def test_trees_beyond_one_launch(ctx, state, prec, n):
    shape, u = TYPES[prec]
    modes = gi.random_modes(60, n, 5 + n)
    ref, ref_abs = oracle_tor(gbs.sigma_inv_block(ctx, state, modes, "real"))
    seen, launches = set(), set()
    for d_top, q_drop in SHAPES:
        ctx.set_tuning(shape, "real", 6, d_top, 0, 1 << 18, q_drop, 0)
        before = ctx.launch_count
        r = gbs.torontonian(ctx, state, modes, prec, "real")
        launches.add(ctx.launch_count - before)
        seen.add(bits(r))
        # (two closed-form evaluations of the block differ by some 2^-52 of an entry)
        assert abs(float(frac3(r.tor) - ref.to_fraction())) <= 8 * n * max(u, 2.0 ** -50) * ref_abs
    ctx.set_tuning(shape, "real", 6, 10, 0, 1 << 18, 0, 0)
    assert len(seen) == 1
    assert min(launches) > 8 and len(launches) >= 4  # click block, top, levels, leaf, final; by shape


@pytest.mark.parametrize("prec", ["fxn", "fx", "fxw"])
@pytest.mark.parametrize("d_top,q_drop", [(0, 2), (6, 1), (7, 0), (10, 2)])
def test_the_same_matrix_as_the_oracle(ctx, state, prec, d_top, q_drop):
    # subset_sum takes the very matrix that the oracle is given: the type's own error model
    n = 18
    G = gbs.sigma_inv_block(ctx, state, gi.random_modes(60, n, 5 + n), "real")
    ref, ref_abs = oracle_tor(G)
    ctx.set_tuning(prec, "real", 6, d_top, 0, 1 << 18, q_drop, 0)
    _, _, tor, a = gbs.subset_sum(ctx, G, "real", prec)
    ctx.set_tuning(prec, "real", 6, 10, 0, 1 << 18, 0, 0)
    assert abs(float(frac3(tor) - ref.to_fraction())) <= 8 * n * TYPES[prec][1] * ref_abs
    assert abs(a - ref_abs) <= 1e-12 * ref_abs


@pytest.mark.parametrize("prec", TYPES)
def test_small_trees_among_many(ctx, state, prec):
    shape, _ = TYPES[prec]
    pats = [gi.random_modes(60, n, 30 + n) for n in range(1, 18)]
    many = pats + [gi.random_modes(60, 12, 100 + i) for i in range(60)]
    alone = [bits(gbs.torontonian(ctx, state, p, prec, "real")) for p in pats]
    launches = set()
    for d_top, q_drop in SHAPES:
        ctx.set_tuning(shape, "real", 6, d_top, 0, 1 << 18, q_drop, 0)
        before = ctx.launch_count
        got = gbs.torontonian_batch(ctx, [state] * len(many), many, prec, "real")
        launches.add(ctx.launch_count - before)
        assert [bits(g) for g in got[:len(pats)]] == alone, (d_top, q_drop)
    ctx.set_tuning(shape, "real", 6, 10, 0, 1 << 18, 0, 0)
    # levels; q_drop shows in the launches, d_top is at its least in so large a batch
    assert min(launches) > 8 and len(launches) >= 2
