"""Trees of the fixed-point engine where the context has less memory left than their workspace's limit:
the same bits in smaller chunks, or a part of the batch at a time."""
import numpy as np
import pytest

import gbs_inputs as gi
import paper_1810_00900_gb300 as gbs

pytestmark = pytest.mark.gpu

MB = 1 << 20


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_1810_00900_gb300 import build
    build.build()


def small_state(ctx):
    p = gi.uniform_squeezed_state(40, 0.8, seed=5, eta=0.9)
    return gbs.build_state(ctx, p.U, p.r, p.eta)


def crowded(budget, left):
    """A context of which other states hold all but `left` bytes."""
    ctx = gbs.Context(0, hbm_budget_bytes=budget)
    st = small_state(ctx)
    gbs.torontonian(ctx, st, [0, 1, 2], "fx")  # the arenas every call needs
    M = int(((budget - left - ctx.bytes_in_use) / 16) ** 0.5)
    other = gbs.build_state(ctx, np.eye(M, dtype=complex), np.full(M, 0.1), 1.0)
    return ctx, st, other


# levels of one tree of 18 modes: 16 MB with 64 fraction bits, 33, 39 and 46 MB with 128, 160 and 192
@pytest.mark.parametrize("prec", ["fp64", "fxn", "fx", "fxw"])
@pytest.mark.parametrize("left", [28 * MB, 12 * MB])
def test_a_tree_takes_the_chunks_that_fit_what_is_left(prec, left):
    modes = gi.random_modes(40, 18, 3)
    with gbs.Context(0) as ctx:
        want = gbs.torontonian(ctx, small_state(ctx), modes, prec)
    ctx, st, other = crowded(120 * MB, left)
    got = gbs.torontonian(ctx, st, modes, prec)
    assert (got.tor, got.abs_sum, got.p) == (want.tor, want.abs_sum, want.p)
    assert ctx.bytes_in_use <= 120 * MB
    ctx.close()


@pytest.mark.parametrize("prec", ["fp64", "fx"])
def test_a_batch_goes_in_the_parts_that_fit_what_is_left(prec):
    # 18-mode trees of 16 and 39 MB beside small ones, 54 of 60 MB of the limit at once
    modes = [gi.random_modes(40, n, 7 + i) for i, n in enumerate([18, 9, 3, 17, 12, 1] if prec == "fx"
                                                                  else [18, 9, 18, 3, 18, 12])]
    with gbs.Context(0) as ctx:
        st = small_state(ctx)
        want = [gbs.torontonian(ctx, st, m, prec) for m in modes]
    ctx, st, other = crowded(120 * MB, 24 * MB)
    for a, b in zip(want, gbs.torontonian_batch(ctx, [st] * len(modes), modes, prec)):
        assert (a.tor, a.abs_sum, a.p) == (b.tor, b.abs_sum, b.p)
    assert ctx.bytes_in_use <= 120 * MB
    ctx.close()


def test_fp64_without_room_for_a_chunk_runs_in_floating_point():
    # 20 modes: chunks of 64-bit trees need 5 MB, the floating-point engine 2
    modes = gi.random_modes(40, 20, 3)
    with gbs.Context(0) as ctx:
        want = gbs.torontonian(ctx, small_state(ctx), modes, "fp64")
    ctx, st, other = crowded(120 * MB, 4 * MB)
    got = gbs.torontonian(ctx, st, modes, "fp64")
    assert abs(got.p - want.p) <= got.err_bound + want.err_bound
    ctx.close()
