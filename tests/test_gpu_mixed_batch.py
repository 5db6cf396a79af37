"""FP64 batches whose trees run on both engines (states that bound them, and others)."""
import numpy as np
import pytest

import gbs_inputs as gi
import paper_1810_00900_gb300 as gbs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    from paper_1810_00900_gb300 import build
    build.build()
    c = gbs.Context(0)
    yield c
    c.close()


def states(ctx):
    # sigma_max 2.5 and 22.9, on either side of the 64-bit engine's limit of 16
    out = []
    for r in (0.7, 1.9):
        p = gi.uniform_squeezed_state(40, r, seed=5, eta=1.0)
        out.append(gbs.build_state(ctx, p.U, p.r, p.eta))
    return out


@pytest.mark.parametrize("sizes", [[1, 1], [3, 9, 5, 6], [12, 7, 18, 11, 2, 17], [5 + i % 9 for i in range(200)]])
def test_mixed_batch_waits_once_and_gives_each_requests_own_bits(ctx, sizes):
    dim, bright = states(ctx)
    reqs = [((dim, bright)[i % 2], gi.random_modes(40, n, 50 + i)) for i, n in enumerate(sizes)]
    sts, pats = [s for s, _ in reqs], [m for _, m in reqs]

    def waits(sts):
        gbs.torontonian_batch(ctx, sts, pats, "fp64")  # workspaces
        ctx.host_gaps()
        out = gbs.torontonian_batch(ctx, sts, pats, "fp64")
        return out, ctx.host_gaps()[1]

    got, n = waits(sts)
    assert n == waits([dim] * len(sts))[1] == waits([bright] * len(sts))[1]
    for (st, m), b in list(zip(reqs, got))[:12]:
        a = gbs.torontonian(ctx, st, m, "fp64")
        assert (a.tor, a.abs_sum, a.p, a.err_bound) == (b.tor, b.abs_sum, b.p, b.err_bound)
    dim.free()
    bright.free()


@pytest.mark.parametrize("left_mb", [24, 9, 3])
def test_mixed_batch_with_little_memory_left(ctx, left_mb):
    # two workspaces at once: chunks, parts or one engine after the other where they do not fit
    dim, bright = states(ctx)
    mb = 1 << 20
    with gbs.Context(0, hbm_budget_bytes=96 * mb) as tight:
        pair = states(tight)
        gbs.torontonian_batch(tight, pair, [[0, 1], [2, 3]], "fp64")
        M = int(((96 - left_mb) * mb - tight.bytes_in_use) ** 0.5 / 4)
        gbs.build_state(tight, np.eye(M, dtype=complex), np.full(M, 0.1), 1.0)
        pats = [gi.random_modes(40, n, 9 + i) for i, n in enumerate([18, 18, 19, 17, 3, 9])]
        for i, got in enumerate(gbs.torontonian_batch(tight, pair * 3, pats, "fp64")):
            want = gbs.torontonian(ctx, (dim, bright)[i % 2], pats[i], "fp64")
            if left_mb > 3 or i % 2:  # too little for a chunk of 19 modes: floating point
                assert (got.tor, got.abs_sum, got.p) == (want.tor, want.abs_sum, want.p)
            assert abs(got.p - want.p) <= got.err_bound + want.err_bound
        assert tight.bytes_in_use <= 96 * mb
    dim.free()
    bright.free()
