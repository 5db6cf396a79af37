"""The fixed-point tree engine where its index arithmetic can go wrong: trees smaller than a tile
of 32 nodes, one level and one tile more, every depth of the top kernel, batches of uneven trees,
and a tree taken in chunks because its levels exceed the context's budget.  Sums are exact, so
every launch shape and split gives the same bits."""
import threading

import numpy as np
import pytest

import gbs_inputs as gi
import oracle
import paper_1810_00900_gb300 as gbs
from helpers import frac3, oracle_tor, real_basis_block

pytestmark = pytest.mark.gpu

# model units of tests/test_gpu_tree.py: |Tor - exact| <= 8 n u sum|terms|
U_OF = {"fxn": 2.0 ** -108, "fx": 2.0 ** -140, "fxw": 2.0 ** -158}


@pytest.fixture(scope="module")
def ctx():
    from paper_1810_00900_gb300 import build
    build.build()
    c = gbs.Context(0)
    yield c
    c.close()


def block(n, seed, r=0.7, eta=0.8):
    st = gi.uniform_squeezed_state(80, r, seed=seed, eta=eta)
    Sig = oracle.sigma(oracle.covariance(st.U, st.r, st.eta))
    return real_basis_block(oracle.sigma_inv_block(Sig, gi.random_modes(80, n, seed=seed)))


@pytest.mark.parametrize("prec", ["fxn", "fx", "fxw"])
@pytest.mark.parametrize("n", [1, 2, 3, 4, 7, 8, 9, 10, 12])
def test_shapes_give_the_oracles_value_and_the_same_bits(ctx, prec, n):
    G = block(n, 40 + n)
    ref, ref_abs = oracle_tor(G)
    seen = set()
    for d_top in (0, 6, 7, 10):
        for q_drop in (0, 1, 2):
            ctx.set_tuning(prec, "real", 6, d_top, 0, 1 << 18, q_drop, 0)
            inc, exc, tor, a = gbs.subset_sum(ctx, G, "real", prec)
            seen.add((tuple(inc), tuple(exc), tuple(tor), a))
            assert abs(float(frac3(tor) - ref.to_fraction())) <= 8 * n * U_OF[prec] * ref_abs
            assert abs(a - ref_abs) <= 1e-12 * ref_abs
    ctx.set_tuning(prec, "real", 6, 10, 0, 1 << 18, 0, 0)
    assert len(seen) == 1


def test_uneven_batch_gives_each_trees_own_bits(ctx):
    st_p = gi.uniform_squeezed_state(60, 0.7, seed=3, eta=0.7)
    st = gbs.build_state(ctx, st_p.U, st_p.r, st_p.eta)
    pats = [gi.random_modes(60, n, seed=100 + i) for i, n in enumerate([9, 1, 14, 2, 8, 3, 11, 9, 1, 16, 5, 7])]
    alone = [gbs.torontonian(ctx, st, p, "fx") for p in pats]
    for p, a, b in zip(pats, alone, gbs.torontonian_batch(ctx, [st] * len(pats), pats, "fx")):
        assert a.tor == b.tor and a.abs_sum == b.abs_sum, len(p)
    st.free()


@pytest.mark.parametrize("prec", ["fp64", "fxn", "fx", "fxw"])
def test_one_launch_and_level_paths_agree(ctx, prec):
    # alone, trees of up to 16 modes take one launch (one CTA up to 9 or 10 modes, several
    # beyond); among enough others they go by levels: the same bits
    st_p = gi.uniform_squeezed_state(60, 0.7, seed=5, eta=0.7)
    st = gbs.build_state(ctx, st_p.U, st_p.r, st_p.eta)
    pats = [gi.random_modes(60, n, seed=300 + n) for n in range(1, 17)]
    many = pats + [gi.random_modes(60, 12, seed=400 + i) for i in range(120)]
    for p, b in zip(pats, gbs.torontonian_batch(ctx, [st] * len(many), many, prec)):
        a = gbs.torontonian(ctx, st, p, prec)
        assert a.tor == b.tor and a.abs_sum == b.abs_sum and a.p == b.p, len(p)
    st.free()


@pytest.mark.parametrize("n", [3, 8, 10, 11, 13, 17])
def test_fp64_of_a_bounded_state_is_no_worse_than_its_estimate(ctx, n):
    # FP64 trees of bounded states run in 64-bit fixed point; bright states, where FP64 carries
    # the cancellation: within the FP64 error model of the exact value of the same block, and
    # as close to it as the FP64 pipe's own tree (gbs_subset_sum on the block) or 1e-13
    st_p = gi.uniform_squeezed_state(n + 1, 1.4, seed=60 + n, eta=0.9)
    st = gbs.build_state(ctx, st_p.U, st_p.r, st_p.eta)
    modes = gi.random_modes(n + 1, n, seed=n)
    G = gbs.sigma_inv_block(ctx, st, modes, "real")
    ref, ref_abs = oracle_tor(G)
    want = float(ref.to_fraction())
    pr = gbs.torontonian(ctx, st, modes, "fp64", "real")
    err = abs(float(frac3(pr.tor) - ref.to_fraction()))
    assert err <= (4 * n + 24) * 2.0 ** -53 * ref_abs
    _, _, tor, _ = gbs.subset_sum(ctx, G, "real", "fp64")
    assert err <= max(abs(float(frac3(tor) - ref.to_fraction())), 1e-13 * abs(want))
    assert abs(pr.abs_sum - ref_abs) <= 1e-12 * ref_abs
    st.free()


@pytest.mark.parametrize("prec", ["fxn", "fx", "fxw"])
def test_chunks_of_a_tree_beyond_the_budget(ctx, prec):
    # 18 modes (beyond the trees that run in one launch) need ~40 MB of levels at once; half
    # of a budget of 24 and 40 MB makes chunks
    G = block(18, 77)
    want = gbs.subset_sum(ctx, G, "real", prec)
    for budget in (24 << 20, 40 << 20):
        for d_top in (6, 10):
            c = gbs.Context(0, hbm_budget_bytes=budget)
            c.set_tuning(prec, "real", 6, d_top, 0, 1 << 18, 0, 0)
            got = gbs.subset_sum(c, G, "real", prec)
            assert all(tuple(np.atleast_1d(x)) == tuple(np.atleast_1d(y)) for x, y in zip(want, got))
            assert c.launch_count > 15 and c.bytes_in_use <= budget
            c.close()


@pytest.mark.parametrize("dense", [False, True])
@pytest.mark.parametrize("M", [1, 2, 15, 16, 17, 33, 66])
def test_many_requests_get_the_roots_of_each_alone(ctx, M, dense):
    """Enough requests for a CTA each: the bits of a few of them alone, whose mode pairs are
    spread over lanes."""
    p = gi.uniform_squeezed_state(M, 0.5, seed=M, eta=0.8)
    st = gbs.build_state(ctx, p.U, p.r, p.eta)
    if dense:
        st.free()
        st = gbs.state_from_V(ctx, oracle.covariance(p.U, p.r, p.eta))
    rng = np.random.default_rng(M)
    pats = [rng.permutation(M)[:rng.integers(1, min(M, 20 if i < 4 else 9) + 1)] for i in range(640)]
    many = gbs.torontonian_batch(ctx, [st] * len(pats), pats, "fp64")
    for i in list(range(4)) + [5, 639]:
        for basis in ("real", "complex"):
            a = gbs.torontonian(ctx, st, pats[i], "fp64", basis)
            b = many[i] if basis == "real" else gbs.torontonian_batch(ctx, [st] * 320, [pats[i]] * 320, "fp64", basis)[7]
            assert (a.tor, a.abs_sum, a.p) == (b.tor, b.abs_sum, b.p), (len(pats[i]), basis)
    st.free()


def test_threads_with_trees_of_different_sizes_at_once():
    """Four contexts in four threads, each with trees of other sizes in turn: the same kernels launched
    with different amounts of shared memory at the same time give every thread its own results."""
    p = gi.uniform_squeezed_state(40, 0.8, seed=5, eta=0.8)
    sizes = [1, 3, 6, 8, 9, 10, 12, 14]

    def run(ctx, order):
        st = gbs.build_state(ctx, p.U, p.r, p.eta)
        out = {}
        for _ in range(6):
            for prec in ("fp64", "fx", "dd"):
                for n in order:
                    out[n, prec] = gbs.torontonian(ctx, st, gi.random_modes(40, n, n), prec).tor
        st.free()
        return out

    with gbs.Context(0) as ctx:
        ref = run(ctx, sizes)
    got = [None] * 4

    def work(i):
        with gbs.Context(0) as ctx:
            got[i] = run(ctx, sizes[2 * i:] + sizes[:2 * i])

    ts = [threading.Thread(target=work, args=(i,)) for i in range(4)]
    [t.start() for t in ts]
    [t.join() for t in ts]
    assert all(g == ref for g in got)


@pytest.mark.parametrize("M", [30, 230])
@pytest.mark.parametrize("n", [1, 3, 20, 40, 80])
def test_sampler_steps_give_the_same_bits_with_any_number_of_trajectories(ctx, M, n):
    """1, 2, 4 or 8 CTAs condition a trajectory, by how many there are: sample 0's bits alone and
    among n."""
    p = gi.uniform_squeezed_state(M, 0.6, seed=M, eta=0.8)
    st = gbs.build_state(ctx, p.U, p.r, p.eta)
    clicks = [sorted(np.random.default_rng(i).permutation(M)[:6].tolist()) for i in range(n)]
    one = gbs.sample(ctx, st, 1, 9, 6, 1, forced_clicks=clicks[:1], want_p0=True)
    many = gbs.sample(ctx, st, n, 9, 6, 1, forced_clicks=clicks, want_p0=True)
    assert np.array_equal(one[0][0], many[0][0]) and np.array_equal(one[1][0], many[1][0])
    st.free()
