"""Launch shapes act on the engine that they name: FP64 trees of bounded states have one of their own."""
import pytest

import gbs_inputs as gi
import paper_1810_00900_gb300 as gbs

pytestmark = pytest.mark.gpu

KEYS = ("sub_e", "d_top", "grid_per_sm", "level_threads", "q_drop", "mid_e")


@pytest.fixture
def ctx():
    from paper_1810_00900_gb300 import build
    build.build()
    with gbs.Context(0) as c:
        yield c


def launches(ctx, st, modes):
    before = ctx.launch_count
    pr = gbs.torontonian(ctx, st, modes, "fp64", "real")
    return ctx.launch_count - before, (pr.tor, pr.abs_sum, pr.p)


def test_each_engine_takes_its_own_shape(ctx):
    # 18 modes: levels on the fixed-point engine, where q_drop = 2 ends the leaf's own levels
    # at one mode in place of three, two launches later
    p = gi.uniform_squeezed_state(40, 0.8, seed=1)
    st = gbs.build_state(ctx, p.U, p.r, p.eta)
    modes = gi.random_modes(40, 18, 2)
    n, bits = launches(ctx, st, modes)
    for prec in ("fp64", "fxn"):
        ctx.set_tuning(prec, "real", 3, 4, 0, 1 << 17, 2, 0)
        assert launches(ctx, st, modes) == (n, bits), prec
    ctx.set_tuning("fp64_fixed", "real", 6, 10, 0, 1 << 17, 2, 0)
    assert launches(ctx, st, modes) == (n + 2, bits)
    assert ctx.tuning("fp64_fixed")["q_drop"] == 2 and ctx.tuning("fxn")["sub_e"] == 3
    # a state without the bound: the floating-point engine's
    p = gi.uniform_squeezed_state(40, 1.9, seed=1)
    hot = gbs.build_state(ctx, p.U, p.r, p.eta)
    n, _ = launches(ctx, hot, modes)
    ctx.set_tuning("fp64_fixed", "real", 6, 10, 0, 1 << 17, 0, 0)
    assert launches(ctx, hot, modes)[0] == n
    ctx.set_tuning("fp64", "real", 0, 4, 0, 1 << 17, 2, 0)
    assert launches(ctx, hot, modes)[0] != n


def test_autotune_of_fp64_reaches_both_engines(ctx):
    ctx.set_tuning("fp64_fixed", "real", 7, 16, 5, 123, 2, 8)
    rep = ctx.autotune("fp64", "real", 10)
    t = ctx.tuning("fp64_fixed")
    assert t["level_threads"] != 123 and t["d_top"] in (6, 8, 9, 10) and t["q_drop"] in (0, 1)
    assert {tuple(r[k] for k in KEYS) for r in rep} >= {tuple(ctx.tuning("fp64")[k] for k in KEYS)}
    assert 0 < len(ctx.autotune("fp64_fixed", "real", 10)) < len(rep)


def test_a_shape_is_no_precision(ctx):
    with pytest.raises(gbs.GbsError):
        ctx.set_tuning("fp64_fixed", "complex")
    with pytest.raises(gbs.GbsError):
        ctx.autotune("fp64_fixed", "complex", 10)
    p = gi.uniform_squeezed_state(4, 0.8, seed=1)
    st = gbs.build_state(ctx, p.U, p.r, p.eta)
    with pytest.raises(KeyError):
        gbs.torontonian(ctx, st, [0, 1], "fp64_fixed")
