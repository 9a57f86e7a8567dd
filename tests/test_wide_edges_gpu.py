"""The wide schedule's launches per level against the per-hand kernel (level schedule), bit for bit.  Chunks
of two hands keep both from running as staged tiles: the wide handle's launch count shows that its levels
are launches of their own.  Odd hand counts (a thread's second hand missing), more hands than a block
takes, one to eight actions at a node, chance nodes, and both update orders."""
import numpy as np
import pytest

from paper_2605_19928_gb300 import capi, synth
from test_gpu_parity import _state, kuhn_random, leduc_random

pytestmark = pytest.mark.gpu

ALL_IN = synth.ALL_IN


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_2605_19928_gb300 import build as pbuild
    pbuild.build()
    capi.load()
    capi.use_torch_allocator()


def _river(hands, seed, sizes=(0.5, 1.0, ALL_IN), **kw):
    return synth.river_subgame(n_hands=hands, seed=seed, range_seed=seed + 1, bet_sizes=sizes, **kw)


def _turn(hands, seed, sizes=(1.0, ALL_IN), raises=2):
    return synth.turn_subgame(n_hands=hands, seed=seed, range_seed=seed + 1, bet_sizes=sizes, max_raises=raises)


CASES = {
    "kuhn": kuhn_random,                       # 3 hands
    "leduc": leduc_random,                     # 6 hands, chance nodes
    "no_bets": lambda: _river(7, 3, max_raises=0),
    "two_to_eight_actions": lambda: _river(45, 5, (0.33, 0.5, 0.75, 1.0, 2.0, ALL_IN), max_raises=2, stack=900.0),
    "turn_odd": lambda: _turn(41, 7),
    "turn_four_actions": lambda: _turn(65, 9, (0.5, 1.0, ALL_IN), 2),
    "two_blocks_a_node": lambda: _river(515, 11, (0.33, 0.75, 1.25, ALL_IN), max_raises=3),
    "three_blocks_a_node": lambda: _turn(1127, 13, (ALL_IN,), 1),
}


def _run(spec, schedule, variant, alternating, precision):
    opts = capi.make_opts(variant, alternating=alternating, precision=precision, schedule=schedule, chunk_hands=2)
    tree = capi.cfr_tree_create(spec, opts)
    try:
        l0 = capi.cfr_counters(tree)["kernel_launches"]
        capi.cfr_iterate(tree, 4)
        launches = (capi.cfr_counters(tree)["kernel_launches"] - l0) // 4
        state = _state(tree, 1, with_pred=variant == "pcfr+")
        expl, br = capi.cfr_exploitability(tree)
        nodes = range(capi.cfr_tree_info(tree)[0])
        state += [capi.cfr_read_values(tree, what, n, player=p) for n in nodes for p in (0, 1)
                  for what in (capi.CFR_READ_CFV, capi.CFR_READ_BR_CFV, capi.CFR_READ_AVG_REACH)]
        return state, br, launches
    finally:
        capi.cfr_tree_destroy(tree)


@pytest.mark.parametrize("precision", ["single", "pairs"])
@pytest.mark.parametrize("case", list(CASES))
@pytest.mark.parametrize("variant,alternating", [("dcfr", True), ("pcfr+", True), ("cfr+", False)])
def test_wide_levels_keep_the_bits(case, variant, alternating, precision):
    spec = CASES[case]()
    want, br_want, level = _run(spec, "level", variant, alternating, precision)
    got, br, wide = _run(spec, "wide", variant, alternating, precision)
    passes = 2 if alternating else 1
    assert level == 2 * passes and wide > 4 * passes
    for x, y in zip(got, want, strict=True):
        assert np.array_equal(x, y)
    np.testing.assert_allclose(br, br_want, rtol=1e-12, atol=1e-12 * spec.pot)  # root sums in another order


def test_trees_that_fit_a_tile_take_one_launch_a_pass():
    for schedule in ("level", "wide"):
        tree = capi.cfr_tree_create(_river(203, 15), capi.make_opts("dcfr", schedule=schedule))
        try:
            l0 = capi.cfr_counters(tree)["kernel_launches"]
            capi.cfr_iterate(tree, 3)
            assert capi.cfr_counters(tree)["kernel_launches"] - l0 == 3 * 4
        finally:
            capi.cfr_tree_destroy(tree)


@pytest.mark.parametrize("precision", ["single", "pairs"])
def test_resident_schedule_takes_these_trees(precision):
    many = tuple(0.2 * k for k in range(1, 11)) + (ALL_IN,)
    for specs in ([synth.leduc()], [_river(27, 45), synth.kuhn()], [_river(19, 41, many, max_raises=1, stack=800.0)],
                  [_river(1081, 1)]):
        tree = capi.cfr_batch_create(specs, capi.make_opts("dcfr", schedule="resident", precision=precision))
        capi.cfr_tree_destroy(tree)
