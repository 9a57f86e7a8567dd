"""The throughput forms against the one-node terminal launch and the level schedule, bit for bit, at
full hand counts (the longest runs of a scan, ragged last tiles), on trees from one decision to
hundreds of nodes (every tile width), and at the edges of a terminal group (1 to 4 nodes) and of a
block's stretch of groups."""
import numpy as np
import pytest

from paper_2605_19928_gb300 import capi, synth
from test_gpu_parity import _state

pytestmark = pytest.mark.gpu

ALL_IN = synth.ALL_IN


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_2605_19928_gb300 import build as pbuild
    pbuild.build()
    capi.load()
    import torch
    assert torch.cuda.is_available()
    capi.use_torch_allocator()


def river(hands, seed, **kw):
    return synth.river_subgame(n_hands=hands, seed=seed, range_seed=seed + 1, **kw)


BATCHES = {
    "full_hands": lambda: [river(1081, 1), river(1081, 3, bet_sizes=(0.33, 0.75, 1.5, ALL_IN), stack=300.0)],
    # one decision (no bets: check or check down), an all-in only, a few hands, one hand past a tile
    "small_trees": lambda: [river(33, 5, max_raises=0), river(64, 7, bet_sizes=(ALL_IN,), max_raises=1), river(5, 9),
                            river(97, 11, bet_sizes=(0.5, ALL_IN), max_raises=2)],
    # the largest trees of batch_rivers and larger: narrower tiles
    "large_trees": lambda: [river(70, 13, bet_sizes=(0.33, 0.5, 0.75, 1.0, 2.0, ALL_IN), max_raises=3, stack=900.0),
                            river(70, 15, bet_sizes=(0.33, 0.5, 1.0, ALL_IN), max_raises=4, stack=1000.0), river(41, 17)],
    # chance nodes inside the tiles, run-outs below all-ins, several board tables
    "turns": lambda: [synth.turn_subgame(n_hands=37, seed=19, range_seed=20, bet_sizes=(ALL_IN,), max_raises=1),
                      synth.turn_subgame(n_hands=12, seed=21, range_seed=22, bet_sizes=(ALL_IN,), max_raises=1),
                      synth.leduc(), synth.kuhn()],
    "full_turn": lambda: [synth.turn_subgame(n_hands=1128, seed=23, range_seed=24, bet_sizes=(ALL_IN,), max_raises=1)],
}


def _solve(specs, opts):
    tree = capi.cfr_batch_create(specs, opts)
    try:
        capi.cfr_iterate(tree, 3)
        capi.cfr_iterate(tree, 2)
        capi.cfr_sync(tree)
        state = _state(tree, len(specs), with_pred=opts.variant == capi.VARIANTS["pcfr+"])
        expl, br = capi.cfr_exploitability(tree, len(specs))
        reach = [capi.cfr_read_values(tree, capi.CFR_READ_AVG_REACH, n, player=p, game=g)
                 for g in range(len(specs)) for n in range(0, capi.cfr_tree_info(tree, g)[0], 7) for p in (0, 1)]
        return state, expl, br, reach
    finally:
        capi.cfr_tree_destroy(tree)


@pytest.mark.parametrize("precision", ["single", "pairs"])
@pytest.mark.parametrize("case", list(BATCHES))
@pytest.mark.parametrize("variant,alternating", [("dcfr", True), ("pcfr+", True), ("cfr+", False), ("cfr", True)])
def test_stream_schedule_and_terminal_groups_keep_the_bits(case, variant, alternating, precision):
    specs = BATCHES[case]()
    kw = dict(alternating=alternating, precision=precision)
    want = _solve(specs, capi.make_opts(variant, schedule="level", term_nodes=1, **kw))
    for schedule, nodes in (("stream", 1), ("stream", 2), ("stream", 4), ("level", 8)):
        got = _solve(specs, capi.make_opts(variant, schedule=schedule, term_nodes=nodes, **kw))
        for x, y in zip([*got[0], got[1], got[2], *got[3]], [*want[0], want[1], want[2], *want[3]], strict=True):
            assert np.array_equal(x, y)


@pytest.mark.parametrize("precision", ["single", "pairs"])
@pytest.mark.parametrize("variant,alternating", [("dcfr", True), ("pcfr+", False), ("cfr+", True)])
def test_latency_forms_keep_the_bits(variant, alternating, precision):
    """The staged tiles (4 hands or more) and the resident schedule's phases against the per-hand
    kernel (chunks of 2 hands take it), with 12 actions at a node, and trees wider than a block."""
    many = tuple(0.2 * k for k in range(1, 11)) + (ALL_IN,)
    for specs in ([river(19, 41, bet_sizes=many, max_raises=1, stack=800.0)],
                  [river(45, 43, bet_sizes=(0.33, 0.5, 0.75, 1.0, ALL_IN), max_raises=3, stack=900.0)],
                  [synth.leduc()], [river(27, 45), synth.kuhn()], BATCHES["turns"]()[:2]):
        kw = dict(alternating=alternating, precision=precision)
        want = _solve(specs, capi.make_opts(variant, schedule="level", chunk_hands=2, **kw))
        runs = [("level", 4), ("level", 8), ("level", 32), ("resident", 1), ("resident", 8)]
        if len(specs) == 1 and specs[0].bet_sizes != many:
            runs.append(("wide", 8))
        for schedule, chunk in runs:
            try:
                got = _solve(specs, capi.make_opts(variant, schedule=schedule, chunk_hands=chunk, **kw))
            except capi.CfrError as e:
                assert schedule == "resident" and e.code == capi.CFR_EINVAL  # too large for shared memory
                continue
            for x, y in zip([*got[0], *got[3]], [*want[0], *want[3]], strict=True):
                assert np.array_equal(x, y), (schedule, chunk)
            assert np.allclose(got[1], want[1], rtol=1e-13, atol=1e-15)  # FP64 root sums over other chunks
            assert np.allclose(got[2], want[2], rtol=1e-13, atol=1e-15)


@pytest.mark.parametrize("precision", ["single", "pairs"])
def test_many_groups_per_block(precision):
    """Stretches of several groups over games of different hand counts (shared memory laid out anew)."""
    specs = [river(40 + 29 * k % 170, 100 + k, stack=100.0 + 37.0 * k, max_raises=2 + k % 2) for k in range(70)]
    want = _solve(specs, capi.make_opts("dcfr", schedule="stream", term_nodes=1, precision=precision))
    got = _solve(specs, capi.make_opts("dcfr", schedule="stream", term_nodes=4, precision=precision))
    for x, y in zip(got[0], want[0], strict=True):
        assert np.array_equal(x, y)
    assert np.array_equal(got[1], want[1]) and np.array_equal(got[2], want[2])


@pytest.mark.parametrize("precision", ["single", "pairs"])
def test_fold_groups_at_1176_hands(precision):
    spec = synth.flop_subgame(n_hands=1176, seed=31, range_seed=32, bet_sizes=(ALL_IN,), max_raises=1, depth_limit=1)
    out = []
    for nodes in (1, 4):
        tree = capi.cfr_tree_create(spec, capi.make_opts("dcfr", schedule="wide", term_nodes=nodes, precision=precision))
        try:
            capi.cfr_set_leaf_net(tree, [np.zeros(s, np.uint16) for s in capi.LEAF_SHAPES],
                                  [np.zeros(s[0], np.float32) for s in capi.LEAF_SHAPES])
            capi.cfr_iterate(tree, 2)
            n_nodes = capi.cfr_tree_info(tree)[0]
            out.append([capi.cfr_read_values(tree, capi.CFR_READ_CFV, n, player=p) for n in range(0, n_nodes, 11)
                        for p in (0, 1)])
        finally:
            capi.cfr_tree_destroy(tree)
    for x, y in zip(*out):
        assert np.array_equal(x, y)
