"""What a handle keeps, sends and reads back between calls: the rows of the last leaf evaluation, whatever
ran or was set since; the current strategy; the tables its kernels read."""
import numpy as np
import pytest

from paper_2605_19928_gb300 import capi, leafnet_train, synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_2605_19928_gb300 import build as pbuild
    pbuild.build()
    capi.load()
    capi.use_torch_allocator()


def _leaf_tree(alternating=True):
    spec = synth.turn_subgame(n_hands=200, seed=3, range_seed=4, bet_sizes=(1.0, synth.ALL_IN), max_raises=2)
    spec.depth_limit = 1
    return capi.cfr_tree_create(spec, capi.make_opts("dcfr", precision="single", alternating=alternating))


def _nets():
    W, b = leafnet_train.load_weights()
    other = [np.roll(w, 1, axis=0) for w in W]  # other finite weights of the same shapes
    return (W, b), (other, [np.roll(x, 1) for x in b])


def _outputs(tree):
    return capi.cfr_read_leaf_rows(tree, 1, 0, 48 * len(capi.cfr_leaf_info(tree)))


def _launches(tree):
    return capi.cfr_counters(tree)["kernel_launches"]


@pytest.mark.parametrize("alternating", [True, False])
def test_leaf_outputs_are_the_last_evaluations_after_the_network_is_replaced(alternating):
    first, second = _nets()
    a, b = _leaf_tree(alternating), _leaf_tree(alternating)
    try:
        for t in (a, b):
            capi.cfr_set_leaf_net(t, *first)
            capi.cfr_iterate(t, 3)
        want = _outputs(a)  # read before the weights change
        capi.cfr_set_leaf_net(a, *second)
        capi.cfr_set_leaf_net(b, *second)
        assert np.array_equal(_outputs(a), want)
        assert np.array_equal(_outputs(b), want)
        for t in (a, b):
            capi.cfr_iterate(t, 1)
        new = _outputs(a)
        assert not np.array_equal(new, want)
        assert np.array_equal(_outputs(b), new)
    finally:
        capi.cfr_tree_destroy(a)
        capi.cfr_tree_destroy(b)


def test_reading_complete_leaf_outputs_launches_nothing():
    net, _ = _nets()
    tree = _leaf_tree()
    n = 48 * 3
    try:
        capi.cfr_set_leaf_net(tree, *net)
        capi.cfr_iterate(tree, 2)
        l0 = _launches(tree)
        row = capi.cfr_read_leaf_rows(tree, 1, 0, 1)
        assert _launches(tree) == l0 + 1  # the other player's outputs, once
        assert np.array_equal(capi.cfr_read_leaf_rows(tree, 1, 0, n)[:1], row)
        assert _launches(tree) == l0 + 1
        evaluations = [lambda: capi.cfr_eval_leaves(tree, average=True), lambda: capi.cfr_exploitability(tree),
                       lambda: capi.cfr_stage_times(tree, 1), lambda: capi.cfr_eval_leaves(tree)]
        for evaluate in evaluations:  # each evaluates both players
            capi.cfr_iterate(tree, 1)
            evaluate()
            l0 = _launches(tree)
            rows = [capi.cfr_read_leaf_rows(tree, 1, k, 1) for k in range(n)]
            assert _launches(tree) == l0
            assert np.array_equal(np.concatenate(rows), capi.cfr_read_leaf_rows(tree, 1, 0, n))
    finally:
        capi.cfr_tree_destroy(tree)


def test_a_read_that_launches_reports_a_wait_that_gave_up():
    net, _ = _nets()
    tree = _leaf_tree()
    try:
        capi.cfr_set_leaf_net(tree, *net)
        capi.cfr_sync(tree)
        capi.cfr_debug_first_wait_polls(0)
        try:
            capi.cfr_iterate(tree, 1)
            with pytest.raises(capi.CfrError) as e:
                capi.cfr_read_leaf_rows(tree, 1, 0, 48)
            assert e.value.code == capi.CFR_ETIMEOUT
        finally:
            capi.cfr_debug_first_wait_polls(-1)
    finally:
        capi.cfr_tree_destroy(tree)


@pytest.mark.parametrize("variant", ["dcfr", "pcfr+"])
def test_current_strategy_of_hand_tiles_is_read_where_it_is_kept(variant):
    specs = [synth.river_subgame(n_hands=60 + 7 * k, seed=3 * k, range_seed=3 * k + 1) for k in range(3)]
    rows = {}
    for schedule in ("level", "stream"):
        tree = capi.cfr_batch_create(specs, capi.make_opts(variant, precision="single", schedule=schedule))
        try:
            capi.cfr_iterate(tree, 4)
            l0 = _launches(tree)
            rows[schedule] = [capi.cfr_strategy(tree, 0, game=g) for g in range(3)]
            assert _launches(tree) == l0
        finally:
            capi.cfr_tree_destroy(tree)
    for x, y in zip(rows["level"], rows["stream"]):
        assert np.array_equal(x, y)


def test_only_walked_trees_upload_their_programs():
    spec = synth.river_subgame(n_hands=64, seed=3, range_seed=4)
    sent = {}
    for schedule, warp_hands, chunk in (("level", 0, 2), ("stream", 0, 0), ("stream", 64, 0)):
        opts = capi.make_opts("dcfr", precision="single", schedule=schedule, warp_hands=warp_hands, chunk_hands=chunk)
        tree = capi.cfr_tree_create(spec, opts)
        sent[schedule, warp_hands] = capi.cfr_counters(tree)["h2d_bytes"]
        capi.cfr_tree_destroy(tree)
    # the per-hand kernels' handle sends less than the one that walks its tree, although its chunks are more
    assert sent["level", 0] < sent["stream", 64]


def test_kernel_names_follow_what_the_handle_runs():
    A = synth.ALL_IN
    small = synth.river_subgame(n_hands=64, seed=3, range_seed=4)
    large = synth.river_subgame(n_hands=64, seed=3, range_seed=4, bet_sizes=(0.33, 0.5, 0.75, 1.0, 2.0, A), max_raises=4,
                                stack=3000.0)
    batch = synth.batch_rivers(256, n_hands=40)
    cases = [([small], dict(schedule="level"), ("k_terminal", "k_tile")),
             ([small], dict(schedule="level", chunk_hands=2), ("k_terminal", "k_hand")),
             ([large], dict(schedule="wide"), ("k_terminal_vec", "k_wide_back")),
             ([small], dict(schedule="stream", warp_hands=64), ("k_terminal", "k_stream_update")),
             ([small], dict(schedule="resident"), ("k_resident", "k_resident")),
             (batch, dict(schedule="stream"), ("k_terminal_vec", "k_tile")),
             (batch, dict(schedule="stream", precision="pairs"), ("k_terminal_run", "k_tile"))]
    for specs, kw, want in cases:
        tree = capi.cfr_batch_create(specs, capi.make_opts("dcfr", **{"precision": "single", **kw}))
        try:
            assert capi.cfr_kernel_names(tree) == want
        finally:
            capi.cfr_tree_destroy(tree)
