"""The terminal launch's throughput forms against its one-node form, bit for bit, where their work lists
end: runs of one to eight nodes over tables of few showdowns, and stretches of groups beyond one wave of
blocks."""
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
    capi.use_torch_allocator()


def _river(hands, seed, **kw):
    return synth.river_subgame(n_hands=hands, seed=seed, range_seed=seed + 1, **kw)


CASES = {
    # 20,520 fold and showdown nodes: groups of four in stretches of two waves of blocks
    "waves": lambda: [_river(9, 3 * k, bet_sizes=(0.33, 0.5, 0.75, 1.0, 2.0, ALL_IN), max_raises=3, stack=900.0)
                      for k in range(40)],
    # 2,352 boards of seven showdowns, most of them below a dealt card: runs cut at every board
    "boards": lambda: [synth.flop_subgame(n_hands=45, seed=5, range_seed=6, bet_sizes=(ALL_IN,), max_raises=1)],
    # games of different hand counts and kinds side by side
    "mixed": lambda: [synth.leduc(), _river(33, 7), synth.kuhn(),
                      synth.turn_subgame(n_hands=301, seed=9, range_seed=10, bet_sizes=(ALL_IN,), max_raises=1)],
    # hand counts at which a thread's run of the prefix sums is 7, 8 and 9 entries, and few showdowns a board
    "eights": lambda: [_river(h, h, bet_sizes=(ALL_IN,), max_raises=1) for h in (559, 561, 640, 896, 897, 900, 1024, 1025, 1081)]
    + [synth.turn_subgame(n_hands=h, seed=9, range_seed=10, bet_sizes=(ALL_IN,), max_raises=1) for h in (1120, 1121, 1128)],
}


@pytest.mark.parametrize("precision", ["single", "pairs"])
@pytest.mark.parametrize("case", list(CASES))
def test_throughput_forms_keep_the_bits(case, precision):
    specs = CASES[case]()
    want = None
    for nodes in (1, 0, 2, 3, 5, 8):
        tree = capi.cfr_batch_create(specs, capi.make_opts("dcfr", precision=precision, term_nodes=nodes))
        try:
            capi.cfr_iterate(tree, 3)  # one player a launch
            got = _state(tree, len(specs))
            got.append(capi.cfr_exploitability(tree, len(specs))[1])  # both in one
        finally:
            capi.cfr_tree_destroy(tree)
        if want is None:
            want = got
        for x, y in zip(got, want, strict=True):
            assert np.array_equal(x, y), nodes
