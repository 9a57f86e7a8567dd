"""Run-out table values at the edges of their kernel's tiles (4 hands a thread, 256 a block, 64
opponent hands a chunk, 8 rows ahead; 8 tops a thread on 8-bit tables, 2 on 16-bit ones): every
top's best-response value against u E q in FP64 from the reach the pass used, E counted from
the strengths.  A value is one chain of H FP32 FMAs, one product with u (itself rounded to FP32)
and exact E, so it is within (H + 3) 2^-24 of u sum |E| q."""
import numpy as np
import pytest

from paper_2605_19928_gb300 import capi, synth
from test_runout_gpu import built, opts, runouts  # noqa: F401

pytestmark = pytest.mark.gpu


def table(spec, board):
    """E over every completion of `board` (ordered cards), for the subgame's hands."""
    H = spec.n_hands
    live = [c for c in range(52) if c not in board]
    boards = [(c,) for c in live] if len(board) == 4 else [(a, b) for a in live for b in live if a != b]
    holds = np.zeros((H, 52), bool)
    for h, (a, b) in enumerate(spec.hands):
        holds[h, [a, b]] = True
    ok = (holds.astype(int) @ holds.T.astype(int)) == 0
    on = holds[:, list(board)].any(axis=1)  # a card dealt above the top is in the hand
    ok &= ~(on[:, None] | on[None, :])
    E = np.zeros((H, H))
    for cards in boards:
        if len(spec.board) == 4:
            row = cards[0]
        else:
            row = board[3] * 52 + cards[0] if len(board) == 4 else cards[0] * 52 + cards[1]
        s = spec.strength[row].astype(np.int64)
        free = ~holds[:, list(cards)].any(axis=1)
        E += np.sign(s[:, None] - s[None, :]) * (free[:, None] & free[None, :])
    return E * ok


@pytest.mark.parametrize("street,hands", [("turn", h) for h in (3, 31, 64, 65, 72, 255, 256, 257, 1128)] +
                         [("flop", h) for h in (3, 65, 262)])
def test_every_top_at_tile_edges(street, hands):
    kw = dict(n_hands=hands, seed=hands, range_seed=2, bet_sizes=(0.5, synth.ALL_IN) if street == "turn" else (synth.ALL_IN,),
              max_raises=2 if street == "turn" else 1)
    spec = synth.turn_subgame(**kw) if street == "turn" else synth.flop_subgame(depth_limit=1, **kw)
    tree = capi.cfr_tree_create(spec, opts())
    try:
        if street == "flop":  # an all-zero network: the run-outs do not depend on it
            capi.cfr_set_leaf_net(tree, [np.zeros(s, np.uint16) for s in capi.LEAF_SHAPES],
                                  [np.zeros(s[0], np.float32) for s in capi.LEAF_SHAPES])
        capi.cfr_iterate(tree, 2)
        capi.cfr_exploitability(tree)
        r = spec.ranges.astype(np.float64)
        r /= r.sum(axis=1, keepdims=True)
        holds = np.zeros((hands, 52))
        np.put_along_axis(holds, spec.hands.astype(int), 1.0, axis=1)
        Z = r[0] @ (holds @ holds.T == 0) @ r[1]
        tops, _ = runouts(tree)
        tables, wide = {}, set()
        for n in tops:
            info = capi.cfr_node_info(tree, n)
            board, m, chance = [int(c) for c in spec.board], n, 1.0
            while m > 0:  # the card dealt above the top, if any
                up = capi.cfr_node_info(tree, m)
                if up["deal"] >= 0:
                    board.append(up["deal"])
                    chance /= 52 - len(spec.board) - 4
                m = up["parent"]
            for k in range(len(board), 5):
                chance /= 52 - k - 4
            wide.add(5 - len(board))
            E = tables.setdefault(tuple(board), table(spec, board))
            u = info["contrib"][0] * chance / Z
            for i in (0, 1):
                q = capi.cfr_read_values(tree, capi.CFR_READ_AVG_REACH, n, player=1 - i)
                got = capi.cfr_read_values(tree, capi.CFR_READ_BR_CFV, n, player=i)
                assert np.all(np.abs(got - u * (E @ q)) <= (hands + 3) * 2.0 ** -24 * u * (np.abs(E) @ q)), (n, i)
        assert wide == ({1} if street == "turn" else {1, 2})
    finally:
        capi.cfr_tree_destroy(tree)
