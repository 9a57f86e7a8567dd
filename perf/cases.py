"""The work that users of this framework have it do, as cases that can be timed and compared.

A case is a dict of plain values.  Three kinds:

  solve   a handle (one subgame or a batch) solved from scratch: reset, `iters` iterations, the
          exploitability of the result and the average strategy at every subgame's root -- what
          `bench.py` times as a step, with fewer iterations a step;
  serve   one request of a serving loop: a handle created from host arrays, solved, its root
          strategy read, and the handle released;
  layer   one dense layer of the leaf network (`cfr_gemm_bf16`).

Trees, sizes and options are those of `synth.py`, `bench.py` and the tests.  `exact` restates a
solve in 64 bits from the rules alone: a betting tree per street, one H x H matrix of showdown
signs per board, and CFR by matrix products.
"""
import functools
import math

import numpy as np
import torch

from paper_2605_19928_gb300 import capi, leafnet_train, synth

ALL_IN = synth.ALL_IN
# bet menus (pot fractions) of the generators and the benchmark's trees
MENUS = {
    "half,all-in": (0.5, ALL_IN),
    "half,pot,all-in": (0.5, 1.0, ALL_IN),
    "third,3/4,5/4,all-in": (0.33, 0.75, 1.25, ALL_IN),
    "all-in": (ALL_IN,),
}
# the leaf network's layers as it runs them: (N, K, GELU, output type)
LAYERS = {1: (512, 2752, True, torch.bfloat16), 2: (512, 512, True, torch.bfloat16), 4: (2688, 512, False, torch.float32)}


def _solve(game, **kw):
    case = {"kind": "solve", "game": game, "games": 1, "hands": 1081, "shape_seed": 0, "menu": "half,pot,all-in",
            "stack": 400.0, "raises": 3, "variant": "dcfr", "alternating": True, "precision": "single",
            "schedule": "auto", "term_nodes": 0, "iters": 100}
    case.update(kw)
    return case


def listed():
    return [
        # the smallest call: Leduc hold'em, 6 one-card hands, with the library's default options
        _solve("leduc", name="leduc", hands=6, precision="pairs", iters=100),
        # a river subgame with the default options (double-float values, one launch per phase)
        _solve("river", name="river_default", precision="pairs", iters=100),
        # the same subgame for lowest latency: the layout and values the autotuner and bench.py use;
        # 240 iterations take it to 1 mbb/hand
        _solve("river", name="river_resident", schedule="resident", iters=240),
        # one request of a real-time player: a new subgame, 240 iterations, its root strategy
        {**_solve("river", name="river_request", schedule="resident", iters=240), "kind": "serve"},
        # a few uneven subgames with part of the hands (403 of 1081), both players updated at once
        _solve("batch", name="batch8_ragged", games=8, hands=403, alternating=False, variant="cfr+", iters=50),
        # batched serving, double-float values, Predictive CFR+
        _solve("batch", name="batch64_pcfr", games=64, precision="pairs", variant="pcfr+", iters=20),
        # batched serving as bench.py measures it: 256 uneven rivers, the autotuner's layout
        _solve("batch", name="batch256", games=256, term_nodes=4, iters=100),
        # an exact turn subgame: 15,195 public nodes, river cards dealt by chance
        _solve("turn", name="turn_exact", hands=1128, iters=20),
        # the same turn cut at the river card, 13 leaves valued by the leaf network
        _solve("turn_leaf", name="turn_leaf", hands=1128, iters=10),
        # a flop subgame cut at the river card: 102,124 public nodes, 1,029 network leaves, all-in
        # run-outs by their tables
        _solve("flop_leaf", name="flop_leaf", hands=1176, menu="third,3/4,5/4,all-in", stack=150.0, raises=4,
               schedule="wide", iters=5),
        # the leaf network's first layer on 16,384 rows, and its output layer on the rows of 261 leaves
        {"kind": "layer", "name": "layer_in", "layer": 1, "rows": 16384},
        {"kind": "layer", "name": "layer_out", "layer": 4, "rows": 12528},
    ]


def _log_int(rng, a, b):
    return int(round(math.exp(rng.uniform(math.log(a), math.log(b)))))


def draw(rng):
    """One more case of the same ranges (no dearer than the largest listed one)."""
    kind = rng.choice(["river", "river", "request", "batch", "batch", "batch", "turn", "turn_leaf", "flop_leaf", "layer"])
    variant = rng.choice(["dcfr", "dcfr", "dcfr", "cfr+", "pcfr+", "cfr"])
    precision = rng.choice(["single", "single", "pairs"])
    alternating = rng.random() < 0.8
    if kind == "layer":
        return {"kind": "layer", "layer": rng.choice([1, 2, 4]), "rows": _log_int(rng, 48, 49392)}
    if kind in ("river", "request"):
        case = _solve("river", hands=_log_int(rng, 60, 1081), menu=rng.choice(["half,all-in", "half,pot,all-in"]),
                      stack=float(rng.randint(100, 900)), raises=rng.randint(2, 3), variant=variant, precision=precision,
                      alternating=alternating, schedule=rng.choice(["auto", "resident"]), iters=rng.randint(40, 240))
        return {**case, "kind": "serve"} if kind == "request" else case
    if kind == "batch":
        return _solve("batch", games=_log_int(rng, 3, 256), hands=_log_int(rng, 200, 1081), shape_seed=rng.randint(0, 9),
                      variant=variant, precision=precision, alternating=alternating,
                      term_nodes=rng.choice([0, 0, 4]), iters=rng.randint(10, 50))
    if kind == "turn":
        return _solve("turn", hands=_log_int(rng, 150, 1128), menu=rng.choice(["half,all-in", "half,pot,all-in"]),
                      stack=float(rng.randint(100, 400)), raises=rng.randint(2, 3), variant=variant, precision=precision,
                      schedule=rng.choice(["auto", "wide"]), iters=rng.randint(5, 20))
    if kind == "turn_leaf":
        return _solve("turn_leaf", hands=_log_int(rng, 300, 1128), menu=rng.choice(["half,all-in", "half,pot,all-in"]),
                      stack=float(rng.randint(100, 400)), variant=variant, precision=precision, iters=rng.randint(3, 10))
    return _solve("flop_leaf", hands=_log_int(rng, 300, 1176), menu=rng.choice(["half,all-in", "half,pot,all-in"]),
                  stack=float(rng.randint(60, 150)), raises=rng.randint(2, 3), variant=variant, schedule="wide",
                  iters=rng.randint(2, 5))


# ------------------------------------------------------------------ inputs

def _specs(case, seed):
    """The subgames of a solve: trees from the case, boards, strengths and ranges from the seed."""
    hands, menu = case["hands"], MENUS[case["menu"]]
    kw = dict(seed=seed, range_seed=seed + 1, stack=case["stack"], bet_sizes=menu, max_raises=case["raises"])
    if case["game"] == "leduc":
        g = synth.leduc()
        g.ranges = synth.random_ranges(6, seed)
        return [g]
    if case["game"] == "river":
        return [synth.river_subgame(n_hands=hands, **kw)]
    if case["game"] == "turn":
        return [synth.turn_subgame(n_hands=hands, **kw)]
    if case["game"] == "turn_leaf":
        return [synth.ranked_turn_subgame(n_hands=hands, depth_limit=1, **kw)]
    if case["game"] == "flop_leaf":  # strengths drawn per board: ranking 1,176 boards takes the host seconds
        return [synth.flop_subgame(n_hands=hands, depth_limit=1, **kw)]
    out = []
    for k, g in enumerate(_batch_shapes(case)):
        out.append(synth.river_subgame(n_hands=hands, seed=seed + 7 * k, range_seed=seed + 7 * k + 3, pot=g[0], stack=g[1],
                                       bet_sizes=g[2], max_raises=g[3]))
    return out


def _batch_shapes(case):
    """(pot, stack, bet sizes, raises) of each subgame of a batch, as synth.batch_rivers draws them."""
    return [(g.pot, g.stack, g.bet_sizes, g.max_raises)
            for g in synth.batch_rivers(case["games"], seed=case["shape_seed"], n_hands=4)]


def _opts(case):
    return capi.make_opts(case["variant"], alternating=case["alternating"], precision=case["precision"],
                          schedule=case["schedule"], term_nodes=case["term_nodes"],
                          runout_tables=case["game"] == "flop_leaf")


class Handle:
    """A solver handle, released with its owner."""

    def __init__(self, tree):
        self.tree = tree

    def __del__(self):
        capi.cfr_tree_destroy(self.tree)


@functools.lru_cache(None)
def _start():
    """Once per process, as a program starts: the library, with PyTorch's allocator behind it."""
    torch.cuda.set_device(0)
    capi.load()
    capi.use_torch_allocator()


def prepare(case, seed):
    _start()
    if case["kind"] == "layer":
        N, K, act, dtype = LAYERS[case["layer"]]
        A, B, bias = _layer_inputs(case, seed)
        return {"case": case, "A": A, "B": B, "bias": bias, "act": act,
                "C": torch.empty(case["rows"], N, dtype=dtype, device="cuda"),
                "err": torch.zeros(1, dtype=torch.int32, device="cuda")}
    specs, opts = _specs(case, seed), _opts(case)
    if case["kind"] == "serve":
        return {"case": case, "specs": specs, "opts": opts}
    batch = case["game"] == "batch"
    tree = capi.cfr_batch_create(specs, opts) if batch else capi.cfr_tree_create(specs[0], opts)
    state = {"case": case, "handle": Handle(tree), "games": len(specs)}
    if case["game"].endswith("_leaf"):
        capi.cfr_set_leaf_net(tree, *leafnet_train.load_weights())
    return state


def _layer_inputs(case, seed):
    N, K, _, _ = LAYERS[case["layer"]]
    g = torch.Generator(device="cuda").manual_seed(seed)
    if case["layer"] == 1:  # two ranges that sum to 1, as the network's inputs
        A = torch.rand(case["rows"], K, device="cuda", generator=g)
        A = A / (0.25 * K * 0.5)
    else:  # activations after GELU
        A = torch.nn.functional.gelu(torch.randn(case["rows"], K, device="cuda", generator=g))
    B = torch.randn(N, K, device="cuda", generator=g) / K ** 0.5
    bias = torch.randn(N, device="cuda", generator=g)
    return A.to(torch.bfloat16), B.to(torch.bfloat16), bias


def _roots(tree, games):
    """The average strategy at every subgame's root, one after the other."""
    return np.concatenate([capi.cfr_strategy(tree, 0, average=True, game=g).ravel() for g in range(games)])


def run(state):
    case = state["case"]
    if case["kind"] == "layer":
        capi.cfr_gemm_bf16(state["A"], state["B"], state["bias"], state["C"], state["act"], state["err"])
        return state["C"]
    if case["kind"] == "serve":
        tree = capi.cfr_tree_create(state["specs"][0], state["opts"])
        try:
            capi.cfr_iterate(tree, case["iters"])
            return {"root_average_strategy": _roots(tree, 1)}
        finally:
            capi.cfr_tree_destroy(tree)
    tree = state["handle"].tree
    capi.cfr_reset(tree)
    capi.cfr_iterate(tree, case["iters"])
    _, br = capi.cfr_exploitability(tree, state["games"])
    # a solve in FP32 values has FP32 best-response values, one in double-float pairs FP64
    return {"root_average_strategy": _roots(tree, state["games"]),
            "best_response": br.astype(np.float32) if case["precision"] == "single" else br}


# ------------------------------------------------------------------ what a pass cannot do without

def work(case):
    if case["kind"] == "layer":
        N, K, _, dtype = LAYERS[case["layer"]]
        M = case["rows"]
        return {"bytes": 2.0 * (M * K + N * K) + 4.0 * N + M * N * (2 if dtype == torch.bfloat16 else 4),
                "flops": 2.0 * M * N * K}
    H, V = case["hands"], 4 if case["precision"] == "single" else 8
    total, flops = 0.0, 0.0
    for rules in _rules(case):
        c = _count(rules, H)
        # per iteration: R, S (and the prediction) read and written once per (row, hand); reach written
        # and read and values written and read once per (terminal or leaf, hand) and player
        state = 32 if case["variant"] != "pcfr+" else 48
        per_iter = H * (c["rows"] * state + 2 * c["ends"] * 4 * V)
        # the exploitability pass: S read once, both players' terminals once more
        total += case["iters"] * per_iter + H * (c["rows"] * 8 + 2 * c["ends"] * 4 * V)
        # per iteration and (row, hand) about 12 operations; per (end, hand) and player about 12
        flops += (case["iters"] + 1) * H * 12.0 * (c["rows"] + 2 * c["ends"])
        if c["leaf_rows"]:  # network rows, both players' updates
            times = 2 if case["alternating"] else 1
            flops += (case["iters"] * times + 1) * c["leaf_rows"] * 2.0 * (2752 * 512 + 2 * 512 * 512 + 512 * 2688 / times)
    return {"bytes": total, "flops": flops}


# ------------------------------------------------------------------ betting trees

class Rules:
    def __init__(self, game, deck, n_board, hand_size, streets, pot, stack, sizes, raises, depth_limit):
        self.game, self.deck, self.n_board, self.hand_size, self.streets = game, deck, n_board, hand_size, streets
        self.pot, self.cap, self.sizes, self.raises, self.depth_limit = pot, pot / 2 + stack, sizes, raises, depth_limit


class Node:
    """A node of the betting tree; a chance node has one child, the subtree of every card."""

    def __init__(self, kind, player=-1, c=(0.0, 0.0), dealt=0, prob=1.0):
        self.kind, self.player, self.c, self.dealt, self.prob, self.kids = kind, player, c, dealt, prob, []


def _rules(case):
    menu = MENUS[case["menu"]]
    if case["game"] == "leduc":
        return [Rules("leduc", 6, 0, 1, 2, 2.0, 0.0, (), 2, 0)]
    if case["game"] == "batch":
        return [Rules("holdem", 52, 5, 2, 1, p, s, z, r, 0) for p, s, z, r in _batch_shapes(case)]
    board = {"river": 5, "turn": 4, "turn_leaf": 4, "flop_leaf": 3}[case["game"]]
    return [Rules("holdem", 52, board, 2, 6 - board, 100.0, case["stack"], menu, case["raises"],
                  int(case["game"].endswith("_leaf")))]


def _tree(R):
    """Betting tree of one subgame: player 0 acts first on every street; a fraction x facing a call
    of d raises by d + x (pot + d); sizes reaching the stack are all-in, duplicates are dropped."""
    def street_over(c, street, dealt, prob):
        if street + 1 >= R.streets:
            return Node("showdown", c=c, dealt=dealt, prob=prob)
        n = Node("chance", c=c, dealt=dealt, prob=prob)
        all_in = R.game == "holdem" and max(c) >= R.cap
        left = R.deck - R.n_board - dealt - 2 * R.hand_size  # cards the two hands and the board leave
        if R.depth_limit and R.n_board + dealt == 4 and not all_in:
            n.kind, n.prob = "leaf", prob / left
            return n
        if all_in:  # nobody can bet: the cards still to come are run out at once
            n.kind = "runout"
            for k in range(dealt, dealt + R.streets - 1 - street):
                n.prob /= R.deck - R.n_board - k - 2 * R.hand_size
            return n
        n.kids = [decide(0, c, street + 1, 0, False, dealt + 1, prob / left)]
        return n

    def decide(p, c, street, raises, checked, dealt, prob):
        n, q = Node("decision", p, c, dealt, prob), 1 - p
        if c[q] > c[p]:
            n.kids.append(Node("fold", p, c, dealt, prob))
            n.kids.append(street_over((c[q], c[q]), street, dealt, prob))
        elif p == 1 or checked:
            n.kids.append(street_over(c, street, dealt, prob))
        else:
            n.kids.append(decide(q, c, street, raises, True, dealt, prob))
        to = []
        if raises < R.raises:
            if R.game == "leduc":
                to = [c[q] + (2.0, 4.0)[street]]
            elif c[q] < R.cap and c[p] < R.cap:
                d, pot = c[q] - c[p], c[0] + c[1]
                for x in R.sizes:
                    t = min(c[p] + (d + x * (pot + d)), R.cap) if x > 0 else R.cap
                    if t > c[q] and t not in to:
                        to.append(t)
        for t in sorted(to):
            k = (t, c[1]) if p == 0 else (c[0], t)
            n.kids.append(decide(q, k, street, raises + 1, False, dealt, prob))
        return n

    return decide(0, (R.pot / 2, R.pot / 2), 0, 0, False, 0, 1.0)


def _count(R, H):
    """Decision rows, end nodes (a run-out's boards not counted) and network rows of the public tree."""
    out = {"rows": 0, "ends": 0, "leaf_rows": 0}

    def walk(n, times):
        if n.kind == "decision":
            out["rows"] += times * len(n.kids)
        elif n.kind == "chance":
            times *= R.deck - R.n_board - n.dealt
        else:
            out["ends"] += times
            if n.kind == "leaf":
                out["leaf_rows"] += times * 48
        for k in n.kids:
            walk(k, times)

    walk(_tree(R), 1)
    return out


# ------------------------------------------------------------------ the same solve in 64 bits

def exact(case, seed):
    f64 = torch.float64
    if case["kind"] == "layer":
        A, B, bias = _layer_inputs(case, seed)
        y = A.to(f64) @ B.to(f64).T + bias.to(f64)
        return torch.nn.functional.gelu(y) if LAYERS[case["layer"]][2] else y
    rules = _rules(case)
    # seconds, roughly: small tensor operations for the trees, matrix products for the boards
    if sum(_size(_tree(R)) for R in rules) * case["iters"] > 60_000:
        return None
    roots, brs = [], []
    for spec, R in zip(_specs(case, seed), rules):
        s = Solve(spec, R, case)
        for t in range(1, case["iters"] + 1):
            s.iterate(t)
        roots.append(s.average(s.root).reshape(-1))
        if case["kind"] == "solve":
            brs.append(s.best_responses())
    out = {"root_average_strategy": torch.cat(roots)}
    if brs:
        out["best_response"] = torch.stack(brs)
    return out


def _size(n):
    return 1 + sum(_size(k) for k in n.kids)


class Solve:
    """CFR over the betting tree in FP64; below a dealt card every array has the card as its first index."""

    def __init__(self, spec, R, case):
        self.R, self.case, dev, f64 = R, case, "cuda", torch.float64
        hands = torch.as_tensor(np.asarray(spec.hands, dtype=np.int64), device=dev)
        H = hands.shape[0]
        holds = torch.zeros(H, R.deck, dtype=f64, device=dev).scatter_(1, hands, 1.0)
        self.K = (holds @ holds.T == 0).to(f64)  # pairs of hands that share no card
        board = [int(c) for c in spec.board] if R.game == "holdem" else []
        self.cards = [c for c in range(R.deck) if c not in board]
        self.live = (1.0 - holds[:, self.cards]).T.contiguous()  # [card, hand]: the hand does not hold it
        self.hands, self.board, self.spec, self.H = hands, board, spec, H
        r = torch.as_tensor(np.asarray(spec.ranges, dtype=np.float64), device=dev)
        self.range = r / r.sum(dim=1, keepdim=True)
        self.kappa = 1.0 / (self.range[0] @ self.K @ self.range[1])
        self.E = {}
        self.net = None
        if R.depth_limit:
            W, b = leafnet_train.load_weights()
            self.net = [((torch.as_tensor(w.astype(np.int32), device=dev) << 16).view(torch.float32).to(f64),
                         torch.as_tensor(np.asarray(x), device=dev).to(f64)) for w, x in zip(W, b)]
        self.root = _tree(R)
        self.nodes = []

        def walk(n):
            self.nodes.append(n)
            if n.kind == "decision":
                shape = (len(n.kids),) + ((len(self.cards),) if n.dealt else ()) + (H,)
                n.R, n.S = torch.zeros(shape, dtype=f64, device=dev), torch.zeros(shape, dtype=f64, device=dev)
                n.M = torch.zeros_like(n.R)
                n.sigma = torch.full_like(n.R, 1.0 / len(n.kids))
            for k in n.kids:
                walk(k)

        walk(self.root)
        self.reach = [None, None]
        for p in (0, 1):
            self.reach[p] = self.forward(p, lambda n: n.sigma)

    def signs(self, dealt):
        """E[h][o]: boards on which h beats o less those on which it loses (0 where they share a card),
        over the boards of one river, of every river card (dealt 1 of a turn), or of a run-out."""
        key = dealt
        if key not in self.E:
            R, s = self.R, self.spec.strength
            if R.game == "leduc":
                h = torch.arange(6, device="cuda")
                st = torch.stack([torch.where(h // 2 == c // 2, 10 + h // 2, h // 2) for c in range(6)])
                self.E[key] = self._sign(st)
            else:
                st = torch.as_tensor(np.asarray(s), device="cuda")
                if R.n_board == 5:
                    self.E[key] = self._sign(st)[0]
                elif R.n_board == 4:
                    self.E[key] = self._sign(st[self.cards])
                    if dealt == 0:  # a run-out from the turn: its boards summed
                        self.E[key] = self._board_sum(self.E[key])
                else:  # flop: run-outs from every turn card, or from the flop
                    rows = []
                    for i, t in enumerate(self.cards):
                        e = self._sign(st[[t * 52 + c for c in self.cards]])
                        e[i] = 0.0
                        rows.append(self._board_sum(e))
                    self.E[key] = torch.stack(rows)
                    if dealt == 0:
                        self.E[key] = self._board_sum(self.E[key])
        return self.E[key]

    def _sign(self, st):
        return torch.sign(st[:, :, None] - st[:, None, :]).to(torch.float64) * self.K

    def _board_sum(self, e):  # over the dealt card, for the pairs of hands that do not hold it
        return torch.einsum("cij,ci,cj->ij", e, self.live, self.live)

    def forward(self, p, strategy):
        reach = {self.root: self.range[p]}
        for n in self.nodes:
            x = reach[n]
            for a, k in enumerate(n.kids):
                if n.kind == "chance":
                    reach[k] = x[None, :] * self.live
                else:
                    reach[k] = x * strategy(n)[a] if n.player == p else x
        return reach

    def end_value(self, n, i, reach):
        q = reach[1 - i][n]
        own = self.live if n.dealt else 1.0
        if n.kind == "fold":
            u = n.c[n.player] * n.prob * self.kappa * (-1.0 if n.player == i else 1.0)
            return u * (q @ self.K) * own
        if n.kind == "showdown" or n.kind == "runout":
            E = self.signs(n.dealt)
            v = torch.einsum("cij,cj->ci", E, q) if n.dealt else E @ q
            return n.c[0] * n.prob * self.kappa * v * own
        return self.leaf_value(n, i, reach)

    def leaf_value(self, n, i, reach):
        pot, cap = n.c[0] + n.c[1], self.R.cap
        behind = cap - n.c[0]
        feat = torch.tensor([pot / (pot + 2 * behind), behind / (pot + 2 * behind)], dtype=torch.float64, device="cuda")
        lo, hi = self.hands.min(dim=1).values, self.hands.max(dim=1).values
        slot = hi * (hi - 1) // 2 + lo
        out = []
        for b in range(len(self.cards) if n.dealt else 1):
            board = self.board + ([self.cards[b]] if n.dealt else [])
            rivers = [k for k, c in enumerate(self.cards) if c not in board]
            ok = self.live[rivers] * (self.live[b] if n.dealt else 1.0)  # hands without the river card
            x = torch.zeros(len(rivers), 2752, dtype=torch.float64, device="cuda")
            for p in (0, 1):
                q = (reach[p][n][b] if n.dealt else reach[p][n]) * ok
                tot = q.sum(dim=1, keepdim=True)
                q = torch.where(tot > 0, q / tot, ok / ok.sum(dim=1, keepdim=True))
                x[:, p * 1326 + slot] = q
            for row, k in enumerate(rivers):
                x[row, [2652 + c for c in board + [self.cards[k]]]] = 1.0
            x[:, 2704:2706] = feat
            for k, (W, bias) in enumerate(self.net):
                x = x @ W.T + bias
                if k < 3:
                    x = torch.nn.functional.gelu(x)
            y = x[:, i * 1326 + slot]
            opp = (reach[1 - i][n][b] if n.dealt else reach[1 - i][n]) * ok
            out.append(((opp @ self.K) * y * ok).sum(dim=0))
        v = torch.stack(out) if n.dealt else out[0]
        return pot * n.prob * self.kappa * v

    def values(self, i, reach, pick):
        """Counterfactual values of player i; pick(n, kids' values) at i's own decisions."""
        v = {}
        for n in reversed(self.nodes):
            if not n.kids:
                v[n] = self.end_value(n, i, reach)
            elif n.kind == "chance":
                v[n] = (v[n.kids[0]] * self.live).sum(dim=0)
            else:
                kids = torch.stack([v[k] for k in n.kids])
                v[n] = pick(n, kids) if n.player == i else kids.sum(dim=0)
        return v

    def iterate(self, t):
        for players in ((0,), (1,)) if self.case["alternating"] else ((0, 1),):
            found = {p: self.values(p, self.reach, lambda n, kids: (n.sigma * kids).sum(dim=0)) for p in players}
            for p in players:
                for n in self.nodes:
                    if n.kind == "decision" and n.player == p:
                        r = torch.stack([found[p][k] for k in n.kids]) - found[p][n]
                        self.update(n, t, r, self.reach[p][n])
            for p in players:
                self.reach[p] = self.forward(p, lambda n: n.sigma)

    def update(self, n, t, r, pi):
        variant, contrib = self.case["variant"], pi * n.sigma
        n.R = n.R + r
        if variant == "dcfr":
            n.R = n.R * torch.where(n.R > 0, t ** 1.5 / (t ** 1.5 + 1.0), 0.5)
            n.S = n.S * (t / (t + 1.0)) ** 2 + contrib
        elif variant == "cfr":
            n.S = n.S + contrib
        else:
            n.R = n.R.clamp(min=0.0)
            n.S = n.S + (t if variant == "cfr+" else t * t) * contrib
        n.sigma = self.match(n.R + r if variant == "pcfr+" else n.R)

    @staticmethod
    def match(x):
        x = x.clamp(min=0.0)
        tot = x.sum(dim=0)
        return torch.where(tot > 0, x / torch.where(tot > 0, tot, 1.0), 1.0 / x.shape[0])

    def average(self, n):
        return self.match(n.S)

    def best_responses(self):
        reach = [self.forward(p, self.average) for p in (0, 1)]
        out = []
        for i in (0, 1):
            v = self.values(i, reach, lambda n, kids: kids.max(dim=0).values)
            out.append(self.range[i] @ v[self.root])
        return torch.stack(out)
