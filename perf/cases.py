"""The work a user of this library has it do, as measurable cases.

A case is a dict of plain values; `path` says which public entry points it
goes through, the other keys are sizes and options.  `listed` gives the cases
that are looked at one by one, `draw` more of the same ranges, `prepare` what
a program holds before the call, `run` one pass, `work` the bytes and
operations a pass cannot do without and `exact` the results in 64-bit
arithmetic from plain torch and numpy (own betting trees, dense card
matrices, own network).
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2112_03804_gb300 import kps, synth

DT = {"f32": torch.float32, "f64": torch.float64, "bf16": torch.bfloat16, "f16": torch.float16}
SIZE = {"f32": 4, "f64": 8, "bf16": 2, "f16": 2}
DIN, WIDTH, DOUT, HIST = 1232, 256, 12, 1081


def listed():
    return [
        # one solver iteration's gradient on one endgame: latency and launches
        dict(name="product_f32_1", path="product", game="river", dtype="f32", direction="A", batch=1),
        # a handful of strategies evaluated against one endgame, a ragged batch, the other direction
        dict(name="product_f32_37", path="product", game="river", dtype="f32", direction="AT", batch=37),
        # the library's headline: many strategy pairs, one A y and one A^T x
        dict(name="step_f32_1024", path="product", game="river", dtype="f32", direction="both", batch=1024),
        # the same products with strategies stored in 16 bits
        dict(name="product_bf16_1000", path="product", game="river", dtype="bf16", direction="A", batch=1000),
        # 64-bit products: reference values and exploitability of many strategies
        dict(name="product_f64_100", path="product", game="river", dtype="f64", direction="AT", batch=100),
        # the large betting tree (247 sequences a player), a moderate batch
        dict(name="libratus_f32_250", path="product", game="libratus", dtype="f32", direction="A", batch=250),
        # uneven endgames (boards of 3 to 5 cards, 13 to 209 terminals) in one launch, both directions
        dict(name="batch_f32_512", path="batch", dtype="f32", games=512, mix=4),
        # a turn endgame: 240 river blocks and the turn round, both directions
        dict(name="turn_f32", path="turn", dtype="f32", turn_cap=2, river_cap=2),
        # the batched solver from a cold start: a few iterations and its averages.  (Few, because a
        # regret within rounding of the matching floor decides a strategy entry either way, and
        # such entries grow with the iterations; every iteration is the same work.)
        dict(name="solve_f32_256", path="solve", games=256, iters=3),
        # the stopping test: averages, FP64 products and best responses
        dict(name="exploit_f64_64", path="exploit", games=64),
        # training the warm-start network: losses and gradients of eight minibatches, then a prediction.
        # (No weight update in between: Adam divides a gradient by its own size, so weights that a
        # rounding moved say nothing about a later gradient.)
        dict(name="train_8x4096", path="train", rows=4096, steps=8),
        # the network's strategy at every query of a batch of endgames
        dict(name="predict_128", path="predict", games=128),
    ]


def _log(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    path = rng.choice(["product"] * 5 + ["batch", "turn", "solve", "exploit", "train", "predict"])
    if path == "product":
        game = rng.choice(["river", "river", "river", "turn4", "libratus"])
        dtype = rng.choice(["f32", "f32", "f32", "bf16", "f16", "f64"])
        top = 1024 if game != "libratus" else 250
        if dtype == "f64":
            top //= 4
        direction = rng.choice(["A", "AT", "both"])
        return dict(path=path, game=game, dtype=dtype, direction=direction, batch=_log(rng, 1, top))
    if path == "batch":
        return dict(path=path, dtype=rng.choice(["f32", "f32", "bf16", "f16"]), games=_log(rng, 8, 512),
                    mix=rng.randint(1, 1000))
    if path == "turn":
        return dict(path=path, dtype=rng.choice(["f32", "f32", "bf16"]), turn_cap=rng.choice([1, 2]),
                    river_cap=rng.choice([1, 2, 3]))
    if path == "solve":
        return dict(path=path, games=_log(rng, 8, 256), iters=rng.randint(2, 4))
    if path == "exploit":
        return dict(path=path, games=_log(rng, 4, 64))
    if path == "train":
        return dict(path=path, rows=_log(rng, 256, 4096), steps=rng.randint(2, 8))
    return dict(path=path, games=_log(rng, 4, 128))


# ---- betting trees (first principles; used by work and exact) ----------------
class Tree:
    """Terminals (s1, s2, is_showdown, payoff to player 1) and per player the
    node and parent sequence of every sequence, numbered depth first."""

    def __init__(self, spec):
        self.node, self.parent, self.nact = ([], []), ([], []), ([], [])
        self.terms, self.payoff = [], 0.0
        self.spec = spec
        self.top = min(spec["contrib0"][p] + spec["stack"][p] for p in (0, 1))
        self._walk(0, [float(c) for c in spec["contrib0"]], [-1, -1], 0, False)

    def _end(self, last, show, value, c):
        self.terms.append((last[0], last[1], show, value))
        self.payoff = max(self.payoff, c[0], c[1])

    def _walk(self, me, c, last, aggressive, checked):
        opp, sp = 1 - me, self.spec
        facing = c[opp] > c[me]
        if sp.get("menu") is not None:
            k = min(aggressive, 3) + 1 if facing else (1 if checked else 0)
            fracs = sp["menu"][me][k]
        else:
            fracs = sp["bet_frac"]
        high = max(c)
        sizes = set()
        cap = sp.get("raise_cap", -1)
        if high < self.top and (cap < 0 or aggressive < cap):
            for f in fracs:
                sizes.add(min(high + f * 2.0 * high, self.top))
            if sp.get("allow_allin"):
                sizes.add(self.top)
        acts = (["fold"] if facing else []) + ["call"] + sorted(sizes)
        node, first = len(self.nact[me]), len(self.node[me])
        self.nact[me].append(len(acts))
        for _a in acts:
            self.node[me].append(node)
            self.parent[me].append(last[me])
        for i, a in enumerate(acts):
            now = list(last)
            now[me] = first + i
            if a == "fold":
                self._end(now, False, c[1] if me == 1 else -c[0], c)
            elif a == "call":
                cc = list(c)
                cc[me] = high
                if facing or checked:
                    self._end(now, True, min(cc), cc)
                else:
                    self._walk(opp, cc, now, aggressive, True)
            else:
                cc = list(c)
                cc[me] = a
                self._walk(opp, cc, now, aggressive + 1, checked)

    def n(self, p):
        return len(self.node[p])


def _hands(spec, device="cpu"):
    """Card pairs in canonical order."""
    left = [c for c in range(spec["ranks"] * spec["suits"]) if c not in set(spec["board"])]
    a, b = np.triu_indices(len(left), 1)
    left = np.asarray(left)
    return torch.from_numpy(np.stack([left[a], left[b]], 1)).to(device)


def _order(strength):
    s = np.asarray(strength)
    return np.lexsort((np.arange(len(s)), s))


class Cards:
    """Dense card matrices of one endgame in 64 bits, hands in strength order."""

    def __init__(self, spec, order=None, strength=None, beta_scale=None, mask=None):
        dev = "cuda"
        strength = np.asarray(spec["strength"] if strength is None else strength)
        self.order = _order(strength) if order is None else order
        self.hand = _hands(spec, dev)[torch.from_numpy(self.order).to(dev)]
        s = torch.from_numpy(strength[self.order].astype(np.int64)).to(dev)
        h = self.hand
        share = (h[:, None, :, None] == h[None, :, None, :]).any(-1).any(-1)
        self.C = (~share).double()
        self.W = torch.sign(s[:, None] - s[None, :]).double() * self.C
        mu = [torch.from_numpy(np.asarray(spec[k], np.float64)[self.order]).to(dev) for k in ("mu1", "mu2")]
        if mask is not None:
            mu = [m * mask(h) for m in mu]
        beta = float((mu[0] @ self.C @ mu[1]).item()) if beta_scale is None else beta_scale
        self.beta, self.mu = beta, mu
        self.lam = [m / math.sqrt(beta) for m in mu]
        self.H = len(self.order)


def _apply(tree, cards, v, out_player):
    """[B, n_in, H] (64 bits) -> [B, n_out, H]: the payoff product."""
    p, q = out_player, 1 - out_player
    x = v * cards.lam[q]
    out = torch.zeros(v.shape[0], tree.n(p), cards.H, dtype=torch.float64, device=v.device)
    sgn = 1.0 if p == 0 else -1.0
    for show, M in ((False, cards.C), (True, cards.W)):
        t = [(a[p], a[q], a[3]) for a in tree.terms if a[2] == show and a[3] != 0.0]
        if not t:
            continue
        rows = torch.tensor([a[0] for a in t], device=v.device)
        cols = torch.tensor([a[1] for a in t], device=v.device)
        coef = torch.tensor([a[2] * (sgn if show else 1.0) for a in t], dtype=torch.float64, device=v.device)
        for b in range(0, v.shape[0], 128):
            out[b:b + 128].index_add_(1, rows, (x[b:b + 128][:, cols] @ M.T) * coef[:, None])
    return out * cards.lam[p]


# ---- inputs ----------------------------------------------------------------
def _spec(kind, seed):
    if kind == "river":
        return synth.river_spec(seed=seed)
    if kind == "turn4":                     # four board cards, 1128 hands
        return synth.river_spec(seed=seed, nboard=4)
    return synth.libratus_spec(seed=seed)


def _levels(tree, p):
    depth = []
    for s in tree.parent[p]:
        depth.append(0 if s < 0 else depth[s] + 1)
    return [torch.tensor([i for i, d in enumerate(depth) if d == k], device="cuda") for k in range(max(depth) + 1)]


def _strategies(tree, p, H, hs, batch, gen, sequence_form=True):
    """Random strategies: per node and hand a uniform draw from the simplex,
    in sequence form (products along the path) or behavioural."""
    n = tree.n(p)
    e = torch.zeros(batch, n, hs, device="cuda")
    e[..., :H] = torch.empty(batch, n, H, device="cuda").exponential_(generator=gen)
    tot, at = torch.empty_like(e), 0
    for na in tree.nact[p]:                 # a node's sequences are consecutive
        tot[:, at:at + na] = e[:, at:at + na].sum(1, keepdim=True)
        at += na
    e /= tot.clamp_min_(1e-30)
    if sequence_form:
        par = torch.tensor(tree.parent[p], device="cuda")
        for lv in _levels(tree, p)[1:]:
            e[:, lv] *= e[:, par[lv]]
    return e


def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    return g


def _players(case):
    return {"A": (0,), "AT": (1,), "both": (0, 1)}[case.get("direction", "both")]


def _batch_specs(case, seed):
    """Board sizes and betting menus by the case, cards and beliefs by the seed."""
    out = []
    for i, s in enumerate(synth.batch_specs(seed=case["mix"], n=case["games"])):
        new = synth.river_spec(seed=1000003 * (seed + 1) + i, nboard=len(s["board"]))
        out.append(dict(s, **{k: new[k] for k in ("board", "strength", "mu1", "mu2")}))
    return out


def _river_specs(case, seed):
    return [synth.river_spec(seed=1000003 * (seed + 1) + i) for i in range(case["games"])]


def _menu_key(spec):
    return (tuple(spec["bet_frac"]), spec["raise_cap"], bool(spec["allow_allin"]), spec["stack"][0], spec["contrib0"][0])


def _trees(specs):
    seen = {}
    for s in specs:
        if _menu_key(s) not in seen:
            seen[_menu_key(s)] = Tree(s)
    return [seen[_menu_key(s)] for s in specs]


def _hs(H):
    return (H + 7) // 8 * 8


def _flat(specs, trees, player, gen, sequence_form=True):
    """One strategy per game, concatenated in game order."""
    out = [None] * len(specs)
    groups = {}
    for i, (s, t) in enumerate(zip(specs, trees)):
        groups.setdefault((id(t), len(s["strength"])), []).append(i)
    for (_, H), idx in groups.items():
        v = _strategies(trees[idx[0]], player, H, _hs(H), len(idx), gen, sequence_form)
        for k, i in enumerate(idx):
            out[i] = v[k].reshape(-1)
    return torch.cat(out)


def _turn_spec(case, seed):
    return synth.turn_spec(seed=seed, raise_cap_t=case["turn_cap"], raise_cap_r=case["river_cap"])


def _turn_games(spec):
    """(ending contribution, river card) and betting tree of every game of a
    turn endgame's layout, the turn round first."""
    N = spec["ranks"] * spec["suits"]
    cards = [c for c in range(N) if c not in set(spec["board"])]
    turn = Tree(dict(spec, bet_frac=spec["bet_frac_t"], raise_cap=spec["raise_cap_t"], allow_allin=False))
    games = [(None, None, turn)]
    trees = {}
    for _s1, _s2, show, c in turn.terms:
        if not show:
            continue
        if c not in trees:
            trees[c] = Tree(dict(spec, bet_frac=spec["bet_frac_r"], raise_cap=spec["raise_cap_r"], allow_allin=False,
                                 contrib0=[c, c], stack=[spec["contrib0"][p] + spec["stack"][p] - c for p in (0, 1)]))
        games += [(c, r, trees[c]) for r in cards]
    turn.terms = [t if not t[2] else (t[0], t[1], True, 0.0) for t in turn.terms]
    return games


# feature rows of the network as a training program has them: board one-hot,
# opponent histogram, node part, hand part
def _train_data(case, seed):
    gen, rows, steps = _gen(seed), case["rows"], case["steps"]
    n, G = rows * steps, 64
    X = torch.zeros(n, DIN, device="cuda")
    board = torch.rand(G, 52, device="cuda", generator=gen).argsort(1)[:, :5]
    hist = torch.rand(G, HIST, device="cuda", generator=gen) + 0.5
    hist /= hist.sum(1, keepdim=True)
    g = torch.randint(G, (n,), device="cuda", generator=gen)
    X[:, :52].scatter_(1, board[g], 1.0)
    X[:, 52:52 + HIST] = hist[g]
    node = torch.randint(15, (n, 1), device="cuda", generator=gen)
    X[:, 1133:1165].scatter_(1, node, 1.0)
    nact = torch.randint(2, 5, (n,), device="cuda", generator=gen).to(torch.int32)
    X[:, 1165] = torch.randint(2, (n,), device="cuda", generator=gen).float()
    X[:, 1166] = nact / 12.0
    X[:, 1167] = torch.randint(4, (n,), device="cuda", generator=gen) / 8.0
    X[:, 1173] = torch.rand(n, device="cuda", generator=gen)
    X[:, 1174] = 1.0 / 32
    X[:, 1175] = torch.rand(n, device="cuda", generator=gen) + 0.5
    two = torch.rand(n, 52, device="cuda", generator=gen).argsort(1)[:, :2]
    X[:, 1177:1229].scatter_(1, two, 1.0)
    live = torch.arange(DOUT, device="cuda")[None] < nact[:, None]
    T = torch.empty(n, DOUT, device="cuda").exponential_(generator=gen) * live
    T /= T.sum(1, keepdim=True)
    w = torch.rand(n, device="cuda", generator=gen) + 1e-3
    return [tuple(a[k * rows:(k + 1) * rows].contiguous() for a in (X, nact, T, w)) for k in range(steps)]


def _params(seed):
    r = np.random.default_rng(seed)
    out = []
    for a, b in ((DIN, WIDTH), (WIDTH, WIDTH), (WIDTH, DOUT)):
        out += [r.normal(0.0, math.sqrt(2.0 / a), size=a * b), r.normal(0.0, 0.05, size=b)]
    return np.concatenate(out).astype(np.float32)


def _split(flat):
    out, k = [], 0
    for a, b in ((DIN, WIDTH), (WIDTH, WIDTH), (WIDTH, DOUT)):
        out.append(flat[k:k + a * b].reshape(a, b))
        out.append(flat[k + a * b:k + a * b + b])
        k += a * b + b
    return out


# ---- the cases ----------------------------------------------------------------
def prepare(case, seed):
    gen, path = _gen(seed), case["path"]
    if path == "product":
        spec = _spec(case["game"], seed)
        tree, H = Tree(spec), len(spec["strength"])
        game = kps.Game(spec)
        game.upload()
        work = []
        for p in _players(case):
            v = _strategies(tree, 1 - p, H, _hs(H), case["batch"], gen).to(DT[case["dtype"]])
            work.append((p, v, torch.empty(case["batch"], tree.n(p), _hs(H), device="cuda", dtype=DT[case["dtype"]])))
        return dict(path=path, game=game, work=work, batch=case["batch"])
    if path == "batch":
        specs = _batch_specs(case, seed)
        trees = _trees(specs)
        batch = kps.Batch([kps.Game(s) for s in specs])
        v = [_flat(specs, trees, p, gen).to(DT[case["dtype"]]) for p in (0, 1)]
        return dict(path=path, batch=batch, v=v, out=[torch.empty_like(a) for a in v])
    if path == "turn":
        spec = _turn_spec(case, seed)
        turn, games = kps.Turn(spec), _turn_games(spec)
        H = spec["strength"].shape[1]
        one = dict(strength=np.zeros(H))
        v = [_flat([one] * len(games), [g[2] for g in games], p, gen).to(DT[case["dtype"]]) for p in (0, 1)]
        return dict(path=path, turn=turn, v=v, out=[torch.empty_like(a) for a in v])
    if path == "solve":
        specs = _river_specs(case, seed)
        batch = kps.Batch([kps.Game(s) for s in specs])
        solver = kps.Solver(batch, kps.F32)
        avg = [torch.zeros(int(batch.offsets(p)[-1]), dtype=torch.float64, device="cuda") for p in (0, 1)]
        return dict(path=path, batch=batch, solver=solver, avg=avg, iters=case["iters"])
    if path == "exploit":
        specs = _river_specs(case, seed)
        trees = _trees(specs)
        batch = kps.Batch([kps.Game(s) for s in specs])
        solver = kps.Solver(batch, kps.F64)
        beh = [_flat(specs, trees, p, gen, False) for p in (0, 1)]
        solver.reset(beh[0], beh[1])
        torch.cuda.synchronize()
        avg = [torch.zeros(b.numel(), dtype=torch.float64, device="cuda") for b in beh]
        e = [torch.zeros(case["games"], dtype=torch.float64, device="cuda") for _ in range(3)]
        return dict(path=path, batch=batch, solver=solver, avg=avg, e=e)
    if path == "train":
        mlp = kps.MLP(seed=seed)
        mlp.set(_params(seed))
        data = [d + (float(d[3].sum().item()),) for d in _train_data(case, seed)]
        return dict(path=path, mlp=mlp, data=data, rows=case["rows"], loss=torch.zeros(case["steps"], device="cuda"),
                    P=torch.zeros(case["rows"], DOUT, device="cuda"))
    specs = _river_specs(case, seed)
    batch = kps.Batch([kps.Game(s) for s in specs])
    mlp = kps.MLP(seed=seed)
    mlp.set(_params(seed))
    kps.warm_num_queries(batch)
    beh = [torch.zeros(int(batch.offsets(p)[-1]), device="cuda") for p in (0, 1)]
    return dict(path=path, batch=batch, mlp=mlp, beh=beh)


def run(state):
    path = state["path"]
    if path == "product":
        for p, v, out in state["work"]:
            (kps.matvec_A if p == 0 else kps.matvec_AT)(state["game"], v, out, state["batch"])
        return [out for _, _, out in state["work"]]
    if path in ("batch", "turn"):
        obj, v, out = state[path], state["v"], state["out"]
        obj.matvec_A(v[1], out[0])
        obj.matvec_AT(v[0], out[1])
        return out
    if path == "solve":
        s, avg = state["solver"], state["avg"]
        s.reset()
        s.step(state["iters"])
        s.average(avg[0], avg[1])
        return [a.float() for a in avg]
    if path == "exploit":
        s, avg, e = state["solver"], state["avg"], state["e"]
        s.average(avg[0], avg[1])
        s.exploitability(e[0], e[1], e[2])
        return {"x": avg[0], "y": avg[1], "expl": e[0], "br1": e[1], "br2": e[2]}
    if path == "train":
        m, rows, loss = state["mlp"], state["rows"], state["loss"]
        for k, (X, nact, T, w, wsum) in enumerate(state["data"]):
            m.gradients(X, rows, nact, T, w, wsum, loss[k:k + 1])
        m.forward(X, rows, nact, state["P"])
        return {"grad": m.get(1), "loss": loss, "P": state["P"]}
    kps.warm_predict(state["batch"], state["mlp"], state["beh"][0], state["beh"][1])
    return state["beh"]


def work(case):
    path = case["path"]
    if path == "product":
        spec = _spec(case["game"], 0)
        t, H, d = Tree(spec), len(spec["strength"]), len(_players(case))
        # per terminal and hand: scale, running mass, two cards in, two out, combine
        return {"bytes": d * case["batch"] * SIZE[case["dtype"]] * H * (t.n(0) + t.n(1)),
                "flops": d * case["batch"] * 8.0 * H * len(t.terms)}
    if path == "batch":
        specs = _batch_specs(case, 0)
        sizes = [(len(s["strength"]), t) for s, t in zip(specs, _trees(specs))]
        return {"bytes": sum(2 * SIZE[case["dtype"]] * H * (t.n(0) + t.n(1)) for H, t in sizes),
                "flops": sum(16.0 * H * len(t.terms) for H, t in sizes)}
    if path == "turn":
        games = _turn_games(_turn_spec(case, 0))
        H = 1128
        return {"bytes": sum(2 * SIZE[case["dtype"]] * H * (g[2].n(0) + g[2].n(1)) for g in games),
                "flops": sum(16.0 * H * len(g[2].terms) for g in games)}
    spec = synth.river_spec(seed=1)
    t, H = Tree(spec), len(spec["strength"])
    seq = t.n(0) + t.n(1)
    if path == "solve":
        # per iteration, sequence and hand: the products read and write one value each, the
        # update reads value, regret, sum and strategy and writes the last three; then the averages
        return {"bytes": case["games"] * H * seq * (case["iters"] * 4.0 * 9 + 4 + 8 + 8 + 4),
                "flops": case["games"] * H * case["iters"] * (16.0 * len(t.terms) + 12.0 * seq)}
    if path == "exploit":
        # averages out, read by the products, whose results the best responses read
        return {"bytes": case["games"] * H * seq * 8.0 * 5, "flops": case["games"] * H * (16.0 * len(t.terms) + 4.0 * seq)}
    macs = DIN * WIDTH + WIDTH * WIDTH + WIDTH * DOUT
    if path == "train":
        return {"bytes": case["steps"] * (4.0 * case["rows"] * (DIN + DOUT + 2) + 6.0 * macs),
                "flops": case["rows"] * (case["steps"] * (6.0 * macs - 2.0 * DIN * WIDTH) + 2.0 * macs)}
    q = case["games"] * H * (len(t.nact[0]) + len(t.nact[1]))
    # the first layer's sparse hand part, the two dense layers
    return {"bytes": 4.0 * case["games"] * H * seq, "flops": q * 2.0 * (5 * WIDTH + WIDTH * WIDTH + WIDTH * DOUT)}


# ---- exact results --------------------------------------------------------
def _pad(v, hs):
    return torch.nn.functional.pad(v, (0, hs - v.shape[-1]))


def _exact_products(games, v):
    """games: (tree, cards) per game; v: flat player vectors; both products."""
    out = ([], [])
    off = [0, 0]
    for tree, cards in games:
        hs = _hs(cards.H)
        x = []
        for p in (0, 1):
            n = tree.n(p) * hs
            x.append(v[p][off[p]:off[p] + n].double().view(1, tree.n(p), hs)[..., :cards.H])
            off[p] += n
        out[0].append(_pad(_apply(tree, cards, x[1], 0), hs).reshape(-1))
        out[1].append(_pad(_apply(tree, cards, x[0], 1), hs).reshape(-1))
    return [torch.cat(o) for o in out]


def _exact_turn(spec, v):
    N, k = spec["ranks"] * spec["suits"] - len(spec["board"]), 2
    H = spec["strength"].shape[1]
    canon = _hands(spec).numpy()
    base = Cards(spec, strength=np.arange(H))
    beta, memo = base.beta * (N - 2 * k), {}

    def games():
        for c, r, tree in _turn_games(spec):
            if c is None:
                yield tree, base
                continue
            if r not in memo:
                holds = (canon == r).any(1)
                s = np.where(holds, -1 - np.arange(H), spec["strength"][r])
                memo[r] = Cards(spec, strength=s, beta_scale=beta, mask=lambda h, r=r: (h != r).all(1))
            yield tree, memo[r]

    return _exact_products(games(), v)


def _sequence_form(beh, tree, p):
    x = beh.clone()
    for lv in _levels(tree, p)[1:]:
        x[:, lv] *= x[:, torch.tensor(tree.parent[p], device="cuda")[lv]]
    return x


class _Many:
    """Endgames of one betting tree, stacked."""

    def __init__(self, specs):
        self.tree = Tree(specs[0])
        self.cards = [Cards(s) for s in specs]
        self.C = torch.stack([c.C for c in self.cards])
        self.W = torch.stack([c.W for c in self.cards])
        self.lam = [torch.stack([c.lam[p] for c in self.cards])[:, None] for p in (0, 1)]
        self.H = self.cards[0].H

    def product(self, v, p):
        tree, q = self.tree, 1 - p
        x = v * self.lam[q]
        out = torch.zeros(v.shape[0], tree.n(p), self.H, dtype=torch.float64, device=v.device)
        for show, M in ((False, self.C), (True, self.W)):
            t = [(a[p], a[q], a[3]) for a in tree.terms if a[2] == show]
            rows, cols = (torch.tensor([a[k] for a in t], device=v.device) for k in (0, 1))
            coef = torch.tensor([a[2] * (-1.0 if show and p else 1.0) for a in t], dtype=torch.float64, device=v.device)
            out.index_add_(1, rows, torch.bmm(x[:, cols], M.transpose(1, 2)) * coef[:, None])
        return out * self.lam[p]


def _exact_solve(case, specs):
    m = _Many(specs)
    tree, G, H = m.tree, len(specs), m.H
    theta = []
    for p in (0, 1):
        theta.append(torch.tensor([tree.payoff * float(c.mu[p].max()) * float(c.mu[1 - p].sum()) / c.beta / 65536.0
                                   for c in m.cards], dtype=torch.float64, device="cuda")[:, None, None])
    nodes = []
    for p in (0, 1):
        first = {}
        for s, k in enumerate(tree.node[p]):
            first.setdefault(k, []).append(s)
        nodes.append([(first[k], tree.parent[p][first[k][0]]) for k in range(len(first))])
    R = [torch.zeros(G, tree.n(p), H, dtype=torch.float64, device="cuda") for p in (0, 1)]
    S = [torch.zeros_like(r) for r in R]
    beh = [torch.zeros_like(r) for r in R]

    def play(p):
        for seqs, _ in nodes[p]:
            r = R[p][:, seqs].clamp_min(0.0)
            tot = r.sum(1, keepdim=True)
            beh[p][:, seqs] = torch.where(tot > theta[p], r / tot, 1.0 / len(seqs))
        return _sequence_form(beh[p], tree, p)

    x = [play(0), play(1)]
    weight = 0.0
    for t in range(1, case["iters"] + 1):
        weight += t
        for p in (0, 1):
            S[p] += float(t) * x[p]
            q = m.product(x[1 - p], p) * (1.0 if p == 0 else -1.0)
            for seqs, par in reversed(nodes[p]):
                v = (beh[p][:, seqs] * q[:, seqs]).sum(1, keepdim=True)
                R[p][:, seqs] = (R[p][:, seqs] + q[:, seqs] - v).clamp_min(0.0)
                if par >= 0:
                    q[:, par] += v[:, 0]
            x[p] = play(p)
    return [_pad(s / weight, _hs(H)).reshape(-1) for s in S]


def _exact_exploit(specs, beh):
    m = _Many(specs)
    tree, G, H = m.tree, len(specs), m.H
    hs = _hs(H)
    x = [_sequence_form(beh[p].double().view(G, tree.n(p), hs)[..., :H], tree, p) for p in (0, 1)]
    br = []
    for p in (0, 1):
        q = m.product(x[1 - p], p) * (1.0 if p == 0 else -1.0)
        root = torch.zeros(G, H, dtype=torch.float64, device="cuda")
        for k in reversed(range(len(tree.nact[p]))):
            seqs = [s for s, n in enumerate(tree.node[p]) if n == k]
            best = q[:, seqs].max(1).values
            par = tree.parent[p][seqs[0]]
            if par >= 0:
                q[:, par] += best
            else:
                root += best
        br.append(root.sum(1))
    pot = [s["contrib0"][0] + s["contrib0"][1] for s in specs]
    e = (br[0] + br[1]) / 2 / torch.tensor(pot, dtype=torch.float64, device="cuda")
    return {"x": _pad(x[0], hs).reshape(-1), "y": _pad(x[1], hs).reshape(-1), "expl": e, "br1": br[0], "br2": br[1]}


def _bf(a):
    return a.float().to(torch.bfloat16).double()


def _exact_train(case, seed):
    W1, b1, W2, b2, W3, b3 = _split(torch.from_numpy(_params(seed)).cuda().double())
    W1, W2, W3 = _bf(W1), _bf(W2), _bf(W3)
    losses = []
    for X, nact, T, w in _train_data(case, seed):
        X, T, w = X.double(), T.double(), w.double()
        a1 = X @ W1 + b1
        h1 = a1.clamp_min(0)
        a2 = h1 @ W2 + b2
        h2 = a2.clamp_min(0)
        z = h2 @ W3 + b3
        live = torch.arange(DOUT, device="cuda")[None] < nact[:, None]
        lp = torch.log_softmax(z.masked_fill(~live, -math.inf), 1).masked_fill(~live, 0.0)
        wn = (w / w.sum())[:, None]
        losses.append(-(wn * T * lp).sum())
    P = lp.exp() * live
    dz = wn * (P * T.sum(1, keepdim=True) - T) * live
    dh2 = (dz @ W3.T) * (a2 > 0)
    dh1 = (dh2 @ W2.T) * (a1 > 0)
    g = torch.cat([t.reshape(-1) for t in (X.T @ dh1, dh1.sum(0), h1.T @ dh2, dh2.sum(0), h2.T @ dz, dz.sum(0))])
    return {"grad": g, "loss": torch.stack(losses), "P": P}


def _exact_predict(case, specs, seed):
    W1, b1, W2, b2, W3, b3 = _split(torch.from_numpy(_params(seed)).cuda().double())
    W1, W2, W3 = _bf(W1), _bf(W2), _bf(W3)
    tree = Tree(specs[0])
    depth = []
    for p in (0, 1):
        d = []
        for k in range(len(tree.nact[p])):
            par = tree.parent[p][tree.node[p].index(k)]
            d.append(0 if par < 0 else d[tree.node[p][par]] + 1)
        depth.append(d)
    out = ([], [])
    for spec in specs:
        order = _order(spec["strength"])
        H, s = len(order), np.asarray(spec["strength"])[order]
        hand = _hands(spec, "cuda")[torch.from_numpy(order).cuda()]
        _, inv, cnt = np.unique(s, return_inverse=True, return_counts=True)
        board = torch.zeros(52, dtype=torch.float64, device="cuda")
        board[torch.tensor(spec["board"], device="cuda")] = 1.0
        mu = [torch.from_numpy(np.asarray(spec[k])[order]).cuda() for k in ("mu1", "mu2")]
        pos = torch.arange(H, device="cuda")
        hf = torch.zeros(H, 56, dtype=torch.float64, device="cuda")
        hf[:, 0] = pos / (H - 1.0)
        hf[:, 1] = torch.from_numpy(cnt[inv] / 32.0).cuda()
        hf.scatter_(1, hand + 4, 1.0)
        for p in (0, 1):
            hist = torch.zeros(HIST, dtype=torch.float64, device="cuda")
            hist.index_add_(0, pos * HIST // H, mu[1 - p] / mu[1 - p].sum())
            hf[:, 2] = mu[p] * H / mu[p].sum()
            nf = torch.zeros(len(tree.nact[p]), 40, dtype=torch.float64, device="cuda")
            for k, na in enumerate(tree.nact[p]):
                nf[k, k] = 1.0
                nf[k, 32], nf[k, 33], nf[k, 34] = p, na / 12.0, depth[p][k] / 8.0
            a1 = (torch.cat([board, hist]) @ W1[:1133] + b1) + (hf @ W1[1173:1229])[None] + (nf @ W1[1133:1173])[:, None]
            z = (a1.clamp_min(0) @ W2 + b2).clamp_min(0) @ W3 + b3
            res = torch.zeros(tree.n(p), _hs(H), dtype=torch.float64, device="cuda")
            at = 0
            for k, na in enumerate(tree.nact[p]):
                res[at:at + na, :H] = torch.softmax(z[k, :, :na], 1).T
                at += na
            out[p].append((tree, res))
    return [_by_sequence(o, p) for p, o in enumerate(out)]


def _by_sequence(parts, p):
    """Rows node after node -> rows in sequence order."""
    tree = parts[0][0]
    at, where = 0, [0] * tree.n(p)
    for k, na in enumerate(tree.nact[p]):
        for s in [s for s, n in enumerate(tree.node[p]) if n == k]:
            where[s] = at
            at += 1
    idx = torch.tensor(where, device="cuda")
    return torch.cat([r[idx].reshape(-1) for _, r in parts])


def exact(case, seed):
    path = case["path"]
    s = _inputs(case, seed) if path in ("product", "batch", "turn", "exploit") else None
    if path == "product":
        spec = _spec(case["game"], seed)
        tree, cards = Tree(spec), Cards(spec)
        return [_pad(_apply(tree, cards, v.double()[..., :cards.H], p), _hs(cards.H))
                for p, v in zip(_players(case), s)]
    if path == "batch":
        specs = _batch_specs(case, seed)
        return _exact_products(((t, Cards(sp)) for sp, t in zip(specs, _trees(specs))), s)
    if path == "turn":
        return _exact_turn(_turn_spec(case, seed), s)
    if path == "solve":
        return _exact_solve(case, _river_specs(case, seed))
    if path == "exploit":
        return _exact_exploit(_river_specs(case, seed), s)
    if path == "train":
        return _exact_train(case, seed)
    return _exact_predict(case, _river_specs(case, seed), seed)


def _inputs(case, seed):
    """The vectors prepare() draws, without the library's objects."""
    gen, path = _gen(seed), case["path"]
    if path == "product":
        spec = _spec(case["game"], seed)
        tree, H = Tree(spec), len(spec["strength"])
        return [_strategies(tree, 1 - p, H, _hs(H), case["batch"], gen).to(DT[case["dtype"]]) for p in _players(case)]
    if path == "turn":
        spec = _turn_spec(case, seed)
        games = _turn_games(spec)
        specs, trees = [dict(strength=np.zeros(spec["strength"].shape[1]))] * len(games), [g[2] for g in games]
    else:
        specs = _batch_specs(case, seed) if path == "batch" else _river_specs(case, seed)
        trees = _trees(specs)
    form = path != "exploit"
    return [_flat(specs, trees, p, gen, form).to(DT[case.get("dtype", "f32")]) for p in (0, 1)]
