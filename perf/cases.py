"""Performance cases: exact two-terminal reliability as programs ask for it.

A case names a network (its size, its recipe and the seed that fixes its
arcs), the reliabilities' range, the outputs wanted and the entry point:

  call      reliability_net with host arrays: one question, one answer
  plan      a kept Plan: execute, then read
  autograd  PBATReliability on a CUDA tensor, forward and backward
  batch     reliability_batched: many networks, many reliability vectors

The network belongs to the case -- a program studies one network, or one set
of networks, under many reliability vectors -- and the vectors are drawn from
the seed given to prepare().  Sizes and recipes are those of this
repository's benchmark and tests: random connected undirected graphs (a
random spanning tree, then uniform non-edges), random directed graphs (a
random arborescence out of the source, then uniform ordered pairs) and
rectangular grids.
"""
import random
from types import SimpleNamespace

import numpy as np
import torch

import paper_2209_09711_gb300 as pb


def listed():
    return [
        # One reliability of a small network, asked for on its own: the call's
        # latency is all there is (2^9 states).
        dict(name="call R, n6 m9", kind="call", graph="undirected", n=6, m=9, net=11, plo=0.80, phi=0.99,
             grad=False, prune=1, tune=0, range_bits=0),
        # A reliability inside a loss that is minimised: R and its gradient
        # through autograd on a CUDA tensor (2^16 states, twice).
        dict(name="autograd, n8 m16", kind="autograd", graph="undirected", n=8, m=16, net=12, plo=0.80, phi=0.99,
             grad=True, prune=1, tune=0, range_bits=0),
        # The 3x6 grid of 27 arcs, corner to corner: R alone in one call, and
        # the importance of every arc from a kept plan.  No tuning, as in a
        # program that meets many structures.
        dict(name="call R, grid 3x6", kind="call", graph="grid", n=18, m=27, net=3, plo=0.85, phi=0.95,
             grad=False, prune=1, tune=0, range_bits=0),
        dict(name="plan grad, grid 3x6", kind="plan", graph="grid", n=18, m=27, net=3, plo=0.85, phi=0.95,
             grad=True, prune=1, tune=0, range_bits=0),
        # Directed networks of 34 arcs (2^34 states): the gradient from a kept
        # plan with prune-aware planning, and R alone with the default planning.
        dict(name="plan grad, directed n20 m34", kind="plan", graph="directed", n=20, m=34, net=13, plo=0.85, phi=0.99,
             grad=True, prune=2, tune=0, range_bits=0),
        dict(name="call R, directed n20 m34", kind="call", graph="directed", n=20, m=34, net=13, plo=0.85, phi=0.99,
             grad=False, prune=1, tune=0, range_bits=0),
        # The largest: 24 nodes, 40 arcs (2^40 states).  The gradient from a
        # kept plan; R alone in one call with every default, tuned once.
        dict(name="plan grad, n24 m40", kind="plan", graph="undirected", n=24, m=40, net=14, plo=0.90, phi=0.999,
             grad=True, prune=2, tune=0, range_bits=0),
        dict(name="call R tuned, n24 m40", kind="call", graph="undirected", n=24, m=40, net=14, plo=0.90, phi=0.999,
             grad=False, prune=1, tune=1, range_bits=0),
        # A dense network, where few prefixes decide the sink's fate and most
        # states are walked (2^31 states, an odd number of arcs and nodes).
        dict(name="call grad, dense n11 m31", kind="call", graph="undirected", n=11, m=31, net=15, plo=0.60, phi=0.95,
             grad=True, prune=1, tune=0, range_bits=0),
        # Unreliable arcs: R is so small that the exact kernel answers (2^23 states).
        dict(name="call grad, unreliable n9 m23", kind="call", graph="undirected", n=9, m=23, net=16, plo=0.01, phi=0.04,
             grad=True, prune=1, tune=0, range_bits=0),
        # Design-space sweeps: 64 networks x 16 vectors for R, every default
        # (tuned once); a smaller ragged set, 20 x 7, with every gradient.
        dict(name="batch R tuned, 64 x 16", kind="batch", graph="undirected", graphs=64, vectors=16, nlo=8, nhi=20,
             mlo=20, mhi=32, net=17, plo=0.60, phi=0.999, grad=False, prune=1, tune=1),
        dict(name="batch grad, 20 x 7", kind="batch", graph="undirected", graphs=20, vectors=7, nlo=7, nhi=16,
             mlo=15, mhi=29, net=18, plo=0.60, phi=0.999, grad=True, prune=1, tune=0),
    ]


def draw(rng):
    """One more case of the same ranges (never more than the 2^40 network's work)."""
    kind = rng.choice(["call", "call", "plan", "plan", "autograd", "batch"])
    case = dict(kind=kind, net=rng.randrange(1000, 1 << 20), tune=0)
    if kind == "batch":
        lo = rng.randint(10, 20)
        case.update(graph="undirected", graphs=rng.randint(2, 24), vectors=rng.choice([1, 3, 5, 8, 13, 16, 17]),
                    nlo=6, nhi=rng.randint(9, 16), mlo=lo, mhi=lo + rng.randint(1, 8), plo=0.6, phi=0.999,
                    grad=rng.random() < 0.5, prune=rng.choice([1, 2]))
        return case
    unreliable = kind == "call" and rng.random() < 0.25
    top = 24 if unreliable else 28 if kind == "autograd" else 34
    m = rng.randint(6, top)
    graph = rng.choice(["undirected", "undirected", "directed"])
    # from trees with a few extra arcs (sparse) to close to complete (dense)
    least = 3
    while least * (least - 1) // (2 if graph == "undirected" else 1) < m:
        least += 1
    n = rng.randint(least, max(least, min(26, (2 * m) // 3)))
    case.update(graph=graph, n=n, m=m, grad=kind == "autograd" or rng.random() < 0.6, prune=rng.choice([1, 1, 2]),
                range_bits=rng.choice([0, 0, 0, 2, 3]) if m >= 20 and not unreliable and kind != "autograd" else 0)
    case.update(plo=0.01, phi=0.05) if unreliable else case.update(plo=0.85, phi=0.99)
    return case


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------

def _random_arcs(graph, n, m, rng):
    if graph == "grid":
        rows, cols = 3, n // 3
        arcs = []
        for r in range(rows):
            for c in range(cols):
                arcs += [(r * cols + c, r * cols + c + 1)] * (c + 1 < cols)
                arcs += [(r * cols + c, r * cols + c + cols)] * (r + 1 < rows)
        assert len(arcs) == m
        return arcs
    order = list(range(1, n))
    if graph == "directed":
        rng.shuffle(order)
    order = [0] + order
    arcs, seen = [], set()
    for i in range(1, n):
        arcs.append((order[rng.randrange(i)], order[i]))
        seen.add(arcs[-1] if graph == "directed" else tuple(sorted(arcs[-1])))
    while len(arcs) < m:
        u, v = rng.randrange(n), rng.randrange(n)
        key = (u, v) if graph == "directed" else (min(u, v), max(u, v))
        if u != v and key not in seen:
            seen.add(key)
            arcs.append((u, v))
    return arcs[:m]


def _network(graph, n, m, rng):
    arcs = _random_arcs(graph, n, m, rng)
    return SimpleNamespace(n=n, m=len(arcs), tail=[a for a, _ in arcs], head=[b for _, b in arcs], source=0,
                           sink=n - 1, directed=graph == "directed")


def _networks(case):
    """The networks of a case (one, unless it is a batch)."""
    if case["kind"] != "batch":
        n = case["n"]
        if case["graph"] != "grid" and case["m"] < n - 1:
            n = case["m"] + 1
        return [_network(case["graph"], n, case["m"], random.Random(case["net"]))]
    rng, nets = random.Random(case["net"]), []
    for _ in range(case["graphs"]):
        m = rng.randint(case["mlo"], case["mhi"])
        n = rng.randint(case["nlo"], case["nhi"])
        while n * (n - 1) // 2 < m:
            n += 1
        nets.append(_network("undirected", min(n, m + 1), m, rng))
    return nets


def _vectors(case, nets, seed):
    """Per network, one row of reliabilities per vector."""
    rng = np.random.RandomState(seed % (1 << 32))
    rows = case.get("vectors", 1)
    return [case["plo"] + (case["phi"] - case["plo"]) * rng.random_sample((rows, g.m)) for g in nets]


def _range(case, seed):
    """The equal division asked for: block `seed` of 2^range_bits, as one of several machines would take it."""
    bits = case.get("range_bits", 0)
    return (bits, seed % (1 << bits)) if bits else (0, 0)


def _options(case, seed):
    bits, block = _range(case, seed)
    more = dict(range_bits=bits, range_lo=block, range_hi=block + 1) if bits else {}
    return pb.options(prune=case["prune"], autotune=case["tune"], **more)


def prepare(case, seed):
    nets = _networks(case)
    vectors = _vectors(case, nets, seed)
    state = dict(kind=case["kind"], grad=case["grad"], nets=nets, opts=_options(case, seed))
    if case["kind"] == "batch":
        state["p"] = [[list(row) for row in v] for v in vectors]
    elif case["kind"] == "autograd":
        state["p"] = torch.tensor(vectors[0][0], dtype=torch.float64, device="cuda", requires_grad=True)
    elif case["kind"] == "plan":
        state["plan"] = pb.Plan(nets[0], p=vectors[0][0], grad=case["grad"], opts=state["opts"])
    else:
        state["p"] = vectors[0][0]
    return state


def run(state):
    kind, grad = state["kind"], state["grad"]
    if kind == "batch":
        R, Nk, grads = pb.reliability_batched(state["nets"], state["p"], grad=grad, opts=state["opts"])
        out = {"R": R, "Nk": np.concatenate([np.array(c, dtype=np.int64) for c in Nk])}
        if grad:
            out["grad"] = np.concatenate([g.ravel() for g in grads])
        return out
    if kind == "autograd":
        R = pb.PBATReliability.apply(state["p"], state["nets"][0], state["opts"])
        (g,) = torch.autograd.grad(R, state["p"])
        return {"R": R.detach(), "grad": g}
    if kind == "plan":
        state["plan"].execute()
        res = state["plan"].read()
    else:
        res = pb.reliability_net(state["nets"][0], p=state["p"], grad=grad, opts=state["opts"])
    out = {"R": np.array([res.R]), "Nk": np.array(res.Nk, dtype=np.int64)}
    if grad:
        out["grad"] = np.array(res.grad)
    return out


def work(case):
    """Reliabilities in, R, N_k and the gradient out; and for every 32 states
    (a word of them) one operation that decides each arc's word, the least a
    visit of all states 32 at a time can do."""
    ops = bytes_ = 0.0
    per = case.get("vectors", 1)
    for g in _networks(case):
        states = 2.0 ** (g.m - case.get("range_bits", 0))
        ops += states / 32 * (2 if case["kind"] == "autograd" else 1)
        bytes_ += 8.0 * (per * g.m + per + g.m + 1 + (per * g.m if case["grad"] else 0))
    return {"bytes": bytes_, "flops": ops}


def tolerance(case):
    """R and dR/dp are sums of integers, off by at most 2^-57 of the enumerated
    mass before they are rounded to doubles once, at the end: against exact()
    the vectors' relative error is up to 2e-16, and 2^-57 over a gradient of
    0.004 is 2e-15.  N_k is whole and exact."""
    return {"rel": 2e-15, "max": 2e-14, "differ": 0.0}


# ---------------------------------------------------------------------------
# the same values from a dynamic program over the arcs, in 64 bits
# ---------------------------------------------------------------------------

_MOST_RECORDS = 400_000


def _arc_order(net):
    """Arcs node by node, the next node being the one that leaves the fewest open."""
    arcs = list(zip(net.tail, net.head))
    left, order, opened = set(range(net.m)), [], {net.source, net.sink}
    while left:
        best = None
        for v in range(net.n):
            mine = [k for k in left if v in arcs[k]]
            if not mine:
                continue
            rest = left - set(mine)
            nodes = opened | {x for k in mine for x in arcs[k]}
            live = {x for k in rest for x in arcs[k]}
            score = (len(nodes & live), len(mine))
            if best is None or score < best[0]:
                best = (score, mine, nodes)
        order += sorted(best[1])
        left -= set(best[1])
        opened = best[2]
    return order


def _layers(net):
    """Per arc, where each record of what the earlier arcs joined goes when
    the arc fails and when it works; None when there are too many records.

    A record holds, for the source, the sink and every node that still has
    arcs to come, the set of these it reaches.  -1: the sink is reached, -2:
    it cannot be any more."""
    order, arcs = _arc_order(net), list(zip(net.tail, net.head))
    s, t = net.source, net.sink
    last = {}
    for i, k in enumerate(order):
        for v in arcs[k]:
            last[v] = i
    records, layers, total = {(): 0}, [], 0   # a record: sorted ((a, b), ...) with a reaching b
    for i, k in enumerate(order):
        u, v = arcs[k]
        gone = [x for x in (u, v) if last[x] == i and x not in (s, t)]
        live = {x for x, at in last.items() if at > i}
        nxt, moves = {}, []

        def close(rel, pairs):
            rel = set(rel)
            for a, b in pairs:
                if (a, b) in rel or b == s or a == t:
                    continue
                before = {x for x, y in rel if y == a} | {a}
                after = {y for x, y in rel if x == b} | {b}
                rel |= {(x, y) for x in before for y in after if x != y and y != s and x != t}
            if (s, t) in rel:
                return -1
            # what the source reaches needs no other way in, what reaches the
            # sink no other way out
            got, wins = {y for x, y in rel if x == s}, {x for x, y in rel if y == t}
            rel = {(x, y) for x, y in rel if x not in gone and y not in gone and
                   not (y in got and x != s) and not (x in wins and y != t) and
                   (x == s or x in live or x in wins)}
            if not (got & live) and s not in live:
                return -2
            if not (wins & live) and t not in live:
                return -2
            key = tuple(sorted(rel))
            return nxt.setdefault(key, len(nxt))

        both = [(u, v)] if net.directed else [(u, v), (v, u)]
        for key in records:
            moves.append((close(key, []), close(key, both)))
        total += len(moves)
        if total > _MOST_RECORDS:
            return None
        layers.append((k, np.array(moves, dtype=np.int64).reshape(-1, 2), len(nxt)))
        records = nxt
    return layers


def _values(net, layers, P):
    """R and dR/dp for every row of P (rows x arcs), each as sums of positive terms."""
    rows = P.shape[0]
    forward = [np.ones((1, rows))]
    for k, moves, count in layers:
        now, nxt = forward[-1], np.zeros((count, rows))
        for works, w in ((0, 1 - P[:, k]), (1, P[:, k])):
            to = moves[:, works]
            np.add.at(nxt, to[to >= 0], now[to >= 0] * w)
        forward.append(nxt)
    # the chance that the sink is reached (up) or not (down) from each record
    up, down = np.zeros((0, rows)), np.zeros((0, rows))
    grad, R = np.zeros_like(P), None
    for (k, moves, count), now in zip(reversed(layers), reversed(forward[:-1])):
        up = np.concatenate([up, np.zeros((1, rows)), np.ones((1, rows))])      # ..., [-2], [-1]
        down = np.concatenate([down, np.ones((1, rows)), np.zeros((1, rows))])
        u0, u1, d0, d1 = up[moves[:, 0]], up[moves[:, 1]], down[moves[:, 0]], down[moves[:, 1]]
        grad[:, k] = (now * np.where(u1 < 0.5, u1 - u0, d0 - d1)).sum(0)
        up = u0 * (1 - P[:, k]) + u1 * P[:, k]
        down = d0 * (1 - P[:, k]) + d1 * P[:, k]
    return up[0], grad


def exact(case, seed):
    nets = _networks(case)
    vectors = _vectors(case, nets, seed)
    bits, block = _range(case, seed)
    Rs, grads, built = [], [], 0
    for net, P in zip(nets, vectors):
        layers = _layers(net)
        if layers is None:
            return None
        built += sum(len(m) for _, m, _ in layers)
        if built > _MOST_RECORDS:
            return None
        # a block fixes its first arcs: their chances are a factor of the rest
        F, chance = P.copy(), np.ones(P.shape)
        for i in range(bits):
            on = (block >> (bits - 1 - i)) & 1
            F[:, i], chance[:, i] = on, P[:, i] if on else 1 - P[:, i]
        R, g = _values(net, layers, F)
        g *= chance.prod(1, keepdims=True)
        for i in range(bits):
            sign = 1 if (block >> (bits - 1 - i)) & 1 else -1
            g[:, i] = sign * np.delete(chance, i, 1).prod(1) * R
        R = R * chance.prod(1)
        Rs.append(R)
        grads.append(g.ravel())
    if case["kind"] == "autograd":
        return {"R": torch.tensor(Rs[0][0], dtype=torch.float64), "grad": torch.from_numpy(grads[0])}
    out = {"R": np.stack(Rs) if case["kind"] == "batch" else Rs[0], "Nk": None}
    if case["grad"]:
        out["grad"] = np.concatenate(grads)
    return out
