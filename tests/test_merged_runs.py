"""Merged runs of the bit-sliced kernels: items whose prefixes leave the same
network share one walk.  On the CPU, the generated signature program is
evaluated in Python and compared with the connectivity it stands for; on the
GPU, merged runs are compared with one-launch runs and the oracle at the
sizes where blocks of items, words of signatures and tables change shape."""
import re

import pytest

import oracle
import synth

FULL = 0xFFFFFFFF


@pytest.fixture(scope="module")
def pb():
    from paper_2209_09711_gb300 import build
    build.build()
    import paper_2209_09711_gb300 as mod
    return mod


def _signature_program(src):
    perm = [int(x) for x in src.splitlines()[0].split(":")[1].split()]
    defs = {k: v for k, v in re.findall(r"#define (BS_\w+) (-?\w+)", src)}
    body = src[src.index("void bs_sig("):]
    return perm, defs, body[:body.index("\n}\n")]


def _evaluate(body, a, n):
    env, z = {"a": a}, [0] * n
    for line in body.splitlines()[1:]:
        line = re.sub(r"\b(0x[0-9a-f]+|0)u\b", r"\1", line)
        m = re.match(r"\s*const u32 (\w+) = (.*);$", line)
        if m:
            env[m.group(1)] = eval(m.group(2), {}, env) & FULL
            continue
        m = re.match(r"\s*(z\[(\d+)\]|dn|up) = (.*);$", line)
        value = eval(m.group(3), {}, env) & FULL
        if m.group(2):
            z[int(m.group(2))] = value
        else:
            env[m.group(1)] = value
    return z, env["dn"], env["up"]


def _residual(net, prefix, on, free):
    """What the working prefix arcs leave between the boundary nodes: who
    reaches whom, without what the source reaches and what reaches the sink
    already say."""
    s, t = net.source, net.sink
    bound = sorted({s, t} | {v for k in free for v in (net.tail[k], net.head[k])})
    reach = {v: {v} for v in range(net.n)}
    grew = True
    while grew:
        grew = False
        for k, works in zip(prefix, on):
            if not works:
                continue
            u, v = net.tail[k], net.head[k]
            for x, y in ((u, v),) if net.directed else ((u, v), (v, u)):
                if net.directed and (y == s or x == t):
                    continue
                for r in reach.values():
                    if x in r and y not in r:
                        r.add(y)
                        grew = True
    pairs = {(x, y) for x in bound for y in bound if x != y and y in reach[x]}
    if net.directed:
        pairs = {(x, y) for x, y in pairs
                 if x == s or y == t or not ((s, x) in pairs or (s, y) in pairs or (x, t) in pairs)}
    return frozenset(pairs)


@pytest.mark.parametrize("directed", [False, True])
@pytest.mark.parametrize("prune", [1, 2])
def test_signature_is_the_residual_network(pb, directed, prune):
    """Over 32 random items at a time, those whose prefix does not join source
    and sink: equal signatures exactly where the prefix leaves the same
    connectivity.  And both ends of the prune, for every item."""
    for seed in range(10):
        rng = synth.SplitMix64(8100 + seed)
        n, m = 3 + rng.below(9), 14 + rng.below(14)
        net = synth.random_small(8200 + seed, n=n, m=m, directed=directed)
        src = pb.kernel_source(net, pb.options(walk_bits=seed % 3, prune=prune, launches=2))
        perm, D, body = _signature_program(src)
        top, nsig = int(D["BS_TOP"]), int(D["BS_NSIG"])
        assert int(D["BS_MERGE"]) == 1 and 0 <= nsig <= 63
        words = [rng.next_u64() & FULL for _ in range(m)]
        z, dn, up = _evaluate(body, [0] * top + words[top:], nsig)
        items = [[(words[k] >> i) & 1 for k in range(top, m)] for i in range(32)]
        sig = [tuple((w >> i) & 1 for w in z) for i in range(32)]
        res = [_residual(net, perm[top:], on, perm[:top]) for on in items]
        st = (net.source, net.sink)   # items that join these are not classed
        for i, on in enumerate(items):
            rest = sum(1 << (m - 1 - a) for a in perm[:top])
            x = sum(1 << (m - 1 - a) for a, works in zip(perm[top:], on) if works)
            assert bool((dn >> i) & 1) == oracle.connected(net, x)
            assert bool((up >> i) & 1) == oracle.connected(net, x | rest)
        left = [i for i in range(32) if st not in res[i]]
        for i in left:
            for j in left:
                assert (sig[i] == sig[j]) == (res[i] == res[j]), (seed, i, j)


@pytest.mark.parametrize("m, bits, lo, hi, items_log2, merged", [
    # as many items as their walks are meant to leave, whatever the division:
    # the whole space, one division of it, an eighth in several divisions
    (36, 0, 0, 0, 20, True), (36, 3, 1, 2, 18, True), (39, 3, 0, 8, 23, True), (36, 6, 8, 16, 18, True),
    # not fewer than ten prefix arcs outside the range, for whole merge blocks
    (32, 12, 0, 1 << 12, 22, True), (34, 12, 0, 1 << 12, 22, True), (40, 10, 0, 1 << 10, 24, True),
    # wide ranges of many bits: more than 2^14 blocks of items, or more than 2^24
    # items -- one launch, and its long walks
    (36, 16, 0, 1 << 16, 16, False), (36, 16, 1 << 15, 1 << 16, 15, False), (36, 20, 0, 1 << 18, 18, False),
    (48, 10, 0, 1 << 10, 28, False),
    # narrow ranges: about 2^10 items in one launch, fewer where there are no more
    (36, 16, 7, 9, 10, False), (36, 24, 5, 6, 2, False), (30, 10, 0, 3, 10, False),
])
@pytest.mark.parametrize("grad", [False, True])
def test_walk_length_of_ranges(pb, m, bits, lo, hi, items_log2, merged, grad):
    """The planner's walk length follows the number of items of the range
    asked for, not that of one division."""
    tail, head, rng = synth.random_connected_undirected(12, m, 31)
    net = synth.Network(12, tail, head, synth.uniform_p(rng, m, 0.7, 0.95), 0, 11)
    src = pb.kernel_source(net, pb.options(range_bits=bits, range_lo=lo, range_hi=hi), grad=grad)
    D = {k: int(v) for k, v in re.findall(r"#define (BS_\w+) (-?\d+)", src)}
    width = (hi - lo) if bits else 1
    items = width << (D["BS_D"] - bits)
    assert (items - 1).bit_length() == items_log2, D
    assert D["BS_MERGE"] == merged


@pytest.mark.parametrize("m, n, walk, merged", [(26, 9, 4, 1), (39, 9, 5, 1), (40, 9, 5, 0), (34, 12, 5, 0)])
@pytest.mark.parametrize("grad", [False, True])
def test_walk_length_of_batches(pb, m, n, walk, merged, grad):
    """Untuned batches walk four arcs where they are merged, five where that
    makes the items few enough to be (39 arcs), and five as ever where they are
    not: too many items (40 arcs), too long a signature (directed, 12 nodes)."""
    net = synth.random_small(8600 + m, n=n, m=m, directed=n == 12, p_lo=0.2, p_hi=0.9)
    small = synth.random_small(8700, n=6, m=12, p_lo=0.2, p_hi=0.9)
    # (the sum of the items is limited: 39 arcs reach the limit alone)
    nets = [net] if m == 39 else [net, small]
    o = pb.options(autotune=0)
    src = (pb.batch_grad_kernel_source(nets, [[g.p] * 3 for g in nets], o) if grad
           else pb.batch_kernel_source(nets, 3, o))
    assert f"#define BSB_LMAX {walk}\n" in src and f"#define BSB_MERGE {merged}\n" in src
    # without the prune nothing is merged
    src = pb.batch_kernel_source(nets, 3, pb.options(autotune=0, prune=0))
    assert "#define BSB_LMAX 5\n" in src and "#define BSB_MERGE 0\n" in src


def _merged_sources(pb):
    """The kernels of a merged run, of one network and of a batch, R and gradient."""
    tail, head, rng = synth.random_connected_undirected(12, 30, 77)
    net = synth.Network(12, tail, head, synth.uniform_p(rng, 30, 0.7, 0.95), 0, 11)
    for grad in (False, True):
        batch = (pb.batch_grad_kernel_source([net, net], [[net.p] * 3] * 2) if grad
                 else pb.batch_kernel_source([net, net], 3))
        for src in (pb.kernel_source(net, pb.options(launches=2), grad=grad), batch):
            assert re.search(r"#define BSB?_MERGE 1", src)
            yield src


def _openers(src, at):
    """The statement at a position, and the headers of the blocks around it."""
    out, depth, i = [src[max(src.rfind(c, 0, at) for c in ";{}"):at]], 0, at
    while i > 0:
        i -= 1
        if src[i] == "}":
            depth += 1
        elif src[i] == "{":
            depth -= 1
            if depth < 0:
                depth = 0
                out.append(src[max(src.rfind(c, 0, i) for c in ";{}"):i])
    return out


def test_a_warp_reads_the_clock_in_one_lane(pb):
    """The time limit: what follows a check are collectives of the whole warp,
    so one lane decides for all.  Every comparison with the clock is made by
    lane 0 or thread 0 alone (the kernels are not run for this)."""
    for src in _merged_sources(pb):
        places = [m.start() for m in re.finditer(r"bs_timer\(\) -|(?<!bool )(?<!return )bs_(?:run_)?late\(", src)]
        assert places
        for at in places:
            assert any("lane == 0" in o or "threadIdx.x == 0" in o for o in _openers(src, at)), src[at - 200:at + 60]


def test_a_block_or_a_warp_reads_the_status_in_one_thread(pb):
    """The word that says that a run was given up, which other blocks of the
    same launch may be setting: only the two functions that read it for a whole
    block or warp do, and a thread that does not return goes on to barriers or
    collectives (the kernels are not run for this)."""
    for src in _merged_sources(pb):
        reads = list(re.finditer(r"(?<!u32)\*(?:\(volatile (?:const )?u32\*\))?(?:W\.)?status", src))
        assert len(reads) == 2
        for m in reads:
            assert any("_given_up(" in o for o in _openers(src, m.start())), src[m.start() - 200:m.end()]


def _same(a, b, tol):
    return abs(a - b) <= tol


def _check(pb, net, p=None, grad=True, ref=None, merged=True, **opt):
    one = pb.reliability_net(net, p=p, grad=grad, opts=pb.options(launches=1, algo=pb.ALGO_BITSLICE, **opt))
    two = pb.reliability_net(net, p=p, grad=grad, opts=pb.options(launches=2, algo=pb.ALGO_BITSLICE, **opt))
    assert one.stats[5] == 1
    if merged:
        assert two.stats[5] == (3 if grad else 2)
    assert two.Nk == one.Nk
    # the bit-sliced bounds: R within 2^-61 + 2^-59 (+ the R kernel's walk
    # masses, 2^(L-64) with L <= 10), each gradient entry within 2^-57, either
    # run, and their rounding to doubles
    assert _same(two.R, one.R, 2 * 2.0**-53 * one.R + 2.0**-53)
    if grad:
        for x, y in zip(two.grad, one.grad):
            assert _same(x, y, 2 * 2.0**-53 * abs(y) + 2.0**-56), (x, y)
    if ref is not None:
        assert two.Nk == ref.Nk
        assert _same(two.R, ref.R, 1e-12 * ref.R + 1e-300)


@pytest.mark.gpu
@pytest.mark.parametrize("m", [11, 12, 15, 16, 19, 20, 21, 22])
@pytest.mark.parametrize("directed", [False, True])
def test_merged_runs_at_block_edges(pb, m, directed):
    """One to twelve prefix arcs: blocks of two items up to full ones, one
    block and several, with and without walk arcs."""
    for seed in range(2):
        net = synth.random_small(9300 + 10 * m + seed, n=4 + (m + seed) % 7, m=m, directed=directed, p_lo=0.2, p_hi=0.99)
        for grad in (False, True):
            ref = oracle.enumerate_states(net) if m < 20 else None
            for walk in {0, min(3, m - 11)}:
                _check(pb, net, grad=grad, ref=ref, walk_bits=walk, prune=1 + seed)


@pytest.mark.gpu
def test_merged_runs_of_ranges_and_extreme_reliabilities(pb):
    """Equal divisions whose blocks are smaller than a word, and arcs that
    always work or never do among the prefix arcs (with too many of them the
    fused kernel is not merged)."""
    net = synth.random_small(611, n=7, m=20, p_lo=0.1, p_hi=0.95)
    for bits in (1, 6, 9):
        for lo in (0, 1):
            for grad in (False, True):
                ref = oracle.enumerate_states(net, prefix_bits=bits, prefix_lo=lo, prefix_hi=lo + 1)
                _check(pb, net, grad=grad, ref=ref, walk_bits=0, range_bits=bits, range_lo=lo, range_hi=lo + 1)
    for bad in (1, 4, 11, 16):
        p = [(1.0 if k % 3 else 0.0) if k < bad else q for k, q in enumerate(net.p)]
        ref = oracle.enumerate_states(net, p=p)
        for grad in (False, True):
            _check(pb, net, p=p, grad=grad, ref=ref, merged=not grad, walk_bits=0)


@pytest.mark.gpu
@pytest.mark.parametrize("wide_first", [False, True])
@pytest.mark.parametrize("grad", [False, True])
def test_ranges_of_other_widths_plan_for_themselves(pb, wide_first, grad):
    """One network's ranges of the same number of bits, narrow and wide, in
    either order: each takes the route of its own number of items, whatever
    range was planned before."""
    # (a network of its own for each order and kernel: plans are kept by network)
    seed = 640 + 2 * wide_first + grad
    # by default: 2^10 items a division, merged from 2^13 on
    net = synth.random_small(seed, n=12, m=30, p_lo=0.3, p_hi=0.95)
    merged = 3 if grad else 2
    widths = [(0, 1, 1), (5, 12, 1), (8, 16, merged), (0, 64, merged), (7, 7, 1), (9, 42, merged)]
    for lo, hi, launches in reversed(widths) if wide_first else widths:
        opt = dict(range_bits=6, range_lo=lo, range_hi=hi, walk_bits=4, algo=pb.ALGO_BITSLICE)
        res = pb.reliability_net(net, grad=grad, opts=pb.options(**opt))
        assert res.stats[5] == launches, (lo, hi)
        one = pb.reliability_net(net, grad=grad, opts=pb.options(launches=1, **opt))
        assert res.Nk == one.Nk and _same(res.R, one.R, 2 * 2.0**-53 * one.R + 2.0**-53)
        for x, y in zip(res.grad if grad else (), one.grad if grad else ()):
            assert _same(x, y, 2 * 2.0**-53 * abs(y) + 2.0**-56), (lo, hi, x, y)
    # merged when asked for: 2^18 items a division, at most 2^24 merged
    net = synth.random_small(seed + 10, n=9, m=36, p_lo=0.3, p_hi=0.95)
    widths = [(3, 4, merged), (64, 128, merged), (64, 129, 1), (0, 256, 1), (5, 30, merged)]
    for lo, hi, launches in reversed(widths) if wide_first else widths:
        opt = dict(range_bits=8, range_lo=lo, range_hi=hi, prune=2, walk_bits=0, algo=pb.ALGO_BITSLICE)
        res = pb.reliability_net(net, grad=grad, opts=pb.options(launches=2, **opt))
        assert res.stats[5] == launches, (lo, hi)
        one = pb.reliability_net(net, grad=grad, opts=pb.options(launches=1, **opt))
        assert res.Nk == one.Nk and _same(res.R, one.R, 2 * 2.0**-53 * one.R + 2.0**-53)
        for x, y in zip(res.grad if grad else (), one.grad if grad else ()):
            assert _same(x, y, 2 * 2.0**-53 * abs(y) + 2.0**-56), (lo, hi, x, y)


@pytest.mark.gpu
def test_more_classes_than_the_table_holds(pb):
    """A network of 2^24 items in more than 2^18 classes: the merged run is
    given up and every item walked, with the same counts and reliability, for
    a kept plan from its first read on."""
    tail, head, rng = synth.random_connected_undirected(20, 38, 902)
    net = synth.Network(20, tail, head, synth.uniform_p(rng, 38, 0.7, 0.95), 0, 19)
    want = pb.reliability_net(net, opts=pb.options(autotune=0, launches=1, walk_bits=4))
    plan = pb.Plan(net, opts=pb.options(autotune=0, launches=2, walk_bits=4))
    for _ in range(2):
        plan.execute()
        res = plan.read()
        assert res.stats[5] == 1
        assert res.Nk == want.Nk and _same(res.R, want.R, 1e-12 * want.R)


@pytest.mark.gpu
def test_time_limit_of_merged_runs(pb):
    """A limit far below the run's length ends merged runs, plain, with the
    gradient and in batches, with the error that says so; the next call is
    right.  So does one that no launch of the run reaches by itself: the
    launches count from the first one's start."""
    net = synth.workload_random_24_40()
    for grad in (False, True):
        opt = dict(autotune=0, launches=2, walk_bits=6, prune=2)
        with pytest.raises(pb.PbatError, match="PBAT_ETIMEOUT"):
            pb.reliability_net(net, grad=grad, opts=pb.options(time_budget_s=1e-9, **opt))
        for _ in range(2):
            res = pb.reliability_net(net, grad=grad, opts=pb.options(time_budget_s=10.0, **opt))
        assert res.stats[5] == (3 if grad else 2) and sum(res.Nk) == sum(pb.reliability_net(net).Nk)
        if grad:   # (about a fifth, half and 0.3 of the run)
            with pytest.raises(pb.PbatError, match="PBAT_ETIMEOUT"):
                pb.reliability_net(net, grad=True, opts=pb.options(time_budget_s=0.7e-9 * res.stats[4], **opt))
    nets, pvecs = synth.workload_batched()
    for grad in (False, True):
        with pytest.raises(pb.PbatError, match="PBAT_ETIMEOUT"):
            pb.reliability_batched(nets, pvecs, grad=grad, opts=pb.options(autotune=0, time_budget_s=1e-9))
        for _ in range(2):
            o = pb.options(autotune=0, time_budget_s=10.0)
            R, Nk, _ = pb.reliability_batched(nets, pvecs, grad=grad, opts=o)
        if grad:   # (the fold, last, takes a tenth to a quarter of the run)
            with pytest.raises(pb.PbatError, match="PBAT_ETIMEOUT"):
                pb.reliability_batched(nets, pvecs, grad=True,
                                       opts=pb.options(autotune=0, time_budget_s=0.92e-9 * o.stats[4]))
        one = pb.reliability_net(nets[0], p=pvecs[0][3], grad=False)
        assert Nk[0] == one.Nk and _same(R[0][3], one.R, 1e-12 * one.R)


@pytest.mark.gpu
@pytest.mark.parametrize("p, launches", [(0.5, 3), (0.7, 3), (0.75, 1), (0.95, 1)])
def test_small_gradients_keep_their_split(pb, p, launches):
    """The fused kernel of the complete graph of 8 nodes: six other arcs at
    the source fail with (1 - p)^6, above 2^-11 merged, below in one launch
    with that route's very results."""
    arcs = [(u, v) for u in range(8) for v in range(u)]
    net = synth.Network(8, [u for u, _ in arcs], [v for _, v in arcs], [p] * 28, 7, 0)
    res = pb.reliability_net(net, grad=True, opts=pb.options(autotune=0))
    one = pb.reliability_net(net, grad=True, opts=pb.options(autotune=0, launches=1))
    assert res.stats[5] == launches
    assert res.Nk == one.Nk and _same(res.R, one.R, 2 * 2.0**-53 * one.R)
    for x, y in zip(res.grad, one.grad):
        assert x == y if launches == 1 else _same(x, y, 2 * 2.0**-53 * abs(y) + 2.0**-56)
    assert pb.reliability_net(net, opts=pb.options(autotune=0)).stats[5] == 2


@pytest.mark.gpu
def test_replay_after_the_class_table_overflowed(pb):
    """A capture of a merged plan's launches stays valid when a read has found
    too many classes and taken the plan to one launch: its replays write to
    the captured job's own buffers, not to memory given back."""
    import torch
    tail, head, rng = synth.random_connected_undirected(20, 38, 902)
    net = synth.Network(20, tail, head, synth.uniform_p(rng, 38, 0.7, 0.95), 0, 19)
    # (another block size than the test above, whose plan is known not to merge)
    plan = pb.Plan(net, opts=pb.options(autotune=0, launches=2, walk_bits=4, block_threads=64))
    stream = torch.cuda.Stream()
    plan.execute(stream.cuda_stream)   # loads the kernels
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=stream):
        plan.execute(stream.cuda_stream)
    graph.replay()
    torch.cuda.synchronize()
    first = plan.read(stream.cuda_stream)
    other = pb.reliability_net(net, opts=pb.options(autotune=0, launches=1, walk_bits=4))
    graph.replay()
    torch.cuda.synchronize()
    plan.execute(stream.cuda_stream)
    again = plan.read(stream.cuda_stream)
    assert first.Nk == again.Nk == other.Nk
    assert first.R == again.R and _same(first.R, other.R, 1e-12 * other.R)


@pytest.mark.gpu
@pytest.mark.parametrize("vectors", [1, 7, 17, 40])
@pytest.mark.parametrize("grad", [False, True])
def test_merged_batches(pb, vectors, grad):
    """Networks from ones without prefix arcs to several blocks of items, in
    one batch, against batches that walk every item (the prune off) and the
    oracle."""
    nets = [synth.random_small(4400 + m, n=4 + m % 6, m=m, directed=bool(m & 1), p_lo=0.3, p_hi=0.99)
            for m in (6, 10, 11, 13, 16, 17, 19, 22)]
    rng = synth.SplitMix64(90 + vectors)
    pvecs = [[synth.uniform_p(rng, net.m, 0.3, 0.99) for _ in range(vectors)] for net in nets]
    for prune, walk in ((1, -1), (1, 0), (2, 1)):
        opts = dict(autotune=0, algo=pb.ALGO_BITSLICE, walk_bits=walk)
        R, Nk, g = pb.reliability_batched(nets, pvecs, grad=grad, opts=pb.options(prune=prune, **opts))
        R0, Nk0, g0 = pb.reliability_batched(nets, pvecs, grad=grad, opts=pb.options(prune=0, **opts))
        assert Nk == Nk0
        for i, net in enumerate(nets):
            if net.m < 17 and prune == 1:
                ref = oracle.enumerate_states(net, p=pvecs[i][0])
                assert Nk[i] == ref.Nk and _same(R[i][0], ref.R, 1e-12 * ref.R)
            for k in range(vectors):   # the bounds of _check; walk masses 2^(5-64) at most
                assert _same(R[i][k], R0[i][k], 2 * 2.0**-53 * R0[i][k] + 2.0**-57)
                if grad:
                    for x, y in zip(g[i][k], g0[i][k]):
                        assert _same(x, y, 2 * 2.0**-53 * abs(y) + 2.0**-56), (net.name, k)


@pytest.mark.gpu
def test_batches_give_their_class_memory_back(pb):
    """Sets of networks one after another, of about 1 GB of class memory each
    (38 arcs, 2^24 items): what the library keeps stays bounded, and the first
    set is answered again, its memory taken and its graph captured anew.  A
    batch with more classes than fit keeps none of it."""
    import torch
    free0 = torch.cuda.mem_get_info()[0]
    nets = [synth.random_small(8900 + i, n=9, m=38, p_lo=0.3, p_hi=0.95) for i in range(7)]
    opt = dict(autotune=0, algo=pb.ALGO_BITSLICE)
    first = []
    for net in nets + nets[:2]:
        R, Nk, _ = pb.reliability_batched([net], [[net.p] * 2], opts=pb.options(**opt))
        first.append((R[0][0], Nk[0]))
        assert R[0][0] == R[0][1]
    assert first[:2] == first[7:]
    one = pb.reliability_net(nets[0], opts=pb.options(autotune=0))
    assert first[0][1] == one.Nk and _same(first[0][0], one.R, 1e-12 * one.R)
    held = free0 - torch.cuda.mem_get_info()[0]
    assert held < (5 << 30), held
    tail, head, rng = synth.random_connected_undirected(20, 38, 902)
    net = synth.Network(20, tail, head, synth.uniform_p(rng, 38, 0.7, 0.95), 0, 19)
    free1 = torch.cuda.mem_get_info()[0]
    for _ in range(2):
        R, Nk, _ = pb.reliability_batched([net], [[net.p] * 64], opts=pb.options(**opt))
        one = pb.reliability_net(net, opts=pb.options(autotune=0, launches=1))
        assert Nk[0] == one.Nk and _same(R[0][63], one.R, 1e-12 * one.R)
    assert free1 - torch.cuda.mem_get_info()[0] < (256 << 20)


@pytest.mark.gpu
def test_no_room_for_the_classes(pb, monkeypatch):
    """Where the class memory of a merged run cannot be had, every item is
    walked by itself, with the same results; a kept plan too."""
    net = synth.random_small(8950, n=9, m=28, p_lo=0.3, p_hi=0.95)
    small = synth.random_small(8951, n=6, m=14, p_lo=0.3, p_hi=0.95)
    nets, pvecs = [net, small], [[net.p] * 3, [small.p] * 3]
    o = dict(autotune=0)
    want = [pb.reliability_net(net, grad=g, opts=pb.options(**o)) for g in (False, True)]
    assert [w.stats[5] for w in want] == [2, 3]
    monkeypatch.setenv("PBAT_FAULT", "classes")
    for grad in (False, True):
        one = pb.reliability_net(net, grad=grad, opts=pb.options(**o))
        plan = pb.Plan(net, grad=grad, opts=pb.options(launches=2, **o))
        plan.execute()
        kept = plan.read()
        R, Nk, gr = pb.reliability_batched(nets, pvecs, grad=grad, opts=pb.options(**o))
        for res in (one, kept):
            assert res.stats[5] == 1 and res.Nk == want[grad].Nk == Nk[0]
            assert _same(res.R, want[grad].R, 2 * 2.0**-53 * res.R) and _same(R[0][2], res.R, 2.0**-52)
            if grad:
                for x, y, z in zip(res.grad, want[1].grad, gr[0][2]):
                    assert _same(x, y, 2 * 2.0**-53 * abs(y) + 2.0**-56) and _same(z, y, 2 * 2.0**-53 * abs(y) + 2.0**-56)
    monkeypatch.delenv("PBAT_FAULT")
    for grad in (False, True):
        res = pb.reliability_net(net, grad=grad, opts=pb.options(**o))
        assert res.stats[5] == want[grad].stats[5] and res.R == want[grad].R
        R2, Nk2, _ = pb.reliability_batched(nets, pvecs, grad=grad, opts=pb.options(**o))
        assert Nk2 == Nk and _same(R2[0][2], R[0][2], 2.0**-52)


@pytest.mark.gpu
@pytest.mark.parametrize("grad", [False, True])
def test_divisions_of_tiny_mass(pb, grad):
    """A division of mass 1e-44 that comes after one of 1e-4: the scale of the
    classes' masses is its own."""
    tail, head, _ = synth.random_connected_undirected(14, 40, 12)
    p = [0.9999] * 12 + [0.95] * 28
    net = synth.Network(14, tail, head, p, 0, 13)
    for lo in (0, 1, 1 << 11, (1 << 11) + (1 << 10)):
        opt = dict(range_bits=12, range_lo=lo, range_hi=lo + 1, autotune=0, algo=pb.ALGO_BITSLICE)
        res = pb.reliability_net(net, grad=grad, opts=pb.options(launches=2, **opt))
        one = pb.reliability_net(net, grad=grad, opts=pb.options(launches=1, **opt))
        assert res.stats[5] == (3 if grad else 2) and res.Nk == one.Nk
        assert one.R > 0 and abs(res.R - one.R) <= 1e-15 * one.R, (lo, res.R, one.R)
        if grad:   # (of the range's mass: the gradient of a fixed arc is R / p or - R / (1 - p))
            for x, y in zip(res.grad, one.grad):
                assert abs(x - y) <= 1e-15 * max(abs(y), one.R)


@pytest.mark.gpu
@pytest.mark.parametrize("grad", [False, True])
def test_description_of_a_merged_plan(pb, grad):
    """Blocks of the launch that walks the classes: three nodes leave at most
    eight signatures, two blocks of four warps, for 2^10 items."""
    arcs = [(k % 3, (k + 1) % 3) for k in range(20)]
    net = synth.Network(3, [u for u, _ in arcs], [v for _, v in arcs], [0.5] * 20, 0, 2)
    for launches, blocks in ((2, 2), (1, 256)):
        plan = pb.Plan(net, grad=grad, opts=pb.options(launches=launches, walk_bits=0, block_threads=128))
        plan.execute()
        assert plan.read().stats[5] == ((3 if grad else 2) if launches == 2 else 1)
        d = plan.describe()
        assert d["blocks"] == blocks and d["prefix_bits"] == 10, d


@pytest.mark.gpu
@pytest.mark.parametrize("bits, lo, hi, merged", [(10, 0, 1 << 10, True), (12, 700, 3100, True), (3, 2, 7, True),
                                                  (16, 5, 50001, False), (20, 3, 1 << 18, False)])
def test_default_plans_of_wide_ranges(pb, bits, lo, hi, merged):
    """Ranges by the planner's own lengths, whole, ragged and of more blocks
    than are merged, against one launch."""
    tail, head, rng = synth.random_connected_undirected(14, 34, 77)
    net = synth.Network(14, tail, head, synth.uniform_p(rng, 34, 0.6, 0.95), 0, 13)
    for grad in (False, True):
        opt = dict(range_bits=bits, range_lo=lo, range_hi=hi, autotune=0, algo=pb.ALGO_BITSLICE)
        res = pb.reliability_net(net, grad=grad, opts=pb.options(**opt))
        one = pb.reliability_net(net, grad=grad, opts=pb.options(launches=1, **opt))
        assert res.stats[5] == ((3 if grad else 2) if merged else 1)
        assert res.Nk == one.Nk and _same(res.R, one.R, 2 * 2.0**-53 * one.R + 2.0**-53)
        for x, y in zip(res.grad if grad else (), one.grad if grad else ()):
            assert _same(x, y, 2 * 2.0**-53 * abs(y) + 2.0**-56), (x, y)
