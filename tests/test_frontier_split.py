"""The frontier kernel's integer warp sums and its split of the space, against
the oracle: one item to several thousand, prefixes of more than 32 arcs, and
reliabilities so small that only sums relative to their own size keep any
digit of R."""
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pb():
    from paper_2209_09711_gb300 import build
    build.build()
    import paper_2209_09711_gb300 as mod
    return mod


def _check(pb, net, **opt):
    bits, lo = opt.get("range_bits", 0), opt.get("range_lo", 0)
    part = dict(prefix_bits=bits, prefix_lo=lo, prefix_hi=lo + 1) if bits else {}
    ref = oracle.enumerate_states(net, grad=True, **part)
    for grad in (False, True):
        res = pb.reliability_net(net, grad=grad, opts=pb.options(algo=pb.ALGO_FRONTIER, **opt))
        assert res.Nk == ref.Nk, net.name
        # the sums are good to 2^-98 of the items' masses, each of which is a
        # product good to 2^-100: one rounding to double, on either side
        assert abs(res.R - ref.R) <= 4 * 2.0**-53 * ref.R, (net.name, res.R, ref.R)
        if grad:
            for a, b, t1, t0 in zip(res.grad, ref.grad_t1t0, ref.T1, ref.T0):
                # the double-double sums A / p - B / (1 - p) of an arc cancel;
                # the oracle's own T1 - T0 is good to 2^-62 of them
                assert abs(a - b) <= 4 * 2.0**-53 * abs(b) + 2.0**-60 * (t1 + t0), (net.name, a, b)


@pytest.mark.parametrize("p_lo,p_hi", [(0.05, 0.95), (0.95, 0.9999), (1e-4, 1e-2), (1e-9, 1e-8)])
@pytest.mark.parametrize("walk", [-1, 0, 3])
def test_frontier_sums(pb, p_lo, p_hi, walk):
    for m in (1, 4, 5, 6, 11, 12, 16, 18):
        net = synth.random_small(7100 + m, n=3 + m % 6, m=m, directed=bool(m & 1), p_lo=p_lo, p_hi=p_hi)
        _check(pb, net, walk_bits=walk)


def test_frontier_prefix_past_a_warp(pb):
    """48 arcs, of which a division fixes 36: prefix arcs on both halves of
    the lanes."""
    net = synth.random_small(7300, n=9, m=48, p_lo=0.3, p_hi=0.9)
    for lo in (0, 0x123456789, 2**36 - 1):
        _check(pb, net, range_bits=36, range_lo=lo, range_hi=lo + 1)


def test_frontier_at_the_shared_memory_limit(pb):
    """64 nodes, walks of nine arcs, blocks of 256 threads and the gradient:
    231,936 bytes of shared memory without the lane masses' table, with it
    above the limit of 232,448.  The table then stays in the parameters."""
    net = synth.random_small(7400, n=64, m=63, p_lo=0.3, p_hi=0.9)
    # a path from source to sink, so that the division reaches it
    tail = list(range(63))
    net = synth.Network(64, tail, [k + 1 for k in tail], net.p, 0, 63)
    for nthr in (256, 128):
        res = pb.reliability_net(net, grad=True, opts=pb.options(algo=pb.ALGO_FRONTIER, walk_bits=9, block_threads=nthr,
                                                                 range_bits=44, range_lo=2**44 - 1, range_hi=2**44))
        want = 1.0
        for p in net.p:
            want *= p
        # one state of the division's 2^19 reaches the sink
        assert sum(res.Nk) == res.Nk[63] == 1
        assert abs(res.R - want) <= 1e-14 * want
        for g, p in zip(res.grad, net.p):
            assert abs(g - want / p) <= 1e-14 * want / p
