"""The forms of networks and reliability vectors that a batch takes, as numpy
converts them: nested lists, arrays, and elements that are arrays (CPU only)."""
from types import SimpleNamespace

import numpy as np
import pytest

import paper_2209_09711_gb300 as pb

ROWS = {
    "lists": ([[0.1, 0.2], [0.3, 0.4]], 2),
    "tuples": (((0.1, 0.2), [0.3, 0.4]), 2),
    "array": (np.array([[0.1, 0.2], [0.3, 0.4]]), 2),
    "rows of float32": ([np.array([0.1, 0.2], np.float32), np.array([0.3, 0.4], np.float32)], 2),
    "end to end": ([0.1, 0.2, 0.3, 0.4], 2),
    "whole numbers": ([[1, 0], [0, 1]], 2),
    "a list deeper": ([[[0.1], [0.2]], [[0.3], [0.4]]], 2),
    "one more list around": ([[[0.1, 0.2, 0.3]]], 1),
    "arrays of one element": ([[np.array([0.1]), np.array([0.2])]], 1),
    "arrays of no dimension": ([[np.array(0.1), np.float32(0.2)]], 1),
}


@pytest.mark.parametrize("form", ROWS)
def test_vectors(form):
    pv, K = ROWS[form]
    want = np.asarray(pv, dtype=np.float64).reshape(K, -1).ravel()
    assert np.array_equal(pb._rows(pv, K), want)


@pytest.mark.parametrize("pv", [[[0.1], [0.2, 0.3]], [["x", 0.1]], [[1j, 0.1]]])
def test_refused_vectors(pv):
    with pytest.raises((TypeError, ValueError)):
        pb._rows(pv, len(pv))


@pytest.mark.parametrize("form", [list, tuple, np.array, lambda x: np.array(x, np.int64)[:, None],
                                  lambda x: [[v] for v in x], lambda x: [np.array([v]) for v in x],
                                  lambda x: [np.int64(v) for v in x], lambda x: range(x[0], x[0] + len(x))])
def test_networks(form):
    nets = [SimpleNamespace(n=4, tail=form([0, 1, 2]), head=form([1, 2, 3]), directed=True, source=0, sink=3),
            SimpleNamespace(n=3, tail=form([0, 1]), head=form([1, 2]), directed=False, source=0, sink=2)]
    graphs, keep, ms = pb._graphs(nets)
    assert list(ms) == [3, 2] and keep
    got = [(g.n_nodes, g.n_arcs, g.tail[:g.n_arcs], g.head[:g.n_arcs], g.directed, g.source, g.sink) for g in graphs[:2]]
    assert got == [(4, 3, [0, 1, 2], [1, 2, 3], 1, 0, 3), (3, 2, [0, 1], [1, 2], 0, 0, 2)]
