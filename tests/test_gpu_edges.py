"""RPQ evaluation where a size decides which path a level or a row takes: rows
at the borders of the chunk classes (32, 128 and 256 edges), frontiers around
the 512 edges that one block expands alone, vertex counts around an emission
segment, source counts around a word, a row and a group of lanes.  Rows, digest and
work counter equal the CPU oracle's exactly, for automatic, all top-down and
all bottom-up levels."""

import numpy as np
import pytest

import oracle
from paper_2602_20748_gb300 import synth
from test_gpu_rpq import MODES, check

pytestmark = pytest.mark.gpu

rpq = pytest.importorskip("paper_2602_20748_gb300.rpq")

DEGREES = (1, 31, 32, 33, 127, 128, 129, 255, 256, 257, 511, 512, 513)


def star_edges():
    """13 vertices with exactly DEGREES[i] out-edges on label a, 13 with as
    many in-edges on it, and two random edges per vertex on labels b and c."""
    n = 2100
    rng = np.random.Generator(np.random.PCG64(11))
    src, dst, lab = [], [], []
    for i, d in enumerate(DEGREES):
        src += [i] * d
        dst += rng.choice(np.arange(100, n), d, replace=False).tolist()
        src += rng.choice(np.arange(100, n), d, replace=False).tolist()
        dst += [40 + i] * d
        lab += [0] * (2 * d)
    src += rng.integers(0, n, 4 * n).tolist()
    dst += rng.integers(0, n, 4 * n).tolist()
    lab += [1, 2] * (2 * n)
    return n, 3, np.array(src, np.uint32), np.array(dst, np.uint32), np.array(lab, np.uint16)


@pytest.fixture(scope="module")
def stars():
    g = star_edges()
    c = rpq.Context(device=0)
    return c, rpq.load_graph(c, *g), oracle.Graph(*g)


@pytest.mark.parametrize("count", [1, 31, 32, 64, 65, 256, 257, 600])
@pytest.mark.parametrize("regex", ["a", "a.b.c*", "(a|b)+.c", "a?.b*.a"])
def test_row_lengths_and_source_counts(stars, regex, count):
    c, g, og = stars
    sources = np.arange(count, dtype=np.uint32)  # the stars first
    want = oracle.rpq(og, regex, sources=sources)
    for mode in MODES.values():
        check(c, g, og, regex, sources=sources, mode=mode, want=want)


@pytest.mark.parametrize("n", [1, 2, 31, 32, 33, 255, 256, 257, 511, 513, 1023, 1025])
def test_vertex_counts_around_emission_segments(n):
    """Two accepting states, both lane widths, rows kept and counted only."""
    src, dst, lab = synth.random_graph(n, 3 * n, 2, seed=500 + n)
    c = rpq.Context(device=0)
    g, og = rpq.load_graph(c, n, 2, src, dst, lab), oracle.Graph(n, 2, src, dst, lab)
    for sources in (np.arange(min(n, 64), dtype=np.uint32), None):
        want = oracle.rpq(og, "a.b?", sources=sources)
        rows, _ = check(c, g, og, "a.b?", sources=sources, want=want)
        q = rpq.compile_rpq(c, "a.b?")
        r = rpq.run_rpq(c, g, q, sources, flags=rpq.RPQ_COUNT_ONLY)
        assert rpq.result_info(r)[0] == len(rows) and rpq.result_info(r)[2:4] == oracle.pair_digest(want.rows)[1:]


@pytest.mark.parametrize("flags", [rpq.RPQ_MATERIALIZE, rpq.RPQ_PER_QUERY])
@pytest.mark.parametrize("regex", ["a", "a.a", "(a|b)+.c?"])
def test_batch_row_lengths(stars, regex, flags):
    """A query per star: the lists of a push hold 1 to 513 edges, and several
    rows meet in one warp."""
    c, g, og = stars
    sources = np.arange(len(DEGREES) + 40, dtype=np.uint32)
    r = rpq.run_rpq_batch(c, g, [rpq.compile_rpq(c, regex)] * len(sources), sources, flags=flags)
    rows, W = [], 0
    for i, s in enumerate(sources):
        want = oracle.rpq(og, regex, sources=[int(s)])
        W += want.W
        rows += [(i, int(y)) for y in want.rows[:, 1]]
        if flags == rpq.RPQ_PER_QUERY:
            assert rpq.result_query_stats(r, i) == oracle.pair_digest(want.rows)
    assert rpq.result_stats(r)["product_edges"] == W
    if flags == rpq.RPQ_MATERIALIZE:
        assert np.array_equal(rpq.fetch_pairs(r), np.array(rows, np.uint32).reshape(-1, 2))


def test_smallest_budget_that_is_accepted():
    """At the smallest memory budget a count is accepted with, the emission's
    scratch is what its longest segments need, and the result is the same."""
    n = 65536
    src, dst, lab = synth.random_graph(n, 2 * n, 2, seed=77)
    sources = np.arange(64, dtype=np.uint32)
    want = oracle.rpq(oracle.Graph(n, 2, src, dst, lab), "a.b*", sources=sources)

    def count(budget):
        c = rpq.Context(device=0, mem_budget_bytes=budget)
        try:
            r = rpq.run_rpq(c, rpq.load_graph(c, n, 2, src, dst, lab), rpq.compile_rpq(c, "a.b*"), sources,
                            flags=rpq.RPQ_COUNT_ONLY)
        except rpq.RPQError:
            return None
        return rpq.result_info(r)[0], rpq.result_info(r)[2], rpq.result_info(r)[3]

    refused, accepted = 1 << 16, 1 << 30
    assert count(refused) is None and count(accepted) == oracle.pair_digest(want.rows)
    while accepted - refused > 1 << 14:
        b = (refused + accepted) // 2
        got = count(b)
        if got is None:
            refused = b
        else:
            assert got == oracle.pair_digest(want.rows)
            accepted = b


@pytest.mark.parametrize("evict_at", [2.0**59, 2.0**60, 2.0**62])
def test_a_bound_no_query_reaches_evicts_none(stars, evict_at):
    og = stars[2]
    c = rpq.Context(device=0)
    rpq.rpq_set_option(c, "batch_evict", evict_at)
    g = rpq.load_graph(c, *star_edges())
    sources = np.arange(40, dtype=np.uint32)
    r = rpq.run_rpq_batch(c, g, [rpq.compile_rpq(c, "(a|b)+.c")] * 40, sources, flags=rpq.RPQ_PER_QUERY)
    assert rpq.result_stats(r)["evicted"] == 0
    for i in range(40):
        assert rpq.result_query_stats(r, i) == oracle.pair_digest(oracle.rpq(og, "(a|b)+.c", sources=[i]).rows)


@pytest.mark.parametrize("flags,launches", [(rpq.RPQ_COUNT_ONLY, 5), (rpq.RPQ_MATERIALIZE, 9)])
def test_launches_of_a_call(stars, flags, launches):
    """Start, traversal, counts, scan, read-back; with rows also their writing,
    their offsets, the digest and its read-back."""
    c, g, _ = stars
    r = rpq.run_rpq(c, g, rpq.compile_rpq(c, "a.b"), np.arange(20, dtype=np.uint32), flags=flags)
    assert rpq.result_stats(r)["launches"] == launches
