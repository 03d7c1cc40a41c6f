"""What the memory limits of the entry points accept, at the limits."""

import numpy as np
import pytest

from paper_2602_20748_gb300 import synth

pytestmark = pytest.mark.gpu

rpq = pytest.importorskip("paper_2602_20748_gb300.rpq")


def up(x, to):
    return -(-x // to) * to


def scan_words(n):
    tiles = -(-n // 2048)
    return 1 if tiles <= 1 else tiles + scan_words(tiles)


def static_bytes(states, n):
    """The static scratch of one lane word: control block, totals, start
    vertices and a spare word, five arrays of a word per (state, vertex), and a
    count and an offset per lane and 4,096 vertices with the scan's scratch."""
    k = 64 * -(-n // 4096)
    return sum(up(b, 256) for b in (2592, 32, 256, 8, *[8 * states * n] * 5, 4 * k, 8 * k, 8 * scan_words(k)))


@pytest.mark.parametrize("regex,states", [("a*", 1), ("a.b.c", 4)])
def test_static_takes_what_its_array_holds(regex, states):
    torch = pytest.importorskip("torch")
    n = next(n for n in range((64 << 20) // (40 * states), 0, -1) if static_bytes(states, n) <= 64 << 20)
    src, lab = np.array([0, 1, 2, n - 2], np.uint32), np.array([0, 1, 2, 0], np.uint16)
    dst = np.array([1, 2, n - 1, n - 1], np.uint32)
    c = rpq.Context(device=0)
    q = rpq.compile_rpq(c, regex)
    assert rpq.query_info(q)[0] == states
    out = torch.zeros(64, dtype=torch.int32, device="cuda")
    rows = rpq.run_rpq_static(c, rpq.load_graph(c, n, 3, src, dst, lab), q, np.array([0], np.uint32),
                              out.data_ptr(), 32)
    want = [[0, 0], [0, 1]] if regex == "a*" else [[0, n - 1]]
    assert out.cpu().numpy()[: 2 * rows].reshape(-1, 2).tolist() == want
    with pytest.raises(rpq.RPQError) as e:
        rpq.run_rpq_static(c, rpq.load_graph(c, n + 1, 3, src, dst, lab), q, np.array([0], np.uint32),
                           out.data_ptr(), 32)
    assert e.value.code == rpq.RPQ_ERR_OUT_OF_BUDGET


def smallest(accepts, low, high):
    """The smallest budget in (low, high] that is accepted, to the byte."""
    assert accepts(high) and not accepts(low)
    while high - low > 1:
        b = (low + high) // 2
        low, high = (low, b) if accepts(b) else (b, high)
    return high


def run_with(budget, graph, regex, sources, flags):
    """(count, digest sum, digest xor) under a memory budget, None when it refuses."""
    c = rpq.Context(device=0, mem_budget_bytes=budget)
    try:
        r = rpq.run_rpq(c, rpq.load_graph(c, *graph), rpq.compile_rpq(c, regex), sources, flags=flags)
    except rpq.RPQError as e:
        assert e.code == rpq.RPQ_ERR_OUT_OF_BUDGET
        return None
    return [rpq.result_info(r)[k] for k in (0, 2, 3)]


@pytest.mark.parametrize("reach", [40, 20000])
def test_rows_need_no_more_than_the_counts_and_themselves(reach):
    """100 start vertices (four words of lanes), `reach` rows each.  A budget
    that holds the count with the longest segments' scratch and, beside it, the
    rows' buffers is enough, and so is every larger one: also where the scratch
    of shorter segments fits, but not with the rows beside it."""
    n = 1 << 20
    src = np.concatenate([np.arange(100), np.full(reach, 200)]).astype(np.uint32)
    dst = np.concatenate([np.full(100, 200), np.arange(1000, 1000 + reach)]).astype(np.uint32)
    graph = (n, 2, src, dst, (src == 200).astype(np.uint16))
    sources = np.arange(100, dtype=np.uint32)
    count = lambda b: run_with(b, graph, "a.b", sources, rpq.RPQ_COUNT_ONLY)
    want = count(1 << 33)
    assert want[0] == 100 * reach
    low = smallest(lambda b: count(b) == want, 1 << 28, 1 << 30)
    rows = 4 * 256 + 8 * 257 + 4 * 100 * reach
    for more in (0, 1, 1 << 19, 1 << 20, (1 << 21) + rows // 2, 1 << 22):
        assert run_with(low + rows + more, graph, "a.b", sources, rpq.RPQ_MATERIALIZE) == want
    assert run_with(low + rows - 1, graph, "a.b", sources, rpq.RPQ_MATERIALIZE) is None


def test_lists_of_shorter_rows_take_nothing_from_the_budget():
    """As many edges in rows of 16 and in rows of 64: what a budget accepts is
    the same, and so are the rows of 64 at its limit, by bottom-up levels."""
    n, m = 1 << 20, 1 << 18
    sources = np.arange(100, dtype=np.uint32)
    lows = []
    for row in (16, 64):
        src = np.repeat(np.arange(m // row, dtype=np.uint32), row)
        dst = (np.arange(m, dtype=np.uint64) * 2654435761 % n).astype(np.uint32)
        for graph in ((n, 1, src, dst, np.zeros(m, np.uint16)), (n, 1, dst, src, np.zeros(m, np.uint16))):
            flags = rpq.RPQ_COUNT_ONLY | rpq.RPQ_FORCE_PULL
            want = run_with(1 << 33, graph, "a.a", sources, rpq.RPQ_COUNT_ONLY)
            lows.append(smallest(lambda b: run_with(b, graph, "a.a", sources, flags) == want, 1 << 28, 1 << 30))
    assert len(set(lows)) == 1


def test_lists_given_back_while_other_contexts_read_them():
    """A call that the budget refuses gives the lists of shorter rows back, in
    the middle of a server's requests on the same graph; replies and later calls
    are what they were."""
    n = 12000
    rng = np.random.default_rng(7)
    graph = (n, 3, *(rng.integers(0, k, 120 * n).astype(t) for k, t in ((n, np.uint32), (n, np.uint32), (3, np.uint16))))
    c = rpq.Context(device=0, mem_budget_bytes=500 << 20)
    g = rpq.load_graph(c, *graph)
    queries = [rpq.compile_rpq(c, x) for x in ("a.b*", "(a|b)+.c", "c.a?.b")]

    def summary(q, sources, flags=rpq.RPQ_COUNT_ONLY):
        return [rpq.result_info(rpq.run_rpq(c, g, q, sources, flags=flags))[k] for k in (0, 2, 3)]

    def batch():
        r = rpq.run_rpq_batch(c, g, queries * 40, rng2, flags=rpq.RPQ_PER_QUERY)
        return [rpq.result_query_stats(r, i) for i in range(120)]

    rng2 = np.arange(120, dtype=np.uint32) * 97
    rpq.rpq_set_option(c, "batch_direct", 1)
    modes = (0, rpq.RPQ_REVERSE, rpq.RPQ_FORCE_PULL, rpq.RPQ_FORCE_PUSH)
    lists = (np.arange(40, dtype=np.uint32), np.arange(600, dtype=np.uint32))
    before = [summary(q, s, rpq.RPQ_COUNT_ONLY | f) for q in queries for s in lists for f in modes] + batch()
    singles = [(q, int(s), summary(q, [int(s)])) for q in queries for s in rng.integers(0, n, 60)]
    everything = [summary(q, None) for q in queries]
    server = rpq.Server(c, g, mem_budget_bytes=8 << 30)
    try:
        tickets = [(server.submit_allpairs(q), w) for q, w in zip(queries, everything)]
        tickets += [(server.submit_single(q, s), w) for q, s, w in singles]
        with pytest.raises(rpq.RPQError) as e:
            rpq.run_rpq(c, g, queries[0], None, flags=rpq.RPQ_MATERIALIZE)  # 140 million rows
        assert e.value.code == rpq.RPQ_ERR_OUT_OF_BUDGET
        tickets += [(server.submit_single(q, s), w) for q, s, w in singles]
        for t, want in tickets:
            rep = server.wait(t, timeout_s=60)
            assert [rep["status"], rep["count"], rep["digest_sum"], rep["digest_xor"]] == [0, *want]
    finally:
        server.close()
    assert [summary(q, s, rpq.RPQ_COUNT_ONLY | f) for q in queries for s in lists for f in modes] + batch() == before


def test_a_batch_is_accepted_again_after_its_lane_launches(monkeypatch):
    """The workspace that the lane-mode launches of a batch leave does not stand
    in the way of the next batch's shared launch."""
    monkeypatch.setenv("RPQ_BATCH_LIST_CAP", str(1 << 24))  # 256 MiB of lists
    n = 1 << 18
    src, dst, lab = synth.rmat_graph(18, 4 << 18, 4, 1.2, seed=11)
    regexes, sources = synth.batch_queries(512, 4, 1.2, src, n, seed=12)

    def batches(budget, times):
        c = rpq.Context(device=0, mem_budget_bytes=budget)
        rpq.rpq_set_option(c, "batch_evict", 64)
        try:
            g = rpq.load_graph(c, n, 4, src, dst, lab)
            qs = [rpq.compile_rpq(c, x) for x in regexes]
            out = []
            for _ in range(times):
                r = rpq.run_rpq_batch(c, g, qs, sources, flags=rpq.RPQ_PER_QUERY)
                out.append([rpq.result_query_stats(r, i) for i in range(len(qs))])
                assert rpq.result_stats(r)["evicted"] > 64
            return out
        except rpq.RPQError as e:
            assert e.code == rpq.RPQ_ERR_OUT_OF_BUDGET
            return None

    want = batches(8 << 30, 1)
    low = smallest(lambda b: batches(b & ~0xFFFFF, 1) == want, 64 << 20, 2 << 30) & ~0xFFFFF
    assert batches(low, 2) == want * 2
