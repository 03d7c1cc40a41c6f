"""What the memory limits of the entry points accept, at the limits."""

import numpy as np
import pytest

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
