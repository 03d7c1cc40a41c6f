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
