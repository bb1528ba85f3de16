"""The streaming greedy and the enumerator at the edges of their work split: group, ring and slot
remainders, more patterns than slots, shared searches, the edge set and the counted last level.  All
quantities are integers: equality is exact."""
from __future__ import annotations

import threading
import time

import numpy as np
import pytest
import scipy.sparse as sp

import oracle
import paper_2404_01585_gb300 as fx
from workloads import make_graph, random_patterns

pytestmark = pytest.mark.gpu
EARLY, FULL = fx.FLEXIS_MODE_EARLY, fx.FLEXIS_MODE_FULL
COUNT, NO_MIS = fx.FLEXIS_MODE_COUNT_MAPS, fx.FLEXIS_MODE_NO_MIS
ALL_SHAPES = ["tree", "cycle", "clique", "path", "star"]


@pytest.fixture(scope="module", autouse=True)
def built():
    import __graft_entry__
    __graft_entry__.build()


def key(r):
    return (r["status"], r["tau"], r["mis"], r["mni"], bool(r["frequent"]))


def er(nv, ne, nl, seed):
    return make_graph(kind="er", nv=nv, ne=ne, nl=nl, law="uniform", zipf_s=None, gamma=None, seed=seed)


# one label: every vertex is a root; a batch of 1 has groups of 8 roots, of 700 of 8 or 16, of 3000 of 32
@pytest.mark.parametrize("count", [1, 700, 3000])
@pytest.mark.parametrize("nv", [7, 33, 1025])
def test_streamed_equals_windowed_and_oracle(nv, count):
    lab, src, dst = er(nv, 3 * nv, 1, nv)
    pats = random_patterns(count, range(2, 7), ALL_SHAPES, lab, 3)
    g = fx.Graph(lab, src, dst)
    w = fx.Graph(lab, src, dst, window_min=16, window_max=256)
    for mode in (EARLY, FULL):
        got = [key(r) for r in g.support_batch(pats, 4, 0.5, mode)]
        assert got == [key(r) for r in w.support_batch(pats, 4, 0.5, mode)]
    og = oracle.Graph(lab, src, dst)
    for (pl, pe), k in list(zip(pats, got))[:6]:
        o = og.support(pl, pe, sigma=4, lam=0.5, mode="full", tier=1)
        assert k == (0, o["tau"], o["mis"], o["mni"], o["frequent"])
    g.close()
    w.close()


@pytest.mark.parametrize("record", [1, 5000])
def test_selection_log_of_streamed_rounds(record):
    lab, src, dst = er(2000, 9000, 2, 8)
    g = fx.Graph(lab, src, dst, record_selected=record)
    w = fx.Graph(lab, src, dst, record_selected=record, window_min=16, window_max=256)
    pats = random_patterns(9, range(2, 6), ALL_SHAPES, lab, 4)
    a, b = (x.support_batch(pats, 3, 0.5, FULL) for x in (g, w))
    for i in range(len(pats)):
        assert key(a[i]) == key(b[i])
        assert g.selected_maps(i, len(pats[i][0])) == w.selected_maps(i, len(pats[i][0])), i
    g.close()
    w.close()


# few patterns whose roots need long searches: they are cut into tasks, and cut again
@pytest.mark.parametrize("n", [5, 6, 7])
def test_shared_searches(n):
    lab, src, dst = make_graph(kind="cl", nv=60000, ne=240000, nl=3, law="zipf", zipf_s=1.0, gamma=2.3, seed=12)
    cyc = np.array([[i, (i + 1) % n] for i in range(n)], np.int32)
    pats = [(np.array([(i * k) % 3 for i in range(n)], np.int32), cyc) for k in (0, 1, 2)]
    g = fx.Graph(lab, src, dst)
    w = fx.Graph(lab, src, dst, window_min=16, window_max=4096)
    for sigma in (50, 1000):
        a, b = (x.support_batch(pats, sigma, 0.5, EARLY) for x in (g, w))
        assert [key(r) for r in a] == [key(r) for r in b]
    g.close()
    w.close()


# a warp of the enumerator takes 1 .. 32 rows; frontier_rows cuts the frontier in the middle of a group
@pytest.mark.parametrize("nv,rows", [(2, 0), (31, 0), (33, 64), (1000, 100), (70000, 5000), (70000, 0)])
def test_counts_in_closed_form(nv, rows):
    rng = np.random.default_rng(nv)
    m = min(4 * nv, nv * (nv - 1) // 2)
    e = np.unique(np.sort(rng.integers(0, nv, (m, 2)), axis=1), axis=0)
    hub = np.stack([np.zeros(nv - 1, np.int64), np.arange(1, nv)], 1)[: 3000]  # one long slice
    e = np.unique(np.concatenate([e[e[:, 0] != e[:, 1]], hub]), axis=0)
    g = fx.Graph(np.zeros(nv, np.int32), e[:, 0], e[:, 1], frontier_rows=rows)
    A = sp.csr_matrix((np.ones(len(e)), (e[:, 0], e[:, 1])), shape=(nv, nv), dtype=np.int64)
    A = A + A.T
    d = np.asarray(A.sum(1)).ravel()
    tri = int((A @ A).multiply(A).sum())  # closed walks of three steps: six a triangle
    s = lambda *x: np.zeros(x[0], np.int32)
    pats = [(s(2), [(0, 1)]), (s(3), [(0, 1), (0, 2)]), (s(4), [(0, 1), (0, 2), (0, 3)]),
            (s(4), [(0, 1), (1, 2), (2, 3)]), (s(3), [(0, 1), (1, 2), (2, 0)])]
    want = [int(d.sum()), int((d * (d - 1)).sum()), int((d * (d - 1) * (d - 2)).sum()),
            int(((d[e[:, 0]] - 1) * (d[e[:, 1]] - 1)).sum() * 2 - tri), tri]
    res = g.support_batch([(pl, np.array(pe, np.int32)) for pl, pe in pats], 1, 0.5, FULL | COUNT | NO_MIS)
    assert [r["n_maps"] for r in res] == [min(x, 1 << 32) for x in want]  # counts saturate at maps_cap
    g.close()


# Few slots and caps of one to a few maps: a pattern that reaches its cap aborts the searches ahead of it, and
# its slot goes to the next pattern at once.  What the aborted searches knew of the old pattern must not
# reach the new one; the patterns share labels, so that an old dead candidate would be one of the new.
@pytest.mark.parametrize("blocks", [1, 2])
@pytest.mark.parametrize("sigma", [1, 40])
def test_slots_reused_after_aborted_searches(blocks, sigma):
    lab, src, dst = make_graph(kind="cl", nv=20000, ne=120000, nl=2, law="zipf", zipf_s=1.0, gamma=2.3, seed=31)
    pats = random_patterns(600, range(4, 7), ALL_SHAPES, lab, 17)
    g = fx.Graph(lab, src, dst, search_blocks=blocks)
    w = fx.Graph(lab, src, dst, window_min=16, window_max=256)
    mode = EARLY | fx.FLEXIS_MODE_NO_MNI
    want = [key(r) for r in w.support_batch(pats, sigma, 0.5, mode)]
    for _ in range(3):
        assert [key(r) for r in g.support_batch(pats, sigma, 0.5, mode)] == want
    g.close()
    w.close()


# Roots that lanes decide in a few steps: no search is long enough to look at the clock, so the deadline has to be
# seen between groups.  The call after it starts from buffers that the stopped one left as they were.
@pytest.mark.parametrize("record", [0, 2])
def test_deadline_stops_many_cheap_patterns(record):
    lab, src, dst = er(20000, 40000, 4, 6)
    pats = random_patterns(2000, range(3, 5), ["tree", "path"], lab, 8)
    many = pats * 10
    mode, sigma = EARLY | fx.FLEXIS_MODE_NO_MNI, 100_000  # never reached: every root is searched
    ref = fx.Graph(lab, src, dst)
    want = [key(r) for r in ref.support_batch(pats, sigma, 0.5, mode)]
    ref.close()
    g = fx.Graph(lab, src, dst, deadline_ms=2, record_selected=record)
    for _ in range(2):
        res = g.support_batch(many, sigma, 0.5, mode)
        stopped = 0
        for i, r in enumerate(res):
            if r["status"] == fx.FLEXIS_E_TIMEOUT:
                stopped += 1
                assert 0 <= r["mis"] <= want[i % len(pats)][2] and r["mni"] == -1 and not r["frequent"]
            else:
                assert key(r) == want[i % len(pats)]
        assert 0 < stopped
        alone = [key(g.support(pl, pe, sigma, 0.5, mode=mode)) for pl, pe in pats[:8]]
        decided = [k == w for k, w in zip(alone, want) if k[0] == 0]
        assert decided and all(decided)
    g.close()


# A batch of some hundred milliseconds leaves SMs to other streams: requests served meanwhile are done before it,
# also when the server is at work as the batch is launched (the last delays: after its host part of some 40 ms).
def test_server_beside_a_batch():
    lab, src, dst = make_graph("mico")
    mode = EARLY | fx.FLEXIS_MODE_NO_MNI
    big = random_patterns(6000, range(5, 7), ALL_SHAPES, lab, 7)
    small = random_patterns(8, range(3, 5), ["tree", "path"], lab, 9)
    g = fx.Graph(lab, src, dst)
    want = [key(r) for r in g.support_batch(small, 300, 0.5, mode)]
    first = [key(r) for r in g.support_batch(big, 1000, 0.5, mode)]
    srv = fx.Server(g, slots=8)
    for delay in (0.1, 0.08, 0.07, 0.06, 0.055, 0.05, 0.045, 0.04, 0.035, 0.03):
        out, ended = [], threading.Event()

        def batch():
            out.extend(key(r) for r in g.support_batch(big, 1000, 0.5, mode))
            ended.set()

        t = threading.Thread(target=batch)
        t.start()
        time.sleep(delay)
        for turn in range(4):
            got = {}
            for i, (pl, pe) in enumerate(small):
                assert srv.submit(i, pl, pe, 300, 0.5, mode) == 0
            while len(got) < len(small):
                got.update((rid, r) for rid, r, _ in srv.poll())
                time.sleep(1e-4)
            assert [key(got[i]) for i in range(len(small))] == want
        beside = not ended.is_set()
        t.join()
        assert out == first
        assert beside, delay
    srv.stop()
    g.close()


# A call of a few patterns is captured when it comes a second time; calls of two kinds in turn are launched singly.
def test_small_calls_are_captured_on_their_second_launch():
    lab, src, dst = er(3000, 12000, 4, 5)
    g = fx.Graph(lab, src, dst)
    tree = (np.array([0, 1, 2], np.int32), np.array([[0, 1], [1, 2]], np.int32))
    ring = (np.array([0, 1, 2], np.int32), np.array([[0, 1], [1, 2], [2, 0]], np.int32))
    w = fx.Graph(lab, src, dst, window_min=16, window_max=256)

    def replays(calls):
        out = []
        for (pl, pe), mode in calls:
            assert key(g.support(pl, pe, 50, 0.5, mode=mode)) == key(w.support(pl, pe, 50, 0.5, mode=mode))
            out.append(g.stats()["graph_launches"])
        return out

    plain = EARLY | fx.FLEXIS_MODE_NO_MNI
    assert replays([(tree, FULL)] * 3) == [0, 1, 1]
    # the edge set is built for the first cycle; from then on trees and cycles are one kind
    assert replays([(ring, FULL), (tree, FULL), (ring, FULL)]) == [0, 1, 1]
    assert replays([(tree, plain), (tree, FULL), (ring, plain), (ring, FULL)]) == [0, 1, 0, 1]
    assert replays([(tree, plain), (ring, plain), (tree, FULL), (tree, plain)]) == [0, 1, 0, 1]
    g.close()
    w.close()


# Two graphs evaluated at once from two threads: the second launch finds only the SMs that the first has left alone.
def test_two_batches_at_once():
    mode = EARLY | fx.FLEXIS_MODE_NO_MNI
    lab, src, dst = make_graph("mico")
    pats = [random_patterns(n, range(4, 7), ALL_SHAPES, lab, s) for n, s in ((3000, 7), (700, 8))]
    gs = [fx.Graph(lab, src, dst) for _ in pats]
    want = [[key(r) for r in g.support_batch(p, 1000, 0.5, mode)] for g, p in zip(gs, pats)]
    for _ in range(3):
        out = [None, None]

        def batch(i):
            out[i] = [key(r) for r in gs[i].support_batch(pats[i], 1000, 0.5, mode)]

        ts = [threading.Thread(target=batch, args=(i,)) for i in (0, 1)]
        for t in ts:
            t.start()
        for t in ts:
            t.join()
        assert out == want
    for g in gs:
        g.close()
