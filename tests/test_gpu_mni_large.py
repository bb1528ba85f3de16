"""MNI of a batch whose candidate vertices, over all patterns and orbits, pass 2^31: the same batch in parts, whose
sums stay below, is the reference."""
from __future__ import annotations

import pytest

import paper_2404_01585_gb300 as fx
from workloads import make_graph, random_patterns

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    import __graft_entry__
    __graft_entry__.build()


def test_candidate_segments_past_31_bits():
    nv = 3_600_000
    lab, src, dst = make_graph(kind="er", nv=nv, ne=1_080_000, nl=1, law="uniform", zipf_s=None, gamma=None, seed=3)
    pats = random_patterns(128, [8], ["tree"], lab, 5)
    g = fx.Graph(lab, src, dst)
    mode = fx.FLEXIS_MODE_FULL
    res = g.support_batch(pats, 100, 0.5, mode)
    total, want = g.stats()["mni_items"], []
    for i in range(0, len(pats), 16):  # 16 patterns of at most 8 orbits: 2^28.8 candidates
        want += g.support_batch(pats[i:i + 16], 100, 0.5, mode)
    assert total > 1 << 31
    assert [(r["status"], r["mis"], r["mni"]) for r in res] == [(r["status"], r["mis"], r["mni"]) for r in want]
    assert all(r["status"] == 0 and r["mni"] >= r["mis"] for r in res)
    g.close()
