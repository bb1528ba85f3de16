"""Plans in device memory (flexis_support_plans_device): records are as far apart as the caller's type
says, whatever the library keeps of them."""
from __future__ import annotations

import ctypes as C

import pytest
import torch

import paper_2404_01585_gb300 as fx
from workloads import make_graph, random_patterns

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    import __graft_entry__
    __graft_entry__.build()


@pytest.mark.parametrize("count", [1, 2, 33, 700])
def test_device_plans_equal_batch(count):
    lab, src, dst = make_graph(kind="er", nv=3000, ne=12000, nl=4, law="uniform", zipf_s=None, gamma=None, seed=5)
    g = fx.Graph(lab, src, dst)
    pats = random_patterns(count, range(2, 6), ["tree", "cycle", "path"], lab, 9)
    want = g.support_batch(pats, 40, 0.5, fx.FLEXIS_MODE_FULL)
    d = torch.from_numpy(g.compile(pats, 40, 0.5, fx.FLEXIS_MODE_FULL)).cuda()
    out = torch.zeros(count * C.sizeof(fx.flexis_support_result), dtype=torch.uint8, device="cuda")
    g.support_plans_device(d.data_ptr(), count, out.data_ptr())
    raw = out.cpu().numpy().tobytes()
    got = (fx.flexis_support_result * count).from_buffer_copy(raw)
    for i in range(count):
        r = got[i].as_dict()
        assert [r[k] for k in ("status", "tau", "mis", "mni", "frequent")] == \
               [want[i][k] for k in ("status", "tau", "mis", "mni", "frequent")], i
    g.close()
