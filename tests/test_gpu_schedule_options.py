"""free_sms: what it does to the plans that take it, and the schedules of the
persistent level-0 products, which a default plan of a dense domain does not
run (it goes by sibling groups)."""
import ctypes

import numpy as np
import pytest

torch = pytest.importorskip("torch")

import paper_1402_6081_gb300 as lgfm
import workloads as W
from paper_1402_6081_gb300 import build as lgf_build

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    lgf_build.build()
    lgfm.library()


class _Attr(ctypes.Union):
    _fields_ = [("priority", ctypes.c_int), ("pad", ctypes.c_char * 64)]


def priorities(solver, f, u):
    """Launch priorities of a solve's kernels, read from a captured solve."""
    rt = ctypes.CDLL("libcudart.so.13")
    ok = lambda e: pytest.fail(f"CUDA runtime error {e}") if e else None
    st = torch.cuda.Stream()
    graph = ctypes.c_void_p()
    ok(rt.cudaStreamBeginCapture(ctypes.c_void_p(st.cuda_stream), 2))   # relaxed
    solver(f, u, st)
    ok(rt.cudaStreamEndCapture(ctypes.c_void_p(st.cuda_stream), ctypes.byref(graph)))
    n = ctypes.c_size_t()
    ok(rt.cudaGraphGetNodes(graph, None, ctypes.byref(n)))
    nodes = (ctypes.c_void_p * n.value)()
    ok(rt.cudaGraphGetNodes(graph, nodes, ctypes.byref(n)))
    out = []
    for node in nodes:
        kind = ctypes.c_int()
        ok(rt.cudaGraphNodeGetType(ctypes.c_void_p(node), ctypes.byref(kind)))
        if kind.value == 0:   # kernel
            a = _Attr()
            ok(rt.cudaGraphKernelNodeGetAttribute(ctypes.c_void_p(node), 8, ctypes.byref(a)))   # priority
            out.append(a.priority)
    ok(rt.cudaGraphDestroy(graph))
    return out


def test_grouped_plan_that_leaves_room_takes_no_precedence():
    p = W.torus_box(seed=2, nb=6, n_b=8, radius=14.0, sigma=3.0, n_levels=3)
    f = torch.from_numpy(p.f).float().cuda()
    us = []
    for free, first in ((0, True), (-1, True), (32, False)):
        s = lgfm.Solver(p.blocks, p.n_b, p.n_levels, p.order, lgfm.LGF_FP32, free_sms=free)
        assert s.stats()["persistent_ctas"] == 0
        us.append(s(f).clone())
        lgfm.lgf_plan_sync(s.plan)
        pr = priorities(s, f, torch.empty_like(f))
        assert len(pr) == lgfm.lgf_plan_kernel_launches(s.plan) and max(pr) == 0
        assert (min(pr) < 0) == first, (free, pr)
        s.close()
    assert torch.equal(us[0], us[1]) and torch.equal(us[0], us[2])   # a schedule only


_refs = {}


@pytest.mark.parametrize("n_b", [6, 12, 16, 18])
@pytest.mark.parametrize("opts", [{"free_sms": -1}, {"free_sms": 24}, {"free_sms": 24, "single_stream": 1}])
def test_persistent_level0_schedules(n_b, opts):
    # before and after the products (-1), and beside them; FP32, against the
    # grouped form, each within 1e-5 of the exact method
    nb = 6 if n_b <= 12 else 5
    p = W.torus_box(seed=n_b, nb=nb, n_b=n_b, radius=0.3 * nb * n_b, sigma=0.06 * nb * n_b, n_levels=3)
    f = torch.from_numpy(p.f).float().cuda()

    def solve(**o):
        s = lgfm.Solver(p.blocks, p.n_b, p.n_levels, min(8, n_b), lgfm.LGF_FP32, **o)
        st, u = s.stats(), s(f)
        lgfm.lgf_plan_sync(s.plan)
        s.close()
        return st, u.double()

    if n_b not in _refs:
        _refs[n_b] = solve()
    st, u = solve(interval_kernel=5, **opts)
    ref_st, ref = _refs[n_b]
    assert st["persistent_ctas"] > 0 and st["top_product_level"] >= 2 and ref_st["persistent_ctas"] == 0
    assert float((u - ref).abs().max()) <= 2e-5 * float(ref.abs().max())
