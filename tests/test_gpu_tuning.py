"""The plan's launch tuning reaches the launches: grids read from a captured graph."""
import ctypes as C

import pytest

from paper_2503_22695_gb300 import inputs as I

from helpers import Case

pytestmark = pytest.mark.gpu


class _KernelNode(C.Structure):   # CUDA_KERNEL_NODE_PARAMS
    _fields_ = [("func", C.c_void_p), ("grid", C.c_uint * 3), ("block", C.c_uint * 3),
                ("smem", C.c_uint), ("params", C.c_void_p), ("extra", C.c_void_p),
                ("kern", C.c_void_p), ("ctx", C.c_void_p)]


def _grids(fn):
    """[(kernel name, CTAs)] of the kernels that fn launches."""
    import torch
    drv = C.CDLL("libcuda.so.1")

    def check(code):
        assert code == 0, code

    graph = torch.cuda.CUDAGraph(keep_graph=True)
    with torch.cuda.graph(graph):
        fn()
    g, n = C.c_void_p(graph.raw_cuda_graph()), C.c_size_t()
    check(drv.cuGraphGetNodes(g, None, C.byref(n)))
    nodes = (C.c_void_p * n.value)()
    check(drv.cuGraphGetNodes(g, nodes, C.byref(n)))
    out = []
    for node in nodes:
        kind = C.c_int()
        check(drv.cuGraphNodeGetType(C.c_void_p(node), C.byref(kind)))
        if kind.value != 0:       # CU_GRAPH_NODE_TYPE_KERNEL
            continue
        k, name = _KernelNode(), C.c_char_p()
        check(drv.cuGraphKernelNodeGetParams_v2(C.c_void_p(node), C.byref(k)))
        check(drv.cuFuncGetName(C.byref(name), C.c_void_p(k.func)) if k.func else
              drv.cuKernelGetName(C.byref(name), C.c_void_p(k.kern)))
        out.append((name.value.decode(), k.grid[0]))
    return out


@pytest.mark.parametrize("fp64", [False, True])
def test_interpolation_cap(fp64):
    import torch
    c = Case(I.block_problem(fp64=fp64))
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    ref = c.ibfe.ib_interp(c.plan, c.pos, c.u)
    U = torch.empty_like(ref)
    seen = {}
    for cap in (1, 2, 3, 8):
        c.ibfe.ib_plan_set_tuning(c.plan, [1024, 4, 8, cap])
        grids = _grids(lambda: c.ibfe.ib_interp(c.plan, c.pos, c.u, U))
        seen[cap], = [n for name, n in grids if "k_interp" in name]
        assert torch.equal(c.ibfe.ib_interp(c.plan, c.pos, c.u), ref)
    if fp64:      # by component: four CTAs per SM at most, four thirds of the cap
        assert seen == {k: min(4 * sms, (4 * k * sms + 2) // 3) for k in seen}
    else:
        assert all(seen[k] <= k * sms for k in seen) and seen[1] < seen[3]
