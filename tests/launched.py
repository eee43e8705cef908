"""Which kernels a call launches, and with how many CTAs: for tests that have to reach one form of a dispatch.

The call is captured into a CUDA graph, which is looked at and thrown away: nothing of the call runs."""
import math

import torch
from cuda.bindings import driver


def launched(call):
    """[(kernel name, CTAs)] in launch order.  The call must have run once before (kernels are loaded on their first launch)."""
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph(keep_graph=True)
    with torch.cuda.graph(graph):
        call()
    handle = graph.raw_cuda_graph()
    _, _, n = driver.cuGraphGetNodes(handle, 0)
    err, nodes, n = driver.cuGraphGetNodes(handle, n)
    assert err == driver.CUresult.CUDA_SUCCESS, err
    out = []
    for node in nodes[:n]:
        if driver.cuGraphNodeGetType(node)[1] != driver.CUgraphNodeType.CU_GRAPH_NODE_TYPE_KERNEL:
            continue
        err, p = driver.cuGraphKernelNodeGetParams(node)
        assert err == driver.CUresult.CUDA_SUCCESS, err
        err, name = driver.cuFuncGetName(p.func)
        assert err == driver.CUresult.CUDA_SUCCESS, err
        out.append((name.decode(), math.prod((p.gridDimX, p.gridDimY, p.gridDimZ))))
    return out


def ran(call, kernel):
    """CTAs of the launches of `kernel` in the call, 0 if there is none."""
    return sum(ctas for name, ctas in launched(call) if kernel in name)
