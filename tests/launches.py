"""Which kernels a call launches, read from a stream capture of it."""
import re

import torch


def _identifiers(mangled):
    """The nested names at the head of an Itanium-mangled symbol: _ZN 6 kvswap 14 combine_kernel I..E .."""
    at, names = re.match(r"_ZN?", mangled).end(), []
    while at < len(mangled) and mangled[at].isdigit():
        digits = re.match(r"\d+", mangled[at:]).group(0)
        at += len(digits)
        names.append(mangled[at:at + int(digits)])
        at += int(digits)
    return names


def launched(call):
    """Names of the kernels that `call()` enqueues, without template arguments, in the order they were captured."""
    from cuda.bindings import driver as cu
    graph = torch.cuda.CUDAGraph(keep_graph=True)
    side = torch.cuda.Stream()
    side.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(side):
        call()                                               # what a first call sets up is not part of the capture
        side.synchronize()
        with torch.cuda.graph(graph, stream=side):
            call()
    torch.cuda.current_stream().wait_stream(side)

    def ok(result):
        assert result[0] == cu.CUresult.CUDA_SUCCESS, result[0]
        return result[1]

    raw = cu.CUgraph(graph.raw_cuda_graph())
    err, _, n = cu.cuGraphGetNodes(raw)
    assert err == cu.CUresult.CUDA_SUCCESS
    err, nodes, n = cu.cuGraphGetNodes(raw, n)
    assert err == cu.CUresult.CUDA_SUCCESS
    names = []
    for node in nodes[:n]:
        if ok(cu.cuGraphNodeGetType(node)) != cu.CUgraphNodeType.CU_GRAPH_NODE_TYPE_KERNEL:
            continue
        params = ok(cu.cuGraphKernelNodeGetParams(node))
        mangled = ok(cu.cuFuncGetName(params.func) if int(params.func) else cu.cuKernelGetName(params.kern)).decode()
        names.append(_identifiers(mangled)[-1])
    return names
