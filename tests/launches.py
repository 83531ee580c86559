"""The kernels that a call launches, read from a CUDA graph that captures it."""
import re
from collections import namedtuple

import torch

Launch = namedtuple("Launch", "kernel numbers blocks threads cluster")   # numbers: the integer template arguments


def launched(call):
    """[Launch] of the library's kernels in the order of their launches, without those of torch.  The graph is run once, so that the
    call's outputs hold what they should."""
    from cuda.bindings import driver

    def ok(result):
        assert result[0] == driver.CUresult.CUDA_SUCCESS, result[0]
        return result[1:]

    call()                                               # (torch's own first-time work stays out of the capture)
    graph = torch.cuda.CUDAGraph(keep_graph=True)
    with torch.cuda.graph(graph):
        kept = call()
    handle = driver.CUgraph(graph.raw_cuda_graph())
    _, n = ok(driver.cuGraphGetNodes(handle))
    nodes, n = ok(driver.cuGraphGetNodes(handle, n))
    out = []
    for node in nodes[:n]:
        if ok(driver.cuGraphNodeGetType(node))[0] != driver.CUgraphNodeType.CU_GRAPH_NODE_TYPE_KERNEL:
            continue
        params, = ok(driver.cuGraphKernelNodeGetParams(node))
        mangled = ok(driver.cuFuncGetName(params.func))[0].decode()
        name = re.search(r"\d(walk_cluster|walk_stream|verify_tree_ring|draw_target|scan_topk|scan_level|sbs_epilogue|sbs_chain|filter_rows|clear_status)_kernel", mangled)
        if name:
            attribute, = ok(driver.cuGraphKernelNodeGetAttribute(node, driver.CUkernelNodeAttrID.CU_LAUNCH_ATTRIBUTE_CLUSTER_DIMENSION))
            out.append(Launch(name.group(1), tuple(int(i) for i in re.findall(r"L[ib](\d+)E", mangled)), params.gridDimX, params.blockDimX, attribute.clusterDim.x))
    graph.instantiate()
    graph.replay()
    torch.cuda.synchronize()
    del kept
    return out
