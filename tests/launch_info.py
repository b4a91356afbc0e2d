"""Which kernels a call launches, and how: from the nodes of a CUDA graph that the call is captured into."""
import torch


def kernels(call):
    """[{"name", "grid", "local_bytes"}] of the kernels that call() launches on the current stream."""
    from cuda.bindings import driver as cu

    def ok(result):
        assert result[0] == cu.CUresult.CUDA_SUCCESS, result[0]
        return result[1:] if len(result) > 2 else result[1]

    call()                                                # (loads the kernels)
    graph = torch.cuda.CUDAGraph(keep_graph=True)
    with torch.cuda.graph(graph):
        call()
    raw = cu.CUgraph(graph.raw_cuda_graph())
    n = ok(cu.cuGraphGetNodes(raw, 0))[1]
    out = []
    for node in ok(cu.cuGraphGetNodes(raw, n))[0][:n]:
        if ok(cu.cuGraphNodeGetType(node)) != cu.CUgraphNodeType.CU_GRAPH_NODE_TYPE_KERNEL:
            continue
        p = ok(cu.cuGraphKernelNodeGetParams(node))
        func = p.func if int(p.func) else ok(cu.cuKernelGetFunction(p.kern))
        local = cu.CUfunction_attribute.CU_FUNC_ATTRIBUTE_LOCAL_SIZE_BYTES
        out.append(dict(name=ok(cu.cuFuncGetName(func)).decode(), grid=(p.gridDimX, p.gridDimY, p.gridDimZ),
                        local_bytes=ok(cu.cuFuncGetAttribute(local, func))))
    return out
