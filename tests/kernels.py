"""Which kernels of the library a call launches, for tests that are about one of several forms."""
import re

import torch


def launched(call):
    """(result of call(), names of the kernels it launches), read from the nodes of a captured graph of the call.  Templates carry
    their integer arguments: k_forward_fused<0,1,256,128,2>."""
    from cuda.bindings import driver
    result = call()                                          # also the one-time look-ups, which a capture may not contain
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph(keep_graph=True)
    with torch.cuda.graph(graph):
        call()
    raw = driver.CUgraph(graph.raw_cuda_graph())
    n = driver.cuGraphGetNodes(raw)[2]
    names = set()
    for node in driver.cuGraphGetNodes(raw, n)[1][:n]:
        if driver.cuGraphNodeGetType(node)[1] != driver.CUgraphNodeType.CU_GRAPH_NODE_TYPE_KERNEL:
            continue
        symbol = driver.cuFuncGetName(driver.cuGraphKernelNodeGetParams(node)[1].func)[1].decode()
        m = re.match(r"_ZN6psattn(\d+)(k_.*)", symbol)
        if m is None:
            continue
        name, rest = m.group(2)[:int(m.group(1))], m.group(2)[int(m.group(1)):]
        ints = re.findall(r"L[bi](\d+)E", rest.split("Ev", 1)[0]) if rest.startswith("I") else []
        names.add(name + ("<%s>" % ",".join(ints) if ints else ""))
    return result, names
