import os
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
if ROOT not in sys.path:
    sys.path.insert(0, ROOT)


def pytest_configure(config):
    config.addinivalue_line("markers", "gpu: needs a CUDA device (B200)")


def load_golden(name):
    """Parse a tests/golden text fixture: 'name rows cols' headers followed by rows of numbers."""
    import numpy as np
    out = {}
    path = os.path.join(ROOT, "tests", "golden", name)
    with open(path) as f:
        lines = [ln.strip() for ln in f if ln.strip() and not ln.startswith("#")]
    i = 0
    while i < len(lines):
        key, r, c = lines[i].split()
        r, c = int(r), int(c)
        vals = [[float(v) for v in lines[i + 1 + j].split()] for j in range(r)]
        out[key] = np.array(vals, dtype=np.float64).reshape(r, c)
        i += 1 + r
    return out


def kernels_launched(call):
    """What `call` enqueues on the current stream, from a capture of it: [(mangled kernel name, CTAs per cluster)]."""
    import torch
    from cuda.bindings import driver as d

    def ok(r):
        assert r[0] == d.CUresult.CUDA_SUCCESS, r[0]
        return r[1:] if len(r) > 2 else r[1]

    graph, side = torch.cuda.CUDAGraph(keep_graph=True), torch.cuda.Stream()
    side.wait_stream(torch.cuda.current_stream())
    with torch.cuda.graph(graph, stream=side):
        call()
    raw, out = d.CUgraph(graph.raw_cuda_graph()), []
    count = ok(d.cuGraphGetNodes(raw, 0))[1]
    for node in ok(d.cuGraphGetNodes(raw, count))[0]:
        if ok(d.cuGraphNodeGetType(node)) != d.CUgraphNodeType.CU_GRAPH_NODE_TYPE_KERNEL:
            continue
        p = ok(d.cuGraphKernelNodeGetParams(node))
        name = ok(d.cuFuncGetName(p.func)) if int(p.func) else ok(d.cuKernelGetName(p.kern))
        a = ok(d.cuGraphKernelNodeGetAttribute(node, d.CUkernelNodeAttrID.CU_LAUNCH_ATTRIBUTE_CLUSTER_DIMENSION))
        out.append((name.decode(), max(1, a.clusterDim.x * a.clusterDim.y * a.clusterDim.z)))
    return out
