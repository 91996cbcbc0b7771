"""qcams_debug_run_plan against the kernels that a captured run holds."""
import ctypes as C

import numpy as np
import pytest

from paper_2304_02731_gb300 import workloads as W

MORSE, GENERIC = W.SYS_H2_CA_MORSE, W.SYS_H2_CA_LJ12


def _kernel_nodes(graph):
    """Kernel nodes of a kept torch graph (cuGraphGetNodes, cuGraphNodeGetType)."""
    cu = C.CDLL("libcuda.so.1")
    handle, n = C.c_void_p(graph.raw_cuda_graph()), C.c_size_t(0)
    assert cu.cuGraphGetNodes(handle, None, C.byref(n)) == 0
    nodes = (C.c_void_p * n.value)()
    assert cu.cuGraphGetNodes(handle, nodes, C.byref(n)) == 0
    kinds = []
    for node in nodes:
        kind = C.c_int(-1)
        assert cu.cuGraphNodeGetType(C.c_void_p(node), C.byref(kind)) == 0
        kinds.append(kind.value)
    return kinds.count(0)                        # CU_GRAPH_NODE_TYPE_KERNEL


@pytest.mark.gpu
@pytest.mark.parametrize("system,precision,mode,per_sm,more,lanes", [
    (MORSE, 64, 1, 20, 0, [6]), (MORSE, 64, 0, 20, 1, [3, 6]), (MORSE, 64, 1, 80, 1, [3, 3, 6]),
    (GENERIC, 64, 1, 512, 0, [3, 3, 6]), (MORSE, 64, 1, 511, 0, [3, 3, 6]),
    (MORSE, 64, 0, 512, 0, [1, 3, 3, 6]), (MORSE, 64, 2, 1, 0, [3]), (MORSE, 64, 3, 600, 0, [6]),
    (MORSE, 32, 1, 1792, 0, [1]), (MORSE, 32, 1, 1792, 1, [1]), (GENERIC, 32, 1, 1024, 1, [1]),
    (GENERIC, 32, 0, 1024, 1, [1])])
def test_plan_is_what_runs(system, precision, mode, per_sm, more, lanes):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    from paper_2304_02731_gb300 import qcams as Q
    n = per_sm * Q.device_info()[0] + more
    kw = W.INTEG_FP64 if precision == 64 else W.INTEG_FP32
    integ = Q.make_integ(**kw, precision=precision, persistent=mode)
    kernels, got = Q.debug_run_plan([system], integ, n)
    assert got == lanes
    b = Q.Batch.empty(n, "cuda", sys_id=np.zeros(n, np.int32), keep_u=False)
    Q.levels([system], [0], [0], [0])            # the context, before the capture
    graph = torch.cuda.CUDAGraph(keep_graph=True)
    with torch.cuda.graph(graph):
        Q.run_batch([system], b, integ)
    assert _kernel_nodes(graph) == kernels + 2   # the potential shapes and the analysis
