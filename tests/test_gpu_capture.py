"""FP64 operator products recorded in a CUDA graph: kernels only, so that the
graph can be instantiated twice and cloned, and replays act on new inputs.  Sizes:
the few-site kernel, the batched one, odd extents, the Schur operator.  The
replays run the kernels of the recording: two replays agree to the bit, and with
the direct call to its rounding (64 units of 2^-53 of the largest entry, as for any two
forms of the product)."""
import ctypes

import numpy as np
import pytest

from inputs import lattice as L

from .gpu_util import cuda, host

pytestmark = pytest.mark.gpu

KERNEL = 0   # CU_GRAPH_NODE_TYPE_KERNEL


@pytest.fixture(scope="module")
def wdl():
    import paper_0710_1988_gb300 as wdl
    wdl.lib()
    return wdl


@pytest.mark.parametrize("dims,nrhs,even_odd", [((4, 4, 4, 4), 1, False), ((16, 16, 16, 8), 3, False),
                                                ((13, 9, 7, 15), 2, False), ((8, 8, 8, 16), 2, True)])
def test_captured_product(wdl, dims, nrhs, even_odd):
    import torch
    cu = ctypes.CDLL("libcuda.so.1")
    op = wdl.WilsonOperator(dims, cuda(L.gauge_field(dims, 0.5, 61)), 0.13, 0.05)
    op.set_operator(even_odd)
    x = cuda(L.gaussian_spinor(dims, 62, nrhs=nrhs).reshape(nrhs, -1)[:, : op.op_n])
    out, direct = torch.empty_like(x), torch.empty_like(x)
    op.apply(x, direct)                      # sizes the handle's own buffers
    torch.cuda.synchronize()
    st = torch.cuda.Stream()
    s, graph = ctypes.c_void_p(st.cuda_stream), ctypes.c_void_p()
    assert cu.cuStreamBeginCapture_v2(s, ctypes.c_int(1)) == 0
    try:
        op.apply(x, out, stream=st.cuda_stream)
    finally:
        assert cu.cuStreamEndCapture(s, ctypes.byref(graph)) == 0
    n = ctypes.c_size_t()
    assert cu.cuGraphGetNodes(graph, None, ctypes.byref(n)) == 0 and n.value > 0
    nodes = (ctypes.c_void_p * n.value)()
    assert cu.cuGraphGetNodes(graph, nodes, ctypes.byref(n)) == 0
    kind = ctypes.c_int()
    for node in nodes:
        assert cu.cuGraphNodeGetType(ctypes.c_void_p(node), ctypes.byref(kind)) == 0 and kind.value == KERNEL
    clone = ctypes.c_void_p()
    assert cu.cuGraphClone(ctypes.byref(clone), graph) == 0
    got = []
    for g in (graph, graph, clone):
        ex = ctypes.c_void_p()
        assert cu.cuGraphInstantiateWithFlags(ctypes.byref(ex), g, ctypes.c_ulonglong(0)) == 0
        out.zero_()
        torch.cuda.synchronize()
        assert cu.cuGraphLaunch(ex, s) == 0
        st.synchronize()
        got.append(host(out).copy())
        if len(got) == 2:                    # the third replay reads other inputs
            x.mul_(2.0)
    assert np.array_equal(got[0], got[1]) and np.array_equal(2.0 * got[0], got[2])
    d = host(direct)
    assert np.abs(got[0] - d).max() <= 64 * 2.0 ** -53 * np.abs(d).max()
    op.close()
