"""Which sampler a network has: k_sample_pipe from L = 8 and for up to four hidden layers, k_sample elsewhere.  The first
also needs the compiler to give it exactly the registers its split is written for, and the library falls back without
a word: the kernel is read off a captured call."""
import ctypes

import pytest

import paper_0903_3053_gb300 as mc

pytestmark = pytest.mark.gpu


def kernel_names(rt, graph):
    n = ctypes.c_size_t()
    assert rt.cudaGraphGetNodes(graph, None, ctypes.byref(n)) == 0
    nodes = (ctypes.c_void_p * n.value)()
    assert rt.cudaGraphGetNodes(graph, nodes, ctypes.byref(n)) == 0
    names = []
    for node in nodes:
        kind = ctypes.c_int()
        assert rt.cudaGraphNodeGetType(ctypes.c_void_p(node), ctypes.byref(kind)) == 0
        if kind.value == 0:  # a kernel; its parameters start with the function
            params = (ctypes.c_void_p * 16)()
            assert rt.cudaGraphKernelNodeGetParams(ctypes.c_void_p(node), params) == 0
            name = ctypes.c_char_p()
            assert rt.cudaFuncGetName(ctypes.byref(name), ctypes.c_void_p(params[0])) == 0
            names.append(name.value.decode())
    return names


@pytest.mark.parametrize("L,depth,pipe", [(64, 6, True), (8, 3, True), (128, 6, True), (10, 4, True), (6, 4, False),
                                          (2, 6, False), (16, 7, False)])
def test_sampler_kernel(L, depth, pipe):
    import torch
    rt = ctypes.CDLL("libcudart.so.13")  # the one libmc.so is linked with
    s = torch.cuda.Stream()
    with torch.cuda.stream(s):
        net = mc.VAN(L, batch=32, depth=depth, seed=1)
        net.sample(32, 0)
        net.sync()
        h, g = ctypes.c_void_p(s.cuda_stream), ctypes.c_void_p()
        assert rt.cudaStreamBeginCapture(h, 2) == 0  # relaxed: the outputs are allocated in the call
        net.sample(32, 1)
        assert rt.cudaStreamEndCapture(h, ctypes.byref(g)) == 0
        names = kernel_names(rt, g)
        assert rt.cudaGraphDestroy(g) == 0
        net.close()
    assert len(names) == 1 and ("k_sample_pipe" in names[0]) == pipe and "k_sample" in names[0]
