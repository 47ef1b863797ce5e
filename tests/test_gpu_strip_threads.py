"""The column pass runs with the threads that fhd_set_cta_threads asks for: its block size read from the kernel nodes
of a captured call, at a strip that leaves room for one CTA to an SM (where the launch's own choice is 1024)."""
import ctypes

import pytest
import torch

import paper_2505_07158_gb300 as fhd

pytestmark = pytest.mark.gpu

KERNEL_NODE = 0


class KernelNodeParams(ctypes.Structure):
    _fields_ = [("func", ctypes.c_void_p), ("grid", ctypes.c_uint * 3), ("block", ctypes.c_uint * 3),
                ("shared", ctypes.c_uint), ("params", ctypes.c_void_p), ("extra", ctypes.c_void_p),
                ("kern", ctypes.c_void_p), ("ctx", ctypes.c_void_p)]


def block_sizes(call):
    """Threads per block of the kernels that call(stream) launches, in no order."""
    cu = ctypes.CDLL("libcuda.so.1")
    s, graph, n = torch.cuda.Stream(), ctypes.c_void_p(), ctypes.c_size_t()
    call(s)
    torch.cuda.synchronize()
    assert cu.cuStreamBeginCapture_v2(ctypes.c_void_p(s.cuda_stream), 2) == 0   # relaxed
    try:
        call(s)
    finally:
        assert cu.cuStreamEndCapture(ctypes.c_void_p(s.cuda_stream), ctypes.byref(graph)) == 0
    assert cu.cuGraphGetNodes(graph, None, ctypes.byref(n)) == 0
    nodes = (ctypes.c_void_p * n.value)()
    assert cu.cuGraphGetNodes(graph, nodes, ctypes.byref(n)) == 0
    out = []
    for node in nodes:
        kind = ctypes.c_int()
        assert cu.cuGraphNodeGetType(ctypes.c_void_p(node), ctypes.byref(kind)) == 0
        if kind.value == KERNEL_NODE:
            p = KernelNodeParams()
            assert cu.cuGraphKernelNodeGetParams_v2(ctypes.c_void_p(node), ctypes.byref(p)) == 0
            out.append(p.block[0] * p.block[1] * p.block[2])
    assert cu.cuGraphDestroy(graph) == 0
    return sorted(out)


@pytest.mark.parametrize("chosen,P,threads", [(512, 64, 512), (256, 64, 256), (0, 64, 1024), (512, 16, 512), (0, 16, 512)])
def test_threads_of_the_column_pass(chosen, P, threads):
    h, w, c = 1080, 1920, 3
    g = torch.Generator(device="cuda").manual_seed(P)
    F, B = (torch.randint(0, 256, (h, w, c), dtype=torch.uint8, device="cuda", generator=g) for _ in range(2))
    D = torch.randint(-32768, 32768, (c * (h + w),), dtype=torch.int16, device="cuda", generator=g)
    E = torch.empty_like(F)
    fhd.fhd_set_strip_width(h, w, c, P)
    fhd.fhd_set_cta_threads(h, w, c, chosen, 128)
    try:
        assert block_sizes(lambda s: fhd.fhd_permute_encrypt(F, D, B, out=E, stream=s)) == sorted([128, threads])
        assert block_sizes(lambda s: fhd.fhd_permute_decrypt(E, D, B, out=F, stream=s)) == sorted([128, threads])
    finally:
        fhd.fhd_set_strip_width(h, w, c, 0)
        fhd.fhd_set_cta_threads(h, w, c, 0, 0)
