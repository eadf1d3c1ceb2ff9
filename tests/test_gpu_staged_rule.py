"""Which half-passes run the staged 16-bit kernel without any hook: those whose
rounds of 1024-site tiles over the 152 SMs are more than five and at least 0.9
filled.  The kernel is read off the graph of a captured call.

The staged arithmetic is that of the register-fed FX16 kernel: equal bits.
FP16 runs one site per thread elsewhere: equal to 2e-3, FP16's rounding order.
"""
import ctypes

import numpy as np
import pytest
import torch

import gen
import paper_1111_0125_gb300 as stg
from paper_1111_0125_gb300 import Gauge

pytestmark = pytest.mark.gpu


def _links(dims):
    """Random SU(3) links out of 4096 Haar matrices."""
    r = np.random.default_rng(3)
    pool = gen.haar_su3(r, 4096)
    lx, ly, lz, lt = dims
    return pool[r.integers(0, len(pool), (lt, lz, ly, lx, 4))]


def _kernels(call):
    """Names of the kernels that call(stream) launches, by capturing it."""
    cu = ctypes.CDLL("libcuda.so.1")

    def ok(err):
        assert err == 0, err

    s = torch.cuda.Stream()
    stream = ctypes.c_void_p(s.cuda_stream)
    graph, n = ctypes.c_void_p(), ctypes.c_size_t()
    ok(cu.cuStreamBeginCapture_v2(stream, 2))  # relaxed
    call(s)
    ok(cu.cuStreamEndCapture(stream, ctypes.byref(graph)))
    ok(cu.cuGraphGetNodes(graph, None, ctypes.byref(n)))
    nodes = (ctypes.c_void_p * n.value)()
    ok(cu.cuGraphGetNodes(graph, nodes, ctypes.byref(n)))
    names = []
    for node in nodes:
        params = (ctypes.c_void_p * 32)()  # CUDA_KERNEL_NODE_PARAMS: the function first
        ok(cu.cuGraphKernelNodeGetParams_v2(ctypes.c_void_p(node), params))
        name = ctypes.c_char_p()
        ok(cu.cuFuncGetName(ctypes.byref(name), ctypes.c_void_p(params[0])))
        names.append(name.value.decode())
    ok(cu.cuGraphDestroy(graph))
    return " ".join(names)


@pytest.mark.parametrize("dims, staged", [
    ((30, 30, 32, 60), True),    # 843.75 tiles: six rounds, 0.93 filled, the last tile ragged
    ((30, 30, 32, 56), False),   # 787.5 tiles: six rounds, 0.86 filled
    ((30, 30, 32, 50), False),   # 703.1 tiles: five rounds, 0.93 filled
])
@pytest.mark.parametrize("prec", [stg.STG_FP16, stg.STG_FX16])
def test_rule(monkeypatch, dims, staged, prec):
    U = _links(dims)
    chi = torch.from_numpy(gen.source(dims, seed=9)).cuda()
    g = Gauge(dims, U, sloppy=prec, recon=12)
    monkeypatch.setenv("STG_FX16_TILED", "0")
    plain = Gauge(dims, U, sloppy=prec, recon=12)
    try:
        f = g.pack(chi, prec)
        out, want, spare = torch.empty_like(f), torch.empty_like(f), torch.empty_like(f)
        stg.stg_dslash(g.handle, 0, f, out, prec)
        stg.stg_dslash(plain.handle, 0, f, want, prec)
        torch.cuda.synchronize()
        names = _kernels(lambda s: stg.stg_dslash(g.handle, 0, f, spare, prec, s))
        assert "k_dslash" in names and ("k_dslash_fx2_staged" in names) == staged, names
        names = _kernels(lambda s: stg.stg_dslash(plain.handle, 0, f, spare, prec, s))
        assert "k_dslash" in names and "staged" not in names, names
        if prec == stg.STG_FX16 or not staged:
            assert torch.equal(out, want)
        else:
            a, b = g.unpack(out, prec), g.unpack(want, prec)
            assert float(torch.linalg.vector_norm(a - b) / torch.linalg.vector_norm(b)) < 2e-3
    finally:
        g.close()
        plain.close()
