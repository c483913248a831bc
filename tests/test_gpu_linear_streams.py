"""Calls on one layer from several streams: up to eight tokens share nothing, with or without a workspace, and from nine on calls with
workspaces of their own (the binding's) share nothing either.  Calls without a workspace, and calls of several layers, against
the single calls and the CPU checker."""
import ctypes as C

import pytest
import torch

from oracle import gwq_oracle as orc
from paper_2411_00850_b200 import binding as gwq
from paper_2411_00850_b200 import synth
from tests.gpu_util import assert_linear_close, oracle_w_hat, quantize_on_gpu, x_tensor

pytestmark = pytest.mark.gpu
CODES = {"f16": gwq.GWQ_F16, "bf16": gwq.GWQ_BF16}


def _layer(N, K, bits, group):
    W, G = synth.make_weight_and_grad(N, K, 140 + bits)
    return quantize_on_gpu(W, G, 0.01, bits, group), oracle_w_hat(orc.quantize_layer(W, G, 0.01, bits, group))


def _x(M, K, seed, dtype="f16"):
    bits16, xv = synth.make_activations(M, K, seed=seed, dtype=dtype)
    return x_tensor(bits16, dtype), xv


def _without_workspace(P, x, y):
    xd = gwq.GWQ_F16 if x.dtype == torch.float16 else gwq.GWQ_BF16
    st = gwq.load_library().gwq_linear(P._h, x.data_ptr(), xd, x.shape[0], y.data_ptr(), gwq._dtype_code(y.dtype),
                                       torch.cuda.current_stream().cuda_stream)
    assert st == 0


# 4096 rows of K = 4096: staged activations and the streaming kernel; K = 11008: too long to stage
@pytest.mark.parametrize("K,M,bits,group,workspace", [
    (4096, 8, 4, 128, False), (4096, 5, 3, 128, False), (11008, 8, 4, 128, False), (4096, 4, 4, 16, False),
    (4096, 8, 4, 128, True), (4096, 16, 4, 128, True), (11008, 32, 4, 64, True),
])
def test_two_streams_on_one_layer(K, M, bits, group, workspace):
    W, G = synth.make_weight_and_grad(4096, K, 141)
    P = quantize_on_gpu(W, G, 0.01, bits, group)
    call = (lambda x, y: gwq.gwq_linear(P, x, out=y)) if workspace else (lambda x, y: _without_workspace(P, x, y))
    xs = [_x(M, K, 7)[0], _x(M, K, 8)[0] * 3]
    want = []
    for x in xs:
        want.append(torch.empty(M, 4096, dtype=torch.float32, device=x.device))
        call(x, want[-1])
    torch.cuda.synchronize()
    outs = [[torch.empty_like(want[0]) for _ in range(40)] for _ in range(2)]
    graph, side = torch.cuda.CUDAGraph(), torch.cuda.Stream()   # two branches, so that no call waits for the host
    with torch.cuda.graph(graph):
        side.wait_stream(torch.cuda.current_stream())
        for s, on in enumerate((torch.cuda.current_stream(), side)):
            with torch.cuda.stream(on):
                for y in outs[s]:
                    call(xs[s], y)
        torch.cuda.current_stream().wait_stream(side)
    for _ in range(5):
        graph.replay()
    torch.cuda.synchronize()
    for s in range(2):
        assert sum(not torch.equal(o, want[s]) for o in outs[s]) == 0


@pytest.mark.parametrize("N,K,bits,group", [(1000, 4096, 4, 128), (600, 28672, 3, 128), (520, 11008, 4, 64), (400, 1024, 4, 16),
                                            (400, 1024, 3, 32), (400, 4096, 8, 128), (2600, 2304, 2, 128)])
def test_calls_without_a_workspace(N, K, bits, group):
    P, w_hat = _layer(N, K, bits, group)
    lib = gwq.load_library()
    for M, dtype in ((1, "bf16"), (2, "f16"), (3, "bf16"), (5, "f16"), (7, "bf16"), (8, "f16")):
        x, xv = _x(M, K, M, dtype)
        y = torch.empty(M, N, dtype=torch.float32, device=x.device)
        if group < 64 and M * (128 // group) > 32 and dtype == "bf16":   # the tensor-core kernel's fp16 copy needs memory
            st = lib.gwq_linear(P._h, x.data_ptr(), CODES[dtype], M, y.data_ptr(), gwq.GWQ_F32, None)
            assert st == gwq.GWQ_ERR_WORKSPACE
            continue
        _without_workspace(P, x, y)
        assert_linear_close(y, *orc.linear(xv, w_hat))


@pytest.mark.parametrize("M", [1, 4, 6, 8, 16, 24])
@pytest.mark.parametrize("K", [4096, 11008])
def test_several_layers_without_and_with_a_workspace(M, K):
    layers = [_layer(N, K, 4, 128)[0] for N in (256, 1040)]
    lib = gwq.load_library()
    x, _ = _x(M, K, 9)
    hs = (C.POINTER(gwq.gwq_packed) * 2)(*[P._h for P in layers])
    stream = torch.cuda.current_stream().cuda_stream
    ys = [torch.empty(M, P.N, dtype=torch.float16, device=x.device) for P in layers]
    ptrs = (C.c_void_p * 2)(*[y.data_ptr() for y in ys])
    assert lib.gwq_linear_multi(hs, 2, x.data_ptr(), gwq.GWQ_F16, M, ptrs, gwq.GWQ_F16, stream) == 0
    for P, y in zip(layers, ys):
        one = torch.empty_like(y)
        _without_workspace(P, x, one)
        assert torch.equal(y, one)
    need = lib.gwq_linear_multi_workspace_bytes(hs, 2, gwq.GWQ_F16, M)
    assert need >= max(lib.gwq_linear_workspace_bytes(P._h, gwq.GWQ_F16, M) for P in layers)
    ws = torch.empty(max(need, 1), dtype=torch.uint8, device=x.device)
    assert lib.gwq_linear_multi_ws(hs, 2, x.data_ptr(), gwq.GWQ_F16, M, ptrs, gwq.GWQ_F16, ws.data_ptr(), need, stream) == 0
    for P, y, again in zip(layers, ys, gwq.gwq_linear_multi(layers, x)):
        assert torch.equal(y, gwq.gwq_linear(P, x)) and torch.equal(y, again)
