"""Outliers in the fused tensor-core kernel: taken from the lists by tile of 16 rows and step of 128 columns, or, where K is not a
multiple of 128, from the rows' CSR entries; more of them in a step than are held in registers, ragged tiles, slices of K that
begin in the middle of a step; one-hot activations give the weights themselves."""
import numpy as np
import pytest
import torch

from oracle import gwq_oracle as orc
from paper_2411_00850_b200 import binding as gwq
from paper_2411_00850_b200 import synth
from tests.gpu_util import assert_linear_close, oracle_w_hat, quantize_on_gpu, x_tensor

pytestmark = pytest.mark.gpu


def _fused(P, bits16, dtype):
    """The product by the fused kernel: as much workspace as the fp16 copy of bf16 activations and their scales take, none for fp16."""
    x = x_tensor(bits16, dtype)
    M, xd = x.shape[0], gwq.GWQ_F16 if dtype == "f16" else gwq.GWQ_BF16
    y = torch.zeros((M, P.N), dtype=torch.float32, device=x.device)
    ws_bytes = 0 if dtype == "f16" else (M * P.K * 2 + 255) // 256 * 256 + (M * 4 + 255) // 256 * 256
    ws = torch.empty(max(ws_bytes, 256), dtype=torch.uint8, device=x.device)
    st = gwq.load_library().gwq_linear_ws(P._h, x.data_ptr(), xd, M, y.data_ptr(), gwq.GWQ_F32, ws.data_ptr() if ws_bytes else None, ws_bytes,
                                          torch.cuda.current_stream().cuda_stream)
    assert st == 0 and gwq.gwq_device_status(P) == 0
    return y


# (what the binding's workspace chooses: the same fused kernel, with K in slices, or the two-phase path)
@pytest.mark.parametrize("N,K,frac,bits,group,taken", [
    (137, 128, 0.02, 4, 128, "two-phase"),   # a step, a ragged tile whose last 16 rows are not all there
    (300, 2176, 0.05, 3, 64, "slices"),      # 17 steps: a slice of K begins inside one
    (128, 1152, 0.6, 4, 16, "slices"),       # far more than two per lane and step
    (260, 704, 0.05, 4, 64, "two-phase"),    # 64 columns past a step: the CSR entries
    (20000, 256, 0.01, 8, 128, "any"),       # more tiles than SMs
])
def test_outliers_of_prompts(N, K, frac, bits, group, taken):
    W, G = synth.make_weight_and_grad(N, K, N + K)
    G[:, K // 2:K // 2 + 40] *= np.float32(1e3)   # many of them in few columns
    P = quantize_on_gpu(W, G, frac, bits, group)
    w_hat = oracle_w_hat(orc.quantize_layer(W, G, frac, bits, group))
    expanded = gwq.load_library().gwq_linear_workspace_bytes(P._h, gwq.GWQ_F16, 33) >= N * K * 2
    sliced = K // 64 >= 16 and N <= 74 * 128
    assert taken == "any" or (taken == "slices") == sliced and (taken == "two-phase") == (expanded and not sliced)
    for M, dtype in ((33, "f16"), (80, "bf16")):
        bits16, xv = synth.make_activations(M, K, seed=M, dtype=dtype)
        y_ref, bound = orc.linear(xv, w_hat)
        assert_linear_close(_fused(P, bits16, dtype), y_ref, bound)
        assert_linear_close(gwq.gwq_linear(P, x_tensor(bits16, dtype), out_dtype=torch.float32), y_ref, bound)
        assert gwq.gwq_device_status(P) == 0
    cols = [(K // 2 + 13 * i) % K for i in range(40)]
    bits16, xv = synth.unit_activations(cols, K, "f16")
    assert_linear_close(_fused(P, bits16, "f16"), *orc.linear(xv, w_hat))
    assert_linear_close(gwq.gwq_linear(P, x_tensor(bits16, "f16"), out_dtype=torch.float32), *orc.linear(xv, w_hat))
    P.free()


# Which path a prompt takes, told by the workspace it asks for: the expanded weights, or not.  Both sides of the line measured (us,
# two-phase / fused): 20.5 / 24.9, 98 / 112, 71 / 40, 57 / 52, 76 / 47.
@pytest.mark.parametrize("N,K,bits,group,dtype,M,expanded", [
    (16000, 1024, 4, 32, "bf16", 33, True), (9600, 8192, 8, 32, "bf16", 128, True), (18000, 4096, 4, 128, "f16", 33, False),
    (11008, 4096, 4, 128, "f16", 129, False), (18000, 4096, 8, 128, "f16", 33, False),
])
def test_choice_of_the_prompt_path(N, K, bits, group, dtype, M, expanded):
    W = torch.full((N, K), 0.5, dtype=torch.float16, device="cuda")
    P = gwq.gwq_pack(W, gwq.gwq_select_outliers(W, torch.zeros(N, K, device="cuda"), 0.0), bits, group)
    xd = gwq.GWQ_F16 if dtype == "f16" else gwq.GWQ_BF16
    assert (gwq.load_library().gwq_linear_workspace_bytes(P._h, xd, M) >= 2 * N * K) == expanded
    P.free()
