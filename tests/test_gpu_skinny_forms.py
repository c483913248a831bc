"""The tcgen05 decode kernel on the forms that no mma.sync kernel has (groups of 16 and 32 beyond 32 columns, 3 bits in groups of 64
with bf16) and on small layers of 17 to 32 tokens, where sizes can go wrong: one step, ragged tiles and rows, windows and units cut
by the ends of rows and of shares, more outliers in a window than a slot holds, more tiles than CTAs."""
import ctypes as C

import numpy as np
import pytest
import torch

from oracle import gwq_oracle as orc
from paper_2411_00850_b200 import binding as gwq
from paper_2411_00850_b200 import synth
from tests.gpu_util import assert_linear_close, checker_rows, distinct_rows, oracle_w_hat, quantize_on_gpu, x_tensor

pytestmark = pytest.mark.gpu


def _layer(N, K, frac, bits, group, crowd=False):
    W, G = synth.make_weight_and_grad(N, K, N + K)
    if crowd:
        G[:, K // 2:K // 2 + 128] *= np.float32(1e4)
    return quantize_on_gpu(W, G, frac, bits, group), oracle_w_hat(orc.quantize_layer(W, G, frac, bits, group))


def _close(y, y_ref, bound, K):
    # q - z and outliers are exact, so what is left are FP32 sums: a tensor core cuts every product and the sum so far below 2^-24 or so
    # of the largest (K of them, 2^-25 of the sum of magnitudes each), and some 72 roundings of scales, steps, outliers and pieces.
    # Rounded weights, or a row in a thousand without one outlier, would be 1e-4 off in the 2-norm; these sums are 1e-7 to 4e-7.
    err = np.abs(y.double().cpu().numpy() - y_ref)
    assert np.all(err <= (K / 4 + 72) * 2.0 ** -23 * bound + 1e-30), float((err / bound).max())
    assert np.linalg.norm(err) <= 2e-6 * np.linalg.norm(y_ref)


def _check(P, w_hat, M, dtype):
    bits16, xv = synth.make_activations(M, P.K, seed=M, dtype=dtype, heavy_channels=8 if dtype == "bf16" else 0)
    x = x_tensor(bits16, dtype)
    y = gwq.gwq_linear(P, x, out_dtype=torch.float32)
    assert gwq.gwq_device_status(P) == 0
    _close(y, *orc.linear(xv, w_hat), P.K)
    assert torch.equal(y, gwq.gwq_linear(P, x, out_dtype=torch.float32))
    _check_columns(P, w_hat, M, dtype, np.arange(P.N))


def _check_columns(P, w_hat, M, dtype, rows):
    """One-hot activations read single weights back, exactly: ends of steps and of windows, and the columns between (crowded ones
    among them: entries past what a slot holds)."""
    K = P.K
    cols = sorted({c for c in [0, K - 1, 127, 128 % K, 511 % K, 512 % K] + [K // 2 + 5 * i for i in range(26)] if c < K})
    for at in range(0, len(cols), M):
        mine = (cols[at:at + M] * M)[:M]
        y = gwq.gwq_linear(P, x_tensor(synth.unit_activations(mine, K, dtype)[0], dtype), out_dtype=torch.float32)
        assert np.array_equal(y.cpu().numpy()[:, rows], w_hat[:, mine].T.astype(np.float32))


@pytest.mark.parametrize("N,K,frac,bits,group,crowd,calls", [
    (5, 128, 0.02, 4, 16, False, ((5, "f16"), (16, "bf16"))),                   # one step, a ragged tile of 16 rows
    (300, 1152, 0.01, 3, 16, False, ((8, "bf16"), (9, "f16"))),                 # nine steps: windows of four and of one
    (137, 2176, 0.05, 2, 32, True, ((9, "f16"), (17, "bf16"), (32, "f16"))),    # crowded windows, seventeen steps
    (260, 640, 0.01, 4, 32, False, ((16, "bf16"), (24, "f16"))),
    (1500, 1920, 0.01, 3, 64, True, ((17, "bf16"), (25, "bf16"), (20, "f16"))),   # 12 tiles x 15 steps: one or two steps per CTA
    (2050, 2304, 0.02, 3, 64, False, ((32, "bf16"), (32, "f16"))),                # shares that cut units, a tile of two rows
    (20000, 128, 0.01, 3, 64, False, ((18, "bf16"),)),                            # a step per tile, more tiles than CTAs
    (1100, 4096, 0.3, 4, 128, False, ((17, "f16"), (31, "f16"))),                 # slots that overflow
])
def test_forms(N, K, frac, bits, group, crowd, calls):
    P, w_hat = _layer(N, K, frac, bits, group, crowd)
    for M, dtype in calls:
        _check(P, w_hat, M, dtype)
    P.free()


# bf16 activations are multiplied as they are: a channel 2^70 above the others leaves the rest of a row's sum alone where its weight
# is zero, a common power of two comes out again exactly, and one infinite activation spoils its own token only (fp16 too).
@pytest.mark.parametrize("N,K,frac,bits,group,M", [(300, 1152, 0.01, 3, 16, 8), (260, 640, 0.02, 4, 32, 16), (137, 2176, 0.05, 2, 32, 17),
                                                   (1500, 1920, 0.01, 3, 64, 32)])
def test_range_of_activations(N, K, frac, bits, group, M):
    W, G = synth.make_weight_and_grad(N, K, N + K)
    far, G[:, K // 2 + 3] = K // 2 + 3, 0.0
    W[::2, far] = 0.0
    P, w_hat = quantize_on_gpu(W, G, frac, bits, group), oracle_w_hat(orc.quantize_layer(W, G, frac, bits, group))
    bits16, xv = synth.make_activations(M, K, seed=M, dtype="bf16", heavy_channels=8)
    x = x_tensor(bits16, "bf16")
    y = gwq.gwq_linear(P, x, out_dtype=torch.float32)
    for power in (2.0 ** 112, 2.0 ** -80):
        assert torch.equal(gwq.gwq_linear(P, x * power, out_dtype=torch.float32), y * power)
    x[:, far], xv[:, far] = 2.0 ** 70, 2.0 ** 70
    y_ref, bound = orc.linear(xv, w_hat)
    err = np.abs(gwq.gwq_linear(P, x, out_dtype=torch.float32).double().cpu().numpy() - y_ref)
    assert np.all(err <= (K + 72) * 2.0 ** -23 * bound + 1e-30), float((err / bound).max())
    for dtype in ("f16", "bf16"):
        x = x_tensor(synth.make_activations(M, K, seed=M, dtype=dtype)[0], dtype)
        y = gwq.gwq_linear(P, x)
        x[M - 2, far] = float("inf")
        spoilt = gwq.gwq_linear(P, x)
        assert not bool(torch.isfinite(spoilt[M - 2]).any())
        assert torch.equal(torch.cat((spoilt[:M - 2], spoilt[M - 1:])), torch.cat((y[:M - 2], y[M - 1:])))
    assert gwq.gwq_device_status(P) == 0
    P.free()


def test_layers_of_one_call_give_the_bits_of_the_single_calls():
    layers = [_layer(N, 1152, 0.02, 4, 16)[0] for N in (260, 5, 3000)]
    for M, dtype in ((8, "f16"), (13, "bf16")):
        x = x_tensor(synth.make_activations(M, 1152, seed=M, dtype=dtype)[0], dtype)
        for many, P in zip(gwq.gwq_linear_multi(layers, x), layers):
            assert torch.equal(many, gwq.gwq_linear(P, x))


# Host buffers: fp16 activations are read by the pre-pass where they are, bf16 ones are copied first.
@pytest.mark.parametrize("M,dtype", [(7, "f16"), (20, "bf16")])
def test_host_buffers(M, dtype):
    P, _ = _layer(300, 1152, 0.02, 3, 16 if M <= 16 else 64)
    x = x_tensor(synth.make_activations(M, 1152, seed=M, dtype=dtype)[0], dtype)
    want = gwq.gwq_linear(P, x).cpu()
    for pin in (True, False):
        xh, yh = x.cpu(), torch.zeros_like(want)
        if pin:
            xh, yh = xh.pin_memory(), yh.pin_memory()
        gwq.gwq_linear_host(P, xh, yh)
        assert torch.equal(yh, want)


# Large layers, on both sides of the rule, by a sample of their rows.
@pytest.mark.parametrize("N,K,bits,group,M,dtype", [
    (8192, 8192, 8, 128, 8, "f16"), (8192, 8192, 8, 128, 6, "bf16"), (8192, 8192, 2, 64, 8, "bf16"), (8192, 8192, 4, 128, 16, "bf16"),
    (8100, 8192, 3, 128, 32, "f16"), (8192, 8192, 4, 128, 8, "f16"), (4096, 4096, 4, 128, 32, "bf16"),
])
def test_large_layers(N, K, bits, group, M, dtype):
    g = torch.Generator(device="cuda")
    g.manual_seed(7)
    W = torch.randn(N, K, device="cuda", generator=g).mul_(0.02).half()
    P = gwq.gwq_pack(W, gwq.gwq_select_outliers(W, torch.randn(N, K, device="cuda", generator=g), 0.01), bits, group)
    a = {k: v.cpu().numpy() for k, v in P.arrays().items()}
    rows = np.array(distinct_rows(N, 7, 300))
    w_hat = checker_rows(W.cpu().numpy(), a["row_ptr"], a["col_idx"], a["val"].view(np.uint16), rows, bits, group)[3]
    bits16, xv = synth.make_activations(M, K, seed=M, dtype=dtype, heavy_channels=8 if dtype == "bf16" else 0)
    x = x_tensor(bits16, dtype)
    y_ref, bound = orc.linear(xv, w_hat)
    y = gwq.gwq_linear(P, x, out_dtype=torch.float32)
    alone = torch.empty_like(y)   # without a workspace: a kernel of the others
    xd = gwq.GWQ_F16 if dtype == "f16" else gwq.GWQ_BF16
    assert gwq.load_library().gwq_linear(P._h, C.c_void_p(x.data_ptr()), xd, M, C.c_void_p(alone.data_ptr()), gwq.GWQ_F32,
                                         C.c_void_p(torch.cuda.current_stream().cuda_stream)) == 0
    assert gwq.gwq_device_status(P) == 0
    if gwq.load_library().gwq_linear_workspace_bytes(P._h, xd, M) > (K // 128) * 2048 * 4 + 65536:   # partial sums: the tcgen05 kernel
        _close(y[:, rows], y_ref, bound, K)
        _check_columns(P, np.broadcast_to(w_hat, w_hat.shape), M, dtype, rows)
    assert_linear_close(y[:, rows], y_ref, bound)
    assert_linear_close(alone[:, rows], y_ref, bound)
    P.free()


# Which kernel a call takes, told by the workspace it asks for (partial sums, or the other kernels' copy of the activations or nothing), on
# both sides of the lines (us, the others' / this kernel's): 14.8 / 16.6, 18.9 / 14.7, 22.2 / 24.4, 27.6 / 25.7, 57.5 / 63.4, 68.7 / 63.3,
# 19.2 / 20.9, 30.8 / 35.2, 35.2 / 33.5; 8-bit codes with bf16 activations have no variant.
@pytest.mark.parametrize("N,K,bits,group,dtype,M,taken", [
    (16384, 2048, 2, 64, "f16", 12, False), (4096, 4096, 2, 64, "f16", 12, True), (16384, 4096, 4, 128, "f16", 12, False),
    (4096, 16384, 4, 128, "f16", 12, True), (8192, 28672, 4, 32, "f16", 2, False), (8192, 28672, 3, 32, "f16", 2, True),
    (11008, 4096, 4, 32, "bf16", 4, False), (16384, 4096, 4, 128, "bf16", 32, False), (8192, 8192, 4, 128, "bf16", 32, True),
    (8192, 8192, 8, 128, "bf16", 8, False), (8192, 8192, 8, 128, "f16", 8, True),
])
def test_choice_of_the_decode_kernel(N, K, bits, group, dtype, M, taken):
    W = torch.full((N, K), 0.5, dtype=torch.float16, device="cuda")
    P = gwq.gwq_pack(W, gwq.gwq_select_outliers(W, torch.zeros(N, K, device="cuda"), 0.0), bits, group)
    asked = gwq.load_library().gwq_linear_workspace_bytes(P._h, gwq.GWQ_F16 if dtype == "f16" else gwq.GWQ_BF16, M)
    assert (asked not in (0, K // 128 * 8576)) == taken
    P.free()
