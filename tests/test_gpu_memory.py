"""Device memory of the library's objects: what the pool keeps is given back on request, and objects in use stay as they are."""
import pytest
import torch

from paper_2411_00850_b200 import binding as gwq
from paper_2411_00850_b200 import synth
from tests.gpu_util import quantize_on_gpu, x_tensor

pytestmark = pytest.mark.gpu


def test_kept_memory_is_given_back():
    W, G = synth.make_weight_and_grad(4096, 4096, 150)
    kept = quantize_on_gpu(W[:256], G[:256], 0.01, 4, 128)
    x = x_tensor(synth.make_activations(4, 4096, seed=150, dtype="f16")[0], "f16")
    want = gwq.gwq_linear(kept, x)
    layers = [quantize_on_gpu(W, G, 0.01, 8, 128) for _ in range(4)]   # 18 MB each
    for P in layers:
        P.free()
    torch.cuda.empty_cache()
    torch.cuda.synchronize()
    before = torch.cuda.mem_get_info()[0]
    gwq.gwq_trim_memory()
    assert torch.cuda.mem_get_info()[0] - before >= 32 << 20
    assert torch.equal(gwq.gwq_linear(kept, x), want)
    again = quantize_on_gpu(W, G, 0.01, 8, 128)   # the pool grows again
    gwq.gwq_trim_memory(1 << 30)                  # more than it keeps: nothing to do
    again.free()
    gwq.gwq_trim_memory(device=0)
    assert torch.equal(gwq.gwq_linear(kept, x), want)
