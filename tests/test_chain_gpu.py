"""Layers back to back on one stream, each reading what the one before wrote:
every launch that overlaps its predecessor's end must still see complete
inputs.  The chained run equals, bit for bit, the same calls with a
synchronisation after each."""
import pytest

from paper_2603_06492_gb300 import binding
from paper_2603_06492_gb300.inputs import Layer, make_layer_inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def lib():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    from paper_2603_06492_gb300.build import build
    build()
    binding.load()


@pytest.mark.parametrize("T,d,r", [(130, 1024, 64), (700, 2048, 128), (5000, 512, 32)])
def test_chain_matches_separate_calls(T, d, r):
    import torch
    n = 4
    devs = [binding.params_to_device(make_layer_inputs(Layer("chain", T, d, d, r, "bf16"), 50 + i), "bf16")
            for i in range(n)]
    bufs = [binding.NobleLinearBuffers(T, d, d, r, "bf16") for _ in range(n)]

    def run(sync):
        x = devs[0]["x"]
        xs = []
        for b, p in zip(bufs, devs):
            xs.append(x)
            x = binding.forward(b, x, p)
            if sync:
                torch.cuda.synchronize()
        g = x
        for b, p, xi in zip(reversed(bufs), reversed(devs), reversed(xs)):
            g, _ = binding.backward(b, xi, g, p)
            if sync:
                torch.cuda.synchronize()
        torch.cuda.synchronize()
        return [t.clone() for b in bufs for t in (b.y, b.dx, b.bucket)]

    want = run(True)
    for _ in range(5):
        for b in bufs:
            b.y.fill_(float("nan"))
            b.dx.fill_(float("nan"))
        assert all(torch.equal(a, w) for a, w in zip(run(False), want))
    binding.noble_get_device_status(None)
