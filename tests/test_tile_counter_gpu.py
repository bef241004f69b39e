"""The tile counter of the backward's grouped launch: a launch that starts before
its counter is published must compute every tile whatever the word held, and a
captured backward must on every replay."""
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


# what an earlier call, or whoever had the memory before, may have left
STALE = {"zero": 0, "spent": (7 << 32) | 5000, "no tag, spent": 5000, "no tag, running": 3, "ones": -1}


@pytest.mark.parametrize("stale", STALE)
@pytest.mark.parametrize("together", [0, 1])  # first tiles given
# two tiles; 76 tiles, all given; 77, one drawn; seven waves of 76 pairs
@pytest.mark.parametrize("M,N,K", [(200, 136, 64), (4864, 512, 64), (19712, 128, 64), (4096, 4096, 256)])
def test_late_counter(M, N, K, together, stale):
    import torch
    g = torch.Generator(device="cuda").manual_seed(M + K)
    A = torch.randn((K, M), generator=g, device="cuda").bfloat16()
    B = torch.randn((K, N), generator=g, device="cuda").bfloat16()
    C = torch.full((M, N), float("nan"), device="cuda")
    word = torch.full((2,), STALE[stale], dtype=torch.int64, device="cuda")
    torch.cuda.synchronize()
    binding.noble_test_late_counter(M, N, K, A, B, C, word, together, 200_000,
                                    torch.cuda.current_stream().cuda_stream)
    torch.cuda.synchronize()
    binding.noble_get_device_status(None)
    ref = A.double().T @ B.double()
    # fp32 accumulation of K products: a few 2^-24 sqrt(K) of the result's scale
    assert (C.double() - ref).abs().max() <= 2e-5 * ref.abs().max()
    assert int(word[0]) == 0


@pytest.mark.parametrize("shape", [(1000, 512, 768, 64), (2048, 1024, 1024, 0)], ids=lambda s: "x".join(map(str, s)))
def test_replays(shape):
    import torch
    T, di, do, r = shape
    dev = binding.params_to_device(make_layer_inputs(Layer("replay", *shape, "bf16"), 11), "bf16")
    buf = binding.NobleLinearBuffers(T, di, do, r, "bf16")

    def step():
        binding.forward(buf, dev["x"], dev)
        binding.backward(buf, dev["x"], dev["dy"], dev)

    step()
    torch.cuda.synchronize()
    want = [t.clone() for t in (buf.y, buf.dx, buf.bucket)]
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        step()
    for _ in range(3):
        buf.dx.fill_(float("nan"))
        buf.grads["dW"].fill_(float("nan"))
        graph.replay()
        graph.replay()
        torch.cuda.synchronize()
        assert all(torch.equal(a, b) for a, b in zip((buf.y, buf.dx, buf.bucket), want))
    binding.noble_get_device_status(None)
