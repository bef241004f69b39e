"""The backward's grouped launch: products of different majorness and output
type as tiles of one launch, handed out by a counter; a K range accumulated in
pieces that are added up in C; token counts that are no multiple of 8 (the last
8-row group in boxes of its own).  Token-summed products and dx against fp64
products of the same bf16 values on the device, and repeats bit for bit."""
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


SHAPES = [
    (4200, 2048, 2048, 64),   # two pieces per tile, no split
    (8193, 1024, 1024, 64),   # pieces and a split; one row past the last whole 8-row group
    (8191, 1024, 1032, 128),  # d_out does not tile by 64: the 2-D layout beside the 4-D one
    (8195, 256, 320, 0),      # no branch: dbias from the ones column, eight K ranges of one piece
    (8195, 1024, 1024, 0),    # ... four ranges of two pieces: added up in column 0
    (32771, 512, 512, 0),     # ... thirteen of two, the last of one
    (131, 768, 2304, 32),     # tiles heavier than the mean: halved
    (7, 64, 64, 16),          # one 8-row group, incomplete
    (65, 64, 128, 256),       # the last k-block holds one row
    (8192, 4096, 4096, 64),   # a K range longer than L2: not started beside the bottleneck kernel
]


@pytest.mark.parametrize("shape", SHAPES, ids=lambda s: "x".join(map(str, s)))
def test_bwd_group(shape):
    import torch
    T, di, do, r = shape
    dev = binding.params_to_device(make_layer_inputs(Layer("group", *shape, "bf16"), 70 + T), "bf16")
    buf = binding.NobleLinearBuffers(T, di, do, r, "bf16")
    binding.forward(buf, dev["x"], dev)
    buf.bucket.fill_(float("nan"))
    buf.workspace.fill_(255)
    binding.backward(buf, dev["x"], dev["dy"], dev)
    torch.cuda.synchronize()
    binding.noble_get_device_status(None)
    got = {k: v.clone() for k, v in buf.grads.items()}
    dx = buf.dx.clone()
    x, dy = dev["x"].double(), dev["dy"].double()
    ref = {"dW": dy.T @ x, "dbias": dy.sum(0)}
    if r:
        c = buf.saved[-((T * r * 2 + 255) // 256 * 256):][:T * r * 2].view(torch.bfloat16).view(T, r).double()
        dh = buf.workspace[:T * r * 2].view(torch.bfloat16).view(T, r).double()
        ref["dW_up"] = dy.T @ c
        ref["dW_down"] = dh.T @ x
        dx_ref = dy @ dev["W"].double() + dh @ dev["W_down"].double()
    else:
        dx_ref = dy @ dev["W"].double()
    for k, v in ref.items():
        # fp32 accumulation of T products: a few 2^-24 sqrt(T) of the result's scale
        err = (got[k].double() - v).abs().max() / v.abs().max()
        assert err <= 2e-5, (k, float(err))
    err = (dx.double() - dx_ref).abs().max() / dx_ref.abs().max()
    assert err <= 2.0**-8, float(err)  # one bf16 rounding
    binding.backward(buf, dev["x"], dev["dy"], dev)
    torch.cuda.synchronize()
    assert torch.equal(buf.dx, dx) and all(torch.equal(buf.grads[k], got[k]) for k in got)
