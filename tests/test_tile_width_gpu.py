"""The forward's tile width (128 or 256 columns per CTA pair, by token count and
weight size) changes no result: the rows of a call equal, bit for bit, those of
a longer call on the other side of the rule, and both the product."""
import pytest

from paper_2603_06492_gb300 import binding

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def lib():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    from paper_2603_06492_gb300.build import build
    build()
    binding.load()


# x of less than 128 KB and of 128 KB; the bottleneck split over CTAs and not;
# the smallest call
@pytest.mark.parametrize("T,T2,sigma", [(15, 16, "cosnet"), (15, 16, "tanh1"), (1, 16, "tanh1")])
def test_rows_do_not_depend_on_the_tile_width(T, T2, sigma):
    import torch
    di, do, r = 4096, 8192, 64
    g = torch.Generator(device="cuda").manual_seed(T + T2)
    n = lambda *s: torch.randn(s, generator=g, device="cuda")  # noqa: E731
    p = {"W": (n(do, di) / 64).bfloat16(), "bias": n(do), "W_down": (n(r, di) / 64).bfloat16(),
         "W_up": (n(do, r) / 8).bfloat16(), "M": n(r, r) / 8}
    for k in ("omega1", "phi1", "omega2", "phi2"):
        p[k] = n(r)
    x = n(T2, di).bfloat16()
    flags = binding.SIGMA_FLAGS[sigma] | binding.NOBLE_FLAG_INFERENCE
    y = []
    for t in (T, T2):
        buf = binding.NobleLinearBuffers(t, di, do, r, "bf16", with_grads=False, flags=flags)
        buf.y.fill_(float("nan"))
        y.append(binding.forward(buf, x[:t].contiguous(), p))
    torch.cuda.synchronize()
    binding.noble_get_device_status(None)
    assert torch.equal(y[0], y[1][:T])
    h = x.double() @ p["W_down"].double().T
    q = {k: v.double() for k, v in p.items()}
    c = (torch.cos(q["omega2"] * (torch.cos(q["omega1"] * h + q["phi1"]) @ q["M"]) + q["phi2"])
         if sigma == "cosnet" else torch.tanh(h))
    ref = x.double() @ q["W"].T + c @ q["W_up"].T + q["bias"]
    assert (y[1].double() - ref).abs().max() <= 1e-2 * ref.abs().max()
