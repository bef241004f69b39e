"""Length of the running fp32 sums of the CUDA-core path: dM (and dM2) over many
like tokens, where every rounding error of a long sum has the same sign."""
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


# one chunk of 1024 tokens, one token past it, many
@pytest.mark.parametrize("T", [1024, 1025, 65536])
@pytest.mark.parametrize("three", [False, True])
def test_dm_of_like_tokens(T, three):
    import torch
    di, do, r = 64, 64, 16
    g = torch.Generator(device="cuda").manual_seed(3)
    u = lambda lo, hi, *s: torch.rand(*s, generator=g, device="cuda") * (hi - lo) + lo  # noqa: E731
    # h = 0, so a and the chain rule are the same for every token
    p = {"W": u(-1, 1, do, di), "W_down": torch.zeros((r, di), device="cuda"), "W_up": u(0.5, 1.5, do, r),
         "M": u(-0.5, 0.5, r, r), "M2": u(-0.5, 0.5, r, r)}
    for i in (1, 2, 3):
        p[f"omega{i}"], p[f"phi{i}"] = u(0.5, 1.5, r), u(-3, 3, r)
    x, dy = u(-1, 1, T, di), u(0, 1, 1, do).expand(T, do).contiguous()
    buf = binding.NobleLinearBuffers(T, di, do, r, "fp32", flags=binding.NOBLE_FLAG_SIGMA_COS3 if three else 0)
    binding.forward(buf, x, p)
    binding.backward(buf, x, dy, p)
    torch.cuda.synchronize()
    q = {k: v.double() for k, v in p.items()}
    a = torch.cos(q["phi1"])
    b = a @ q["M"]
    d, want = dy[0].double() @ q["W_up"], {}
    if three:
        a2 = torch.cos(q["omega2"] * b + q["phi2"])
        db2 = -q["omega3"] * torch.sin(q["omega3"] * (a2 @ q["M2"]) + q["phi3"]) * d
        want["dM2"] = T * torch.outer(a2, db2)
        d = db2 @ q["M2"].T
    want["dM"] = T * torch.outer(a, -q["omega2"] * torch.sin(q["omega2"] * b + q["phi2"]) * d)
    # sums of at most 1024 tokens and of the T / 1024 partials (half an ulp each),
    # 64 2^-24 for the terms themselves
    bound = (1024 + T / 1024 + 64) * 2.0**-24
    for k, v in want.items():
        err = (buf.grads[k].double() - v).abs().max() / v.abs().max()
        assert err <= bound, (k, float(err), bound)
