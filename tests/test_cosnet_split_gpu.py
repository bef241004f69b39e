"""The bottleneck kernels on clusters of four CTAs per token tile (few tiles,
long K) against the fp64 oracle: token counts that leave lane quarters empty,
k-block counts that do not divide by four, every rank, and the last shapes on
either side of the rule."""
import numpy as np
import pytest

from paper_2603_06492_gb300 import binding
from paper_2603_06492_gb300.inputs import Layer, make_cos3_inputs, make_layer_inputs
from tests.gpu_helpers import assert_close, run_gpu, run_oracle
from tests.test_cos3_gpu import oracle_cos3, run_cos3

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
    (1, 2048, 2048, 16),     # one row: three CTAs without rows
    (33, 2056, 2072, 32),    # two quarters live; 33 k-blocks, the last one partial
    (97, 2304, 2176, 64),    # 36 and 34 k-blocks; the last quarter holds one row
    (385, 2048, 2240, 128),  # four tiles, the last of one row
    (513, 2048, 2048, 64),   # five: the forward does not split, the backward does
    (1664, 256, 2048, 32),   # backward: thirteen tiles split, 32 k-blocks
    (1665, 256, 2048, 32),   # ... fourteen do not
    (1600, 256, 1984, 32),   # ... nor thirteen with 31 k-blocks
    (512, 1984, 256, 64),    # forward: 31 k-blocks do not
]


@pytest.mark.parametrize("shape", SHAPES, ids=lambda s: "x".join(map(str, s)))
def test_split_tiles(shape):
    layer = Layer("split", *shape, "bf16")
    inp = make_layer_inputs(layer, 90 + sum(shape), init="strong_branch")
    got = run_gpu(layer, inp)
    assert_close(got, run_oracle(layer, inp), "bf16", ctx=str(shape))
    again = run_gpu(layer, inp)
    assert all(np.array_equal(got[k], again[k]) for k in got)


@pytest.mark.parametrize("shape", [(70, 2048, 2048, 32), (200, 2112, 2048, 128)], ids=lambda s: "x".join(map(str, s)))
def test_split_tiles_cos3(shape):
    layer = Layer("split3", *shape, "bf16")
    inp = dict(make_layer_inputs(layer, 95 + sum(shape), init="strong_branch"), **make_cos3_inputs(shape[3], 5))
    assert_close(run_cos3(layer, inp), oracle_cos3(inp), "bf16", ctx=str(shape))
