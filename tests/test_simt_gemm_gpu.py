"""The CUDA-core path's grouped products at the edges of their tiles (64 x 64,
k-tiles of 32), of the K ranges of a cluster and of the column-sum chunks
(128 rows), against the fp64 oracle."""
import numpy as np
import pytest

from paper_2603_06492_gb300 import binding
from paper_2603_06492_gb300.inputs import Layer, make_layer_inputs
from tests.gpu_helpers import assert_close, run_gpu, run_oracle

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def lib():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    from paper_2603_06492_gb300.build import build
    build()
    binding.load()


EDGES = [
    (1, 8, 8, 16),        # one row, one group of columns, K below one k-tile
    (64, 64, 64, 64),     # exact tiles
    (65, 72, 136, 16),    # one past a tile in every dimension
    (129, 1000, 56, 32),  # K in eight ranges, the last one shorter; a second colsum chunk of one row
    (40, 264, 2056, 128),  # ranges of 33 k-tiles over eight CTAs: the last CTAs have none of segment 0
    (1030, 512, 640, 64),  # more tiles than fit at once: no split
    (257, 136, 72, 0),    # no branch
]


@pytest.mark.parametrize("shape", EDGES, ids=lambda s: "x".join(map(str, s)))
@pytest.mark.parametrize("dtype", ["fp32", "bf16"])
def test_simt_edges(shape, dtype):
    layer = Layer("simt", *shape, dtype)
    inp = make_layer_inputs(layer, 31 + sum(shape), init="strong_branch")
    flags = binding.NOBLE_FLAG_SIMT_ONLY if dtype == "bf16" else 0
    got = run_gpu(layer, inp, flags=flags)
    assert_close(got, run_oracle(layer, inp), dtype, ctx=f"{shape} {dtype}")
    again = run_gpu(layer, inp, flags=flags)
    assert all(np.array_equal(got[k], again[k]) for k in got)  # fixed order of every sum
