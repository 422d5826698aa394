"""Sizes at the edges of the kernels' own tiles, against the fp64 oracle through the C ABI (one B200)."""
import pytest

from paper_2608_06838_b200 import inputs
from paper_2608_06838_b200.inputs import Workload

from helpers import compare, oracle_reference, run_chain, tolerance

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


# The CUDA-core kernels walk a block in tiles of 64 tokens whatever the chunk: blocks shorter than a tile (3 chunks of 16),
# of one tile and a remainder (5 of 16, 3 of 32), of whole tiles; segments that end one token before, at and after a tile.
@pytest.mark.parametrize("chunk,cpb", [(16, 3), (16, 5), (32, 3), (64, 2), (64, 0)])
@pytest.mark.parametrize("dk,dv,dtype", [(32, 32, "f32"), (32, 64, "bf16"), (64, 64, "f32"), (64, 64, "bf16"), (128, 128, "f32")])
def test_cuda_core_tiles_and_blocks(dk, dv, dtype, chunk, cpb):
    w = Workload("tiles-%d-%d-%s-%d-%d" % (dk, dv, dtype, chunk, cpb), 2, 2, dk, dv, [129, 64, 63, 65, 1], chunk, dtype=dtype,
                 g_scale=0.1, s_in_sigma=0.3, ds_out_sigma=0.3, seed=61)
    x = inputs.make_inputs(w, DEV)
    got, _ = run_chain(w, x, chunks_per_block=cpb)
    compare(got, oracle_reference(x), tolerance(w), label=w.name)
