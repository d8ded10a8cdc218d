"""The products that read the heads' tensors contract in half heads at D = 64 (tc_gemm.cu): mixer layer and
gradients against the oracle with several heads and tensors side by side, row tiles in pairs (the last
one short) and one at a time. Tolerance as in test_mixer_tiles_gpu.py."""
import pytest

from test_mixer_tiles_gpu import test_projection_tiles_match_oracle as check

pytestmark = pytest.mark.gpu

SHAPES = [  # B, H, N, M, D, P
    (1, 2, 304 * 128 + 3, 16, 64, 4),  # 305 row tiles: pairs, the last of one tile of three rows
    (2, 6, 200, 16, 64, 2),            # C = 384: three column tiles, row tiles one at a time
]


@pytest.mark.parametrize("shape", SHAPES, ids=[str(s) for s in SHAPES])
def test_half_head_slices_match_oracle(shape):
    check(shape)
