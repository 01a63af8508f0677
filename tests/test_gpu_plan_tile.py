"""The tile that a plan reports is the one that its whole products run."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


# few 256 x 256 tiles run as 128 x 128 ones (at most a quarter of the SMs, 3xTF32 at most 16): 1, 25 and 28 tiles; 64, 49 and 25 do not
@pytest.mark.parametrize("dtype,n,d,tile", [("F32_SPLIT_BF16", 256, 0, 128), ("F32_SPLIT_FP16", 1280, 0, 128),
                                            ("F32_SPLIT_BF16", 1024, 1, 128), ("F32_SPLIT_TF32", 1024, 0, 128),
                                            ("F32_SPLIT_BF16", 2048, 0, 256), ("F32_SPLIT_BF16", 1792, 0, 256),
                                            ("F32_SPLIT_TF32", 1280, 0, 256), ("F32_SPLIT_BF16", 384, 0, 128)])
def test_reported_tile(stark_lib, dtype, n, d, tile):
    S = stark_lib
    with S.Plan(n, d, S.DType[dtype]) as p:
        assert p.tile == (128, tile)
