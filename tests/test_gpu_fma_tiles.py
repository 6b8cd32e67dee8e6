"""The fp32-FMA grouped GEMMs at the edges of their tiles: reductions below, at and beyond one, two and three pieces of 128
or 256, ragged column and row tiles, both tile sizes, empty experts, fp32 layers and bf16 ones without packed weights
(GPU required)."""
import pytest

import dsmoe_inputs as gi
from harness import TOL_BF16, TOL_F32, layer_parity

pytestmark = pytest.mark.gpu

# few rows: 32 x 32 tiles; many: 64 x 64
SHAPES = [(1, 8, 8, 1, 1), (33, 264, 72, 5, 2), (64, 256, 512, 8, 2), (31, 520, 136, 40, 3), (129, 776, 40, 64, 1),
          (700, 136, 264, 16, 3), (1025, 392, 200, 8, 8), (640, 128, 1032, 33, 2)]


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("shape", SHAPES, ids=["x".join(map(str, s)) for s in SHAPES])
def test_edges_of_the_fma_tiles(shape, dtype):
    T, d, H, E, K = shape
    s = gi.LayerSpec("fma" + "x".join(map(str, shape)), T=T, d=d, H=H, E=E, dtype=dtype, mode=gi.MODE_TOPK, K=K, router_gain=4.0)
    r = layer_parity(s, pack=False)
    tol = TOL_F32 if dtype == "f32" else TOL_BF16
    assert r["err_rows"] <= tol, (r["err_rows"], r["err"])
