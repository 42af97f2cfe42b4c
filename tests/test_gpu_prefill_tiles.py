"""Prefill kernels at the edges of their tiles, against the float64 oracle (bf16 tolerance of the parity tests)."""
import pytest

from test_gpu_parity import _prefill_decode_compare, _small, tlf  # noqa: F401  (fixture)

pytestmark = pytest.mark.gpu

# heads, kv heads, head_dim, d_model, ffn_hidden (160 and 176 end inside a 64-feature gate/up group)
SHAPES = {
    "hd32-g2": dict(n_heads=4, n_kv_heads=2, head_dim=32, d_model=128, ffn_hidden=160),
    "hd64-g1": dict(n_heads=4, n_kv_heads=4, head_dim=64, d_model=192, ffn_hidden=176),
    "hd128-g4": dict(n_heads=4, n_kv_heads=1, head_dim=128, d_model=320, ffn_hidden=416),
}


@pytest.mark.parametrize("shape", SHAPES, ids=str)
@pytest.mark.parametrize("lens", [[257], [255, 2, 300], [512, 129]], ids=str)
def test_many_row_projections(tlf, shape, lens):  # noqa: F811
    """Chunks of more than 256 rows: the pair GEMM at full, partial and one-row tiles of every loop."""
    _prefill_decode_compare(tlf, _small(**SHAPES[shape]), lens, steps=1)


def test_many_row_projections_conditioned(tlf):  # noqa: F811
    _prefill_decode_compare(tlf, _small(conditioning=True, d_model=192), [300, 90], steps=1)
