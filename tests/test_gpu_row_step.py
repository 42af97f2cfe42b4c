"""Small float32 models run a step's block one CTA per row: against the oracle around its edges, and against the
launch-per-stage path (which profiled steps keep), with as many launches as each of them has."""
import numpy as np
import pytest

from paper_2609_15160_gb300 import synth

from _parity import rel_err
from test_gpu_parity import _prefill_decode_compare, _small, tlf  # noqa: F401  (fixture)

pytestmark = pytest.mark.gpu

SHAPES = [dict(d_model=64, n_heads=4, n_kv_heads=4, head_dim=16, n_layers=1, ffn_hidden=176),
          dict(d_model=64, n_heads=2, n_kv_heads=1, head_dim=32, n_layers=2, ffn_hidden=80),
          dict(d_model=128, n_heads=2, n_kv_heads=2, head_dim=64, n_layers=1, ffn_hidden=160),
          dict(d_model=192, n_heads=2, n_kv_heads=1, head_dim=128, n_layers=1, ffn_hidden=112),
          dict(d_model=64, n_heads=4, n_kv_heads=2, head_dim=16, n_layers=2, ffn_hidden=48, conditioning=True)]


@pytest.mark.parametrize("shape", SHAPES, ids=lambda s: f"d{s['d_model']}-hd{s['head_dim']}-J{s['n_layers']}")
@pytest.mark.parametrize("lens", [[1], [63, 64, 65, 130]], ids=str)
def test_row_steps_match_oracle(tlf, shape, lens):  # noqa: F811
    _prefill_decode_compare(tlf, _small("f32", **shape), lens, steps=2)


def test_more_rows_than_sms(tlf):  # noqa: F811
    """One CTA per row in more than one wave."""
    _prefill_decode_compare(tlf, _small("f32", **SHAPES[0]), [1 + b % 3 for b in range(170)], steps=1)


def test_long_caches_leave_the_row_kernel(tlf):  # noqa: F811
    """Steps across the longest cache that the row kernel takes (1024 entries) agree with profiled ones."""
    m = _small("f32", **SHAPES[0])
    w = synth.make_weights(m)
    rng = np.random.default_rng(5)
    with tlf.Context(m, w, max_seqs=2, max_batch=2, max_seq_len=1100) as a, \
            tlf.Context(m, w, max_seqs=2, max_batch=2, max_seq_len=1100) as b:
        b.set_profiling(True)
        for i, n in ((0, 1021), (1, 7)):
            snap = synth.make_cache_snapshot(m, n, seed=3 + i)
            a.load_cache(i, snap)
            b.load_cache(i, snap)
        for step in range(6):
            toks = rng.integers(0, m.vocab, size=2).astype(np.int32)
            la, ma, _ = a.decode_step([0, 1], toks)
            lb, mb, _ = b.decode_step([0, 1], toks)
            np.testing.assert_array_equal(ma, mb)
            by_rows = a.last_step_profile()[2] == 4  # router, plan, block, LM head
            assert by_rows == (1021 + step + 1 <= 1024)
            assert rel_err(la, lb) < 1e-5  # float32 sums in another order
