"""Steps of up to 16 rows run the block in one persistent kernel: against the oracle at its batch edges, and against
the launch-per-stage path (which profiled steps keep) over the forms it accepts."""
import numpy as np
import pytest

from paper_2609_15160_gb300 import synth

from _parity import rel_err
from test_gpu_parity import _prefill_decode_compare, _small, tlf  # noqa: F401  (fixture)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("batch", [1, 8, 9, 16, 17])
def test_batch_edges_match_oracle(tlf, batch):  # noqa: F811
    m = _small(d_model=192, n_heads=4, n_kv_heads=4, ffn_hidden=176, max_loops=3, depth_probs=(0.4, 0.3, 0.3))
    _prefill_decode_compare(tlf, m, [1 + (37 * b) % 130 for b in range(batch)], steps=3)


SHAPES = [dict(head_dim=32, n_heads=4, n_kv_heads=2), dict(head_dim=32, n_heads=4, n_kv_heads=4),
          dict(head_dim=64, n_heads=4, n_kv_heads=4), dict(head_dim=64, n_heads=8, n_kv_heads=2),
          dict(head_dim=128, n_heads=2, n_kv_heads=2), dict(head_dim=128, n_heads=4, n_kv_heads=2),
          dict(head_dim=128, n_heads=4, n_kv_heads=1), dict(conditioning=True), dict(exit_rule="survival"),
          dict(router_hidden=64, depth_probs=None), dict(ffn_hidden=1376, d_model=512, n_layers=3)]


@pytest.mark.parametrize("shape", SHAPES, ids=lambda s: "-".join(f"{k}{v}" for k, v in s.items()))
def test_matches_the_launch_per_stage_path(tlf, shape):  # noqa: F811
    """The same steps on two contexts: logits within the rounding of one bf16 operand plane pair, loop counts equal,
    every appended K/V row within one bf16 rounding of the other's."""
    m = _small(**{**dict(max_loops=4), **shape})
    w = synth.make_weights(m)
    lens = [1, 64, 200, 65, 700]
    rng = np.random.default_rng(3)
    ids = list(range(len(lens)))
    with tlf.Context(m, w, max_seqs=5, max_batch=5, max_seq_len=800) as a, \
            tlf.Context(m, w, max_seqs=5, max_batch=5, max_seq_len=800) as b:
        b.set_profiling(True)
        for i, n in zip(ids, lens):
            snap = synth.make_cache_snapshot(m, n, seed=11 + i)
            a.load_cache(i, snap)
            b.load_cache(i, snap)
        for _ in range(3):
            toks = rng.integers(0, m.vocab, size=len(ids)).astype(np.int32)
            la, ma, _ = a.decode_step(ids, toks)
            lb, mb, _ = b.decode_step(ids, toks)
            np.testing.assert_array_equal(ma, mb)
            # both paths keep 16-bit-significant operands (2^-17 relative each, a few dozen of them) and bf16 caches
            assert rel_err(la, lb) < 2e-3
        for i in ids:
            for r in range(1, m.max_loops + 1):
                for j in range(m.n_layers):
                    pa, ka, va = a.read_cache(i, r, j)
                    pb, kb, vb = b.read_cache(i, r, j)
                    np.testing.assert_array_equal(pa, pb)
                    for x, y in ((ka, kb), (va, vb)):
                        if x.size:
                            assert np.max(np.abs(x - y)) <= 2 ** -7 * np.max(np.abs(y))
