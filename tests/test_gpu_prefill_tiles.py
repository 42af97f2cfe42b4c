"""Prefill kernels at the edges of their tiles, against the float64 oracle (bf16 tolerance of the parity tests)."""
import numpy as np
import pytest

from oracle import tlf_oracle as O
from paper_2609_15160_gb300 import synth

from _parity import DepthOracle, check_cache, rel_err, tol_for
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


@pytest.mark.parametrize("shape", SHAPES, ids=str)
@pytest.mark.parametrize("n", [1, 16, 17, 32, 33, 64, 65, 128, 129, 256])
def test_few_row_projections(tlf, shape, n):  # noqa: F811
    """A chunk of up to 256 rows: every token tile at its first and last size, with the CTA sizes that go with it."""
    _prefill_decode_compare(tlf, _small(**SHAPES[shape]), [n], steps=1)


@pytest.mark.parametrize("n", [1, 17, 128, 129, 256, 300])
def test_more_weight_tiles_than_sms(tlf, n):  # noqa: F811
    """A gate/up projection of 154 tiles of 128 features, with few rows and just above."""
    _prefill_decode_compare(tlf, _small(ffn_hidden=9808, n_layers=1, max_loops=2, depth_probs=(0.5, 0.5)), [n], steps=1)


@pytest.mark.parametrize("rows", [33, 64, 65, 128])
def test_long_k_projections(tlf, rows):  # noqa: F811
    """Projections with eight k-tiles a CTA and more (78 gate/up tiles over 8 k-tiles, 78 k-tiles down): two CTAs share an
    SM, in the prompts' chunk and in the decode step."""
    m = _small(d_model=512, ffn_hidden=4992, n_layers=1, max_loops=2, depth_probs=(0.5, 0.5))
    _prefill_decode_compare(tlf, m, [1] * rows, steps=1)


@pytest.mark.parametrize("d,n,cond", [(1024, 200, False), (1024, 200, True), (1088, 32, False), (1088, 33, False),
                                      (192, 255, True)])
def test_split_norms_of_short_prompts(tlf, d, n, cond):  # noqa: F811
    """Pre-norms split between the projections of a one-tile loop, on both sides of the rule, with and without
    conditioning, over more loops and layers than one; feature tiles that end inside 128."""
    m = _small(d_model=d, n_layers=3, max_loops=2, depth_probs=(0.5, 0.5), conditioning=cond)
    _prefill_decode_compare(tlf, m, [n], steps=1)


@pytest.mark.parametrize("hd,heads,kv", [(64, 4, 4), (64, 4, 2), (64, 4, 1), (128, 2, 2), (128, 4, 2), (128, 4, 1)])
def test_pair_attention_blocks(tlf, hd, heads, kv):  # noqa: F811
    """The two-tile prefill attention around its 128-slot key blocks and query tiles, in one chunk and in chunks whose
    queries start inside a key block: last-token logits and every cached K/V row against the oracle."""
    m = _small(n_heads=heads, n_kv_heads=kv, head_dim=hd, d_model=128, max_loops=2, depth_probs=(0.4, 0.6))
    w = synth.make_weights(m)
    om = O.OracleModel.from_config(m, w)
    depth = DepthOracle(om)
    rng = np.random.default_rng(hd + kv)
    lens = [1, 127, 129, 257, 400, 640]
    prompts = [rng.integers(0, m.vocab, size=n).astype(np.int32) for n in lens]
    forced = [depth.forced_for(p) for p in prompts]
    seqs = [O.OracleSequence(om) for _ in prompts]
    want = [O.prefill_gathered(om, s, p, forced=f) for s, p, f in zip(seqs, prompts, forced)]
    ids = list(range(1, 1 + len(lens)))
    for chunk in (8192, 256):
        with tlf.Context(m, w, max_seqs=len(lens), max_batch=len(lens), max_seq_len=700, prefill_chunk=chunk) as ctx:
            lg, loops = ctx.prefill(ids, prompts, forced=forced)
            for b, (olog, oloops) in enumerate(want):
                np.testing.assert_array_equal(loops[b], oloops)
                assert rel_err(lg[b], olog) < tol_for(m), (chunk, lens[b])
                check_cache(ctx, ids[b], seqs[b], m)


@pytest.mark.parametrize("hd,heads,kv", [(64, 4, 4), (64, 4, 1), (128, 4, 2)])
@pytest.mark.parametrize("chunk", [8192, 256])
def test_entries_of_released_pages_do_not_reach_a_prompt(tlf, hd, heads, kv, chunk):  # noqa: F811
    """Prompts on pages that held infinities before: the slots behind a prompt's last token are masked, and what they
    hold must not reach its result, bit for bit (0 x infinity is NaN)."""
    m = _small(n_heads=heads, n_kv_heads=kv, head_dim=hd, d_model=128, max_loops=2, depth_probs=(0.4, 0.6))
    w = synth.make_weights(m)
    rng = np.random.default_rng(hd + kv)
    lens = [1, 15, 66, 127, 130, 257, 390]
    prompts = [rng.integers(0, m.vocab, size=n).astype(np.int32) for n in lens]
    ids = list(range(1, 1 + len(lens)))
    pages = 2 * sum((n + 63) // 64 + 1 for n in lens)
    got = []
    for dirty in (False, True):
        with tlf.Context(m, w, max_seqs=8, max_batch=8, max_seq_len=64 * pages, kv_pool_pages=pages, prefill_chunk=chunk) as ctx:
            if dirty:
                n = 64 * (pages // 2) - 1  # every page of the pool
                bad = np.full((n, m.n_layers, kv, hd), np.inf, np.float32)
                ctx.load_cache(99, {"positions": [np.arange(n, dtype=np.int32)] * 2, "k": [bad] * 2, "v": [bad] * 2})
                assert ctx.stats()[1] == 0
                ctx.release(99)
            lg, _ = ctx.prefill(ids, prompts)
            assert np.isfinite(lg).all()
            got.append(lg)
    np.testing.assert_array_equal(got[0], got[1])
