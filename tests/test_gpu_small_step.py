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


SMALL_LAUNCHES = 6  # router, plan, first norm, block, final norm, LM head


def _pair(tlf, m, snaps, steps=3):  # noqa: F811
    """The same steps on a context that takes the persistent kernel and on one that launches every stage (profiled): the
    contexts' caches after `steps` steps, with loop counts equal and logits within the rounding of the bf16 operand
    planes and caches."""
    w = synth.make_weights(m)
    n = len(snaps)
    ids = list(range(n))
    room = max(len(s["positions"][0]) for s in snaps) + steps + 1
    rng = np.random.default_rng(3)
    with tlf.Context(m, w, max_seqs=n, max_batch=n, max_seq_len=room) as a, \
            tlf.Context(m, w, max_seqs=n, max_batch=n, max_seq_len=room) as b:
        b.set_profiling(True)
        for i, snap in zip(ids, snaps):
            a.load_cache(i, snap)
            b.load_cache(i, snap)
        for _ in range(steps):
            toks = rng.integers(0, m.vocab, size=n).astype(np.int32)
            la, ma, _ = a.decode_step(ids, toks)
            lb, mb, _ = b.decode_step(ids, toks)
            assert a.last_step_profile()[2] == SMALL_LAUNCHES
            assert b.last_step_profile()[2] == 5 + 5 * m.n_layers * m.max_loops
            np.testing.assert_array_equal(ma, mb)
            # both paths keep 16-bit-significant operands (2^-17 relative each, a few dozen of them) and bf16 caches
            assert rel_err(la, lb) < 2e-3
        for i, snap in zip(ids, snaps):
            for r in range(1, m.max_loops + 1):
                old = len(snap["positions"][r - 1])
                for j in range(m.n_layers):
                    pa, ka, va = a.read_cache(i, r, j)
                    pb, kb, vb = b.read_cache(i, r, j)
                    np.testing.assert_array_equal(pa, pb)
                    for x, y in ((ka, kb), (va, vb)):
                        np.testing.assert_array_equal(x[:old], y[:old])  # restored
                        x, y = x[old:], y[old:]
                        if x.size:
                            # appended: the entry's own bf16 rounding (2^-7 of it at most), and what such roundings of
                            # entries before it bring through the attention (2^-8 of the largest)
                            assert (np.abs(x - y) <= 2 ** -7 * np.abs(y) + 2 ** -8 * np.max(np.abs(y))).all()


@pytest.mark.parametrize("shape", SHAPES, ids=lambda s: "-".join(f"{k}{v}" for k, v in s.items()))
def test_matches_the_launch_per_stage_path(tlf, shape):  # noqa: F811
    m = _small(**{**dict(max_loops=4), **shape})
    _pair(tlf, m, [synth.make_cache_snapshot(m, n, seed=11 + i) for i, n in enumerate([1, 64, 200, 65, 700])])


@pytest.mark.parametrize("rows", [1, 8, 9, 16])
def test_long_reductions(tlf, rows):  # noqa: F811
    """Down projections over more K steps than one batch of the token operand holds (3072 for up to 8 rows, 1536 above)."""
    m = _small(ffn_hidden=3248, max_loops=2, depth_probs=(0.5, 0.5))
    _pair(tlf, m, [synth.make_cache_snapshot(m, 3 + 5 * i, seed=i) for i in range(rows)], steps=2)


@pytest.mark.parametrize("rows,keys", [(16, 2600), (4, 20000), (1, 33000)])
def test_many_pages_a_group(tlf, rows, keys):  # noqa: F811
    """More than 32 pages for a group of warps: the ring's refills go past the page list that a warp holds at once, and
    items lie over several groups (16 kv heads, 304 groups: 34, 65 and 28 pages of the first loop each)."""
    m = _small(head_dim=32, n_heads=16, n_kv_heads=16, n_layers=1, max_loops=2, depth_probs=(0.3, 0.7))
    _pair(tlf, m, [synth.make_cache_positions(m, keys - i, seed=i) for i in range(rows)], steps=2)


def test_contexts_step_at_the_same_time(tlf):  # noqa: F811
    """Two threads, each with a context and a stream of its own, step at once: one through the persistent kernel, which
    needs every SM, one through it or through the launches. Every step gives what it gives alone."""
    import threading

    import torch
    m = _small()
    w = synth.make_weights(m)
    steps = 60

    def run(rows, stream, out):
        toks = np.random.default_rng(rows).integers(0, m.vocab, size=(steps, rows)).astype(np.int32)
        with tlf.Context(m, w, max_seqs=rows, max_batch=rows, max_seq_len=700) as ctx:
            for i in range(rows):
                ctx.load_cache(i, synth.make_cache_snapshot(m, 30 + 29 * (i % 20), seed=i))
            for t in toks:
                out.append(ctx.decode_step(list(range(rows)), t, stream=stream)[0].copy())

    for pair in ((4, 16), (4, 40)):
        alone, both = [[], []], [[], []]
        for rows, out in zip(pair, alone):
            run(rows, None, out)
        streams = [torch.cuda.Stream() for _ in pair]
        threads = [threading.Thread(target=run, args=(rows, s.cuda_stream, out)) for rows, s, out in zip(pair, streams, both)]
        for t in threads:
            t.start()
        for t in threads:
            t.join()
        for a, b in zip(alone, both):
            assert len(b) == steps
            np.testing.assert_array_equal(np.stack(a), np.stack(b))
