"""Decode attention with one query head a kv head: items merged behind the consumers' backs, at the edges of the split."""
import numpy as np
import pytest

from oracle import tlf_oracle as O

from _attn_problem import args_for, gather_kv, make_problem, out_to_host, to_device
from test_gpu_attn_op import T  # noqa: F401  (fixture)

pytestmark = pytest.mark.gpu

LENS = {
    "one-page": [1, 64, 63, 2] * 64,                    # many items a CTA, each of one page
    "short": [65, 128, 129, 700, 30] * 40,              # items that cross CTAs between whole ones
    "long-first": [9000] + [1, 65] * 60,                # one item over many CTAs, then short ones
    "few": [5, 200],                                    # fewer pages than CTAs
}


@pytest.mark.parametrize("heads,hd,dtype", [(16, 64, "bf16"), (8, 128, "bf16"), (4, 32, "bf16"), (4, 16, "f32"),
                                            (4, 128, "f32")])
@pytest.mark.parametrize("lens", LENS.values(), ids=LENS.keys())
def test_items_of_a_cta(T, lens, heads, hd, dtype):  # noqa: F811
    import torch
    p = make_problem(len(lens), lens, heads, heads, hd, dtype=dtype, seed=hd)
    d = to_device(p)
    a = args_for(T, p, d)
    nbytes = T.tlf_attn_decode_scratch_bytes(a)
    scratch = torch.empty(nbytes, dtype=torch.uint8, device="cuda")
    tol = 1e-4 if dtype == "f32" else 2e-2
    want = [O.attention(p["q"][b].astype(np.float64), *gather_kv(p, b)) for b in range(p["n"])]
    first = None
    for _ in range(2):  # the tickets are back at zero for the second launch
        T.tlf_attn_decode(a, scratch, nbytes)
        torch.cuda.synchronize()
        assert int(d["err"][0].item()) == 0
        got = out_to_host(p, d["out"])
        for b in range(p["n"]):
            assert np.max(np.abs(got[b] - want[b])) < tol * np.max(np.abs(want[b])), b
        first = got if first is None else first
        np.testing.assert_array_equal(got, first)


@pytest.mark.parametrize("hd", [64, 128])
def test_items_of_a_masked_cta(hd):
    """Full-length caches (the dense-cache ablation) with more items a CTA than merge buffers: 250 rows of a page each over
    8 kv heads leave a CTA seven."""
    from paper_2609_15160_gb300 import build, tlf
    from test_gpu_parity import _prefill_decode_compare, _small
    build.build()
    m = _small(n_heads=8, n_kv_heads=8, head_dim=hd, n_layers=1, max_loops=2, depth_probs=(0.5, 0.5))
    _prefill_decode_compare(tlf, m, [1 + b % 3 for b in range(250)], steps=2, ablation="dense_cache")
