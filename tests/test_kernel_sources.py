"""CPU checks on the kernels' sources, for orders that a run cannot be trusted to show wrong."""
import os
import re

import pytest

from paper_2609_15160_gb300 import build


def _kernels():
    """(name, body) of every __global__ function of the library."""
    for src in build.SOURCES:
        text = re.sub(r"//[^\n]*", "", open(os.path.join(build.CSRC, src)).read())
        for part in text.split("__global__")[1:]:
            body = part[:part.index("\n}\n")]
            yield re.search(r"\b(k_\w+)\s*\(", body).group(1), body


TMEM_KERNELS = {name: body for name, body in _kernels() if "tmem_alloc" in body}


def test_the_kernels_with_tensor_memory_are_found():
    assert {"k_gemm_tc", "k_gemm_pf", "k_pf_attn_tc", "k_pf_attn_pair"} <= set(TMEM_KERNELS)


@pytest.mark.parametrize("name", sorted(TMEM_KERNELS))
def test_dependents_start_only_once_tensor_memory_is_allocated(name):
    """tcgen05.alloc waits, without a limit, for columns that CTAs on the same SM hold. A dependent grid that was let
    start before a CTA has its columns could take them and then wait for that CTA's grid: pdl_trigger() comes after the
    barrier that follows the allocation (or right before the CTA leaves)."""
    body = re.sub(r"pdl_trigger\(\);\s*return;", "return;", TMEM_KERNELS[name])
    alloc = re.search(r"tmem_alloc\w*\(", body).start()
    published = body.index("__syncthreads();", alloc)
    assert published < body.index("pdl_trigger();")


COPYING_KERNELS = {name: body for name, body in _kernels() if re.search(r"bulk_g2s|tma_load|ss_fetch", body)}


@pytest.mark.parametrize("name", sorted(COPYING_KERNELS))
def test_a_kernel_whose_wait_ran_out_waits_for_its_copies(name):
    """Copies in flight when a CTA leaves would land in the next CTA's shared memory."""
    assert "drain_copies()" in COPYING_KERNELS[name]
