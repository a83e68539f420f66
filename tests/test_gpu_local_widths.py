"""The local pass's group sizes (128, 256 and 512 threads, chosen by the number
of blocks, a block's tokens and its workspace) at the edges of the choice,
against the input and the oracle.  (-m gpu)"""
import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu

BLOCK = 16384


@pytest.mark.parametrize("more", [None, 0, 1], ids=["one", "2 per SM", "2 per SM + 1"])
@pytest.mark.parametrize("kind", ["dna", "text"])
def test_blocks_at_the_edges_of_the_group_sizes(kind, more):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2608_10188_gb300 as acx
    from gpu_util import gpu_decode
    acx.build.build()
    nb = 1 if more is None else 2 * torch.cuda.get_device_properties(0).multi_processor_count + more
    data = synth.corpus(kind, nb * BLOCK - 5, 17)
    arc = acx.encode(data, segment=32 * BLOCK)
    assert np.array_equal(oracle.decode(arc), data)
    ctx = acx.Context(0)
    try:
        rc, out = gpu_decode(ctx, arc)
        assert rc == 0, ctx.last_error()
        assert np.array_equal(out, data)
    finally:
        ctx.close()
