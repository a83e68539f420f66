"""The entropy stage's tickets: whole blocks, or a block's literals, offsets
and other short streams on warps of their own, at the edge of the choice (all
parts find a warp at once, or one block too many), with tickets taken one and
several at a time, against the input and the oracle.  (-m gpu)"""
import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu

BLOCK = 16384


@pytest.mark.parametrize("chunk", [0, 4])
@pytest.mark.parametrize("more", [0, 1], ids=["last split", "first whole"])
@pytest.mark.parametrize("kind", ["dna", "text"])
def test_blocks_at_the_edge_of_the_split(kind, more, chunk):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2608_10188_gb300 as acx
    from gpu_util import gpu_decode
    acx.build.build()
    warps = 2 * 16 * torch.cuda.get_device_properties(0).multi_processor_count
    data = synth.corpus(kind, (warps // 3 + more) * BLOCK - 5, 19)
    arc = acx.encode(data, segment=64 * BLOCK)
    assert np.array_equal(oracle.decode(arc), data)
    ctx = acx.Context(0, queue_chunk=chunk)
    try:
        rc, out = gpu_decode(ctx, arc)
        assert rc == 0, ctx.last_error()
        assert np.array_equal(out, data)
    finally:
        ctx.close()
