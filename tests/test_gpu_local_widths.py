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


@pytest.mark.parametrize("matches", [1, 4, 63, 64, 65, 129, 400])
def test_in_block_matches_around_the_lane_choice(matches):
    """Blocks with that many in-block matches, plain ones of 4 to 100 bytes and
    periodic ones of 1 to 40 bytes' distance, sources anywhere before them
    (chains of any depth): a lane or eight lanes a match."""
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2608_10188_gb300 as acx
    from fmt_writer import build_archive
    from gpu_util import gpu_decode
    acx.build.build()
    rng = np.random.default_rng(matches)
    blocks, out = [], bytearray()
    for _ in range(3):
        B, toks = len(out), []
        lead = 64
        for k in range(matches):
            lits = rng.integers(0, 256, lead, dtype=np.uint8).tobytes()
            lead = int(rng.integers(0, 4))
            out.extend(lits)
            pos = len(out)
            if rng.random() < 0.25:
                d, ml = int(rng.integers(1, 41)), int(rng.integers(41, 80))
            else:
                d = int(rng.integers(4, pos - B + 1))
                ml = int(rng.integers(4, min(d, 101 if matches < 100 else 24) + 1))
            ml = min(ml, B + BLOCK - pos)
            if ml < 4:
                break
            toks.append({"cmd": 0, "lits": lits, "ml": ml, "src": pos - d})
            for j in range(ml):
                out.append(out[pos - d + j])
        rest = B + BLOCK - len(out)
        if rest:
            lits = rng.integers(0, 256, rest, dtype=np.uint8).tobytes()
            toks.append({"cmd": 5, "lits": lits, "ml": 0})
            out.extend(lits)
        blocks.append(toks)
    arc = build_archive(blocks)
    assert oracle.decode(arc, verify=False).tobytes() == bytes(out)
    ctx = acx.Context(0)
    try:
        rc, got, st = gpu_decode(ctx, arc, stats=True)
        assert rc == 0, ctx.last_error()
        assert got.tobytes() == bytes(out)
        assert st["pending_spans"] == 0  # every chain ends inside its block
    finally:
        ctx.close()
