"""A batch whose archives need workspaces of two sizes (DNA-like ones small,
text large), each kind with enough blocks for a local pass of its own: the
archives take another order on the device, every output and every status must
still be its own archive's, replayed or not, with one and several blocks per
ticket, and a corrupt archive of either kind fails alone.  One block less of a
kind leaves the batch in one pass: the same results.  (-m gpu)"""
import numpy as np
import pytest

import oracle
import synth
from fmt_writer import build_archive

pytestmark = pytest.mark.gpu

BLOCK = 16384
BLOCKS_PER_SM = 32  # of each kind, from which on the batch runs two passes


@pytest.fixture(scope="module")
def acx():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2608_10188_gb300 as acx
    acx.build.build()
    acx.load()
    return acx


@pytest.fixture(scope="module")
def parts(acx):
    """Per kind: an archive of all but 5 of the blocks that make a class, and
    archives of 3 and 4 blocks (the fifth is a corrupt archive's)."""
    import torch
    n = BLOCKS_PER_SM * torch.cuda.get_device_properties(0).multi_processor_count
    out = {}
    for kind, seed in (("dna", 5), ("text", 6)):
        for blocks in (n - 5, 3, 4):
            data = synth.corpus(kind, blocks * BLOCK - 77, seed + blocks)
            out[kind, 1 if blocks > 4 else blocks] = data, acx.encode(data, segment=4 << 20)
    return out


@pytest.mark.parametrize("graph,chunk,small", [(False, 1, 4), (True, 1, 4), (False, 16, 4), (False, 1, 3)])
def test_batch_of_two_workspaces(acx, parts, graph, chunk, small):
    import torch
    # an unknown command, in a block of one token (19 KB of workspace) and of 1,501 (62 KB)
    last = [{"cmd": 6, "lits": b"ACGT", "ml": 4, "src": 0}]
    narrow, wide = build_archive([last]), build_archive([[{"cmd": 0, "lits": b"ACGT", "ml": 4, "src": 0}] * 1500 + last])
    for bad in (narrow, wide):
        assert oracle.decode_status(bad, verify=False)[0] == oracle.E_CORRUPT
    cases = [parts["text", small], (None, wide), parts["dna", small], parts["text", 1], parts["dna", 1], (None, narrow)]
    ctx = acx.Context(0, timeout_us=2_000_000)
    try:
        ctx.set_params(queue_chunk=chunk, timeout_us=2_000_000)
        h = [np.frombuffer(a, np.uint8).copy() for _, a in cases]
        d = [torch.from_numpy(x).cuda() for x in h]
        arcs = [acx.Archive(ctx, t.data_ptr(), x, x.size) for t, x in zip(d, h)]
        outs = [torch.full((A.total + 64,), 0xA5, dtype=torch.uint8, device="cuda") for A in arcs]
        b = acx.Batch(ctx, [(A, o.data_ptr(), A.total) for A, o in zip(arcs, outs)], graph=graph)
        st = torch.cuda.current_stream().cuda_stream
        for rep in range(2):
            for o in outs:
                o.fill_(0xA5)
            rc, per = b.run(st)
            assert rc == -2 and per == [-2 if x is None else 0 for x, _ in cases]
            for (want, _), A, o in zip(cases, arcs, outs):
                got = o.cpu().numpy()
                assert want is None or np.array_equal(got[:A.total], want), rep
                assert np.all(got[A.total:] == 0xA5)
        b.close()
        for A in arcs:
            A.close()
    finally:
        ctx.close()
