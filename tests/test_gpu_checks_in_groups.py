"""Blocks that fail a check which the local pass's threads make on their own (a
repeat distance before the output's start, a source block missing from the
dependency list), one after another among valid blocks of other archives, at
every group size: each such archive fails alone, every valid one decodes exactly,
on every run.  (-m gpu)"""
import numpy as np
import pytest

import oracle
import synth
from fmt_writer import build_archive

pytestmark = pytest.mark.gpu

BLOCK = 16384


def _bad_archives():
    lits = bytes(np.random.default_rng(3).integers(65, 69, BLOCK, dtype=np.uint8))
    full = [{"cmd": 5, "lits": lits, "ml": 0}]
    yield build_archive([[{"cmd": 4, "lits": b"", "ml": 4}]])  # one token: distance 4 at position 0
    yield build_archive([[{"cmd": 4, "lits": b"", "ml": 4}] + [{"cmd": 1, "lits": b"AC", "ml": 5}] * 600])
    yield build_archive([full, [{"cmd": 0, "lits": b"", "ml": 4, "src": 7}]], deps=[[], []])
    yield build_archive([full, [{"cmd": 0, "lits": b"G", "ml": 9, "src": 70}] * 600], deps=[[], []])


# threads of a group: 256 and 512 for at most two blocks per SM, 128 and 256 (text) for more
@pytest.mark.parametrize("kind,blocks", [("dna", 20), ("text", 20), ("dna", 700), ("text", 500)])
@pytest.mark.parametrize("chunk", [1, 3])
def test_failed_checks_stay_in_their_archive(kind, blocks, chunk):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2608_10188_gb300 as acx
    acx.build.build()
    data = synth.corpus(kind, blocks * BLOCK - 99, 23)
    good = acx.encode(data, deps=True, segment=16 * BLOCK)
    assert np.array_equal(oracle.decode(good), data)
    bad = list(_bad_archives())
    for a in bad:
        assert oracle.decode_status(a, verify=False)[0] == oracle.E_CORRUPT
    if kind == "dna":  # (the archives of 600 tokens would widen the groups)
        bad = bad[::2]
    cases = (bad + [good]) * 8
    want = ([oracle.E_CORRUPT] * len(bad) + [0]) * 8
    ctx = acx.Context(0, timeout_us=2_000_000, queue_chunk=chunk)
    try:
        h = [np.frombuffer(a, np.uint8).copy() for a in cases]
        d = [torch.from_numpy(x).cuda() for x in h]
        arcs = [acx.Archive(ctx, t.data_ptr(), x, x.size) for t, x in zip(d, h)]
        outs = [torch.full((A.total + 64,), 0xA5, dtype=torch.uint8, device="cuda") for A in arcs]
        b = acx.Batch(ctx, [(A, o.data_ptr(), A.total) for A, o in zip(arcs, outs)], graph=True)
        ref = torch.from_numpy(data).cuda()
        st = torch.cuda.current_stream().cuda_stream
        for rep in range(20):
            for o in outs:
                o.fill_(0xA5)
            rc, per = b.run(st)
            assert rc == oracle.E_CORRUPT and per == want, rep
            for w, A, o in zip(want, arcs, outs):
                assert w or torch.equal(o[:A.total], ref), rep
                assert bool((o[A.total:] == 0xA5).all())
        b.close()
        for A in arcs:
            A.close()
    finally:
        ctx.close()
