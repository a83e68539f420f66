"""The statuses of a batch are its own: two batches of one context, waited for from
two threads, one with a corrupt archive and one without, each report what their
archives are, however the waits interleave.  (-m gpu)"""
import threading

import numpy as np
import pytest

import oracle
import synth
from fmt_writer import build_archive

pytestmark = pytest.mark.gpu


def test_two_batches_of_a_context_from_two_threads():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2608_10188_gb300 as acx
    acx.build.build()
    good = acx.encode(synth.dna(20_000, 7))
    bad = build_archive([[{"cmd": 6, "lits": b"ACGT", "ml": 4, "src": 0}]])  # unknown command
    assert oracle.decode_status(bad, verify=False)[0] == oracle.E_CORRUPT
    ctx = acx.Context(0)
    keep, batches = [], []
    for arcs in ([good, bad], [good, good, good]):
        items = []
        for a in arcs:
            h = np.frombuffer(a, np.uint8).copy()
            d = torch.from_numpy(h).cuda()
            A = acx.Archive(ctx, d.data_ptr(), h, h.size)
            out = torch.zeros(A.total + 16, dtype=torch.uint8, device="cuda")
            keep.append((A, d, out))
            items.append((A, out.data_ptr(), A.total))
        batches.append(acx.Batch(ctx, items))
    want = [(oracle.E_CORRUPT, [0, oracle.E_CORRUPT]), (0, [0, 0, 0])]
    wrong, start = [], threading.Barrier(2)

    def work(k, stream):
        start.wait(60)
        for rep in range(2000):
            got = batches[k].run(stream.cuda_stream)
            if tuple(got) != want[k]:
                wrong.append((k, rep, got))

    torch.cuda.synchronize()
    streams = [torch.cuda.Stream(), torch.cuda.Stream()]
    threads = [threading.Thread(target=work, args=(k, streams[k])) for k in range(2)]
    try:
        for t in threads:
            t.start()
        for t in threads:
            t.join()
        assert not wrong, (len(wrong), wrong[:3])
    finally:
        for b in batches:
            b.close()
        for A, _, _ in keep:
            A.close()
        ctx.close()
