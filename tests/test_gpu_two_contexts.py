"""Two host threads, each with a context and a stream of its own, decode archives
of small and of large workspaces at the same time: the kernels' shared-memory
limit belongs to the device, not to a launch, so neither thread may narrow it
under the other.  (-m gpu)"""
import threading

import numpy as np
import pytest

import oracle
from fmt_writer import build_archive

pytestmark = pytest.mark.gpu


def _archive(tokens, lits, ml):
    arc = build_archive([[{"cmd": 0, "lits": lits, "ml": ml, "src": 0}] * tokens])
    return arc, oracle.decode(arc, verify=False)


@pytest.mark.parametrize("variant", ["fast", "fused"])
def test_workspaces_of_two_sizes_at_once(variant):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2608_10188_gb300 as acx
    acx.build.build()
    # one block each, of the same kernel (more than 256 tokens): 27 and 97 KB
    cases = [_archive(300, b"ACGT", 4), _archive(3000, b"A", 4)]
    failures, start = [], threading.Barrier(2)

    def work(arc, want):
        ctx = acx.Context(0, variant=acx.lib.VARIANT_FUSED if variant == "fused" else acx.lib.VARIANT_FAST)
        stream = torch.cuda.Stream()
        h = np.frombuffer(arc, np.uint8).copy()
        d = torch.from_numpy(h).cuda()
        out = torch.empty(want.size, dtype=torch.uint8, device="cuda")
        ref = torch.from_numpy(want.copy()).cuda()
        torch.cuda.synchronize()
        A = acx.Archive(ctx, d.data_ptr(), h, h.size)
        try:
            start.wait(60)
            for k in range(1500):
                rc = acx.decode_all(ctx, A, out.data_ptr(), out.numel(), stream.cuda_stream)
                if rc != 0:
                    failures.append((k, rc, ctx.last_error()))
            if not failures and not torch.equal(out, ref):
                failures.append("wrong bytes")
        finally:
            A.close()
            ctx.close()

    threads = [threading.Thread(target=work, args=c) for c in cases]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not failures, (len(failures), failures[:3])
