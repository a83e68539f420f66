"""Device addresses off the 16-byte boundary: the kernels move 16 bytes at a time, so
archives and whole outputs there are refused on the host, before any launch; what
needs no wide access (regions, outputs below 16 bytes, an archive that is only
described, or decoded from host memory) is served.  (-m gpu)"""
import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("off", [1, 4, 8])
def test_unaligned_device_addresses(off):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2608_10188_gb300 as acx
    acx.build.build()
    L = acx.lib
    data = synth.dna(50_001, 9)
    arc = np.frombuffer(acx.encode(data), np.uint8).copy()
    assert np.array_equal(oracle.decode(arc.tobytes()), data)
    room = torch.zeros(arc.size + 64, dtype=torch.uint8, device="cuda")
    room[:arc.size] = torch.from_numpy(arc).cuda()
    out = torch.zeros(data.size + 64, dtype=torch.uint8, device="cuda")
    moved = torch.zeros(arc.size + 64, dtype=torch.uint8, device="cuda")
    moved[off:off + arc.size] = room[:arc.size]
    st = torch.cuda.current_stream().cuda_stream
    ctx = acx.Context(0)
    try:
        good = acx.Archive(ctx, room.data_ptr(), arc, arc.size)
        bad = acx.Archive(ctx, moved.data_ptr() + off, arc, arc.size)
        assert bad.total == data.size
        for variant in (L.VARIANT_FAST, L.VARIANT_PLAIN, L.VARIANT_FUSED):
            ctx.set_params(variant=variant)
            assert acx.decode_all(ctx, good, out.data_ptr() + off, data.size, st) == L.E_ARG
            assert acx.decode_all(ctx, bad, out.data_ptr(), data.size, st) == L.E_ARG
            assert acx.decode_all_async(ctx, bad, out.data_ptr(), data.size, st) == L.E_ARG
        ctx.set_params()
        for a, o in ((good, off), (bad, 0)):
            with pytest.raises(acx.AceapexError) as e:
                acx.Batch(ctx, [(a, out.data_ptr() + o, data.size)])
            assert e.value.status == L.E_ARG
        assert acx.decode_range(ctx, bad, 100, 1000, out.data_ptr(), st) == L.E_ARG
        with pytest.raises(acx.AceapexError):
            bad.build_index()
        with pytest.raises(acx.AceapexError):
            acx.Server(ctx, bad)
        assert L.decode_noalloc(moved.data_ptr() + off, arc.size, out.data_ptr(), data.size, st) == L.E_ARG
        assert L.decode_noalloc(room.data_ptr(), arc.size, out.data_ptr() + off, data.size, st) == L.E_ARG
        torch.cuda.synchronize()
        # what needs no alignment
        assert acx.decode_range(ctx, good, 100, 1000, out.data_ptr() + off, st) == 0, ctx.last_error()
        assert np.array_equal(out[off:off + 1000].cpu().numpy(), data[100:1100])
        host = np.zeros(data.size, np.uint8)
        assert acx.decode_host(ctx, bad, arc, host, st) == 0, ctx.last_error()
        assert np.array_equal(host, data)
        tiny = np.frombuffer(acx.encode(data[:15]), np.uint8).copy()
        d = torch.from_numpy(tiny).cuda()
        a = acx.Archive(ctx, d.data_ptr(), tiny, tiny.size)
        for f in (lambda: acx.decode_all(ctx, a, out.data_ptr() + off, 15, st),
                  lambda: L.decode_noalloc(d.data_ptr(), tiny.size, out.data_ptr() + off, 15, st)):
            out.zero_()
            assert f() == 0, ctx.last_error()
            assert np.array_equal(out[off:off + 15].cpu().numpy(), data[:15])
        for x in (a, good, bad):
            x.close()
    finally:
        ctx.close()
