"""The cross-block pass's copy of one piece by one lane, at every source and
destination alignment and piece length, in its three job forms (one archive,
a batch, a range decode into slots), against the byte-serial copy and the
oracle; with pieces that take the byte path (periodic ones, sources that cross
a block boundary or end in the output's last 16-byte word) among them, and
blocks of few and of very many pieces (parts of the hand-out).  (-m gpu)"""
import numpy as np
import pytest

import oracle
from fmt_writer import build_archive

pytestmark = pytest.mark.gpu

BLOCK = 16384


@pytest.fixture(scope="module")
def acx():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2608_10188_gb300 as acx
    acx.build.build()
    acx.load()
    return acx


def _archive(lens, seed):
    """Block 0 is literals; then, for each length, a match at each of the 16
    source and 8 destination alignments from a random earlier block (so chains
    of any depth form), periodic cross-block fills and boundary-crossing
    sources in between, and a last block of 13 bytes that copies the bytes up
    to its own start."""
    rng = np.random.default_rng(seed)
    out = bytearray(rng.integers(0, 256, BLOCK, dtype=np.uint8).tobytes())
    blocks, toks = [[{"cmd": 5, "lits": bytes(out), "ml": 0}]], []

    def room():
        return BLOCK - len(out) % BLOCK if len(out) % BLOCK or toks == [] else 0

    def close():
        nonlocal toks
        rest = -len(out) % BLOCK
        if rest:
            lits = rng.integers(0, 256, rest, dtype=np.uint8).tobytes()
            toks.append({"cmd": 5, "lits": lits, "ml": 0})
            out.extend(lits)
        blocks.append(toks)
        toks = []

    def match(src, ml, dalign):
        pad = (dalign - len(out)) % 8
        if room() < pad + ml:
            close()
            pad = (dalign - len(out)) % 8
        lits = rng.integers(0, 256, pad, dtype=np.uint8).tobytes()
        out.extend(lits)
        toks.append({"cmd": 0, "lits": lits, "ml": ml, "src": src})
        for j in range(ml):
            out.append(out[src + j])

    for ml in lens:
        for sa in range(16):
            for da in range(8):
                b = int(rng.integers(0, len(out) // BLOCK))
                match(b * BLOCK + 16 * int(rng.integers(0, 1000)) + sa, ml, da)
        nb = len(out) // BLOCK
        match(nb * BLOCK - 1 - ml // 2, ml, 3)       # (its source may cross into this block or end at it)
        if nb > 1:
            match(BLOCK - ml // 2, ml, 5)            # a source across the first block boundary
        d = int(rng.integers(1, 70))                  # a periodic fill whose period was copied from elsewhere
        match(int(rng.integers(0, BLOCK - d)), max(4, d), 0)
        match(len(out) - d, 5 * ml, len(out) % 8)
    if toks:
        close()
    # 13 bytes: 4 literals, then 9 bytes whose source ends in the last 16-byte word of the output
    lits = rng.integers(0, 256, 4, dtype=np.uint8).tobytes()
    src = len(out) - 6
    out.extend(lits)
    toks = [{"cmd": 0, "lits": lits, "ml": 9, "src": src}]
    for j in range(9):
        out.append(out[src + j])
    blocks.append(toks)
    arc = build_archive(blocks)
    assert oracle.decode(arc, verify=False).tobytes() == bytes(out)
    return arc, np.frombuffer(bytes(out), np.uint8)


@pytest.mark.parametrize("lens", [range(4, 12), range(12, 24), range(24, 40), (63, 64, 65, 100)],
                         ids=lambda r: f"{min(r)}-{max(r)}")
def test_piece_copies_at_every_alignment(acx, lens):
    import torch
    arc, want = _archive(lens, min(lens))
    h = np.frombuffer(arc, np.uint8).copy()
    d = torch.from_numpy(h).cuda()
    st = torch.cuda.current_stream().cuda_stream
    ctx = acx.Context(0)
    try:
        A = acx.Archive(ctx, d.data_ptr(), h, h.size)
        out = torch.full((want.size,), 0xA5, dtype=torch.uint8, device="cuda")
        assert acx.decode_all(ctx, A, out.data_ptr(), out.numel(), st) == 0, ctx.last_error()
        assert np.array_equal(out.cpu().numpy(), want)
        out.fill_(0xA5)
        assert acx.decode_range(ctx, A, 0, want.size, out.data_ptr(), st) == 0, ctx.last_error()
        assert np.array_equal(out.cpu().numpy(), want)
        outs = torch.full((3, (want.size + 255) // 256 * 256), 0xA5, dtype=torch.uint8, device="cuda")
        B = acx.Batch(ctx, [(A, outs[i].data_ptr(), want.size) for i in range(3)], graph=True)
        rc, per = B.run(st)
        assert rc == 0 and per == [0, 0, 0], ctx.last_error()
        assert all(np.array_equal(outs[i, :want.size].cpu().numpy(), want) for i in range(3))
        B.close()
        A.close()
    finally:
        ctx.close()


@pytest.mark.parametrize("blocks", [2, 65, 400])
def test_blocks_of_very_different_piece_counts(acx, blocks):
    """Parts of the hand-out: most blocks leave one piece, some thousands."""
    rng = np.random.default_rng(blocks)
    out = bytearray(rng.integers(0, 256, BLOCK, dtype=np.uint8).tobytes())
    bl = [[{"cmd": 5, "lits": bytes(out), "ml": 0}]]
    for b in range(1, blocks):
        toks, B = [], len(out)
        for _ in range(4096 if b % 37 == 1 else 1):
            src = int(rng.integers(0, B - 4))
            toks.append({"cmd": 0, "lits": b"", "ml": 4, "src": src})
            out.extend(out[src:src + 4])
        rest = B + BLOCK - len(out)
        if rest:
            lits = rng.integers(0, 256, rest, dtype=np.uint8).tobytes()
            toks.append({"cmd": 5, "lits": lits, "ml": 0})
            out.extend(lits)
        bl.append(toks)
    arc = build_archive(bl)
    want = oracle.decode(arc, verify=False)
    assert want.tobytes() == bytes(out)
    from gpu_util import gpu_decode
    ctx = acx.Context(0)
    try:
        rc, got, st = gpu_decode(ctx, arc, stats=True)
        assert rc == 0, ctx.last_error()
        assert np.array_equal(got, want)
        # every match was a piece, and the waits of round 0 finished them all
        assert st["pending_spans"] == sum(4096 if b % 37 == 1 else 1 for b in range(1, blocks))
        assert st["wait_polls"] == 0
    finally:
        ctx.close()
