"""The measured workloads of the decoder: what its users have it do, through its public entry points.

A case names an operation, the corpus, the size and the encoder's options:

* ``op``: ``decode`` (device-resident archive -> device buffer), ``host`` (pinned host archive -> pinned host
  buffer), ``noalloc`` (the entry point without allocations), ``range`` (one region of an archive), ``batch``
  (many archives by one graph replay), ``serve`` (a burst of region requests to the region server),
  ``encode`` (host bytes -> archive);
* ``kind``: ``dna`` or ``text``, the two seeded corpora of ``synth``;
* ``size``: decompressed bytes; ``segment``: 0, or the size of the independently generated and parsed parts
  (chromosomes of a genome, files of a collection);
* ``no_rep``, ``levels``, ``deps``, ``lanes``: the encoder's options of the same names.

Every output is bytes, so every comparison is exact.
"""
from __future__ import annotations

import math
from concurrent.futures import ThreadPoolExecutor

import numpy as np
import torch

import paper_2608_10188_gb300 as acx
import synth

KIB, MIB = 1 << 10, 1 << 20
BLOCK = acx.lib.BLOCK_SIZE
RATIO = {"dna": 0.25, "text": 0.36}  # archive bytes per decompressed byte
THREADS = 16


def _case(name, op, kind, size, segment=0, no_rep=False, levels=False, deps=False, lanes=32, **more):
    return {"name": name, "op": op, "kind": kind, "size": size, "segment": segment, "no_rep": no_rep,
            "levels": levels, "deps": deps, "lanes": lanes, **more}


def listed():
    return [
        # a file smaller than a block, decoded and waited for: launches and latency only
        _case("file-10k", "decode", "text", 10_007, sync=True),
        # one region of about a block out of an indexed genome: a seek of a genome browser
        _case("seek-16k", "range", "dna", 32 * MIB, segment=4 * MIB, start=0.6180339, length=16_301, index=True),
        # a small file under a runtime that owns the device's memory
        _case("noalloc-1m", "noalloc", "dna", 1_000_003),
        # the small configuration of the tests and benchmarks: 4 MiB, decoded and waited for
        _case("dna-4m", "decode", "dna", 4 * MIB, sync=True),
        # a mid-size genome encoded without the distance history, queued among other work
        _case("dna-64m-free", "decode", "dna", 64 * MIB + 4_321, segment=8 * MIB, no_rep=True, sync=False),
        # the headline size: a chromosome-sized genome, queued among other work
        _case("genome-254m", "decode", "dna", synth.GENOME_CHR1_SIZE, segment=16 * MIB, sync=False),
        # a large text collection with level bodies, queued among other work
        _case("text-200m-levels", "decode", "text", 200 * MIB, segment=16 * MIB, levels=True, sync=False),
        # a collection of files of mixed sizes, corpora and encodings: one graph replay
        _case("batch-96", "batch", "mixed", 4 * MIB, count=96),
        # end to end from host memory with the archive's plan kept (a loader that reads the same file again)
        _case("host-64m", "host", "dna", 64 * MIB, segment=8 * MIB, keep=True),
        # end to end from host memory, a file seen once: plan, upload, decode, download
        _case("host-once-3m", "host", "text", 3 * MIB + 77, keep=False),
        # a burst of regions to the region server, whose cache holds a quarter of the genome
        _case("serve-256", "serve", "dna", 64 * MIB, segment=8 * MIB, count=256),
        # the encoder on a small file
        _case("encode-1m", "encode", "text", 1 * MIB),
    ]


def _log(rng, lo, hi):
    return min(hi, max(lo, int(math.exp(rng.uniform(math.log(lo), math.log(hi + 1))))))


def _segment(size):
    """Parts of a corpus of that size: none for a small one, else about 16 block-aligned parts of at most 16 MiB."""
    if size <= 2 * MIB:
        return 0
    return min(16 * MIB, max(BLOCK, (size // 16 + BLOCK - 1) // BLOCK * BLOCK))


def draw(rng):
    op = rng.choice(["decode", "decode", "decode", "decode", "host", "noalloc", "range", "range", "batch", "serve"])
    kind = rng.choice(["dna", "text"])
    opt = {"no_rep": rng.random() < 0.4, "levels": rng.random() < 0.3, "deps": rng.random() < 0.2,
           "lanes": rng.choice([8, 16, 32, 32, 32, 64, 128])}
    if op == "decode":
        size = _log(rng, 1, 240 * MIB if kind == "dna" else 192 * MIB)
        more = {"sync": size < 8 * MIB}
    elif op == "host":
        size = _log(rng, 4 * KIB, 128 * MIB)
        more = {"keep": rng.random() < 0.5}
    elif op == "noalloc":
        size, more = _log(rng, 1, 600_000), {}
        opt["lanes"] = 32
    elif op == "range":
        size = _log(rng, 256 * KIB, 48 * MIB)
        index = rng.random() < 0.7
        if not index:
            opt["deps"] = True
        more = {"start": round(rng.random(), 6), "length": _log(rng, 1, min(size, 1 * MIB)), "index": index}
    elif op == "serve":
        size = _log(rng, 8 * MIB, 96 * MIB)
        more = {"count": rng.randint(16, 256)}
    else:
        size = _log(rng, 128 * KIB, 4 * MIB)
        more = {"count": rng.randint(2, 96)}
        return {k: v for k, v in _case("", "batch", "mixed", size, **more).items() if k != "name"}
    c = _case("", op, kind, size, segment=_segment(size), **opt, **more)
    del c["name"]
    return c


# ---- inputs ------------------------------------------------------------------------------------


def _data(kind, size, segment, seed):
    """The corpus: one part, or parts of `segment` bytes, each from a seed of its own."""
    if not segment or segment >= size:
        return synth.corpus(kind, size, seed * 4096)
    out = np.empty(size, np.uint8)
    make = synth.dna if kind == "dna" else synth.text

    def part(i):
        lo = i * segment
        make(min(segment, size - lo), seed * 4096 + i, out=out[lo:lo + segment])

    with ThreadPoolExecutor(THREADS) as pool:
        list(pool.map(part, range((size + segment - 1) // segment)))
    return out


def _encode(case, seed):
    data = _data(case["kind"], case["size"], case["segment"], seed)
    arc = acx.encode(data, no_rep=case["no_rep"], levels=case["levels"], deps=case["deps"], max_lanes=case["lanes"],
                     segment=case["segment"])
    return np.frombuffer(arc, np.uint8)


def _specs(case, seed):
    """The files of a batch: sizes log-uniform in [64 KiB, case size] (the case's own), corpora and encodings in turn."""
    specs = synth.batch_specs(case["count"], lo=64 * KIB, hi=case["size"])
    return [dict(s, seed=seed * 4096 + s["index"]) for s in specs]


def _regions(case, seed):
    """Requests of a burst: uniform starts, lengths (the case's own) lognormal around 16 KiB in [4 KiB, 512 KiB]."""
    ln = np.random.default_rng(55).lognormal(math.log(16 * KIB), 1.0, case["count"])
    ln = np.clip(ln, 4 * KIB, 512 * KIB).astype(np.uint64)
    st = np.random.default_rng(seed).random(case["count"]) * (case["size"] - ln.astype(np.float64))
    st = st.astype(np.uint64)
    return st, ln


def _blank(n):
    return torch.full((max(int(n), 1),), 0xA5, dtype=torch.uint8, device="cuda")


def _pinned(a):
    t = torch.empty(max(int(a.size), 1), dtype=torch.uint8, pin_memory=True)
    t.numpy()[:a.size] = a
    return t


def prepare(case, seed):
    op, s = case["op"], {"op": case["op"], "case": dict(case)}
    if op == "encode":
        s["data"] = _data(case["kind"], case["size"], case["segment"], seed)
        s["out"] = np.zeros(case["size"] + 64 * KIB, np.uint8)  # the program's file buffer
        return s
    if op == "batch":
        specs = _specs(case, seed)
        with ThreadPoolExecutor(THREADS) as pool:
            arcs = list(pool.map(lambda x: np.frombuffer(acx.encode(synth.corpus(x["kind"], x["size"], x["seed"]),
                                                                    no_rep=x["no_rep"], threads=1), np.uint8), specs))
        s["ctx"] = ctx = acx.Context(0)
        s["d_arcs"] = [torch.from_numpy(a.copy()).cuda() for a in arcs]
        at = np.concatenate([[0], np.cumsum([(x["size"] + 255) // 256 * 256 for x in specs])])
        s["out"] = _blank(at[-1])  # the files side by side
        s["arcs"] = [acx.Archive(ctx, d.data_ptr(), a, a.size) for d, a in zip(s["d_arcs"], arcs)]
        s["batch"] = acx.Batch(ctx, [(a, s["out"].data_ptr() + int(o), x["size"])
                                     for a, o, x in zip(s["arcs"], at, specs)], graph=True)
        return s
    arc = _encode(case, seed)
    if op == "host":
        s["ctx"] = ctx = acx.Context(0)
        s["h_arc"] = _pinned(arc)
        s["h_out"] = _pinned(np.full(case["size"], 0xA5, np.uint8))
        s["np_arc"], s["np_out"] = s["h_arc"].numpy()[:arc.size], s["h_out"].numpy()[:case["size"]]
        if case["keep"]:
            s["d_arc"] = torch.from_numpy(arc.copy()).cuda()
            s["arc"] = acx.Archive(ctx, s["d_arc"].data_ptr(), arc, arc.size)
        return s
    s["d_arc"] = torch.from_numpy(arc.copy()).cuda()
    if op == "noalloc":
        s["out"] = _blank(case["size"])
        return s
    s["ctx"] = ctx = acx.Context(0)
    s["arc"] = a = acx.Archive(ctx, s["d_arc"].data_ptr(), arc, arc.size)
    if op == "decode":
        s["out"] = _blank(case["size"])
    elif op == "range":
        if case["index"]:
            a.build_index()
        s["start"] = int(case["start"] * (case["size"] - case["length"]))
        s["out"] = _blank(case["length"])
    elif op == "serve":
        a.build_index()
        s["starts"], s["lens"] = _regions(case, seed)
        s["out"] = _blank(int(s["lens"].sum()))
        s["ptrs"] = s["out"].data_ptr() + np.concatenate([[0], np.cumsum(s["lens"])[:-1]]).astype(np.uint64)
        s["srv"] = acx.Server(ctx, a, cache_bytes=max(case["size"] // 4, 16 * MIB))
    return s


# ---- one pass ----------------------------------------------------------------------------------


def _ok(rc, s):
    if rc != acx.lib.OK:
        raise RuntimeError(f"status {rc}: {s['ctx'].last_error() if 'ctx' in s else ''}")


def run(state):
    s, op = state, state["op"]
    st = torch.cuda.current_stream().cuda_stream
    if op == "decode":
        f = acx.decode_all if s["case"]["sync"] else acx.decode_all_async
        _ok(f(s["ctx"], s["arc"], s["out"].data_ptr(), s["out"].numel(), st), s)
        return s["out"]
    if op == "host":
        _ok(acx.decode_host(s["ctx"], s.get("arc"), s["np_arc"], s["np_out"], st), s)
        return s["np_out"]
    if op == "noalloc":
        _ok(acx.lib.decode_noalloc(s["d_arc"].data_ptr(), s["d_arc"].numel(), s["out"].data_ptr(), s["out"].numel(), st),
            s)
        return s["out"]
    if op == "range":
        _ok(acx.decode_range(s["ctx"], s["arc"], s["start"], s["case"]["length"], s["out"].data_ptr(), st), s)
        return s["out"]
    if op == "batch":
        rc, per = s["batch"].run(st)
        _ok(rc, s)
        return s["out"]
    if op == "serve":
        s["srv"].submit_many(s["starts"], s["lens"], s["ptrs"])
        _ok(s["srv"].drain(), s)
        if any(c["status"] != acx.lib.OK for c in s["srv"].poll(max_n=s["case"]["count"])):
            raise RuntimeError("a request failed: " + s["srv"].last_error())
        return s["out"]
    c = s["case"]
    arc = acx.encode(s["data"], no_rep=c["no_rep"], levels=c["levels"], deps=c["deps"], max_lanes=c["lanes"],
                     segment=c["segment"])
    s["out"][:len(arc)] = np.frombuffer(arc, np.uint8)
    return [len(arc), s["out"]]


# ---- what a pass cannot do without -------------------------------------------------------------


def work(case):
    """Bytes of one pass: the archive bytes of what is decoded, read once, and the output, written once (in the
    other direction for the encoder).  There is no arithmetic to speak of."""
    op = case["op"]
    if op == "range":
        return {"bytes": case["length"] * (1 + RATIO[case["kind"]]), "flops": 0}
    if op == "serve":  # the mean of the clipped lognormal is about 26 KiB
        return {"bytes": case["count"] * 26 * KIB * (1 + RATIO[case["kind"]]), "flops": 0}
    if op == "batch":
        lo, hi = 64 * KIB, case["size"]
        return {"bytes": case["count"] * (hi - lo) / math.log(hi / lo) * 1.3, "flops": 0}
    return {"bytes": case["size"] * (1 + RATIO[case["kind"]]), "flops": 0}


def tolerance(case):
    """Every output is bytes of the one decode (or of the one archive that the encoder's rules give)."""
    return "exact"
