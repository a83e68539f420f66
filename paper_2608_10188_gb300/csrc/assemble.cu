// Parse and match layer of the decode (paper: "parse" and "copy"), in two
// passes separated by a kernel boundary.
//
// k_local (one CTA of 128, 256 or 512 threads per block, persistent, any order):
//   * varint boundaries by compaction: every byte < 0x80 ends a value; a CTA
//     prefix count gives each value its index (LL_i, ML_i).  The paper finds
//     varints make 0.61% of commands sequential in a serial parse ("The Last
//     Sequential Element"); here they are a scan like everything else.
//   * prefix sums of LL+ML, LL and #NEW give every token's output position,
//     literal position and offset index (the paper's 93.94% scan share).
//   * the 4-entry distance history as a monoid scan: each token is a map on
//     the history (NEW pushes a distance, REPk moves entry k to the front);
//     maps compose associatively, so the history before every token is a
//     prefix "sum" too.  Skipped when a block has no repeat code (history-
//     free encoding, where the parse is a dependency-free prefix scan).
//   * literals: runs of up to 32 bytes are copied by one thread each, all
//     threads at once; longer runs by eight lanes with 16-byte funnel-shifted
//     stores.
//   * matches whose source lies inside the block are periodic fills
//     out[dst+k] = out[src + (k mod d)] ("What Does: Periods, Not Chains"),
//     done in rounds as their sources become final; matches whose source
//     chain leaves the block become pending spans.
//   * the block is written with coalesced 16-byte stores; its pending-byte
//     bitmap and pending spans go beside it.
// k_external (warps take parts of blocks in ascending order, a lane per span):
//   after the kernel boundary every literal and every in-block match byte is
//   final, so a pending span waits only on the spans its source really
//   depends on, which lie at lower positions and were taken earlier: the
//   ascending order makes the bounded waits deadlock-free.  Under an explicit
//   wait limit (wait_ns), spans that wait for longer go to work lists, staged
//   per warp in shared memory; barrier-separated rounds walk the lists until
//   they are empty, each round finishing at least the lowest span.
#include <algorithm>

#include <mutex>

#include "launch.h"
#include "local_dev.cuh"

namespace acx {

// CTAs per SM that a kernel is built for.  Blocks of some 900 tokens and more
// (55 KB of workspace) leave room for four CTAs of 256 threads: at 61 registers
// (64 in a batch) they fit (200 MiB text: three 423 us, four 357).  Where the
// workspace leaves room for three, the registers of three are better (a batch of
// 96 small files with the workspace of all kinds: 646 us, 657 built for four).
template <int NT>
constexpr int kLocCtas = NT == kLocThreads ? 6 : NT == kLocWide ? 4 : 1;

template <int NT, Loc kKind, int kCtas>
__global__ void __launch_bounds__(NT, kCtas) k_local(JobDev job) {
    extern __shared__ __align__(128) uint8_t sm[];
    grid_dependency_wait();  // the entropy stage's streams
    local_worker<NT, kKind>(job, sm, 0, threadIdx.x);
}

// ---- cross-block pass --------------------------------------------------------------------
// What the pass needs of the archive that a piece belongs to.  A job over one
// archive keeps it in the kernel's parameters; in a batch each lane holds its
// own piece's.
struct ArcView {
    uint8_t* out;
    uint32_t* pmap;
    const uint32_t* slot;
    uint64_t total;
};
__device__ __forceinline__ ArcView view_of(const ArcJob& J) { return ArcView{J.out, J.pmap, J.slot, J.total}; }
__device__ __forceinline__ uint64_t slot_of(const ArcView& V, uint64_t a) { return V.slot ? V.slot[a] : a; }
__device__ __forceinline__ uint64_t out_off(const ArcView& V, uint64_t pos) {
    return V.slot ? (uint64_t)V.slot[pos >> 14] * kBlock + (pos & (kBlock - 1)) : pos;
}

// Are the bytes [s, e) (absolute, at most 32 of them) final?  The local pass
// writes every block's pending-byte bitmap; a clear bit means a final byte.
// The loads are acquire loads: a lane that sees its piece's source bits clear
// is ordered after the release that cleared them, and the warp barrier before
// a copy by other lanes carries that order to them (no fence per attempt).
// At most two bitmap words, possibly of two blocks: both are loaded before
// either is tested.
__device__ __forceinline__ bool src_final(const ArcView& V, uint64_t s, uint64_t e) {
    const uint64_t l = e - 1;
    const uint64_t s0 = slot_of(V, s >> 14), s1 = slot_of(V, l >> 14);
    if (s0 == kNoSlot || s1 == kNoSlot) return false;  // not in this decode's output: never final
    const uint32_t o0 = (uint32_t)(s & (kBlock - 1)), o1 = (uint32_t)(l & (kBlock - 1));
    const uint32_t* p0 = V.pmap + s0 * (kBlock / 32) + (o0 >> 5);
    const uint32_t* p1 = V.pmap + s1 * (kBlock / 32) + (o1 >> 5);
    const uint32_t lo0 = 0xffffffffu << (o0 & 31);         // bits from o0 on in its word
    const uint32_t hi1 = 0xffffffffu >> (31 - (o1 & 31));  // bits up to o1 in its word
    if (p0 == p1) return (ld_acquire_u32(p0) & lo0 & hi1) == 0;
    const uint32_t w0 = ld_acquire_u32(p0), w1 = ld_acquire_u32(p1);
    return ((w0 & lo0) | (w1 & hi1)) == 0;
}

// One CTA per SM: grid barriers stay cheap, and more warps are no faster (768 x 2
// and 1024 x 2 threads per SM: 1178 and 1338 us on 11 M text pieces, against
// 1108): the pass is bound by the memory system's latency under load.
constexpr int kExtThreads = 1024;
// Pieces a hand-out ticket of round 0 covers, about: a block's pieces are cut
// into as many equal parts as that takes on average over the job.  Handed out
// by whole blocks, a text block's 900 pieces run on one warp, a small file
// leaves most warps without work, and a large one has all of its blocks in
// flight at once, so that chains between them clog the lanes; in parts, the
// pieces in flight are a narrow window of the output, and a wait without limit
// pays at every size.  Zipf text: 1 MiB 195 -> 35 us, 4 MiB 238 -> 55, 16 MiB
// 242 -> 82, 64 MiB 418 -> 295, 200 MiB 1091 (in level order) -> 750; DNA-like
// 4 MiB 43 -> 34, 64 MiB 70 -> 59.  With parts of 32 / 48 / 96 / 128 pieces the
// 200 MiB text takes 881 / 772 / 758 / 832 us, and DNA-like 64 MiB 61 / 59 / 74 / 72.
constexpr uint32_t kPartPieces = 64;

// Are the bytes a piece reads final?  (period 0: [src, src+len); otherwise the
// residues phase.. of the period window [src, src+period), one or two ranges.)
__device__ __forceinline__ bool piece_final(const ArcView& V, uint64_t src, uint32_t phase, uint32_t period,
                                            uint32_t len) {
    uint32_t lo = 0, hi = len, wrap = 0;  // [src + lo, src + hi), then [src, src + wrap)
    if (period) {
        lo = len >= period ? 0 : phase;
        hi = len >= period ? period : min(phase + len, period);
        wrap = len >= period || phase + len <= period ? 0 : phase + len - period;
    }
    return src_final(V, src + lo, src + hi) && (wrap == 0 || src_final(V, src, src + wrap));
}

constexpr int kSlowBatch = 4;  // byte-copied pieces whose loads are in flight together

// Copy len <= 32 bytes from sa to da, any alignments, by one lane: the aligned
// 16-byte words that hold the source bytes (three at most), a barrel shift to
// the destination's 8-byte words, whole words as 8-byte stores, and the ragged
// ends as a 1-, a 2- and a 4-byte store each, as far as they need them.  Only
// words that hold a source byte are read, only the len bytes are written.  (A
// warp's 32 pieces take about 600 instructions in all; moved a byte per lane,
// a piece at a time, they took 1,340, and the output-order pass over 64 MiB of
// text 474 us instead of 426.)
__device__ __forceinline__ void copy_piece(const uint8_t* sa, uint8_t* da, uint32_t len) {
    const uint32_t off = (uint32_t)(uintptr_t)sa & 15, d0 = (uint32_t)(uintptr_t)da & 7, E = d0 + len;
    const uint4* S = reinterpret_cast<const uint4*>(sa - off);
    const uint4 z = make_uint4(0, 0, 0, 0);
    const uint4 a = __ldcg(S), b = off + len > 16 ? __ldcg(S + 1) : z, c = off + len > 32 ? __ldcg(S + 2) : z;
    // w: the source from 8 bytes before S; the destination's word 0 starts at
    // byte e of it
    uint32_t w[18] = {0, 0, a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w, c.x, c.y, c.z, c.w, 0, 0, 0, 0};
    const uint32_t e = off + 8 - d0, q = e >> 2, sh = 8 * (e & 3);
#pragma unroll
    for (int i = 0; i < 14; i++) w[i] = q & 4 ? w[i + 4] : w[i];
#pragma unroll
    for (int i = 0; i < 12; i++) w[i] = q & 2 ? w[i + 2] : w[i];
#pragma unroll
    for (int i = 0; i < 11; i++) w[i] = q & 1 ? w[i + 1] : w[i];
#pragma unroll
    for (int i = 0; i < 10; i++) w[i] = __funnelshift_r(w[i], w[i + 1], sh);
    uint8_t* D = da - d0;
    uint32_t p = d0;  // up to the next 8-byte boundary
    if ((p & 1) && p + 1 <= E) {
        D[p] = (uint8_t)((p & 4 ? w[1] : w[0]) >> (8 * (p & 3)));
        p += 1;
    }
    if ((p & 2) && p + 2 <= E) {
        *reinterpret_cast<uint16_t*>(D + p) = (uint16_t)((p & 4 ? w[1] : w[0]) >> (8 * (p & 3)));
        p += 2;
    }
    if ((p & 4) && p + 4 <= E) {
        *reinterpret_cast<uint32_t*>(D + p) = w[1];
        p += 4;
    }
    uint32_t t0 = w[0], t1 = w[1];  // the word that holds byte p
#pragma unroll
    for (int k = 0; k < 5; k++) {
        if (p >= 8u * k) {
            t0 = w[2 * k];
            t1 = w[2 * k + 1];
        }
        if (p == 8u * k && p + 8 <= E) {
            *reinterpret_cast<uint2*>(D + 8 * k) = make_uint2(t0, t1);
            p += 8;
        }
    }
    if (p + 4 <= E) {
        *reinterpret_cast<uint32_t*>(D + p) = t0;
        p += 4;
    }
    if (p + 2 <= E) {
        *reinterpret_cast<uint16_t*>(D + p) = (uint16_t)((p & 4 ? t1 : t0) >> (8 * (p & 3)));
        p += 2;
    }
    if (p < E) D[p] = (uint8_t)((p & 4 ? t1 : t0) >> (8 * (p & 3)));
}

// A warp's attempt at its lanes' pieces (lane `has` a piece `rec` of the
// block in output slot `dslot`, of archive L).  Each lane checks its own
// piece and copies it when it is ready; after one fence (the release) the
// lanes clear the pieces' pending bits with relaxed atomic ANDs.  Returns true
// on the lanes whose piece is done.
//
// Periodic pieces, pieces whose last 16-byte source word would end beyond the
// output and, in jobs with slots, pieces whose source crosses a block boundary
// go by bytes: their owners publish them in shared memory and the warp walks
// them, lane i moving byte i.
__device__ __forceinline__ bool try_pieces(bool has, const ArcView& L, uint32_t dslot, SpanRec rec, SpanRec* wrec,
                                           uint64_t* wdst, int lane) {
    const uint64_t src = (uint64_t)rec.x | ((uint64_t)(rec.y & 0xff) << 32);
    const uint32_t phase = (rec.y >> 8) & 0xffff, period = rec.w, o = rec.z & 0xffff, len = rec.z >> 16;
    const bool ready = has && piece_final(L, src, phase, period, len);
    const uint32_t rmask = __ballot_sync(ACX_FULL, ready);
    if (!rmask) return false;
    uint8_t* g = L.out;
    uint8_t* dst = g + (uint64_t)dslot * kBlock + o;
    const bool words = ready && period == 0 && (L.slot ? (src >> 14) == ((src + len - 1) >> 14)
                                                      : ((src + len + 15) & ~15ull) <= L.total);
    if (words) copy_piece(g + out_off(L, src), dst, len);
    const uint32_t smask = __ballot_sync(ACX_FULL, ready && !words);
    if (smask) {
        uint64_t* wsa = reinterpret_cast<uint64_t*>(wrec);       // [rank]: source address (jobs with slots: position)
        uint64_t* wda = reinterpret_cast<uint64_t*>(wrec) + 32;  // [rank]: destination address
        uint32_t* wln = reinterpret_cast<uint32_t*>(wdst);       // [rank]: length | phase << 8
        uint32_t* wpp = wln + 32;                                 // [rank]: period | M << 16
        if (ready && !words) {
            const uint32_t r = __popc(smask & ((1u << lane) - 1));
            wsa[r] = L.slot ? src : (uint64_t)(g + src);
            wda[r] = (uint64_t)dst;
            wln[r] = len | phase << 8;
            // a period below 32 takes the residue by a multiply-shift: for
            // x < 64, (x * ceil(2048 / p)) >> 11 is floor(x / p)
            wpp[r] = period | (period && period < 32 ? ((2047 + period) / period) << 16 : 0u);
        }
        __syncwarp();
        const uint32_t ns = __popc(smask);
        // byte k of a periodic piece reads (phase + k) mod period of its window
        // (phase < period, so with a period of 32 or more one subtraction does)
        for (uint32_t b0 = 0; b0 < ns; b0 += kSlowBatch) {
            uint32_t v = 0;
            bool mine[kSlowBatch];
#pragma unroll
            for (int u = 0; u < kSlowBatch; u++) {
                const uint32_t i = (b0 + u) & 31;
                const uint32_t a = wln[i], pp = wpp[i];
                const uint32_t per = pp & 0xffff, M = pp >> 16, x = (uint32_t)lane + (a >> 8);
                const uint32_t k = M ? x - per * ((x * M) >> 11) : (per && x >= per ? x - per : x);
                mine[u] = b0 + u < ns && (uint32_t)lane < (a & 0xff);
                const uint64_t q = wsa[i] + k;
                if (mine[u])
                    v |= (uint32_t)__ldcg(L.slot ? g + out_off(L, q) : reinterpret_cast<const uint8_t*>(q)) << (8 * u);
            }
#pragma unroll
            for (int u = 0; u < kSlowBatch; u++)
                if (mine[u]) reinterpret_cast<uint8_t*>(wda[(b0 + u) & 31])[lane] = (uint8_t)(v >> (8 * u));
        }
    }
    // release: every lane's stores (to other lanes' pieces too) happen before
    // the warp's fence, and the fence before any owner clears its bits
    __syncwarp();
    fence_acq_rel_gpu();
    if (ready) {
        uint32_t* pm = L.pmap + (uint64_t)dslot * (kBlock / 32);
        for (uint32_t w = o >> 5; w <= ((o + len - 1) >> 5); w++) red_and_relaxed(pm + w, ~range_mask(w, o, o + len));
    }
    __syncwarp();
    return ready;
}

// Grid-wide barrier of a cooperative launch (every CTA resident): bounded
// wait; the last CTA to arrive clears the count `reset` before it releases
// the others.  Returns false when the wait ran out.
__device__ bool grid_barrier(uint32_t* counters, uint32_t reset, uint64_t deadline) {
    __syncthreads();
    __shared__ int ok_s;
    if (threadIdx.x == 0) {
        ok_s = 1;
        const uint32_t gen = ld_acquire_u32(counters + kBarGen);
        __threadfence();
        if (atomicAdd(counters + kBarCount, 1u) == gridDim.x - 1) {
            counters[kBarCount] = 0;
            counters[reset] = 0;
            __threadfence();
            atomicAdd(counters + kBarGen, 1u);
        } else {
            uint32_t spins = 0;
            while (ld_acquire_u32(counters + kBarGen) == gen) {
                __nanosleep(32);
                if ((++spins & 255) == 0 && gtimer() > deadline) { ok_s = 0; break; }
            }
        }
    }
    __syncthreads();
    return ok_s != 0;
}

// Appends to a work list go through a per-warp staging buffer in shared
// memory: the list's count is one word that every warp of the grid would
// otherwise hit with an atomic at every step, so a warp reserves space for
// kStage entries at a time.  `sn` (warp-uniform) counts the staged entries.
typedef JobDev::ListEnt ListEnt;
constexpr uint32_t kStage = 64;
__device__ __forceinline__ void stage_flush(ListEnt* buf, uint32_t& sn, ListEnt* list, uint32_t* cnt, int lane) {
    if (sn == 0) return;
    __syncwarp();
    uint32_t base = 0;
    if (lane == 0) base = atomicAdd(cnt, sn);
    base = __shfl_sync(ACX_FULL, base, 0);
    for (uint32_t i = lane; i < sn; i += 32) list[base + i] = buf[i];
    __syncwarp();
    sn = 0;
}
__device__ __forceinline__ void append(bool keep, ListEnt e, ListEnt* buf, uint32_t& sn, ListEnt* list, uint32_t* cnt,
                                       int lane) {
    const uint32_t m = __ballot_sync(ACX_FULL, keep);
    if (!m) return;
    if (sn + __popc(m) > kStage) stage_flush(buf, sn, list, cnt, lane);
    if (keep) buf[sn + __popc(m & ((1u << lane) - 1))] = e;
    sn += __popc(m);
}

// Round trace (diagnostics): work-list size and start time (ns) of every round.
__device__ __forceinline__ void trace_round(const JobDev& job, uint32_t round, uint32_t n) {
    if (round >= kTraceRounds) return;
    job.counters[kTrace + 3 * round] = n;
    const uint64_t t = gtimer();
    job.counters[kTrace + 3 * round + 1] = (uint32_t)t;
    job.counters[kTrace + 3 * round + 2] = (uint32_t)(t >> 32);
}

// A round that finished no piece.  In a valid archive the lowest pending
// piece always has final sources (every source precedes its destination), so
// the pieces left wait on bytes that no piece writes: their archives are
// corrupt.
__device__ void report_stalled(const JobDev& job, uint32_t in, uint32_t n, uint32_t w0, uint32_t nw, int lane) {
    for (uint32_t i = w0 * 32 + lane; i < n; i += nw * 32) {
        const ListEnt e = job.lists[in][i];
        const int a = find_arc(job, e.y);
        const ArcJob J = load_arc(job, a);
        set_err_arc(job, a, kErrCorrupt, kStageSources << 24, item_ref(J, e.y - J.item_base).blk);
    }
}

// One pass over a list of n pieces by warps w0, w0 + nw, ...: every piece is
// attempted once; the unfinished ones go to work list `out`.
template <bool kMulti>
__device__ void round_pass(const JobDev& job, const ListEnt* src, uint32_t out, uint32_t n, uint32_t w0, uint32_t nw,
                           SpanRec* wrec, uint64_t* wdst, ListEnt* sbuf, int lane) {
    uint32_t sn = 0;
    for (uint32_t i0 = w0 * 32; i0 < n; i0 += nw * 32) {
        const uint32_t i = i0 + lane;
        const bool has = i < n;
        ListEnt e{0, 0};
        if (has) e = src[i];
        const ArcJob& J = kMulti ? job.arcs[has ? find_arc(job, e.y) : 0] : job.one;
        SpanRec r{0, 0, 0, 0};
        if (has) r = J.spans[e.x];
        const uint32_t slot = has ? item_ref(J, e.y - J.item_base).slot : 0;
        const bool done = try_pieces(has, view_of(J), slot, r, wrec, wdst, lane);
        append(has && !done, e, sbuf, sn, job.lists[out], &job.counters[kListCnt + out], lane);
    }
    stage_flush(sbuf, sn, job.lists[out], &job.counters[kListCnt + out], lane);
}

// The last rounds on one CTA (the other CTAs have left): list `in` holds n
// entries and the count of the other list is zero.  Rounds are separated by
// CTA barriers; the same progress argument as the grid rounds ends them.
constexpr uint32_t kSoloMax = 4 * kExtThreads;  // lists up to four CTA-wide passes
template <bool kMulti>
__device__ void solo_rounds(const JobDev& job, uint32_t in, uint32_t n, uint32_t round, uint64_t deadline,
                            SpanRec* wrec, uint64_t* wdst, ListEnt* sbuf, int lane) {
    __shared__ uint32_t n_next;
    const uint32_t warp = threadIdx.x >> 5, nw = kExtThreads / 32;
    for (;;) {
        const uint32_t out = in ^ 1u;
        round_pass<kMulti>(job, job.lists[in], out, n, warp, nw, wrec, wdst, sbuf, lane);
        __syncthreads();  // every append of this round is visible to the CTA
        if (threadIdx.x == 0) {
            n_next = *((volatile uint32_t*)&job.counters[kListCnt + out]);
            job.counters[kListCnt + in] = 0;  // list `in` becomes the next output
            trace_round(job, ++round, n_next);
            if (n_next) atomicAdd(&job.counters[kStatPolls], 1u);
        }
        __syncthreads();
        const uint32_t m = n_next;
        if (m == 0) return;
        if (m == n) {
            report_stalled(job, out, m, warp, nw, lane);
            return;
        }
        if (__syncthreads_or(gtimer() > deadline)) {
            if (threadIdx.x == 0) set_err(job.err, kErrTimeout, kStageWait << 24, 0);
            return;
        }
        in = out;
        n = m;
    }
}

// The level list of a level-ordered decode (whole single-archive jobs with
// kJobLevels), built between the local pass and the cross-block pass, so
// that round l walks a contiguous segment with one piece per lane however
// unevenly the level's pieces are spread over the blocks.
//   lvl_off[(l-1) * n + b]: offset of item b's level-l pieces in level l's
//     segment (k_level_scan: one CTA per level, an exclusive scan over items);
//   lvl_off[Lg * n + l - 1]: level l's total; lvl_off[Lg * n + Lg + l - 1]:
//     its segment's base (l = 1 .. Lg + 1, the last being the list's length);
//   lvl_list[base(l) + offset + k] = {span slot, item} of the item's k-th
//     level-l piece in output order (k_level_fill: one warp per item, reading
//     each piece's level from its record).
constexpr int kScanThreads = 1024;
// A decode whose local pass timed out left blocks unprocessed, so their level
// rows, piece counts and records may be stale: the passes after it do nothing.
__device__ __forceinline__ bool local_pass_timed_out(const JobDev& job) {
    return *((volatile const int*)job.err) == kErrTimeout;
}

__global__ void __launch_bounds__(kScanThreads) k_level_scan(JobDev job) {
    __shared__ uint32_t wsum[kScanThreads / 32];
    if (local_pass_timed_out(job)) return;
    const uint32_t l = blockIdx.x + 1, Lg = job.n_levels, n = job.n_items;
    const uint32_t per = (n + kScanThreads - 1) / kScanThreads;
    const uint32_t i0 = min(n, threadIdx.x * per), i1 = min(n, i0 + per);
    auto cnt = [&](uint32_t b) {
        const uint32_t* row = job.lvl_tab + (uint64_t)(job.one.lo + b) * (Lg + 1);
        return row[l] - row[l - 1];
    };
    uint32_t s = 0;
    for (uint32_t b = i0; b < i1; b++) s += cnt(b);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    uint32_t inc = s;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(ACX_FULL, inc, o);
        if (lane >= o) inc += y;
    }
    if (lane == 31) wsum[warp] = inc;
    __syncthreads();
    uint32_t pre = 0, tot = 0;
    for (int w = 0; w < kScanThreads / 32; w++) {
        if (w < warp) pre += wsum[w];
        tot += wsum[w];
    }
    uint32_t off = pre + inc - s;
    uint32_t* out = job.lvl_off + (uint64_t)(l - 1) * n;
    for (uint32_t b = i0; b < i1; b++) {
        out[b] = off;
        off += cnt(b);
    }
    if (threadIdx.x == 0) job.lvl_off[(uint64_t)Lg * n + (l - 1)] = tot;  // level l's total
}

__global__ void __launch_bounds__(256) k_level_fill(JobDev job) {
    __shared__ uint32_t base[kMaxLevel + 1];
    __shared__ uint32_t cursor[8][kMaxLevel + 1];  // per warp: the block's entries written so far, per level
    if (local_pass_timed_out(job)) return;
    const uint32_t Lg = job.n_levels, n = job.n_items;
    const uint32_t* tot = job.lvl_off + (uint64_t)Lg * n;
    if (threadIdx.x == 0) {
        uint32_t c = 0;
        for (uint32_t l = 1; l <= Lg; l++) {
            base[l - 1] = c;
            c += tot[l - 1];
        }
        base[Lg] = c;
    }
    __syncthreads();
    if (blockIdx.x == 0)  // segment bases, read by the cross-block pass
        for (uint32_t l = threadIdx.x; l <= Lg; l += blockDim.x)
            job.lvl_off[(uint64_t)Lg * n + Lg + l] = base[l];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const uint32_t lt = (1u << lane) - 1;
    uint32_t* cur = cursor[warp];
    const uint32_t nw = gridDim.x * (blockDim.x >> 5);
    for (uint32_t b = blockIdx.x * (blockDim.x >> 5) + warp; b < n; b += nw) {
        const uint32_t blk = job.one.lo + b;
        const uint32_t* row = job.lvl_tab + (uint64_t)blk * (Lg + 1);
        const uint32_t total = row[Lg];
        if (total == 0) continue;  // no pending pieces
        const BlockDev& bd = job.one.blk[blk];
        const uint32_t sb = bd.span_base;
        if (total > bd.n_tok + kSpanSlack) {  // more pieces than the block's slots: not this decode's row
            if (lane == 0) set_err(job.err, kErrCorrupt, kStageLimits << 24, blk);
            continue;
        }
        for (uint32_t l = lane; l <= Lg; l += 32) cur[l] = 0;
        __syncwarp();
        // the block's pieces in output order, each to its level's segment
        bool bad = false;
        for (uint32_t k0 = 0; k0 < total; k0 += 32) {
            const uint32_t k = k0 + lane;
            const bool has = k < total;
            const uint32_t l = has ? min(max(job.one.spans[sb + k].y >> 24, 1u), Lg) : 0u;
            const uint32_t peers = __match_any_sync(ACX_FULL, has ? l : 0xffffffffu);
            if (has) {
                const uint32_t r = cur[l] + __popc(peers & lt);
                const uint64_t at = (uint64_t)base[l - 1] + job.lvl_off[(uint64_t)(l - 1) * n + b] + r;
                if (r >= row[l] - row[l - 1] || at >= job.lvl_cap) bad = true;
                else job.lvl_list[at] = JobDev::ListEnt{sb + k, b};
            }
            __syncwarp();
            if (has && (peers & lt) == 0) cur[l] += __popc(peers);  // the group's first lane
            __syncwarp();
        }
        if (__any_sync(ACX_FULL, bad) && lane == 0) set_err(job.err, kErrCorrupt, kStageLimits << 24, blk);
    }
}

cudaError_t launch_level_list(const JobDev& job, cudaStream_t st) {
    const cudaError_t e = launch_kernel(k_level_scan, job.n_levels, kScanThreads, 0, st, job);
    if (e != cudaSuccess) return e;
    const uint32_t grid = std::max(1u, std::min(4096u, (job.n_items + 7) / 8));
    return launch_kernel(k_level_fill, grid, 256, 0, st, job);
}

// Cross-block pass.  Round 0 hands the pieces out in order and a lane waits a
// while for sources that lower pieces are about to finish; each later round
// walks the pieces the previous one could not finish, every piece attempted
// once, so it needs no ordering argument: every round finishes at least the
// lowest pending piece (its sources are final), and the number of rounds is
// bounded by the depth of the cross-block dependency chains.  Pieces finished
// earlier in the same round are visible to later ones.  Rounds are separated
// by a grid barrier (cooperative launch).
template <bool kMulti>
__global__ void __launch_bounds__(kExtThreads) k_external(JobDev job) {
    __shared__ SpanRec recs[kExtThreads];
    __shared__ uint64_t dsts[kExtThreads];
    __shared__ ListEnt stage[kExtThreads / 32][kStage];
    SpanRec* wrec = recs + (threadIdx.x & ~31u);
    uint64_t* wdst = dsts + (threadIdx.x & ~31u);
    ListEnt* sbuf = stage[threadIdx.x >> 5];
    const int lane = threadIdx.x & 31;
    const uint32_t gwarp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const uint32_t nwarps = (gridDim.x * blockDim.x) >> 5;
    const uint64_t deadline = gtimer() + job.timeout_ns;
    if (local_pass_timed_out(job)) return;  // (every CTA returns: no barrier is entered)
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        const uint64_t t = gtimer();
        job.counters[kTrace] = 0;
        job.counters[kTrace + 1] = (uint32_t)t;
        job.counters[kTrace + 2] = (uint32_t)(t >> 32);
    }
    const uint64_t pieces = *((volatile const uint32_t*)&job.counters[kStatPending]);
    if (pieces == 0) return;  // (every CTA reads the same final count)
    // round 0: pieces handed out in order; a lane waits for the sources that
    // lower pieces are about to finish, without limit unless wait_ns sets one:
    // then it defers its piece to the rounds below.  The order is the output
    // order (warps take parts of blocks from a ticket, idle lanes take the
    // part's next pieces), or, for a level-ordered job, the level list's (warps
    // take 32 entries at a time): every level's pieces come after all pieces of
    // the levels below, so with true level hints a lane only waits for pieces
    // already handed out (the paper's waves, without a barrier between them).
    {
        const bool lv = !kMulti && job.lvl_tab;
        const uint64_t wait_ns = job.wait_ns == 0 || job.wait_ns == 0xffffffffu ? ~0ull : job.wait_ns;
        uint32_t spins = 0, nap = 64;
        uint32_t sn0 = 0;  // entries staged for list 0
        uint64_t t0 = 0;   // start of the lane's wait (0: its piece has not been refused yet)
        // after an attempt that left the lanes `has` waiting: pieces that have
        // waited too long go to the rounds; a warp without progress naps.
        // Returns false when the deadline has passed.
        auto settle = [&](bool& has, bool progressed, uint32_t span, uint32_t item) -> bool {
            bool giveup = false;
            if (has) {
                const uint64_t now = gtimer();
                if (t0 == 0) t0 = now;
                giveup = now - t0 > wait_ns;
            }
            append(giveup, ListEnt{span, item}, sbuf, sn0, job.lists[0], &job.counters[kListCnt], lane);
            if (giveup) has = false;
            if (__any_sync(ACX_FULL, progressed || giveup)) {
                spins = 0;
                nap = 64;
                return true;
            }
            __nanosleep(nap);
            if (wait_ns == ~0ull) nap = min(2 * nap, 1024u);  // long waits: fewer polls of the bitmaps
            if ((++spins & 255) == 0 && __any_sync(ACX_FULL, gtimer() > deadline)) {
                if (lane == 0) {
                    const ArcJob& J = kMulti ? job.arcs[find_arc(job, item)] : job.one;
                    set_err_arc(job, kMulti ? find_arc(job, item) : 0, kErrTimeout, kStageWait << 24,
                                item_ref(J, item - J.item_base).blk);
                }
                return false;
            }
            return true;
        };
        uint32_t n_lv = 0;
        if (lv) {
            n_lv = job.lvl_off[(uint64_t)job.n_levels * job.n_items + 2 * job.n_levels];  // the list's length
            if (n_lv > job.lvl_cap) {
                if (threadIdx.x == 0) set_err(job.err, kErrCorrupt, kStageLimits << 24, 0);
                n_lv = 0;
            }
        }
        const uint64_t per_part = (uint64_t)job.n_items * kPartPieces;
        const uint32_t parts = (uint32_t)max((pieces + per_part - 1) / per_part, (uint64_t)1);
        const uint64_t n_tickets = (uint64_t)job.n_items * parts;
        uint32_t dsl = 0, cnt = 0, next = 0, base = 0, item = 0;
        bool exhausted = false, has = false;
        const ArcJob* J = &job.one;
        ArcView V = view_of(job.one);  // of the lane's piece
        SpanRec rec{0, 0, 0, 0};
        uint32_t l_dsl = 0, l_span = 0, l_item = 0;
        const uint32_t lt_mask = (1u << lane) - 1;
        for (;;) {
            uint32_t idle = __ballot_sync(ACX_FULL, !has);
            while (idle && !exhausted) {
                if (next >= cnt) {
                    // a level-ordered job: chunk t * kLvStripes + k of 32 entries
                    // from stripe k's counter, so that the hand-out is not one
                    // counter's atomics in a row (the order stays the list's, up to
                    // how far the stripes drift apart; every CTA has warps on every
                    // stripe).  Otherwise part t % parts of block t / parts.
                    const uint32_t k = (threadIdx.x >> 5) & (kLvStripes - 1);
                    uint32_t t = 0;
                    if (lane == 0) t = atomicAdd(&job.counters[lv ? kLvTickets + k : 2], 1u);
                    t = __shfl_sync(ACX_FULL, t, 0);
                    next = 0;
                    if (lv) {
                        base = (t * kLvStripes + k) * 32;
                        if (base >= n_lv) { exhausted = true; break; }
                        cnt = min(32u, n_lv - base);
                        continue;
                    }
                    if (t >= n_tickets) { exhausted = true; break; }
                    item = t / parts;
                    const uint32_t part = t - item * parts;
                    if (kMulti) J = job.arcs + find_arc(job, item);
                    const ItemRef ir = item_ref(*J, item - J->item_base);
                    dsl = ir.slot;
                    base = ir.span_base;
                    const uint64_t n = J->npend[dsl];
                    next = (uint32_t)(n * part / parts);
                    cnt = (uint32_t)(n * (part + 1) / parts);
                    continue;
                }
                const uint32_t avail = cnt - next;
                const uint32_t r = __popc(idle & lt_mask);
                if ((idle >> lane & 1) && r < avail) {
                    if (lv) {
                        const ListEnt e = job.lvl_list[base + next + r];
                        l_span = e.x;
                        l_item = e.y;
                        l_dsl = J->lo + e.y;  // a whole-archive job: item i is block lo + i, in slot lo + i
                    } else {
                        l_span = base + next + r;
                        l_item = item;
                        l_dsl = dsl;
                    }
                    if (kMulti) V = view_of(*J);
                    rec = J->spans[l_span];
                    t0 = 0;
                    has = true;
                }
                next += min(avail, (uint32_t)__popc(idle));
                idle = __ballot_sync(ACX_FULL, !has);
            }
            if (!__any_sync(ACX_FULL, has)) break;
            const bool done = try_pieces(has, V, l_dsl, rec, wrec, wdst, lane);
            if (done) has = false;
            if (__any_sync(ACX_FULL, has) && !settle(has, done, l_span, l_item)) break;
        }
        stage_flush(sbuf, sn0, job.lists[0], &job.counters[kListCnt], lane);
    }
    uint32_t n_prev = 0xffffffffu;
    for (uint32_t round = 1;; round++) {
        const uint32_t in = (round - 1) & 1, out = round & 1;
        if (!grid_barrier(job.counters, kListCnt + out, deadline)) {
            if (threadIdx.x == 0) set_err(job.err, kErrTimeout, kStageWait << 24, 0);
            return;
        }
        const uint32_t n = *((volatile uint32_t*)&job.counters[kListCnt + in]);
        if (blockIdx.x == 0 && threadIdx.x == 0) trace_round(job, round, n);
        if (n == 0) return;
        if (n == n_prev) {
            report_stalled(job, in, n, gwarp, nwarps, lane);
            return;
        }
        n_prev = n;
        if (blockIdx.x == 0 && threadIdx.x == 0) atomicAdd(&job.counters[kStatPolls], 1u);
        if (n <= kSoloMax) {
            // a short list: one CTA finishes the remaining rounds with CTA
            // barriers instead of grid barriers
            if (blockIdx.x == 0) solo_rounds<kMulti>(job, in, n, round, deadline, wrec, wdst, sbuf, lane);
            return;
        }
        round_pass<kMulti>(job, job.lists[in], out, n, gwarp, nwarps, wrec, wdst, sbuf, lane);
    }
}

size_t local_smem_bytes(uint32_t T, uint32_t LB, uint32_t LIT, bool need, bool lvl) {
    return loc_layout(T, LB, LIT, need, lvl).total;
}

// CTAs of smem bytes of workspace that an SM's shared memory holds.
static int local_fit(size_t smem) { return (int)(kMaxSmem / (smem + 1024)); }

// Threads of a local CTA for a job of n_items blocks of up to T tokens whose
// workspace has `smem` bytes.  A CTA's shared memory sets how many fit an SM:
// with four or fewer (blocks of some 900 tokens and more), 128 threads leave
// most of the SM's issue slots empty (200 MiB text: 487 us; 256 threads 461, and
// 357 since four of them fit; a batch of 96 files 936 -> 825), with five or six they fill it (254 MB genome:
// 322 us; 256 threads 420).  A job of few blocks has every block on an SM at
// once, so only a block's latency counts: 256 threads, or 512 for blocks of
// many tokens (4 MiB DNA-like 34 -> 27 us; 4 MiB text 97 -> 73 -> 60 with 128,
// 256, 512 threads; one 10 KB text block 62 -> 43 -> 35).
static int local_threads(size_t smem, uint32_t n_items, uint32_t T) {
    if (n_items <= 2u * (uint32_t)noted_sm_count()) return T > 256 ? kLocWidest : kLocWide;
    return local_fit(smem) <= 4 ? kLocWide : kLocThreads;
}

bool local_narrow(size_t smem) { return local_threads(smem, 0xffffffffu, 0) == kLocThreads; }

template <int NT, Loc kKind, int kCtas>
static cudaError_t local_attrs() {
    cudaError_t e = allow_max_smem(k_local<NT, kKind, kCtas>);
    if (e == cudaSuccess)  // the whole unified L1 as shared memory: CTAs per SM are set by their workspaces
        e = cudaFuncSetAttribute(k_local<NT, kKind, kCtas>, cudaFuncAttributePreferredSharedMemoryCarveout,
                                 cudaSharedmemCarveoutMaxShared);
    return e;
}

template <int NT, Loc kKind, int kCtas>
static cudaError_t launch_local_ctas(const JobDev& job, int grid, size_t smem, cudaStream_t st) {
    const cudaError_t e = local_attrs<NT, kKind, kCtas>();
    if (e != cudaSuccess) return e;
    return launch_dependent(k_local<NT, kKind, kCtas>, grid, NT, smem, st, job);
}
template <int NT, Loc kKind>
static cudaError_t launch_local_kind(const JobDev& job, int grid, size_t smem, cudaStream_t st) {
    if constexpr (NT == kLocWide) {
        if (kKind == Loc::kAny || local_fit(smem) < kLocCtas<NT>)
            return launch_local_ctas<NT, kKind, 3>(job, grid, smem, st);
    }
    if constexpr (NT != kLocWide || kKind != Loc::kAny)
        return launch_local_ctas<NT, kKind, kLocCtas<NT>>(job, grid, smem, st);
}

template <int NT>
static cudaError_t launch_local_nt(const JobDev& job, int grid, size_t smem, cudaStream_t st) {
    // (a batch's archives have no item tables)
    if (job.flags == 0 && !job.ready && job.arcs) return launch_local_kind<NT, Loc::kBatch>(job, grid, smem, st);
    if (job.flags == 0 && !job.ready && !job.one.items) return launch_local_kind<NT, Loc::kOne>(job, grid, smem, st);
    return launch_local_kind<NT, Loc::kAny>(job, grid, smem, st);
}

cudaError_t launch_local(const JobDev& job_in, int grid, cudaStream_t st) {
    JobDev job = job_in;
    if (job.loc_hi == 0) {  // one pass over all items
        job.loc_hi = job.n_items;
        job.loc_ctr = 1;
    }
    const size_t sm = local_smem_bytes(job.max_tok, job.max_lenb, job.max_lit, (job.flags & kJobNeed) != 0,
                                       (job.flags & kJobLevels) != 0);
    // a small job (a seek, a serving tick) needs no more CTAs than ticket runs
    const uint32_t items = job.loc_hi - job.loc_lo;
    const uint64_t runs = (items + (uint64_t)(job.chunk ? job.chunk : 1) - 1) / (job.chunk ? job.chunk : 1);
    grid = job_grid(grid, runs);
    const int nt = local_threads(sm, items, job.max_tok);
    return nt == kLocWidest ? launch_local_nt<kLocWidest>(job, grid, sm, st)
           : nt == kLocWide ? launch_local_nt<kLocWide>(job, grid, sm, st)
                            : launch_local_nt<kLocThreads>(job, grid, sm, st);
}

// Cooperative launches (the cross-block pass, the fused decode) run one at a
// time on a device.  A cooperative grid waits at its grid barriers (and its
// lanes on one another's pieces) for CTAs that must all be resident; two such
// grids launched on different streams, each holding part of the SMs, could
// wait for CTAs that cannot start until the other grid ends.  So every
// cooperative launch of the process waits for the completion event of the
// previous one on the same device and records it anew.  A stream that is
// being captured into a graph is left alone (its graph runs its passes on one
// stream).
namespace {
std::mutex g_coop_mu;
constexpr int kCoopDevices = 64;
cudaEvent_t g_coop_ev[kCoopDevices] = {};
}  // namespace

cudaError_t coop_ordered(cudaStream_t st, cudaError_t (*launch)(void*), void* arg) {
    cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
    cudaError_t e = cudaStreamIsCapturing(st, &cs);
    if (e != cudaSuccess) return e;
    int dev = 0;
    if (cs != cudaStreamCaptureStatusNone || cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kCoopDevices)
        return launch(arg);
    std::lock_guard<std::mutex> g(g_coop_mu);
    cudaEvent_t& ev = g_coop_ev[dev];
    if (!ev) {
        if ((e = cudaEventCreateWithFlags(&ev, cudaEventDisableTiming)) != cudaSuccess) {
            ev = nullptr;
            return e;
        }
    } else if ((e = cudaStreamWaitEvent(st, ev, 0)) != cudaSuccess) {
        return e;
    }
    if ((e = launch(arg)) != cudaSuccess) return e;
    return cudaEventRecord(ev, st);
}

cudaError_t launch_external(const JobDev& job, int grid, cudaStream_t st) {
    struct Arg {
        const JobDev* job;
        int grid;
        cudaStream_t st;
    } a{&job, grid, st};
    return coop_ordered(st, [](void* p) -> cudaError_t {
        const Arg* a = static_cast<const Arg*>(p);
        cudaLaunchConfig_t cfg{};
        // two CTAs a block take all of its parts at once
        cfg.gridDim = dim3((uint32_t)std::min<uint64_t>((uint64_t)a->grid, 2ull * a->job->n_items));
        cfg.blockDim = dim3(kExtThreads);
        cfg.dynamicSmemBytes = 0;
        cfg.stream = a->st;
        cudaLaunchAttribute attr[1];
        attr[0].id = cudaLaunchAttributeCooperative;
        attr[0].val.cooperative = 1;
        cfg.attrs = attr;
        cfg.numAttrs = 1;
        return a->job->arcs ? cudaLaunchKernelEx(&cfg, k_external<true>, *a->job)
                            : cudaLaunchKernelEx(&cfg, k_external<false>, *a->job);
    }, &a);
}

template <int NT>
static int local_occupancy_nt(size_t smem) {  // (of the kind that runs most CTAs: a grid may exceed what is resident)
    int n = 0;
    if (local_attrs<NT, Loc::kOne, kLocCtas<NT>>() != cudaSuccess ||
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, k_local<NT, Loc::kOne, kLocCtas<NT>>, NT, smem) != cudaSuccess)
        return 0;
    return n;
}

int local_occupancy(size_t smem) {  // (of a job of many blocks: a small one fits an SM or two per block)
    return local_threads(smem, 0xffffffffu, 0) == kLocWide ? local_occupancy_nt<kLocWide>(smem)
                                                           : local_occupancy_nt<kLocThreads>(smem);
}

int external_occupancy() {
    int n = 0;
    int m = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, k_external<false>, kExtThreads, 0) != cudaSuccess ||
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&m, k_external<true>, kExtThreads, 0) != cudaSuccess)
        return 0;
    return std::min(n, m);
}

}  // namespace acx
