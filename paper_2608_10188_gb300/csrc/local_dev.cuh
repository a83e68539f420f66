// Device code of the local pass of the decode (paper: "parse" and the
// in-block part of "copy"), shared by k_local and the fused decode kernel.
// See assemble.cu for the pass as a whole.
#pragma once
#include "common.cuh"

namespace acx {

// Threads of a local group: 128 when a block's workspace leaves room for five
// CTAs or more per SM, else 256 or 512 (see local_threads).
constexpr int kLocThreads = 128, kLocWide = 256, kLocWidest = 512;
constexpr int kLocMaxWarps = kLocWidest / 32;

// A loop of the local pass, rolled or left to the compiler.  Six CTAs of 128
// threads, each at another point of the code, are limited by instruction
// fetch, so their loops stay rolled (254 MB genome: 242 us, with the compiler's
// unrolling 256); wider groups run longer loops on fewer blocks (200 MiB text, at
// three CTAs per SM: 447 and 421).
template <bool kRolled, class F>
__device__ __forceinline__ void each(uint32_t first, uint32_t end, uint32_t step, F f) {
    if constexpr (kRolled) {
#pragma unroll 1
        for (uint32_t i = first; i < end; i += step) f(i);
    } else {
        for (uint32_t i = first; i < end; i += step) f(i);
    }
}

struct LocLayout {
    uint32_t out, pend, tsrc, tpos, tll, tml, tlit, tcmd, tstat, lenb, soff, slit, scan, bar, misc, need, tlvl, tlvk,
        lhist, total;
};

// Shared-memory workspace of one local group for blocks of up to T tokens,
// LB length bytes and LIT literals; need: jobs with wanted-byte intervals; lvl: jobs that
// sort pieces by level (the token levels and a level histogram).
__host__ __device__ inline LocLayout loc_layout(uint32_t T, uint32_t LB, uint32_t LIT, bool need, bool lvl = false) {
    LocLayout L;
    uint32_t o = 0;
    auto take = [&](uint32_t bytes, uint32_t align) {
        o = (o + align - 1) & ~(align - 1);
        const uint32_t r = o;
        o += bytes;
        return r;
    };
    const uint32_t T16 = (T + 15) & ~15u;
    L.out = take(kBlock, 16);
    L.pend = take(kBlock / 8, 16);
    L.tsrc = take(8 * T, 16);
    L.tpos = take(2 * T, 16);
    L.tll = take(2 * T, 16);
    L.tml = take(2 * T, 16);
    L.tlit = take(2 * T, 16);
    L.tcmd = take(T16 + 16, 16);
    L.tstat = take(T16, 16);
    L.lenb = take(((LB + 15) & ~15u) + 16, 16);
    L.soff = take(((5 * T + 15) & ~15u) + 16, 16);
    L.slit = take(((LIT + 15) & ~15u) + 16, 16);
    L.scan = take(kLocMaxWarps * 3 * 4, 16);
    L.bar = take(8, 8);
    L.misc = take(64, 16);
    L.need = need ? take(kBlock / 8, 16) : 0;  // wanted-byte bitmap (jobs with kJobNeed)
    L.tlvl = lvl ? take(T16 + 16, 16) : 0;       // token levels as staged (jobs with kJobLevels)
    L.tlvk = lvl ? take(T16, 16) : 0;            // the block's token levels, kept past the next block's staging
    L.lhist = lvl ? take(4 * (kMaxLevel + 2), 16) : 0;
    L.total = (o + 127) & ~127u;
    return L;
}

// Literal runs up to this many bytes are copied by one thread (a byte at a
// time, every thread of the CTA on its own run); longer ones by eight lanes.
constexpr uint32_t kLaneBytes = 32;

// Does the match at [o, o + ml) of a block touch a wanted byte?
__device__ __forceinline__ bool wanted(const uint32_t* need, uint32_t o, uint32_t ml) {
    for (uint32_t w = o >> 5; w <= ((o + ml - 1) >> 5); w++)
        if (need[w] & range_mask(w, o, o + ml)) return true;
    return false;
}

// Barriers of one group of NT threads: named barrier `bid` (0 in k_local, where
// the group is the whole CTA; 1.. for the groups of a fused CTA).
template <int NT>
__device__ __forceinline__ void grp_sync(uint32_t bid) {
    asm volatile("bar.sync %0, %1;" ::"r"(bid), "n"(NT) : "memory");
}
template <int NT>
__device__ __forceinline__ int grp_or(uint32_t bid, int v) {
    uint32_t r;
    asm volatile(
        "{\n .reg .pred p, q;\n setp.ne.u32 q, %1, 0;\n barrier.cta.red.or.pred p, %2, %3, q;\n"
        " selp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(r)
        : "r"((uint32_t)v), "r"(bid), "n"(NT)
        : "memory");
    return (int)r;
}

// Group-wide exclusive scan of V u32 values per thread (tid: the thread in
// its group).
template <int NT, int V>
__device__ __forceinline__ void block_scan(uint32_t (&v)[V], uint32_t (&tot)[V], uint32_t* buf, uint32_t bid, int tid) {
    const int lane = tid & 31, warp = tid >> 5;
    uint32_t inc[V];
#pragma unroll
    for (int k = 0; k < V; k++) inc[k] = v[k];
#pragma unroll(NT == kLocThreads ? 1 : 5)
    for (int o = 1; o < 32; o <<= 1) {
#pragma unroll
        for (int k = 0; k < V; k++) {
            const uint32_t y = __shfl_up_sync(ACX_FULL, inc[k], o);
            if (lane >= o) inc[k] += y;
        }
    }
    if (lane == 31)
        for (int k = 0; k < V; k++) buf[warp * V + k] = inc[k];
    grp_sync<NT>(bid);
    uint32_t wpre[V], t[V];
#pragma unroll
    for (int k = 0; k < V; k++) wpre[k] = t[k] = 0;
#pragma unroll
    for (int w = 0; w < NT / 32; w++) {
#pragma unroll
        for (int k = 0; k < V; k++) {
            const uint32_t s = buf[w * V + k];
            if (w < warp) wpre[k] += s;
            t[k] += s;
        }
    }
#pragma unroll
    for (int k = 0; k < V; k++) {
        v[k] = wpre[k] + inc[k] - v[k];
        tot[k] = t[k];
    }
    grp_sync<NT>(bid);
}

// The four-entry distance history ("The Last Sequential Element") as a map
// from the history before a run of tokens to the history after it, packed in
// 64 bits: entry k (bits 16k..16k+15) is kHRef | j, "entry j of the history
// before the run", or the index in the block of the NEW token whose distance
// it holds (a block that passes the token checks has at most kBlock / 4 + 1
// tokens, so an index never reaches kHRef).  Maps compose associatively,
// which makes the history a prefix scan.
typedef uint64_t HMap;
constexpr uint32_t kHRef = 0x8000;
constexpr HMap kHIdentity = 0x8003800280018000ull;

// The map followed by token i with command cmd: a NEW token pushes its own
// distance in front; a repeat of entry j moves that entry to the front.
__device__ __forceinline__ HMap hmap_step(HMap m, uint8_t cmd, uint32_t i) {
    if (cmd == kNew) return (m << 16) | i;
    if (cmd >= 2 && cmd <= 4) {  // entry j = cmd - 1 >= 1 (a repeat of entry 0 changes nothing)
        const uint32_t s = 16 * (cmd - 1);
        const uint64_t low = m & ((1ull << s) - 1);   // entries 0 .. j-1
        const uint64_t e = (m >> s) & 0xffff;          // entry j
        const uint64_t high = s == 48 ? 0ull : m & (~0ull << (s + 16));
        return high | (low << 16) | e;
    }
    return m;
}
// (first f, then g): an entry of g that names entry j of its input takes f's entry j
__device__ __forceinline__ HMap hmap_compose(HMap f, HMap g) {
    const uint32_t flo = (uint32_t)f, fhi = (uint32_t)(f >> 32);
    uint32_t v[4];
#pragma unroll
    for (int k = 0; k < 4; k++) {
        const uint32_t x = (uint32_t)(g >> (16 * k)) & 0xffff;
        const uint32_t j = x & 3;
        const uint32_t fj = (j & 2 ? fhi : flo) >> (16 * (j & 1));
        v[k] = (x & kHRef) ? fj & 0xffff : x;
    }
    return (uint64_t)(v[0] | (v[1] << 16)) | ((uint64_t)(v[2] | (v[3] << 16)) << 32);
}

template <bool kRolled>
__device__ __forceinline__ void pend_update_smem(uint32_t* pend, uint32_t s, uint32_t e, bool set) {
    if (s >= e) return;
    each<kRolled>(s >> 5, ((e - 1) >> 5) + 1, 1, [&](uint32_t w) {
        const uint32_t m = range_mask(w, s, e);
        if (set) atomicOr(&pend[w], m); else atomicAnd(&pend[w], ~m);
    });
}

// Literal run out[b, b+L) = lit[a, a+L) (both in shared memory), by the eight
// lanes sl = 0..7 of a lane group: 16-byte stores in the middle, each from five
// funnel-shifted source words, bytes at the ragged ends.  Source words may reach
// 4 bytes past the run (the fifth of an aligned one), inside the literal buffer's
// 16 bytes of padding; those bytes are not used.
template <bool kRolled>
__device__ __forceinline__ void copy_run8(uint8_t* sout, const uint8_t* lit, uint32_t a, uint32_t b, uint32_t L,
                                          uint32_t sl) {
    const uint32_t e = b + L;
    const uint32_t q0 = (b + 15) >> 4, q1 = e >> 4;  // whole 16-byte chunks [q0, q1)
    if (q0 >= q1) {
        each<kRolled>(b + sl, e, 8, [&](uint32_t x) { sout[x] = lit[a + (x - b)]; });
        return;
    }
    each<kRolled>(b + sl, 16 * q0, 8, [&](uint32_t x) { sout[x] = lit[a + (x - b)]; });
    each<kRolled>(16 * q1 + sl, e, 8, [&](uint32_t x) { sout[x] = lit[a + (x - b)]; });
    const uint32_t* lw = reinterpret_cast<const uint32_t*>(lit);
    const uint32_t s0 = a + 16 * q0 - b;  // source of chunk q0
    const uint32_t sh = 8 * (s0 & 3);
    each<kRolled>(q0 + sl, q1, 8, [&](uint32_t q) {
        const uint32_t w = (s0 >> 2) + 4 * (q - q0);
        const uint32_t x0 = lw[w], x1 = lw[w + 1], x2 = lw[w + 2], x3 = lw[w + 3], x4 = lw[w + 4];
        reinterpret_cast<uint4*>(sout)[q] = make_uint4(__funnelshift_r(x0, x1, sh), __funnelshift_r(x1, x2, sh),
                                                       __funnelshift_r(x2, x3, sh), __funnelshift_r(x3, x4, sh));
    });
}

// Copy out[o, o + ml) = out[so, so + ml) (disjoint), by one thread: bytes up to
// a word boundary of the destination, words from two source words each, four
// at a time, bytes at the end.  Words may reach 4 bytes past the source run (the
// second word of an aligned one, loaded and not used), never past the block: a
// source ends at or before its destination, which holds at least 4 bytes.
__device__ __forceinline__ void copy_lane(uint8_t* out, uint32_t so, uint32_t o, uint32_t ml) {
    const uint32_t e = o + ml, q0 = (o + 3) >> 2, q1 = e >> 2;
    const uint32_t head = min(4 * q0, e), tail = max(4 * q1, head);
    for (uint32_t x = o; x < head; x++) out[x] = out[so + x - o];
    const uint32_t* lw = reinterpret_cast<const uint32_t*>(out);
    uint32_t* ow = reinterpret_cast<uint32_t*>(out);
    const uint32_t s0 = so + 4 * q0 - o, sh = 8 * (s0 & 3), w = s0 >> 2;
    for (uint32_t q = q0; q < q1; q += 4) {
        uint32_t x[5];
#pragma unroll
        for (int u = 0; u < 5; u++) x[u] = q + u <= q1 ? lw[w + (q - q0) + u] : 0;
#pragma unroll
        for (int u = 0; u < 4; u++)
            if (q + u < q1) ow[q + u] = __funnelshift_r(x[u], x[u + 1], sh);
    }
    for (uint32_t x = tail; x < e; x++) out[x] = out[so + x - o];
}

// Periodic fill out[o + k] = out[so + (k mod d)], k < ml, d < ml, by the eight
// lanes sl of a lane group: it reads the period window [so, so + d) only, so
// the lanes are independent; whole destination words as one store each.
template <bool kRolled>
__device__ __forceinline__ void fill_run8(uint8_t* out, uint32_t so, uint32_t o, uint32_t ml, uint32_t d, uint32_t sl) {
    const uint32_t e = o + ml, q0 = (o + 3) >> 2, q1 = e >> 2;  // whole words [q0, q1)
    // k mod d with one division: k and d stay below 2^14 + 4, so the rounded-up
    // reciprocal gives the quotient exactly
    const uint32_t M = 0xffffffffu / d + 1;
    auto mod = [&](uint32_t k) { return d == 1 ? 0u : k - d * __umulhi(k, M); };
    // ragged ends of at most 3 bytes: lanes 0..3 the head, 4..7 the tail
    const uint32_t edge = sl < 4 ? o + sl : max(4 * q1, 4 * q0) + sl - 4, edge_end = sl < 4 ? min(4 * q0, e) : e;
    if (edge < edge_end) out[edge] = out[so + mod(edge - o)];
    each<kRolled>(q0 + sl, q1, 8, [&](uint32_t q) {
        uint32_t v = 0, x = mod(4 * q - o);
#pragma unroll
        for (int u = 0; u < 4; u++) {
            v |= (uint32_t)out[so + x] << (8 * u);
            if (++x == d) x = 0;
        }
        reinterpret_cast<uint32_t*>(out)[q] = v;
    });
}

// Plain copy out[o, o + ml) = out[so, so + ml) (disjoint), by the eight lanes sl
// of a lane group: whole destination words from two source words each, bytes
// at the ragged ends.  An in-block match is short (30 bytes on average in a
// genome), where the 16-byte chunks of copy_run8 are mostly ragged ends.
// Words may reach 4 bytes past the source run, never past the block (as in
// copy_lane).
template <bool kRolled>
__device__ __forceinline__ void copy_words8(uint8_t* out, uint32_t so, uint32_t o, uint32_t ml, uint32_t sl) {
    const uint32_t e = o + ml, q0 = (o + 3) >> 2, q1 = e >> 2;  // whole words [q0, q1)
    const uint32_t edge = sl < 4 ? o + sl : max(4 * q1, 4 * q0) + sl - 4, edge_end = sl < 4 ? min(4 * q0, e) : e;
    if (edge < edge_end) out[edge] = out[so + edge - o];
    const uint32_t* lw = reinterpret_cast<const uint32_t*>(out);
    const uint32_t s0 = so + 4 * q0 - o, sh = 8 * (s0 & 3);
    each<kRolled>(q0 + sl, q1, 8, [&](uint32_t q) {
        const uint32_t w = (s0 >> 2) + q - q0;
        const uint32_t x0 = lw[w], x1 = lw[w + 1];
        reinterpret_cast<uint32_t*>(out)[q] = __funnelshift_r(x0, x1, sh);
    });
}

// One pass by one warp over the listed in-block matches act[first + k],
// act[first + stride + k], .., with 32 / G matches at a time (k < 32 / G) and
// G lanes a match.  A match whose source window has no pending byte is filled,
// its bits are cleared and its status becomes 0.  Returns, over the lane's
// matches, bit 0: one is left; bit 1: one was filled.
//
// G = 8 suits blocks of some tens of matches, whose copies are then short; a
// block with hundreds (the first blocks of a text, which hold no earlier
// blocks to copy from) is bound by its number of passes, and G = 1 looks after
// eight times as many in each: a lane copies a short plain match, eight lanes
// each longer or periodic one (one 10 KB text block 35 -> 23 us in the local
// pass, 4 MiB of text 60 -> 42, 64 MiB in 8 MiB segments 189 -> 164).  Groups of 128
// threads, whose blocks have few tokens, go without it: the code alone costs
// them (254 MB genome 318 -> 332 us; with G = 1 at every size 411).
constexpr uint32_t kLaneCopy = 64;
constexpr uint32_t kManyMatches = 64;  // more: G = 1
template <uint32_t G, bool kRolled>
__device__ __forceinline__ uint32_t match_pass(const uint16_t* act, uint32_t n_act, uint32_t first, uint32_t stride,
                                               uint8_t* sout, uint32_t* pend, uint8_t* tstat, const uint16_t* tml,
                                               const uint16_t* tpos, const uint16_t* tll, const uint64_t* tsrc,
                                               uint64_t B, int lane) {
    uint32_t res = 0;
    const uint32_t g = lane / G, sl = lane % G, gmask = (G == 8 ? 0xffu : 1u) << (G * g);
    for (uint32_t base = first; base < n_act; base += stride) {
        const uint32_t i = base + g < n_act ? act[base + g] : 0;
        const bool on = base + g < n_act && tstat[i] == 1;  // the same for the group's lanes
        uint32_t ml = 0, o = 0, so = 0, d = 1, we = 0;
        bool busy = false;
        if (on) {
            ml = tml[i];
            o = tpos[i] + tll[i];
            so = (uint32_t)(tsrc[i] - B);
            d = o - so;
            we = so + min(d, ml);  // periodic source window [so, we)
            each<kRolled>((so >> 5) + sl, ((we - 1) >> 5) + 1, G, [&](uint32_t w) {
                busy |= (((volatile uint32_t*)pend)[w] & range_mask(w, so, we)) != 0;
            });
        }
        const uint32_t bm = __ballot_sync(ACX_FULL, busy);  // every lane, active or not
        const bool ready = on && (bm & gmask) == 0;
        if (on && !ready) res |= 1;
        __threadfence_block();  // source reads after the readiness reads
        if (G == 8) {
            if (ready) {
                if (d >= ml) copy_words8<kRolled>(sout, so, o, ml, sl);
                else fill_run8<kRolled>(sout, so, o, ml, d, sl);
            }
        } else {
            const bool mine = ready && d >= ml && ml <= kLaneCopy;
            if (mine) copy_lane(sout, so, o, ml);
            uint32_t rest = __ballot_sync(ACX_FULL, ready && !mine);
            while (rest) {
                uint32_t k = 32;  // the next four, eight lanes each
#pragma unroll
                for (int u = 0; u < 4; u++) {
                    if (lane >> 3 == u && rest) k = __ffs(rest) - 1;
                    rest &= rest - 1;  // (0 stays 0)
                }
                const uint32_t ml2 = __shfl_sync(ACX_FULL, ml, k & 31), o2 = __shfl_sync(ACX_FULL, o, k & 31),
                               so2 = __shfl_sync(ACX_FULL, so, k & 31);
                if (k < 32) {
                    if (o2 - so2 >= ml2) copy_words8<kRolled>(sout, so2, o2, ml2, lane & 7);
                    else fill_run8<kRolled>(sout, so2, o2, ml2, o2 - so2, lane & 7);
                }
            }
        }
        __syncwarp();
        __threadfence_block();
        if (ready) {
            each<kRolled>((o >> 5) + sl, ((o + ml - 1) >> 5) + 1, G,
                          [&](uint32_t w) { atomicAnd(&pend[w], ~range_mask(w, o, o + ml)); });
            if (sl == 0) tstat[i] = 0;
            res |= 2;
        }
        __syncwarp();
    }
    return res;
}

// The kind of job a local group is built for.  Whole decodes without levels
// (one archive, or a batch of them: no wanted bytes, no level tables, no
// parse-only records, no ready flags, no item tables) get code of their own:
// the local pass loses issue slots to instruction fetch, and what such a job
// never runs is as much again (254 MB genome 314 -> 290 us).
enum class Loc { kAny, kOne, kBatch };
template <Loc kKind>
struct LocJob {
    static constexpr bool kWhole = kKind != Loc::kAny;
    static __device__ __forceinline__ bool flag(const JobDev& job, uint32_t f) { return !kWhole && (job.flags & f); }
    static __device__ __forceinline__ bool fused(const JobDev& job) { return !kWhole && job.ready; }
    // the pass's items [first, end) and its tickets
    static __device__ __forceinline__ uint32_t first(const JobDev& job) { return kKind == Loc::kBatch ? job.loc_lo : 0u; }
    static __device__ __forceinline__ uint32_t end(const JobDev& job) {
        return kKind == Loc::kBatch ? job.loc_hi : job.n_items;
    }
    static __device__ __forceinline__ uint32_t* tickets(const JobDev& job) {
        return job.counters + (kKind == Loc::kBatch ? job.loc_ctr : 1u);
    }
    static __device__ __forceinline__ int arc(const JobDev& job, uint32_t item) {
        return kKind == Loc::kOne ? 0 : find_arc(job, item);
    }
    static __device__ __forceinline__ ArcJob load(const JobDev& job, int a) {
        return kKind == Loc::kOne ? job.one : kKind == Loc::kBatch ? job.arcs[a] : load_arc(job, a);
    }
    static __device__ __forceinline__ ItemRef ref(const ArcJob& J, uint32_t idx) {
        return kWhole ? block_ref(J, idx) : item_ref(J, idx);
    }
};

// Issue the 1-D TMA copies of an item's four decoded streams (16-aligned,
// padded) into the stream buffers (one thread).  Nothing is issued for a
// block beyond the job's shared-memory limits (the caller treats it as bad).
template <Loc kKind>
__device__ __forceinline__ void stage_streams(const JobDev& job, uint32_t item, uint8_t* tcmd, uint8_t* lenb, uint8_t* soff,
                              uint8_t* slit, uint8_t* tlvl, uint64_t* bar) {
    typedef LocJob<kKind> Kind;
    const ArcJob J = Kind::load(job, Kind::arc(job, item));
    const ItemRef ir = Kind::ref(J, item - J.item_base);
    const BlockDev& bd = J.blk[ir.blk];
    const uint32_t n = bd.n_tok, LB = bd.s_raw[kLen], n_new = bd.n_new, n_lit = bd.s_raw[kLit];
    if (n > job.max_tok || LB > job.max_lenb || n_new > job.max_tok || n_lit > job.max_lit) return;
    const uint8_t* scr = J.scratch + ir.scratch;
    const uint32_t sz[4] = {(n + 15) & ~15u, (LB + 15) & ~15u, (5 * n_new + 15) & ~15u, (n_lit + 15) & ~15u};
    uint8_t* dsts[4] = {tcmd, lenb, soff, slit};
    // the level body (stored in the payload, 16-aligned and padded) beside them
    const uint32_t lsz = Kind::flag(job, kJobLevels) && bd.lvl_body ? sz[0] : 0;
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");  // earlier generic use of the buffers
    mbar_arrive_tx(bar, sz[0] + sz[1] + sz[2] + sz[3] + lsz);
    for (int q = 0; q < 4; q++)
        if (sz[q]) tma_load_1d(dsts[q], scr + bd.s_off[q], sz[q], bar);
    if (lsz) tma_load_1d(tlvl, J.arc + bd.payload + bd.lvl_body, lsz, bar);
}

// Item -> ticket order of the local pass: tickets are items, except in a
// fused decode, where the local groups follow the entropy warps' hand-out
// order (most symbols first) so that a ticket's streams are decoded early.
__device__ __forceinline__ uint32_t ticket_item(const JobDev& job, uint32_t t) {
    if (t >= job.n_items || !job.ready || !job.one.order) return t;
    return job.one.order[t];
}

// Wait (bounded) until the entropy stage of a fused decode has published
// item's streams; then generic-proxy writes of other SMs are visible to this
// thread's bulk copies.
__device__ __forceinline__ bool wait_ready(const uint32_t* ready, uint32_t item, uint64_t deadline) {
    uint32_t spins = 0;
    while (ld_acquire_u32(ready + item) == 0) {
        __nanosleep(64);
        if ((++spins & 63) == 0 && gtimer() > deadline) return false;
    }
    asm volatile("fence.proxy.async.global;" ::: "memory");
    return true;
}

// Words of a group's `misc`: 0 its claimed ticket, 2 whether the next block's
// streams are in flight, 3 the listed in-block matches, and one for each check
// of a block that threads make on their own.  A check's word is cleared when
// the block starts, set before the barrier that ends the check and read behind
// it, and no later phase writes it: every thread reads the same verdict, however
// late it leaves the barrier.  (`bad` decides which barriers a thread meets.
// With one word for all checks, a warp that read a verdict late could see the
// next check's, and run one barrier ahead of its group from there on.)
enum : uint32_t { kChkLen = 4, kChkValue, kChkToken, kChkSource, kChkHistory, kChkDeps, kChkEnd };

// The local pass of one group of NT threads (k_local: a whole CTA; k_fused: a
// group of a fused CTA) over the job's tickets, with its workspace at sm and
// named barrier bid; tid is the thread's index in its group.
template <int NT, Loc kKind>
__device__ __forceinline__ void local_worker(const JobDev& job, uint8_t* sm, uint32_t bid, int tid) {
    typedef LocJob<kKind> Kind;
    constexpr bool kRolled = NT == kLocThreads;
    const bool lvl = Kind::flag(job, kJobLevels);
    const LocLayout L = loc_layout(job.max_tok, job.max_lenb, job.max_lit, Kind::flag(job, kJobNeed), lvl);
    uint8_t* tlvl = sm + L.tlvl;                                      // valid in kJobLevels jobs
    uint8_t* tlvk = sm + L.tlvk;
    uint32_t* lhist = reinterpret_cast<uint32_t*>(sm + L.lhist);
    uint8_t* sout = sm + L.out;
    uint32_t* need = reinterpret_cast<uint32_t*>(sm + L.need);  // valid in kJobNeed jobs
    uint32_t* pend = reinterpret_cast<uint32_t*>(sm + L.pend);
    uint64_t* tsrc = reinterpret_cast<uint64_t*>(sm + L.tsrc);
    uint16_t* tpos = reinterpret_cast<uint16_t*>(sm + L.tpos);
    uint16_t* tll = reinterpret_cast<uint16_t*>(sm + L.tll);
    uint16_t* tml = reinterpret_cast<uint16_t*>(sm + L.tml);
    uint16_t* tlit = reinterpret_cast<uint16_t*>(sm + L.tlit);
    uint8_t* tcmd = sm + L.tcmd;
    uint8_t* tstat = sm + L.tstat;
    uint8_t* lenb = sm + L.lenb;
    uint8_t* soff = sm + L.soff;
    uint8_t* slit = sm + L.slit;
    uint32_t* scanbuf = reinterpret_cast<uint32_t*>(sm + L.scan);
    uint64_t* bar = reinterpret_cast<uint64_t*>(sm + L.bar);
    volatile uint32_t* misc = reinterpret_cast<volatile uint32_t*>(sm + L.misc);
    const int lane = tid & 31, warp = tid >> 5;
    const uint64_t deadline = gtimer() + job.timeout_ns;       // waits on published blocks (fused decodes)
    const uint64_t copy_deadline = gtimer() + kCopyWaitNs;    // waits on this group's own bulk copies
    if (tid == 0) mbar_init(bar, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    grp_sync<NT>(bid);
    uint32_t phase = 0;
    const uint32_t chunk = job.chunk ? job.chunk : 1u;
    uint32_t cnext = 0, cleft = 0;  // the group's current run of `chunk` tickets
    uint32_t pf_item = 0xffffffffu;  // the next item, claimed early (group-uniform)

    for (;;) {
        uint32_t item;
        bool prefetched = false;  // its streams are already in flight
        if (pf_item != 0xffffffffu) {
            item = pf_item;
            prefetched = misc[2] != 0;  // written by the thread that issued the item's copies
            pf_item = 0xffffffffu;
        } else {
            if (cleft == 0) {
                if (tid == 0) misc[0] = atomicAdd(Kind::tickets(job), chunk);
                grp_sync<NT>(bid);
                cnext = misc[0];
                cleft = chunk;
            }
            item = Kind::kWhole ? Kind::first(job) + cnext++ : ticket_item(job, cnext++);
            cleft--;
        }
        // the next block's ticket: its atomic goes out now and is read at the
        // prefetch point, so its latency hides behind this block's work
        uint32_t pre_claim = 0;
        bool claimed = cleft == 0;  // group-uniform
        if (claimed && tid == 0) pre_claim = atomicAdd(Kind::tickets(job), chunk);
        // a block that ends before the prefetch point (corrupt, or a parse-only
        // job) hands the claimed tickets on to the next iteration
        auto settle_claim = [&]() {
            if (!claimed) return;
            if (tid == 0) misc[0] = pre_claim;
            grp_sync<NT>(bid);
            cnext = misc[0];
            cleft = chunk;
            claimed = false;
        };
        if (item >= Kind::end(job)) return;
        const int a = Kind::arc(job, item);
        const ArcJob J = Kind::load(job, a);
        const ItemRef ir = Kind::ref(J, item - J.item_base);
        const uint32_t b = ir.blk;
        const BlockDev& bd = J.blk[b];
        const uint64_t B = (uint64_t)b * kBlock;
        const uint32_t R = bd.raw_len, n = bd.n_tok, LB = bd.s_raw[kLen], n_lit = bd.s_raw[kLit];
        const uint32_t n_new = bd.n_new;
        bool bad = n > job.max_tok || LB > job.max_lenb || n_new > job.max_tok || n_lit > job.max_lit;
        int stage = bad ? kStageLimits : 0;
        auto mark = [&](bool cond, int st) {
            if (cond && !bad) { bad = true; stage = st; }
        };

        // ---- stage the four decoded streams with 1-D TMA bulk copies (unless
        //      they were prefetched during the previous block) ----
        if (!bad && tid == 0 && !prefetched && (!Kind::fused(job) || wait_ready(job.ready, item, deadline)))
            stage_streams<kKind>(job, item, tcmd, lenb, soff, slit, tlvl, bar);
        for (uint32_t i = tid; i < kBlock / 128; i += NT) reinterpret_cast<uint4*>(pend)[i] = make_uint4(0, 0, 0, 0);
        if (tid < (int)(kChkEnd - kChkLen)) misc[kChkLen + tid] = 0;
        // wanted bytes of this item (all when it names none)
        const bool partial = Kind::flag(job, kJobNeed) && ir.need_n != 0;
        if (partial) {
            for (uint32_t i = tid; i < kBlock / 32; i += NT) need[i] = 0;
            grp_sync<NT>(bid);
            for (uint32_t q = 0; q < ir.need_n; q++) {
                const uint32_t iv = J.need[ir.need_off + q];
                const uint32_t s0 = iv & 0xffff, e0 = min(iv >> 16, kBlock);
                if (s0 < e0)
                    for (uint32_t w = (s0 >> 5) + tid; w <= ((e0 - 1) >> 5); w += NT)
                        atomicOr(&need[w], range_mask(w, s0, e0));
            }
        }
        bool timed_out = false;
        if (!bad) {
            uint32_t spins = 0;
            while (!mbar_try_wait(bar, phase & 1))
                if ((++spins & 1023) == 0 && gtimer() > copy_deadline) { timed_out = true; break; }
            phase++;
        }
        if (grp_or<NT>(bid, timed_out)) {
            // a copy that never lands: give up on the decode (the barrier phase is lost)
            if (tid == 0) set_err_arc(job, a, kErrTimeout, kStageWait << 24, b);
            return;
        }

        // ---- varints: each byte < 0x80 ends a value ----
        uint32_t v1[1], tot1[1], v3[3], tot3[3], v2[2], tot2[2];
        const uint32_t per = (LB + NT - 1) / NT;
        const uint32_t j0 = min(LB, tid * per), j1 = min(LB, j0 + per);
        {
            uint32_t c = 0;
            bool vbad = false;
            if (!bad)
                each<kRolled>(j0, j1, 1, [&](uint32_t j) {
                    const uint8_t by = lenb[j];
                    if (by < 0x80) c++;
                    // a value has at most three bytes
                    if (by >= 0x80 && j >= 2 && lenb[j - 1] >= 0x80 && lenb[j - 2] >= 0x80) vbad = true;
                });
            if (vbad) misc[kChkLen] = 1;
            v1[0] = c;
            block_scan<NT, 1>(v1, tot1, scanbuf, bid, tid);
        }
        mark(tot1[0] != 2 * n || (LB > 0 && lenb[LB - 1] >= 0x80) || (LB == 0 && n > 0) || misc[kChkLen], kStageVarint);
        if (!bad) {
            uint32_t idx = v1[0];
            each<kRolled>(j0, j1, 1, [&](uint32_t j) {
                const uint8_t by = lenb[j];
                if (by >= 0x80) return;
                uint32_t val = by;
                if (j >= 1 && lenb[j - 1] >= 0x80) {
                    val = (val << 7) | (lenb[j - 1] & 0x7f);
                    if (j >= 2 && lenb[j - 2] >= 0x80) val = (val << 7) | (lenb[j - 2] & 0x7f);
                }
                if (val > kBlock) misc[kChkValue] = 1;
                const uint32_t tk = idx >> 1;
                if (idx & 1) tml[tk] = (uint16_t)min(val, kBlock); else tll[tk] = (uint16_t)min(val, kBlock);
                idx++;
            });
        }
        grp_sync<NT>(bid);
        mark(misc[kChkValue] != 0, kStageVarint);

        // ---- token scans: positions, literal positions, NEW indices ----
        const uint32_t tper = (n + NT - 1) / NT;
        const uint32_t i0 = min(n, tid * tper), i1 = min(n, i0 + tper);
        bool any_rep = false;
        {
            uint32_t s_len = 0, s_ll = 0, s_new = 0;
            bool tbad = false;
            if (!bad)
                each<kRolled>(i0, i1, 1, [&](uint32_t i) {
                    const uint32_t ll = tll[i], ml = tml[i], c = tcmd[i];
                    s_len += ll + ml;
                    s_ll += ll;
                    s_new += c == kNew;
                    if (c > kLitOnly) tbad = true;
                    if (c == kLitOnly) { if (ml != 0 || i != n - 1 || ll == 0) tbad = true; }
                    else if (ml < J.min_match) tbad = true;
                    any_rep |= c >= 1 && c <= 4;
                });
            if (tbad) misc[kChkToken] = 1;
            v3[0] = s_len; v3[1] = s_ll; v3[2] = s_new;
            block_scan<NT, 3>(v3, tot3, scanbuf, bid, tid);
        }
        mark(tot3[0] != R || tot3[1] != n_lit || tot3[2] != n_new || misc[kChkToken], kStageTokens);
        if (!bad) {
            uint32_t pos = v3[0], lp = v3[1], ni = v3[2];
            each<kRolled>(i0, i1, 1, [&](uint32_t i) {
                const uint32_t ll = tll[i], ml = tml[i];
                tpos[i] = (uint16_t)pos;
                tlit[i] = (uint16_t)lp;
                uint64_t src = 0;
                if (tcmd[i] == kNew) {
#pragma unroll
                    for (int p = 0; p < 5; p++) src |= (uint64_t)soff[p * n_new + ni] << (8 * p);
                    ni++;
                    if (src >= B + pos + ll) misc[kChkSource] = 1;  // every absolute offset precedes its destination
                }
                tsrc[i] = src;
                pos += ll + ml;
                lp += ll;
            });
        }
        any_rep = grp_or<NT>(bid, any_rep && !bad);
        mark(misc[kChkSource] != 0, kStageSources);

        // ---- the four-entry history (blocks with repeat codes only) as a
        //      warp-level scan of packed maps by warp 0, while the other warps
        //      place the literals, which need positions only (a parse-only job
        //      places none) ----
        const bool place = !bad && !Kind::flag(job, kJobIndex);
        if (!bad && (any_rep || place)) {
            if (any_rep && warp == 0) {
                const uint32_t per = (n + 31) / 32;
                const uint32_t j0 = min(n, lane * per), j1 = min(n, j0 + per);
                HMap agg = kHIdentity;
                each<kRolled>(j0, j1, 1, [&](uint32_t i) { agg = hmap_step(agg, tcmd[i], i); });
                // inclusive scan of the lanes' maps (earlier maps act first)
                HMap inc = agg;
#pragma unroll 1
                for (int o = 1; o < 32; o <<= 1) {
                    const HMap prev = __shfl_up_sync(ACX_FULL, inc, o);
                    if (lane >= o) inc = hmap_compose(prev, inc);
                }
                const HMap ex = __shfl_up_sync(ACX_FULL, inc, 1);
                const HMap pre = lane > 0 ? ex : kHIdentity;
                // the history before this lane's tokens: the block starts from
                // (1, 2, 3, 4); a NEW token's entry is its distance
                auto entry = [&](int k) -> uint64_t {
                    const uint32_t x = (uint32_t)(pre >> (16 * k)) & 0xffff;
                    return (x & kHRef) ? (uint64_t)((x & 3) + 1) : B + tpos[x] + tll[x] - tsrc[x];
                };
                // the lane's history in four registers (selects, no indexed array)
                uint64_t h0 = entry(0), h1 = entry(1), h2 = entry(2), h3 = entry(3);
                each<kRolled>(j0, j1, 1, [&](uint32_t i) {
                    const uint8_t c = tcmd[i];
                    const uint64_t dst = B + tpos[i] + tll[i];
                    if (c == kNew) {
                        h3 = h2; h2 = h1; h1 = h0; h0 = dst - tsrc[i];
                    } else if (c >= 1 && c <= 4) {
                        const uint32_t j = c - 1u;
                        const uint64_t d = j == 0 ? h0 : j == 1 ? h1 : j == 2 ? h2 : h3;
                        if (d < 1 || d > dst) misc[kChkHistory] = 1;
                        tsrc[i] = dst - d;
                        h3 = j >= 3 ? h2 : h3;
                        h2 = j >= 2 ? h1 : h2;
                        h1 = j >= 1 ? h0 : h1;
                        h0 = d;
                    }
                });
            }
            if (place && (warp > 0 || !any_rep)) {
                // literal placement: a thread copies a tiny run (<= kLaneBytes)
                // by itself, all threads at once; eight lanes copy each longer one
                const int w0 = any_rep ? 1 : 0, nw = (NT / 32) - w0;
#pragma unroll 1
                for (uint32_t i = tid - 32 * w0; i < n; i += 32 * nw) {
                    const uint32_t ll = tll[i];
                    if (ll <= kLaneBytes) {
                        const uint32_t la = tlit[i], lb = tpos[i];
                        for (uint32_t k = 0; k < ll; k++) sout[lb + k] = slit[la + k];
                    }
                }
#pragma unroll 1
                for (uint32_t i = (warp - w0) * 4 + (lane >> 3); i < n; i += nw * 4)
                    if (tll[i] > kLaneBytes) copy_run8<kRolled>(sout, slit, tlit[i], tpos[i], tll[i], lane & 7);
            }
            grp_sync<NT>(bid);
            mark(misc[kChkHistory] != 0, kStageSources);
        }

        // ---- with dependency lists: every block a match reads outside its own
        //      block must be listed (range decodes read only the listed closure) ----
        if (J.deps && !bad) {
            const uint32_t* dl = J.deps + bd.dep_off;
            const uint32_t nd = bd.n_deps;
            bool dbad = false;
            for (uint32_t i = i0; i < i1; i++) {
                const uint32_t ml = tml[i];
                if (!ml || tsrc[i] >= B) continue;
                const uint64_t d = B + tpos[i] + tll[i] - tsrc[i];
                const uint64_t e = tsrc[i] + (d < ml ? d : ml);
                for (uint64_t a = tsrc[i] >> 14; a <= (e - 1) >> 14 && a < b && !dbad; a++)
                    dbad = !listed(dl, nd, (uint32_t)a);
            }
            if (dbad) misc[kChkDeps] = 1;
            grp_sync<NT>(bid);
            mark(misc[kChkDeps] != 0, kStageSources);
        }

        if (Kind::flag(job, kJobIndex)) {
            // parse only: one record per token (source, destination offset,
            // match length, command)
            if (!bad)
                for (uint32_t i = tid; i < n; i += NT)
                    J.spans[ir.span_base + i] = SpanRec{(uint32_t)tsrc[i], (uint32_t)(tsrc[i] >> 32),
                                                        (uint32_t)(tpos[i] + tll[i]) | ((uint32_t)tml[i] << 16), tcmd[i]};
            if (bad && tid == 0) {
                set_err_arc(job, a, kErrCorrupt, stage << 24, b);
                J.npend[ir.slot] = 1;  // per-item status of a parse-only job
            }
            grp_sync<NT>(bid);
            settle_claim();
            continue;
        }

        uint32_t npend = 0, pbytes = 0;
        if (!bad) {
            // ---- every match byte starts unresolved; external sources are pending for good;
            //      the in-block matches are listed (the literal positions are dead now) ----
            uint16_t* act_list = tlit;
            if (tid == 0) misc[3] = 0;
            grp_sync<NT>(bid);
#pragma unroll 1
            for (uint32_t i = tid; i < n; i += NT) {
                const uint32_t ml = tml[i];
                uint8_t st = 0;  // 0: none/done, 1: unresolved in-block, 2: pending
                if (ml) {
                    const uint32_t s = tpos[i] + tll[i];
                    pend_update_smem<kRolled>(pend, s, s + ml, true);
                    st = tsrc[i] >= B ? 1 : 2;
                    if (st == 1) act_list[atomicAdd((uint32_t*)&misc[3], 1u)] = (uint16_t)i;
                }
                tstat[i] = st;
                if (lvl) tlvk[i] = tlvl[i];  // the staging buffer takes the next block's levels below
            }
            grp_sync<NT>(bid);
            // ---- the stream buffers are free from here on: start the next item's
            //      copies, so that they land while this block finishes ----
            settle_claim();
            pf_item = Kind::kWhole ? Kind::first(job) + cnext++ : ticket_item(job, cnext++);
            cleft--;
            // (issued by the last warp, which takes the fewest in-block matches
            // below, so that its loads of the next block's descriptor delay the
            // rounds least)
            if (tid == NT - 32) {
                // in a fused decode, only streams that are already published
                const bool go = pf_item < Kind::end(job) && (!Kind::fused(job) || ld_acquire_u32(job.ready + pf_item) != 0);
                if (go) {
                    if (Kind::fused(job)) asm volatile("fence.proxy.async.global;" ::: "memory");
                    stage_streams<kKind>(job, pf_item, tcmd, lenb, soff, slit, tlvl, bar);
                }
                misc[2] = go;
            }
            // ---- in-block matches: rounds over the listed matches ----
            const uint32_t n_act = misc[3];
            for (;;) {
                const uint32_t r =
                    NT > kLocThreads && n_act > kManyMatches
                        ? match_pass<1, kRolled>(tlit, n_act, 32 * warp, NT, sout, pend, tstat, tml, tpos, tll, tsrc, B, lane)
                        : match_pass<8, kRolled>(tlit, n_act, 4 * warp, NT / 8, sout, pend, tstat, tml, tpos, tll, tsrc, B, lane);
                const int any_left = grp_or<NT>(bid, r & 1);
                const int any_prog = grp_or<NT>(bid, r & 2);
                if (!any_left || !any_prog) break;
            }
            // ---- whatever is still unresolved becomes pending pieces (for a
            //      partial item: the wanted matches only) ----
            if (partial)
#pragma unroll 1
                for (uint32_t i = i0; i < i1; i++)
                    if (tstat[i] && !wanted(need, tpos[i] + tll[i], tml[i])) tstat[i] = 0;
            uint32_t cnt = 0, nbytes = 0;
#pragma unroll 1
            for (uint32_t i = i0; i < i1; i++)
                if (tstat[i]) {
                    cnt += pieces_of(tml[i]);
                    nbytes += tml[i];
                }
            v2[0] = cnt; v2[1] = nbytes;
            block_scan<NT, 2>(v2, tot2, scanbuf, bid, tid);
            npend = tot2[0];
            pbytes = tot2[1];
            if (lvl) {
                // the block's row of the level table (pieces of level <= l,
                // a piece's level being its token's level byte clamped to
                // [1, n_levels]); the pieces themselves stay in output order
                // and carry their level, and the level list is built from
                // them (k_level_fill)
                const uint32_t Lg = job.n_levels;
                for (uint32_t l = tid; l <= Lg; l += NT) lhist[l] = 0;
                grp_sync<NT>(bid);
                for (uint32_t i = i0; i < i1; i++)
                    if (tstat[i]) atomicAdd(&lhist[min(max((uint32_t)tlvk[i], 1u), Lg)], pieces_of(tml[i]));
                grp_sync<NT>(bid);
                if (warp == 0) {
                    uint32_t carry = 0;
                    uint32_t* row = job.lvl_tab + (uint64_t)ir.slot * (Lg + 1);
                    for (uint32_t l0 = 0; l0 <= Lg; l0 += 32) {
                        const uint32_t l = l0 + lane;
                        uint32_t inc = l <= Lg ? lhist[l] : 0;
#pragma unroll
                        for (int o = 1; o < 32; o <<= 1) {
                            const uint32_t y = __shfl_up_sync(ACX_FULL, inc, o);
                            if (lane >= o) inc += y;
                        }
                        if (l <= Lg) row[l] = carry + inc;
                        carry += __shfl_sync(ACX_FULL, inc, 31);
                    }
                }
            }
            {
                uint32_t k = v2[0];
#pragma unroll 1
                for (uint32_t i = i0; i < i1; i++) {
                    if (!tstat[i]) continue;
                    const uint32_t o = tpos[i] + tll[i];
                    const uint32_t lv = lvl ? min(max((uint32_t)tlvk[i], 1u), job.n_levels) : 0u;
                    k += emit_pieces(J.spans + ir.span_base + k, o, tsrc[i], tml[i], B + o - tsrc[i], lv);
                }
            }
        }
        grp_sync<NT>(bid);
        if (bad) {
            if (tid == 0) set_err_arc(job, a, kErrCorrupt, stage << 24, b);
            npend = 0;
            if (lvl)  // an empty row: the level rounds take nothing from this block
                for (uint32_t l = tid; l <= job.n_levels; l += NT)
                    job.lvl_tab[(uint64_t)ir.slot * (job.n_levels + 1) + l] = 0;
        }
        // ---- write the block (pending bytes are filled by the cross-block pass) ----
        uint8_t* gout = J.out + (uint64_t)ir.slot * kBlock;
        const uint32_t nv = R / 16;
        for (uint32_t i = tid; i < nv; i += NT) reinterpret_cast<uint4*>(gout)[i] = reinterpret_cast<uint4*>(sout)[i];
#pragma unroll 1
        for (uint32_t x = 16 * nv + tid; x < R; x += NT) gout[x] = sout[x];
        {
            // the pending bitmap is written for every block (all clear when nothing
            // is pending, a corrupt block included), so readers need no second
            // lookup and never wait on a corrupt block
            uint4* gp = reinterpret_cast<uint4*>(J.pmap + (uint64_t)ir.slot * (kBlock / 32));
            const uint4* sp = reinterpret_cast<const uint4*>(pend);
            const uint4* np4 = reinterpret_cast<const uint4*>(need);
            for (uint32_t i = tid; i < kBlock / 128; i += NT) {
                uint4 v = npend ? sp[i] : make_uint4(0, 0, 0, 0);
                if (partial) {  // unwanted bytes are never read: leave them out of the bitmap
                    const uint4 m = np4[i];
                    v.x &= m.x; v.y &= m.y; v.z &= m.z; v.w &= m.w;
                }
                gp[i] = v;
            }
        }
        if (tid == 0) {
            J.npend[ir.slot] = npend;
            if (npend) {
                atomicAdd(&job.counters[kStatPending], npend);
                atomicAdd(reinterpret_cast<unsigned long long*>(job.counters + kStatPendBytes), (unsigned long long)pbytes);
            }
        }
        grp_sync<NT>(bid);
        settle_claim();
    }
}

}  // namespace acx
