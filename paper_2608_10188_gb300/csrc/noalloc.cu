// Decode entry point that allocates nothing (aceapex_decode_noalloc).
//
// Some callers cannot allocate device memory when they decode: allocators
// that hand the whole device to a framework pool at start-up, or real-time
// paths where an allocation's latency or failure is not acceptable.  For
// small archives they get this entry point: every byte of scratch it needs
// (the decode plan, the dependency lists, the decoded streams, the pending
// bitmaps and pieces, the work lists, the tickets and the error word) lives
// in one file-scope device array, and the archive's plan is built on the
// device by a small kernel, so neither device nor host memory is allocated.
// The call reads the plan summary and the status back to the host and
// synchronises its stream twice, so it cannot be recorded into a CUDA graph.
//
// Limits: at most kNaMaxBlocks blocks (1 MiB of output) and the per-region
// capacities below; valid archives beyond them are rejected with
// ACEAPEX_E_ARG, archives the regular entry point finds corrupt with
// ACEAPEX_E_CORRUPT.  The array is shared by every call in the process on a
// given device: calls that overlap on the GPU (other streams, other host
// threads) race on it.
#include <algorithm>
#include <mutex>

#include "../../include/aceapex.h"
#include "common.cuh"
#include "launch.h"

namespace acx {

namespace {

constexpr uint32_t kNaMaxBlocks = 64;
constexpr size_t kNaStreamBytes = 2u << 20;     // decoded streams
constexpr uint32_t kNaSpanSlots = 96u * 1024;   // pending pieces (and each work list)

// Layout of the static scratch (byte offsets, 256-aligned regions).
constexpr size_t al(size_t x) { return (x + 255) & ~(size_t)255; }
constexpr size_t kOffSummary = 0;
constexpr size_t kOffErr = al(kOffSummary + 64);
constexpr size_t kOffCounters = al(kOffErr + 16);
constexpr size_t kOffPlan = al(kOffCounters + kCounterWords * 4);
constexpr size_t kOffTab = al(kOffPlan + kNaMaxBlocks * sizeof(BlockDev));
constexpr size_t kOffNpend = al(kOffTab + 4 * kM * 4);
constexpr size_t kOffPmap = al(kOffNpend + kNaMaxBlocks * 4);
// dependency lists, copied out of the archive: block b's (at most b ids) at
// [b(b-1)/2, b(b-1)/2 + b), so the kernels read aligned words
constexpr size_t kNaDepWords = (size_t)kNaMaxBlocks * (kNaMaxBlocks - 1) / 2;
constexpr size_t kOffDeps = al(kOffPmap + (size_t)kNaMaxBlocks * (kBlock / 8));
constexpr size_t kOffSpans = al(kOffDeps + kNaDepWords * 4);
constexpr size_t kOffLists = al(kOffSpans + (size_t)kNaSpanSlots * sizeof(SpanRec));
constexpr size_t kOffStreams = al(kOffLists + 2 * (size_t)kNaSpanSlots * sizeof(JobDev::ListEnt));
constexpr size_t kNaBytes = al(kOffStreams + kNaStreamBytes + 64);

}  // namespace

// The scratch of aceapex_decode_noalloc (about 5.3 MiB per device).
static __device__ __align__(256) uint8_t g_noalloc_scratch[kNaBytes];

namespace {

// Plan summary written by k_plan_small and read back by the host.
struct NaSummary {
    int32_t status;       // 0 ok, -2 corrupt, -1 beyond the static limits
    uint32_t n_blocks, min_match, max_tok, max_lenb, max_lit, has_deps;
    uint64_t total, span_slots, stream_bytes;
};
static_assert(sizeof(NaSummary) <= 64, "summary");

__device__ __forceinline__ uint16_t rd16d(const uint8_t* p) { return (uint16_t)(p[0] | (p[1] << 8)); }
__device__ __forceinline__ uint32_t rd32d(const uint8_t* p) {
    return (uint32_t)p[0] | ((uint32_t)p[1] << 8) | ((uint32_t)p[2] << 16) | ((uint32_t)p[3] << 24);
}
__device__ __forceinline__ uint64_t rd64d(const uint8_t* p) { return (uint64_t)rd32d(p) | ((uint64_t)rd32d(p + 4) << 32); }
// N consecutive little-endian words at p, all loads before any use (words when
// p is aligned, bytes otherwise).
template <int N>
__device__ __forceinline__ void rd_words(const uint8_t* p, uint32_t (&w)[N]) {
    if (((uintptr_t)p & 3) == 0) {
#pragma unroll
        for (int i = 0; i < N; i++) w[i] = reinterpret_cast<const uint32_t*>(p)[i];
    } else {
#pragma unroll
        for (int i = 0; i < N; i++) w[i] = rd32d(p + 4 * i);
    }
}

// Validate a format v1 archive held in device memory and build its decode
// plan in the static scratch (one CTA).  The checks are the host plan
// builder's: header, tables, index entries, payload descriptors.
//
// The kernel is bound by load round trips, so they are few and taken side by
// side: a thread a block, its index entry and its four stream descriptors as
// whole loads; the tables are summed and written by warps; offsets and maxima
// over the blocks come from shared memory.  (With serial tables, byte loads and
// one thread's walk over the blocks in global memory it took 135 us, half of a
// 1 MB decode.)
constexpr int kPlanThreads = 256;
__global__ void __launch_bounds__(kPlanThreads) k_plan_small(const uint8_t* a, uint64_t len, uint8_t* base) {
    NaSummary* S = reinterpret_cast<NaSummary*>(base + kOffSummary);
    BlockDev* blk = reinterpret_cast<BlockDev*>(base + kOffPlan);
    uint32_t* tab = reinterpret_cast<uint32_t*>(base + kOffTab);
    uint32_t* deps = reinterpret_cast<uint32_t*>(base + kOffDeps);
    __shared__ int bad;            // 0 ok, -2 corrupt, -1 too large
    __shared__ uint64_t off_tab, off_idx, off_deps, total;
    __shared__ uint32_t nb, min_match, flags;
    __shared__ uint16_t freq[4][256], cum[4][256];
    __shared__ uint32_t ok_tab[4];
    __shared__ uint32_t b_bytes[kNaMaxBlocks], b_slots[kNaMaxBlocks];  // per block: stream bytes, piece slots
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    if (tid == 0) {
        bad = 0;
        if (len < 64) {
            bad = -2;
        } else {
            uint32_t h[14];
            rd_words(a, h);
            // "ACX1", version 1
            if (h[0] != 0x31584341u || (h[1] & 0xffff) != 1 || h[2] != kBlock) {
                bad = -2;
            } else {
                flags = h[1] >> 16;
                min_match = h[3];
                total = h[4] | (uint64_t)h[5] << 32;
                nb = h[6];
                off_tab = h[8] | (uint64_t)h[9] << 32;
                off_idx = h[10] | (uint64_t)h[11] << 32;
                off_deps = h[12] | (uint64_t)h[13] << 32;
                if (min_match < 4 || min_match > kBlock || (uint64_t)nb != (total + kBlock - 1) / kBlock) bad = -2;
                else if (off_tab > len || len - off_tab < 2048) bad = -2;
                else if (off_idx > len || (len - off_idx) / 40 < nb) bad = -2;
                else if (nb > kNaMaxBlocks) bad = -1;
            }
        }
    }
    __syncthreads();
    if (bad) {
        if (tid == 0) S->status = bad;
        return;
    }
    for (uint32_t i = tid; i < 4 * 256; i += kPlanThreads) freq[i >> 8][i & 255] = rd16d(a + off_tab + 2 * i);
    if (tid < (int)kNaMaxBlocks) b_bytes[tid] = b_slots[tid] = 0;
    __syncthreads();
    if (warp < 4) {  // table `warp`: its sum and each symbol's first slot
        uint32_t own = 0;
        for (int k = 0; k < 8; k++) own += freq[warp][8 * lane + k];
        uint32_t inc = own;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_up_sync(ACX_FULL, inc, o);
            if (lane >= o) inc += y;
        }
        const uint32_t sum = __shfl_sync(ACX_FULL, inc, 31);
        uint32_t c = inc - own;
        for (int k = 0; k < 8; k++) {
            cum[warp][8 * lane + k] = (uint16_t)c;  // (used only when the sum is kM)
            c += freq[warp][8 * lane + k];
        }
        if (lane == 0) {
            ok_tab[warp] = sum == kM;
            if (sum != 0 && sum != kM) bad = -2;
        }
    }
    __syncthreads();
    // decode entries sym | (f-1) << 8 | (slot-c) << 20: a slot's symbol is the
    // last one that starts at or before it (symbols that do not occur start
    // where the next one does)
    for (uint32_t i = tid; i < 4 * kM; i += 4 * kPlanThreads) {
        uint32_t k[4] = {0, 0, 0, 0};
#pragma unroll
        for (uint32_t h = 128; h; h >>= 1)
#pragma unroll
            for (int u = 0; u < 4; u++) {
                const uint32_t j = i + u * kPlanThreads;
                if (cum[j / kM][k[u] + h] <= j % kM) k[u] += h;
            }
#pragma unroll
        for (int u = 0; u < 4; u++) {
            const uint32_t j = i + u * kPlanThreads, t = j / kM;
            if (ok_tab[t]) tab[j] = k[u] | (uint32_t)(freq[t][k[u]] - 1) << 8 | (j % kM - cum[t][k[u]]) << 20;
        }
    }
    const uint32_t b = tid;
    BlockDev bd{};
    if (b < nb) {
        uint32_t e[7];
        rd_words(a + off_idx + 40 * (uint64_t)b, e);
        const uint64_t poff = e[0] | (uint64_t)e[1] << 32;
        const uint32_t plen = e[2], n_tok = e[3], raw = e[4], dep_off = e[5], n_deps = e[6];
        const uint64_t B = (uint64_t)b * kBlock;
        const uint64_t R = total - B < kBlock ? total - B : kBlock;
        bool ok = raw == R && !(off_deps == 0 && (dep_off || n_deps));
        // an ascending list of distinct ids below b has at most b entries
        const uint32_t dslot = b * (b - 1) / 2;
        if (ok && off_deps) {
            ok = off_deps <= len && (len - off_deps) / 4 >= (uint64_t)dep_off + n_deps && n_deps <= b;
            uint32_t prev = 0;
            for (uint32_t k = 0; ok && k < n_deps; k++) {
                const uint32_t id = rd32d(a + off_deps + 4 * ((uint64_t)dep_off + k));
                if (id >= b || (k && id <= prev)) ok = false;
                prev = id;
                deps[dslot + k] = id;
            }
        }
        ok = ok && !(poff & 15) && !(plen & 15) && plen >= 48 && poff <= len && len - poff >= plen;
        uint64_t soff = 0;
        if (ok) {
            uint32_t d[12];
            rd_words(a + poff, d);
            bd.payload = poff;
            bd.raw_len = raw;
            bd.n_tok = n_tok;
            if (off_deps) {
                bd.dep_off = dslot;
                bd.n_deps = n_deps;
            }
            uint64_t off = 48;
#pragma unroll
            for (int s = 0; s < 4; s++) {
                const uint32_t sraw = d[3 * s], enc = d[3 * s + 1];
                const uint8_t mode = (uint8_t)d[3 * s + 2], K = (uint8_t)(d[3 * s + 2] >> 8);
                if (d[3 * s + 2] >> 16 || sraw > kMaxStreamRaw || off + enc > plen) ok = false;
                if (mode == 0) {
                    if (enc != sraw || K != 0) ok = false;
                } else if (mode == 1) {
                    const bool lanes_ok = K >= 1 && K <= kMaxLanes && (K & (K - 1)) == 0;
                    const uint32_t hdr = (4u * K + 15) & ~15u;
                    if (sraw == 0 || !lanes_ok || !ok_tab[s] || enc < hdr || ((enc - hdr) & 1)) ok = false;
                    bd.rans_mask |= 1u << s;
                } else {
                    ok = false;
                }
                bd.s_raw[s] = sraw;
                bd.s_body[s] = (uint32_t)off;
                bd.s_enc[s] = enc;
                bd.s_K[s] = K;
                bd.s_off[s] = (uint32_t)soff;
                soff = (soff + sraw + 15) & ~(uint64_t)15;
                off = (off + enc + 15) & ~(uint64_t)15;
            }
            if (flags & 2) {  // the level body (one stored byte per token) after the four streams
                ok = ok && off + n_tok <= plen;
                off = (off + n_tok + 15) & ~(uint64_t)15;
            }
            ok = ok && off == plen && bd.s_raw[kCmd] == n_tok && bd.s_raw[kOff] % 5 == 0 && bd.s_raw[kLit] <= raw;
            // every token but a closing literal run has a match of at least
            // min_match bytes: more tokens than that cannot sum to the block
            // (the regular decode finds such a block corrupt too)
            ok = ok && n_tok <= raw / min_match + 1;
            bd.n_new = bd.s_raw[kOff] / 5;
        }
        if (ok) {
            b_bytes[b] = (uint32_t)soff;  // (four streams of at most kMaxStreamRaw bytes)
            b_slots[b] = n_tok + kSpanSlack;
        } else {
            bad = -2;
        }
    }
    __syncthreads();
    if (bad) {
        if (tid == 0) S->status = bad;
        return;
    }
    if (b < nb) {
        uint32_t scratch = 0, slots = 0;  // (64 blocks: both fit 32 bits)
        for (uint32_t k = 0; k < b; k++) {
            scratch += b_bytes[k];
            slots += b_slots[k];
        }
        bd.scratch = scratch;
        bd.span_base = slots;
        blk[b] = bd;
    }
    if (warp < 2) {  // the summary: block b is lane b & 31 of warp b >> 5
        __shared__ uint32_t part[2][5];
        const uint32_t v[5] = {b < nb ? b_bytes[b] : 0, b < nb ? b_slots[b] : 0, bd.n_tok, bd.s_raw[kLen], bd.s_raw[kLit]};
        uint32_t r[5];
        r[0] = __reduce_add_sync(ACX_FULL, v[0]);
        r[1] = __reduce_add_sync(ACX_FULL, v[1]);
#pragma unroll
        for (int k = 2; k < 5; k++) r[k] = __reduce_max_sync(ACX_FULL, v[k]);
        if (lane == 0)
            for (int k = 0; k < 5; k++) part[warp][k] = r[k];
        asm volatile("bar.sync 1, 64;" ::: "memory");  // (warps 0 and 1)
        if (tid == 0) {
            const uint64_t scratch = (uint64_t)part[0][0] + part[1][0], slots = (uint64_t)part[0][1] + part[1][1];
            S->status = scratch + 64 > kNaStreamBytes || slots > kNaSpanSlots ? -1 : 0;
            S->n_blocks = nb;
            S->min_match = min_match;
            S->max_tok = max(1u, max(part[0][2], part[1][2]));
            S->max_lenb = max(1u, max(part[0][3], part[1][3]));
            S->max_lit = max(part[0][4], part[1][4]);
            S->total = total;
            S->has_deps = off_deps != 0;
            S->span_slots = slots;
            S->stream_bytes = scratch;
        }
    }
}

// Device address of the static scratch, looked up once per device.
std::mutex g_na_mutex;
uint8_t* g_na_base[64];

}  // namespace
}  // namespace acx

using namespace acx;

extern "C" int aceapex_decode_noalloc(const void* d_arc, uint64_t arc_len, void* d_out, uint64_t out_cap,
                                      void* stream) {
    if (!d_arc || !d_out) return ACEAPEX_E_ARG;
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return ACEAPEX_E_CUDA;
    uint8_t* base = nullptr;
    {
        // set-up on the first call on this device (with that device current):
        // the host-side name of the array is not a device address
        std::lock_guard<std::mutex> lock(g_na_mutex);
        if (!g_na_base[dev]) {
            void* p = nullptr;
            if (cudaGetSymbolAddress(&p, g_noalloc_scratch) != cudaSuccess || !p) return ACEAPEX_E_CUDA;
            g_na_base[dev] = static_cast<uint8_t*>(p);
        }
        base = g_na_base[dev];
    }
    cudaStream_t st = (cudaStream_t)stream;
    if (launch_kernel(k_plan_small, 1, kPlanThreads, 0, st, (const uint8_t*)d_arc, arc_len, base) != cudaSuccess)
        return ACEAPEX_E_CUDA;
    NaSummary S;
    if (cudaMemcpyAsync(&S, base + kOffSummary, sizeof S, cudaMemcpyDeviceToHost, st) != cudaSuccess ||
        cudaStreamSynchronize(st) != cudaSuccess)
        return ACEAPEX_E_CUDA;
    if (S.status == -1) return ACEAPEX_E_ARG;  // beyond the static scratch limits
    if (S.status != 0) return ACEAPEX_E_CORRUPT;
    if (out_cap < S.total) return ACEAPEX_E_ARG;
    if (S.n_blocks == 0) return ACEAPEX_OK;
    // the kernels move 16 bytes at a time (see the regular path's check)
    if (((uintptr_t)d_arc & 15) || (S.total >= 16 && ((uintptr_t)d_out & 15))) return ACEAPEX_E_ARG;
    const size_t lsm = local_smem_bytes(S.max_tok, S.max_lenb, S.max_lit);
    if (lsm > kMaxSmem) return ACEAPEX_E_CORRUPT;  // as the regular plan: no valid block needs that much
    JobDev job{};
    ArcJob& J = job.one;
    J.arc = (const uint8_t*)d_arc;
    J.blk = reinterpret_cast<const BlockDev*>(base + kOffPlan);
    J.dtab = reinterpret_cast<const uint32_t*>(base + kOffTab);
    J.scratch = base + kOffStreams;
    J.out = (uint8_t*)d_out;
    J.npend = reinterpret_cast<uint32_t*>(base + kOffNpend);
    J.pmap = reinterpret_cast<uint32_t*>(base + kOffPmap);
    J.spans = reinterpret_cast<SpanRec*>(base + kOffSpans);
    J.total = S.total;
    J.n_blocks = S.n_blocks;
    J.lo = 0;
    J.hi = S.n_blocks;
    J.min_match = S.min_match;
    J.deps = S.has_deps ? reinterpret_cast<const uint32_t*>(base + kOffDeps) : nullptr;
    job.n_arcs = 1;
    job.n_items = S.n_blocks;
    job.counters = reinterpret_cast<uint32_t*>(base + kOffCounters);
    job.err = reinterpret_cast<int*>(base + kOffErr);
    job.timeout_ns = 2000000000ull;
    job.max_tok = S.max_tok;
    job.max_lenb = S.max_lenb;
    job.max_lit = S.max_lit;
    job.lists[0] = reinterpret_cast<JobDev::ListEnt*>(base + kOffLists);
    job.lists[1] = job.lists[0] + kNaSpanSlots;
    int n_sms = 0;
    if (cudaDeviceGetAttribute(&n_sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) return ACEAPEX_E_CUDA;
    note_sm_count(n_sms);
    // the array keeps the previous call's contents: clear the error word; the
    // prologue kernel clears the tickets and statistics
    if (cudaMemsetAsync(job.err, 0, 16, st) != cudaSuccess) return ACEAPEX_E_CUDA;
    if (launch_prologue(job.counters, 3 + 1, st) != cudaSuccess) return ACEAPEX_E_CUDA;
    if (launch_rans(job, std::max(1, rans_occupancy()) * n_sms, st) != cudaSuccess) return ACEAPEX_E_CUDA;
    if (launch_local(job, std::max(1, local_occupancy(lsm)) * n_sms, st) != cudaSuccess) return ACEAPEX_E_CUDA;
    if (launch_external(job, std::max(1, external_occupancy()) * n_sms, st) != cudaSuccess) return ACEAPEX_E_CUDA;
    int err[4] = {0, 0, 0, 0};
    if (cudaMemcpyAsync(err, job.err, sizeof err, cudaMemcpyDeviceToHost, st) != cudaSuccess ||
        cudaStreamSynchronize(st) != cudaSuccess)
        return ACEAPEX_E_CUDA;
    return err[0];
}
