// Entropy stage of the decode (paper, Table 1/2: "ANS"): the persistent
// k_rans kernel (one warp per block, see rans_dev.cuh) and the launchers.
#include <algorithm>
#include <atomic>

#include "launch.h"
#include "rans_dev.cuh"

namespace acx {

// Start of a decode call: every ticket and statistic restarts at zero.
__global__ void k_prologue(uint32_t* counters, uint32_t n_counters, int* errs, uint32_t n_errs) {
    grid_launch_dependents();
    for (uint32_t i = threadIdx.x; i < n_counters; i += blockDim.x) counters[i] = 0;
    for (uint32_t i = threadIdx.x; i < n_errs; i += blockDim.x) errs[i] = 0;
    if (threadIdx.x < kLvStripes) counters[kLvTickets + threadIdx.x] = 0;
    if (threadIdx.x == 0) {
        counters[kStatPending] = 0;
        counters[kStatPolls] = 0;
        counters[kListCnt] = 0;
        counters[kListCnt + 1] = 0;
        counters[kBarCount] = 0;
        counters[kStatPendBytes] = 0;
        counters[kStatPendBytes + 1] = 0;
    }
}

// Each CTA works on one archive at a time (its tables in shared memory);
// its warps take blocks of that archive from the archive's ticket, and when
// the archive is exhausted the CTA moves to the archive with the most blocks
// left.  A lone archive has a kernel of its own, which reads its job from the
// parameters: with the archive's fields in registers the kernel, at its 64 per
// thread, spilled four times as much (254 MB genome 254 -> 240 us).
template <bool kMulti>
__global__ void __launch_bounds__(kRansWarps * 32) k_rans(JobDev job) {
    extern __shared__ __align__(128) uint8_t smraw[];
    RansSmem& S = *reinterpret_cast<RansSmem*>(smraw);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (lane < kSlots) mbar_init(&S.bar[warp][lane], 1);
    if (lane == kSlots) mbar_init(&S.sbar[warp], 1);
    if (threadIdx.x < 4) mbar_init(&S.tbar[threadIdx.x], 1);
    grid_launch_dependents();
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    if (threadIdx.x == 0) {
        const uint64_t target = (uint64_t)blockIdx.x * job.n_items / gridDim.x;
        S.next_arc = kMulti ? find_arc(job, (uint32_t)target) : 0;
        S.arc = -1;
    }
    __syncthreads();
    uint64_t deadline = 0;  // the entropy stage waits only for its copies
    uint32_t seq = 0, sphase = 0, tphase = 1;
    uint32_t* tickets = job.counters + 3;
    const uint32_t ring_s = ring_addr(S, warp);
    for (;;) {
        const int a = S.next_arc;
        if (a < 0) break;
        const ArcJob J = kMulti ? job.arcs[a] : job.one;
        if (S.arc != a) {
            // (every warp has left the tables of the archive before)
            if (threadIdx.x == 0) {
                asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                for (int k = 0; k < 4; k++) {
                    const int s = k == 0 ? kLit : k - 1;  // the literals' first: the longest streams
                    mbar_arrive_tx(&S.tbar[s], 4 * kM);
                    tma_load_1d(S.tab[s], J.dtab + s * kM, 4 * kM, &S.tbar[s]);
                }
            }
            tphase ^= 1;
            __syncthreads();
            if (threadIdx.x == 0) S.arc = a;
        }
        const TabLoad T{S.tbar, tphase};
        if (!deadline) {
            // (plans and tables do not depend on the kernel before, tickets do)
            grid_dependency_wait();
            deadline = gtimer() + kCopyWaitNs;
        }
        // tickets: the blocks, or (rans_parts) their literals, then their other
        // parts; a lone archive's first run of every warp is its own, so that
        // the work starts spread over the SMs however their CTAs come up
        const uint32_t n_blk = J.hi - J.lo, n_a = n_blk * job.rans_parts;
        const uint32_t chunk = job.chunk ? job.chunk : 1u;
        const uint32_t own = kMulti ? 0u : gridDim.x * kRansWarps * chunk;
        uint32_t cnext = (warp * gridDim.x + blockIdx.x) * chunk;  // this warp's current run of `chunk` tickets
        uint32_t cleft = own ? chunk : 0u;
        for (;;) {
            if (cleft == 0) {
                uint32_t t0 = 0;
                if (lane == 0) t0 = atomicAdd(&tickets[a], chunk);
                cnext = own + __shfl_sync(ACX_FULL, t0, 0);
                cleft = chunk;
            }
            const uint32_t tk = cnext++;
            cleft--;
            if (tk >= n_a) break;
            const uint32_t turn = tk / n_blk, i = tk - turn * n_blk;
            const uint32_t part = job.rans_parts == 1 ? kRansAll : kRansParts - 1 - turn;
            rans_block(job, a, J, item_ref(J, J.order ? J.order[i] : i), part, T, smem_u32(&S.tab[0][0]), ring_s,
                       smem_u32(&S.stage[warp][0]), &S.bar[warp][0], &S.sbar[warp], seq, sphase, lane, deadline);
        }
        // a warp without work has not waited for the tables: their copies land
        // before the CTA leaves or the next archive's go out
        if (warp == 0)
            for (int s = 0; s < 4; s++) wait_table(T, s, deadline);
        if (!kMulti) break;
        __syncthreads();
        if (warp == 0) {
            // the archive with the most tickets left, the lowest of equals
            uint32_t best = 0xffffffffu, best_left = 0;
            for (uint32_t k = lane; k < job.n_arcs; k += 32) {
                const uint32_t taken = *((volatile uint32_t*)&tickets[k]);
                const uint32_t n_k = (job.arcs[k].hi - job.arcs[k].lo) * job.rans_parts;
                const uint32_t left = taken < n_k ? n_k - taken : 0;
                if (left > best_left) { best_left = left; best = k; }
            }
            const uint32_t most = __reduce_max_sync(ACX_FULL, best_left);
            best = __reduce_min_sync(ACX_FULL, best_left == most ? best : 0xffffffffu);
            if (lane == 0) S.next_arc = most ? (int)best : -1;
        }
        __syncthreads();
    }
}

size_t rans_smem_bytes() { return sizeof(RansSmem); }

static std::atomic<int> g_sm_count{0};

void note_sm_count(int n_sms) { g_sm_count.store(n_sms); }

int noted_sm_count() { return std::max(g_sm_count.load(), 1); }

int job_grid(int full, uint64_t need) {
    const uint64_t g = std::max<uint64_t>(need, (uint64_t)noted_sm_count());
    return (int)std::max<uint64_t>(1, std::min<uint64_t>((uint64_t)full, g));
}

cudaError_t launch_prologue(uint32_t* counters, uint32_t n_counters, cudaStream_t st, int* errs, uint32_t n_errs) {
    return launch_kernel(k_prologue, 1, 128, 0, st, counters, n_counters, errs, n_errs);
}

cudaError_t launch_rans(const JobDev& job_in, int grid, cudaStream_t st) {
    JobDev job = job_in;
    const size_t sm = rans_smem_bytes();
    const auto kernel = job.arcs ? k_rans<true> : k_rans<false>;
    cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
    if (e != cudaSuccess) return e;
    // When every part of every block finds a warp at once, a block's streams
    // decode on three warps and only the longest counts (one 10 KB text block
    // 47 -> 27 us, 4 MiB of text 62 -> 31, 4 MiB DNA-like 65 -> 54); with more
    // blocks the warps are busy anyway, and a part would only cost a ticket.
    const uint64_t warps = (uint64_t)kRansWarps * (uint64_t)grid;
    job.rans_parts = (uint64_t)job.n_items * kRansParts <= warps ? kRansParts : 1;
    // One CTA per SM while that gives every ticket run a warp (each CTA loads
    // the 64 KiB of tables), else all: with a grid cut to the need, some SMs
    // have twice the warps of others (4,097 blocks: 95 us, 90 with all).
    const uint64_t per_cta = (uint64_t)kRansWarps * (job.chunk ? job.chunk : 1);
    const uint64_t need = ((uint64_t)job.n_items * job.rans_parts + per_cta - 1) / per_cta;
    if (need <= (uint64_t)noted_sm_count()) grid = std::min(grid, noted_sm_count());
    return launch_dependent(kernel, grid, kRansWarps * 32, sm, st, job);
}

int rans_occupancy() {
    const size_t sm = rans_smem_bytes();
    int n = 0, m = 0;
    cudaFuncSetAttribute(k_rans<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
    cudaFuncSetAttribute(k_rans<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, k_rans<false>, kRansWarps * 32, sm) != cudaSuccess ||
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&m, k_rans<true>, kRansWarps * 32, sm) != cudaSuccess)
        return 0;
    return std::min(n, m);
}

}  // namespace acx
