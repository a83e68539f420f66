// Host-side launchers of the decode kernels (defined in the .cu files).
#pragma once
#include <cuda_runtime.h>
#include <stddef.h>
#include <stdint.h>

#include "internal.h"

namespace acx {

// The most shared memory a CTA may have (sm_103a), and a kernel's permission to
// use it.  The permission belongs to the kernel on the device, not to a launch:
// it is always the whole, so that no thread narrows it between another's
// permission and launch (set to each job's own workspace, 657 of 3,000 decodes of
// two threads failed to launch).  A launch still takes what its workspace needs.
constexpr size_t kMaxSmem = 227 * 1024;
template <class K>
cudaError_t allow_max_smem(K kernel) {
    return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kMaxSmem);
}

// Launch a kernel.  The status is this launch's own: reading the runtime's last
// error behind a <<<>>> launch would report an earlier call's failure again.
template <class K, class... A>
cudaError_t launch_kernel(K kernel, dim3 grid, int block, size_t smem, cudaStream_t st, const A&... args) {
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = grid;
    cfg.blockDim = dim3((unsigned)block);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    return cudaLaunchKernelEx(&cfg, kernel, args...);
}

// Launch a kernel that begins with grid_dependency_wait() and may come up while
// the kernel before it on the stream still runs (programmatic dependent launch):
// its launch, and what it does before the wait, hide behind that kernel (10 KB
// file 75 -> 70 us, 1 MB without allocations 154 -> 145, 64 MiB genome 231 -> 224).
template <class K, class... A>
cudaError_t launch_dependent(K kernel, int grid, int block, size_t smem, cudaStream_t st, const A&... args) {
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((unsigned)grid);
    cfg.blockDim = dim3((unsigned)block);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kernel, args...);
}

// Clears counters[0, n_counters) and the statistics/list/barrier words, and
// errs[0, n_errs) (status words that the kernels set).
cudaError_t launch_prologue(uint32_t* counters, uint32_t n_counters, cudaStream_t st, int* errs = nullptr,
                            uint32_t n_errs = 0);
cudaError_t launch_rans(const JobDev& job, int grid, cudaStream_t st);
cudaError_t launch_local(const JobDev& job, int grid, cudaStream_t st);
// Cooperative launch (every CTA resident); recorded as a cooperative kernel
// node when the stream is being captured into a graph.
cudaError_t launch_external(const JobDev& job, int grid, cudaStream_t st);
// Run launch(arg) (a cooperative launch on st) after the previous cooperative
// launch of this process on the current device has completed, and make it the
// one the next waits for (see assemble.cu).
cudaError_t coop_ordered(cudaStream_t st, cudaError_t (*launch)(void*), void* arg);
// The level list of a level-ordered job (kJobLevels): a per-level scan over
// the items, then one warp per item writes its pieces' entries.
cudaError_t launch_level_list(const JobDev& job, cudaStream_t st);
cudaError_t launch_plain(const JobDev& job, int grid, cudaStream_t st);
// Fused entropy stage + local pass of a whole single-archive job (job.ready
// set, its flags cleared): G local groups per CTA, one CTA per SM
// (cooperative).  fused_groups: the most groups whose workspaces fit a CTA
// for blocks of max_tok tokens, max_lenb length bytes and max_lit
// literals (0: none fits).
cudaError_t launch_fused(const JobDev& job, int G, int grid, cudaStream_t st);
int fused_groups(uint32_t max_tok, uint32_t max_lenb, uint32_t max_lit, bool lvl);
int fused_occupancy(int G, uint32_t max_tok, uint32_t max_lenb, uint32_t max_lit, bool lvl);
size_t local_smem_bytes(uint32_t T, uint32_t LB, uint32_t LIT, bool need = false, bool lvl = false);
int rans_occupancy();
// Grid of a persistent kernel for a job that can use `need` CTAs at most:
// no more than `full`, and no fewer than one per SM, so that a mid-size job
// spreads its warps over the whole GPU instead of packing a few SMs.  The SM
// count is recorded when a context is created (no API call at launch time,
// which may be inside a graph capture).
int job_grid(int full, uint64_t need);
void note_sm_count(int n_sms);
int noted_sm_count();
int local_occupancy(size_t smem);
// Does a job of many blocks run the local pass with its narrow CTAs?
bool local_narrow(size_t smem);
int external_occupancy();
int plain_occupancy();
// Copy regions out of block slots (block a at out + slot[a]*kBlock): the one
// request `one` (list == nullptr) or list[0, n_req); max_len sizes the grid.
cudaError_t launch_gather(const GatherReq* one, const GatherReq* list, uint32_t n_req, uint64_t max_len,
                          const uint8_t* out, const uint32_t* slot, cudaStream_t st);

}  // namespace acx
