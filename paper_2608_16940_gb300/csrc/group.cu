// Launches of the group passes (group.cuh): one state, and the batched
// trajectories.
#include <cooperative_groups.h>
#include <cuda_runtime.h>

#include <algorithm>

#include "group.cuh"

namespace qsa {

namespace {

using namespace dev;

extern __shared__ __align__(16) unsigned char smem_raw[];

// Two CTAs per SM: 64 KiB of stages and up to 38 KiB of program each.
__global__ void __launch_bounds__(group::kThreads, 2)
    k_group(float2* psi, const __grid_constant__ GroupPass pass, const unsigned char* progs, uint32_t prog_cap, int zero) {
    __shared__ GroupPass p;
    if (threadIdx.x < sizeof(GroupPass) / sizeof(uint64_t))
        reinterpret_cast<uint64_t*>(&p)[threadIdx.x] = reinterpret_cast<const uint64_t*>(&pass)[threadIdx.x];
    __syncthreads();
    float2* stage = reinterpret_cast<float2*>(smem_raw);
    unsigned char* prog = smem_raw + sizeof(float2) * 2 * group::kAmps;
    group::Tables& tb = *reinterpret_cast<group::Tables*>(prog + prog_cap);
    group::fetch_program(progs + p.prog, p.bytes, prog);
    group::run_pass(p, psi, stage, prog, tb, blockIdx.x, gridDim.x, zero != 0);
}

namespace cg = cooperative_groups;

// Batched trajectories in one persistent launch: a cluster of CTAs pops a
// trajectory from an atomic queue (longest first) and applies its passes from
// |0...0> (the first pass generates it), the CTAs splitting every pass's tiles
// (rank r takes tiles r, r + C, ...) and meeting at a cluster barrier between
// passes.
__global__ void __launch_bounds__(group::kThreads, 2) k_batch_evolve(BatchArgs a) {
    float2* stage = reinterpret_cast<float2*>(smem_raw);
    unsigned char* prog = smem_raw + sizeof(float2) * 2 * group::kAmps;
    group::Tables& tb = *reinterpret_cast<group::Tables*>(prog + kGroupProgBytes);
    // Rank 0 of the cluster pops the queue and makes the watchdog's decision;
    // the others read them from its shared memory after a cluster barrier, so
    // every CTA of a cluster takes the same path and meets the same barriers
    // (s_stop alternates by pass so a value is never rewritten before all have
    // read it; s_slot is rewritten only after the trajectory's barriers).
    __shared__ int s_slot;
    __shared__ int s_stop[2];
    __shared__ GroupPass s_pass;
    cg::cluster_group cluster = cg::this_cluster();
    const unsigned crank = cluster.block_rank(), csize = cluster.num_blocks();
    const long long t_start = clock64();
    for (;;) {
        if (crank == 0 && threadIdx.x == 0) s_slot = static_cast<int>(atomicAdd(a.queue, 1u));
        cluster.sync();
        const int slot = *cluster.map_shared_rank(&s_slot, 0);
        if (slot >= a.n_traj) {
            cluster.sync();   // no CTA leaves while another may still read its shared memory
            break;
        }
        const int traj = a.order[slot];
        float2* psi = a.states + (static_cast<uint64_t>(traj) << a.n);
        const uint32_t p0 = a.pstart[traj], p1 = a.pstart[traj + 1];
        if (p0 == p1) {   // an empty trajectory: |0...0> itself, a share per CTA
            float4* p4 = reinterpret_cast<float4*>(psi);
            const uint64_t npairs = (1ull << a.n) >> 1;
            for (uint64_t i = crank * blockDim.x + threadIdx.x; i < npairs; i += csize * blockDim.x)
                p4[i] = make_float4(i == 0 ? 1.f : 0.f, 0.f, 0.f, 0.f);
            cluster.sync();
        }
        for (uint32_t p = p0; p < p1; ++p) {
            if (threadIdx.x < sizeof(GroupPass) / sizeof(uint64_t))
                reinterpret_cast<uint64_t*>(&s_pass)[threadIdx.x] =
                    reinterpret_cast<const uint64_t*>(a.passes + p)[threadIdx.x];
            __syncthreads();
            group::fetch_program(a.progs + a.prog_base[traj] + s_pass.prog, s_pass.bytes, prog);
            group::run_pass(s_pass, psi, stage, prog, tb, crank, csize, p == p0);
            // the pass's tiles are written before any CTA of the cluster reads
            // them in the next pass; the watchdog's decision travels with it
            if (crank == 0 && threadIdx.x == 0)
                s_stop[p & 1] = (a.budget != 0 && static_cast<unsigned long long>(clock64() - t_start) > a.budget) ? 1 : 0;
            __threadfence();
            cluster.sync();
            if (*cluster.map_shared_rank(&s_stop[p & 1], 0)) {
                if (crank == 0 && threadIdx.x == 0) atomicExch(a.err, 7);
                cluster.sync();
                return;
            }
        }
    }
}

}  // namespace

QSA_BOUNDS_READER(bounds_word_group)

cudaError_t launch_group(float2* psi, int n, const GroupPass& p, const unsigned char* d_progs, bool zero,
                         cudaStream_t st, uint64_t* launches) {
    if (p.T != std::min(kGroupTileBits, n) || p.bytes > kGroupProgBytes) return cudaErrorInvalidValue;
    cudaError_t e = set_smem_attr(reinterpret_cast<const void*>(k_group), static_cast<int>(group::smem_bytes(kGroupProgBytes)));
    if (e != cudaSuccess) return e;
    const uint64_t grid = std::min<uint64_t>(p.ntiles, 2ull * num_sms());
    k_group<<<static_cast<unsigned>(grid), group::kThreads, group::smem_bytes(p.bytes), st>>>(psi, p, d_progs, p.bytes,
                                                                                             zero ? 1 : 0);
    ++*launches;
    return cudaGetLastError();
}

cudaError_t launch_batch_evolve(const BatchArgs& a, cudaStream_t st, uint64_t* launches) {
    const size_t smem = group::smem_bytes(kGroupProgBytes);
    cudaError_t e = set_smem_attr(reinterpret_cast<const void*>(k_batch_evolve), static_cast<int>(smem));
    if (e != cudaSuccess) return e;
    // a trajectory's passes run one after another, so the batch ends when its
    // deepest trajectory does: up to four CTAs share one, as many as it has tiles
    unsigned csize = a.n >= kGroupTileBits + 2 ? 4 : a.n == kGroupTileBits + 1 ? 2 : 1;
    // eight when the trajectories would leave half of the CTA slots empty with four (with more of them
    // than slots, larger clusters only add waiting: 128 at N = 20, 29.5 / 30.0 / 35.2 ms with 4 / 8 / 16)
    if (a.n >= kGroupTileBits + 4 && a.n_traj * 8 <= 2 * num_sms()) csize = 8;
    // one cluster per trajectory in flight (clusters that find the queue empty leave at once)
    unsigned clusters = std::max(1u, static_cast<unsigned>(2 * num_sms()) / csize);
    clusters = std::min(clusters, static_cast<unsigned>(a.n_traj));
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(clusters * csize);
    cfg.blockDim = dim3(group::kThreads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeClusterDimension;
    at.val.clusterDim.x = csize;
    at.val.clusterDim.y = 1;
    at.val.clusterDim.z = 1;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    e = cudaLaunchKernelEx(&cfg, k_batch_evolve, a);
    if (e != cudaSuccess) return e;
    ++*launches;
    return cudaGetLastError();
}

}  // namespace qsa
