// Launches of the resident chain kernel and the frame evaluator (kern_chain.cuh): shared
// memory, cluster sizes. The instantiations of each cluster size are a translation unit of
// their own, so that they compile side by side.
#include "kern_chain.cuh"

namespace scps {

SCPS_RESIDENT_LAUNCHERS(extern, 1, false)
SCPS_RESIDENT_LAUNCHERS(extern, 1, true)
SCPS_RESIDENT_LAUNCHERS(extern, 2, true)
SCPS_RESIDENT_LAUNCHERS(extern, 4, true)
SCPS_RESIDENT_LAUNCHERS(extern, 8, true)
SCPS_EVAL_LAUNCHERS(extern, 1)
SCPS_EVAL_LAUNCHERS(extern, 2)
SCPS_EVAL_LAUNCHERS(extern, 4)
SCPS_EVAL_LAUNCHERS(extern, 8)
SCPS_MAX_CLUSTERS(extern, 4)
SCPS_MAX_CLUSTERS(extern, 8)

// Shared-memory bytes of the resident kernels for nta atom slots (plus the 8 sentinel
// slots): positions with charges and LJ parameters, velocities, the xi array and the two
// parities of force and bias-gradient partials (modular and coarse words).
size_t resident_smem_bytes(int nta) {
    const size_t na8 = (size_t)nta + 8;
    return sizeof(float4) * (na8 + 2 * (size_t)nta) + sizeof(float2) * na8 +
           2 * 4 * 3 * sizeof(int) * na8;
}

// Dynamic shared memory a resident or frame-evaluation CTA may request on the current
// device: the opt-in per-block limit less the static shared block of those kernels.
// 0 when the device cannot be queried (nothing then fits).
size_t resident_smem_limit() {
    int dev = 0, optin = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return 0;
    if (cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev) != cudaSuccess)
        return 0;
    const size_t stat = (kChainStaticSmem + 15) & ~(size_t)15;
    return (size_t)optin > stat ? (size_t)optin - stat : 0;
}

constexpr int kMaxCacheItems = 8192;

// Dynamic shared memory of a launch with CTAs of `threads` threads: the resident state plus
// a cache of pair items (CacheItem, 64 B) in what the state leaves free; CTAs of up to 512
// threads keep room for a second CTA on their SM. Sets *lc_cap to the cache's capacity.
size_t launch_smem(int nta, int threads, int cl, int* lc_cap) {
    const size_t base = resident_smem_bytes(nta);
    size_t lim = resident_smem_limit();
    if (threads <= 512) {
        int dev = 0, per_sm = 0, reserved = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&per_sm, cudaDevAttrMaxSharedMemoryPerMultiprocessor, dev);
        cudaDeviceGetAttribute(&reserved, cudaDevAttrReservedSharedMemoryPerBlock, dev);
        const size_t stat = (kChainStaticSmem + 15) & ~(size_t)15;
        const size_t two = (size_t)per_sm / 2;
        const size_t half = two > (size_t)reserved + stat ? two - (size_t)reserved - stat : 0;
        lim = std::min(lim, half);
    }
    size_t cap = lim > base ? (lim - base) / sizeof(CacheItem) : 0;
    // no more than the lists of compact chains need (about 1.8 x 80 pairs per atom in items
    // of 128, per CTA): shared memory and the L1 cache share the SM's storage, and the L1
    // serves the topology tables; longer tables stay in global memory
    cap = std::min(cap, std::min((size_t)kMaxCacheItems, (size_t)(cl == 1 ? 2 * nta : 2 * nta / cl)));
    *lc_cap = (int)cap;
    return base + cap * sizeof(CacheItem);
}

// Clusters of `cl` CTAs (4 or 8) of the resident kernel that run at once.
int chain_max_clusters(int cl, int nta, int threads) {
    return cl == 8 ? max_clusters_cl<8>(nta, threads) : max_clusters_cl<4>(nta, threads);
}

// Whether `count` lone CTAs run in the wide form: the narrow form's 64 registers spill more
// (300 replicas of 64 atoms 7.1 us per step, 6.6 in the wide form; 128 atoms 13.2 and 12.2), but
// more of its CTAs share an SM, which pays where that saves a wave (600 of 128 atoms 23.4 and
// 26.4; 304 of 560 on 512 threads 68 and 73).
static bool wide_form(int count, int nta, int threads) {
    int dev = 0, n_sm = 0, per_sm = 0, reserved = 0, lc_cap = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&n_sm, cudaDevAttrMultiProcessorCount, dev);
    cudaDeviceGetAttribute(&per_sm, cudaDevAttrMaxSharedMemoryPerMultiprocessor, dev);
    cudaDeviceGetAttribute(&reserved, cudaDevAttrReservedSharedMemoryPerBlock, dev);
    const int smem = (int)(launch_smem(nta, threads, 1, &lc_cap) + kChainStaticSmem) + reserved;
    auto waves = [&](int regs) {
        const int fit = std::max(1, std::min(65536 / (regs * threads), per_sm / smem));
        return (count + fit * n_sm - 1) / std::max(1, fit * n_sm);
    };
    return waves(80) <= waves(64);
}

cudaError_t launch_resident(int elec, int cluster, const TopoDev* topos, const RepDev* reps,
                            const StateDev& st, const RunParams& P, int nta, int threads,
                            cudaStream_t stream) {
    switch (cluster) {
        case 8: return launch_resident_cl<8, true>(elec, topos, reps, st, P, nta, threads, stream);
        case 4: return launch_resident_cl<4, true>(elec, topos, reps, st, P, nta, threads, stream);
        case 2: return launch_resident_cl<2, true>(elec, topos, reps, st, P, nta, threads, stream);
        default: break;
    }
    if (threads <= kMaxThreadsPair && wide_form(P.n_replicas, nta, threads))
        return launch_resident_cl<1, true>(elec, topos, reps, st, P, nta, threads, stream);
    return launch_resident_cl<1, false>(elec, topos, reps, st, P, nta, threads, stream);
}

cudaError_t launch_eval(int elec, const TopoDev* topo, const RunParams& P, const float* X,
                        double* U, float* F, double* Z, long long n_frames, int nta, int threads,
                        int cl, cudaStream_t stream) {
    switch (cl) {
        case 8: return launch_eval_cl<8>(elec, topo, P, X, U, F, Z, n_frames, nta, threads, stream);
        case 4: return launch_eval_cl<4>(elec, topo, P, X, U, F, Z, n_frames, nta, threads, stream);
        case 2: return launch_eval_cl<2>(elec, topo, P, X, U, F, Z, n_frames, nta, threads, stream);
        default: return launch_eval_cl<1>(elec, topo, P, X, U, F, Z, n_frames, nta, threads, stream);
    }
}

}  // namespace scps
