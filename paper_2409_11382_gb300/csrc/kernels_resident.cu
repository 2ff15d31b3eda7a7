// Resident V-cycles of the small coarse levels (sweep_resident.cuh), FP32 and
// FP64 levels in one kernel.  Compiled with --fmad=false: the shared sweep
// arithmetic writes every multiply-add it wants fused, and the FP64 levels must
// round as in the FP64 unit.
#include "sweep_resident.cuh"

cudaError_t biot::launch_resident(const biot::ResParams &P, size_t smem, cudaStream_t s)
{
    if (P.nprog < 1 || P.nprog > RES_MAX_PROGS || P.cs < 1 || P.cs > RES_CLUSTER_MAX || smem > (size_t)RES_SMEM_MAX)
        return cudaErrorInvalidValue;
    return P.ghosts ? launch_resident_kind<true>(P, smem, s) : launch_resident_kind<false>(P, smem, s);
}

int biot::resident_max_cluster()
{
    static DeviceCache found;
    const int n = found.get([](int) {
        cudaLaunchConfig_t cfg;
        cudaLaunchAttribute at[1];
        int clusters = 0;
        if (resident_config<true>(cfg, at[0], 1, RES_CLUSTER_MAX, RES_SMEM_MAX, nullptr) == cudaSuccess &&
            cudaOccupancyMaxActiveClusters(&clusters, k_resident_cycle<true>, &cfg) == cudaSuccess && clusters > 0)
            return RES_CLUSTER_MAX;
        cudaGetLastError();
        return 8;
    });
    return n ? n : 8;
}
