// Instantiations of the 2D particle pass of the plain FP64 form.
#include "pic_gpp_fx.cuh"
#include "pic_launch.h"

namespace pic {

namespace {

template <int L, int KT, bool DET>
__global__ void __launch_bounds__(32 * fx_warps(L), 2) k_gpp2d(const __grid_constant__ RunDev rd)
{
    extern __shared__ __align__(16) char smem[];
    tile_fx<L, KT, DET>(rd, smem, blockIdx.x);
}

template <int L, int KT>
cudaError_t go(const RunDev &rd, cudaStream_t st)
{
    const size_t smem = stage_fx_launch_bytes(rd);
    auto k = rd.det ? k_gpp2d<L, KT, true> : k_gpp2d<L, KT, false>;
    cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    k<<<dim3((unsigned)rd.ntiles, tile_parts(rd)), 32 * fx_warps(L), smem, st>>>(rd);
    return cudaGetLastError();
}

}  // namespace

cudaError_t launch_gpp_f64(const RunDev &rd, int kt, cudaStream_t st)
{
    if (rd.dim != 2) return launch_gpp3d(rd, kt, st);
    const bool wide = kt > rd.l + 1;
    switch (rd.l) {
    case 1: return wide ? go<1, 3>(rd, st) : go<1, 2>(rd, st);
    case 2: return wide ? go<2, 4>(rd, st) : go<2, 3>(rd, st);
    case 3: return wide ? go<3, 5>(rd, st) : go<3, 4>(rd, st);
    case 4: return wide ? go<4, 6>(rd, st) : go<4, 5>(rd, st);
    default: return cudaErrorInvalidValue;
    }
}

// What a 2D launch takes, and what it must have.
size_t gpp_launch_smem_bytes_f64(const RunDev &rd) { return stage_fx_launch_bytes(rd); }

size_t gpp_smem_bytes_f64(const RunDev &rd)
{
    return rd.dim == 2 ? stage_fx_bytes(rd.reg_nodes) : 0;
}

}  // namespace pic
