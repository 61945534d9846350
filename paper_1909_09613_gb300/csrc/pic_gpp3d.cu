// Instantiations of the fused particle pass in 3D, both forms.
#include "pic_gpp3d_fx.cuh"
#include "pic_launch.h"

namespace pic {

namespace {

// FP32 form, l <= 2: four blocks per SM (at most 128 registers; the staged stage of four blocks
// fits in shared memory and the extra warps hide latency); higher orders keep their registers
template <int L, int KT>
__global__ void __launch_bounds__(128, (L <= 2 ? 4 : 1)) k_gpp3d_f32(const __grid_constant__ RunDev rd)
{
    extern __shared__ __align__(16) float sf3[];
    tile_3d<L, KT>(rd, blockIdx.x, sf3);
}

template <int L, int KT, bool DET>
__global__ void __launch_bounds__(128, L <= 2 ? 4 : 2) k_gpp3d_f64(const __grid_constant__ RunDev rd)
{
    tile3_fx<L, KT, DET>(rd, blockIdx.x);
}

// CTAs per tile of the FP64 form, which stages nothing and so splits its tiles freely: eight
// waves of four CTAs per SM, so that the last wave is short, while every part keeps a particle of
// a species per thread.
unsigned tile_parts3(const RunDev &rd)
{
    int dev = 0, sms = 0;
    if (cudaGetDevice(&dev) != cudaSuccess
        || cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
        return 1;
    int64_t n = 0;
    for (int s = 0; s < rd.nsp; ++s) n = rd.sp[s].n > n ? rd.sp[s].n : n;
    const int64_t most = (n / rd.ntiles + 127) / 128;
    const int64_t want = (8 * 4 * (int64_t)sms + rd.ntiles - 1) / rd.ntiles;
    const int64_t parts = want < most ? want : most;
    return (unsigned)(parts > 1 ? parts : 1);
}

template <int L, int KT>
cudaError_t go(const RunDev &rd, cudaStream_t st)
{
    if (rd.prec == 1) {  // FP32 form
        const size_t smem = stage3d_bytes(rd);
        cudaError_t e = cudaFuncSetAttribute(k_gpp3d_f32<L, KT>,
                                             cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
        k_gpp3d_f32<L, KT><<<(unsigned)rd.ntiles, 128, smem, st>>>(rd);
    } else {
        const dim3 grid((unsigned)rd.ntiles, tile_parts3(rd));
        if (rd.det) k_gpp3d_f64<L, KT, true><<<grid, 128, 0, st>>>(rd);
        else k_gpp3d_f64<L, KT, false><<<grid, 128, 0, st>>>(rd);
    }
    return cudaGetLastError();
}

}  // namespace

cudaError_t launch_gpp3d(const RunDev &rd, int kt, cudaStream_t st)
{
    const bool wide = kt > rd.l + 1;
    switch (rd.l) {
    case 1: return wide ? go<1, 3>(rd, st) : go<1, 2>(rd, st);
    case 2: return wide ? go<2, 4>(rd, st) : go<2, 3>(rd, st);
    case 3: return wide ? go<3, 5>(rd, st) : go<3, 4>(rd, st);
    case 4: return wide ? go<4, 6>(rd, st) : go<4, 5>(rd, st);
    default: return cudaErrorInvalidValue;
    }
}

size_t gpp3d_smem_bytes(const RunDev &rd)
{
    return rd.prec == 1 ? stage3d_bytes(rd) : 0;
}

}  // namespace pic
