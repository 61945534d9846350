// Host-side launchers shared by the C-ABI implementation (not part of the public ABI).
#pragma once
#include "pic_common.cuh"

namespace pic {

bool build_ttable(int l, int scheme, double dtt, TTable *t, bool fixed = false);
int ttable_eval_host(const TTable *t, int l, double delta, double *w);

// CTAs per tile of a single run's 2D particle pass (tile_2d's split), from the tile and particle
// counts.  A grid of few tiles left most SMs idle: 64x32 cells are 4 to 8 tiles, 256x128 are 64,
// on 304 CTA slots (two per SM).  Every tile takes as many parts as fill the slots once, down to
// one warp of each species per part (particle kernel, us, one CTA per tile -> this rule: FP64
// 64x32 quadratic at 4 per cell 105 -> 21, FP32 50 -> 23, FP32 250x126 cubic at 8 per cell 85 ->
// 44, FP32 256x128 quartic at 64 per cell 445 -> 173).  The FP64 form, bound by a pipe every CTA
// of the SM shares, also splits a grid of few waves so that its last wave is short, while a part
// keeps 256 particles of a species (512x256 cubic at 64 per cell: 7388 -> 6362 us); the FP32 form
// loses there to the parts' extra stages and flushes (256 tiles: 421 us with one part, 432 with
// two) and stays at one wave.
inline unsigned tile_parts(const RunDev &rd)
{
    int dev = 0, sms = 0;
    if (cudaGetDevice(&dev) != cudaSuccess
        || cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
        return 1;
    int64_t n = 0;
    for (int s = 0; s < rd.nsp; ++s) n = rd.sp[s].n > n ? rd.sp[s].n : n;
    const int64_t slots = 2 * (int64_t)sms, per_tile = (n + rd.ntiles - 1) / rd.ntiles;
    int64_t parts = slots / rd.ntiles;
    if (rd.prec == 0) {
        const int64_t want = (8 * slots + rd.ntiles - 1) / rd.ntiles, most = per_tile / 256;
        const int64_t p = want < most ? want : most;
        if (p > parts) parts = p;
    }
    const int64_t most = (per_tile + 31) / 32;
    if (parts > most) parts = most;
    return (unsigned)(parts > 1 ? parts : 1);
}
// fused gather-push-deposit over all tiles of one run
cudaError_t launch_gpp(const RunDev &rd, int kt, cudaStream_t st);
size_t gpp_smem_bytes(const RunDev &rd);
// the 3D particle pass of either form (pic_gpp3d.cu); dynamic shared memory of its blocks
cudaError_t launch_gpp3d(const RunDev &rd, int kt, cudaStream_t st);
size_t gpp3d_smem_bytes(const RunDev &rd);

// Yee and grid kernels
cudaError_t launch_yee_b(const RunDev &rd, bool first, bool last, cudaStream_t st);
cudaError_t launch_yee_e(const RunDev &rd, bool shadow, cudaStream_t st);
cudaError_t launch_shadow(const RunDev &rd, cudaStream_t st);

// particle packing (load / read back)
// particles p0 .. p0 + m - 1; x[a * xs + i], u[a * us + i] hold particle p0 + i
cudaError_t launch_pack(const RunDev &rd, int s, const double *x, int64_t xs, const double *u,
                        int64_t us, int64_t m, int64_t p0, cudaStream_t st);
// drifting plasma generated on the device: SplitMix64 stream keys of the offsets (per axis),
// the two Box-Muller uniforms of each momentum component and the flip uniform
struct LoadKeys {
    uint64_t pos[3];
    uint64_t mom[6];
    uint64_t flip;
    uint64_t jut[4];  // Sobol's method: the four uniforms of an attempt
    uint64_t dir[2];  // isotropic direction of a Juttner momentum
};
// theta > 0: Juttner-Synge co-moving momenta of temperature theta (u_th unused); else Gaussian
cudaError_t launch_load_plasma(const RunDev &rd, int s, const LoadKeys &keys, int64_t per_cell,
                               double gamma, double u_th, double theta, int64_t n, cudaStream_t st);
// particles p0 .. p0 + m - 1 -> x[a * m + i], u[a * m + i], cell[i]
cudaError_t launch_unpack(const RunDev &rd, int s, double *x, double *u, int64_t *cell,
                          int64_t m, int64_t p0, cudaStream_t st);

// diagnostics (device doubles): out[0] field energy sum, out[1] kinetic energy, out[2] max
// |D.E - rho|, out[3] max |G - gref| (gref != null), out[4] max continuity residual against
// rho_prev (rho_prev != null); rho receives the charge density of the current particles
cudaError_t launch_diag(const RunDev &rd, double *out, double *rho, const double *gref,
                        const double *rho_prev, cudaStream_t st);
// G = D.E - rho of the current state into gref (rho and 3 doubles of scratch overwritten)
cudaError_t launch_gauss_ref(const RunDev &rd, double *rho, double *gref, double *scratch,
                             cudaStream_t st);
// fixed-point current of a deterministic run -> FP64 (after the particle pass)
cudaError_t launch_det_finish(const RunDev &rd, cudaStream_t st);
// FP32 current of a 3D FP32 run (RunDev::J32) -> F[6..8] (after the particle pass)
cudaError_t launch_j32_finish(const RunDev &rd, cudaStream_t st);

// tile sort of species s0 .. s0 + ns - 1 (ns > 1 only with RunDev::sc_more) into their other
// buffers; adds its kernels to *launches
cudaError_t launch_sort(const RunDev &rd, int s0, int ns, cudaStream_t st, int64_t *launches);

}  // namespace pic
