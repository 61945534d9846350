// Host-side launchers shared by the C-ABI implementation (not part of the public ABI).
#pragma once
#include "pic_common.cuh"

namespace pic {

bool build_ttable(int l, int scheme, double dtt, TTable *t, bool fixed = false);
int ttable_eval_host(const TTable *t, int l, double delta, double *w);

// CTA slots of the 2D particle passes (two per SM); 0 if the device does not say.
inline int64_t tile_slots()
{
    int dev = 0, sms = 0;
    if (cudaGetDevice(&dev) != cudaSuccess
        || cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
        return 0;
    return 2 * (int64_t)sms;
}

// particles of the fullest species per tile
inline int64_t tile_load(const RunDev &rd)
{
    int64_t n = 0;
    for (int s = 0; s < rd.nsp; ++s) n = rd.sp[s].n > n ? rd.sp[s].n : n;
    return (n + rd.ntiles - 1) / rd.ntiles;
}

// CTAs per tile of a single FP64 run's 2D particle pass (tile_fx's split).  A grid of few tiles
// left most SMs idle: 64x32 cells are 8 tiles on 304 CTA slots.  Every tile takes as many parts
// as fill the slots once, down to one warp of each species per part (64x32 quadratic at 4 per
// cell 105 -> 21 us).  Bound by a pipe every CTA of the SM shares, this form also splits a grid of
// few waves so that its last wave is short, while a part keeps 256 particles of a species
// (512x256 cubic at 64 per cell: 7388 -> 6362 us).
inline unsigned tile_parts(const RunDev &rd)
{
    const int64_t slots = tile_slots(), per_tile = tile_load(rd);
    int64_t parts = slots / rd.ntiles;
    const int64_t want = (8 * slots + rd.ntiles - 1) / rd.ntiles, full = per_tile / 256;
    const int64_t p = want < full ? want : full;
    if (p > parts) parts = p;
    const int64_t most = (per_tile + 31) / 32;
    if (parts > most) parts = most;
    return (unsigned)(parts > 1 ? parts : 1);
}

// particles of the fullest species a CTA keeps when the tiles are divided evenly (tile_ctas)
constexpr int64_t kEvenMin = 1024;

// CTAs of a single FP32 run's 2D particle pass; every CTA takes the same share of the grid's tiles
// (EvenSplit).  Whole tiles or whole parts of them left slots empty in a grid of few waves: 256
// tiles, or 64 tiles in 4 parts, are 256 CTAs on 304 slots.  A share that crosses a tile border
// stages twice and still wins (particle kernel, us, 512x256 at 32 per cell: quadratic 212 -> 193,
// cubic 229 -> 200; 256x128 quartic at 64 per cell 168 -> 162).  Where the lines lie (whole parts /
// even shares, us, 256x128): 431 particles of a species per CTA quadratic 45.7 / 47.6, 647 cubic 61.0 /
// 63.2, 862 cubic 69.5 / 66.9, 1293 cubic 81.1 / 78.8.  A deterministic run's CTAs are counted for the
// slots of a GB300 whatever the device: its warps add their lanes' FP32 currents before the fixed-point
// word, so which 32 particles meet must not depend on the device.
inline unsigned tile_ctas(const RunDev &rd)
{
    const int64_t slots = rd.det ? 304 : tile_slots(), per_tile = tile_load(rd), nt = rd.ntiles;
    // whole parts per tile, as many as fill the slots once, down to one warp of each species
    int64_t parts = slots / nt;
    const int64_t most = (per_tile + 31) / 32;
    if (parts > most) parts = most;
    if (parts < 1) parts = 1;
    // all slots of the last wave, where that leaves a CTA enough particles to pay for staging a
    // second tile and the waves are few
    if (slots > 0) {
        const int64_t waves = (nt * parts + slots - 1) / slots, g = slots * waves;
        if (waves <= 4 && 16 * g >= 17 * nt * parts && per_tile * nt / g >= kEvenMin) return (unsigned)g;
    }
    return (unsigned)(nt * parts);
}
// fused gather-push-deposit over all tiles of one run
cudaError_t launch_gpp(const RunDev &rd, int kt, cudaStream_t st);
size_t gpp_smem_bytes(const RunDev &rd);
// the 3D particle pass of either form (pic_gpp3d.cu); dynamic shared memory of its blocks
cudaError_t launch_gpp3d(const RunDev &rd, int kt, cudaStream_t st);
size_t gpp3d_smem_bytes(const RunDev &rd);

// Yee and grid kernels
// ahead of a call's first step: B half a step on, the current cleared
cudaError_t launch_yee_start(const RunDev &rd, cudaStream_t st);
// after the particle pass: E, then B to integer time (last step of a call) or half a step past it
cudaError_t launch_yee_step(const RunDev &rd, bool shadow, bool last, cudaStream_t st);
int yee_step_launches(const RunDev &rd);
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
