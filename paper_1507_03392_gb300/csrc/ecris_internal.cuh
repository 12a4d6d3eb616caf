// Internal definitions shared by the CUDA translation units of the ECRIS
// library: the per-run device parameter block, the tally layout and the
// device-side building blocks of the time step (Philox words, field model,
// E-grid gather).  Host-side API code lives in api.cu.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include <utility>

#include "../../include/ecris.h"

namespace ecris {

constexpr int kQSlots = 64;            // charge-state slots per tally array
// Tally words per run (u64): extracted[64], lost[64], kinetic energy of ions
// that left (micro-eV), Coulomb pair collisions.
constexpr int kTallyExtracted = 0;
constexpr int kTallyLost = 64;
constexpr int kTallyKe = 128;
constexpr int kTallyCoulomb = 129;
constexpr int kTallyWords = 132;
// first-passage times: 4 bins per octave of the age in steps (ages < 2^30)
constexpr int kFptdBins = ECRIS_FPTD_BINS;
// [Q][bin] counts, [Q] age sums, [Q] extraction radius sums (nm)
constexpr int kFptdWords = kQSlots * (kFptdBins + 2);
constexpr int kFptdAgeSum = kQSlots * kFptdBins;
constexpr int kFptdRadius = kQSlots * (kFptdBins + 1);

// meta word layout (matches the public header)
constexpr uint32_t kQMask = 0xFFu;
constexpr uint32_t kEvWall = 1u << 8;
constexpr uint32_t kEvExtract = 1u << 9;
constexpr uint32_t kEvIonize = 1u << 10;
constexpr uint32_t kEvCx = 1u << 11;
constexpr uint32_t kEvCoulomb = 1u << 12;
constexpr uint32_t kEvElastic = 1u << 13;
constexpr uint32_t kEvRecomb = 1u << 14;
constexpr uint32_t kStFrozen = 1u << 16;
constexpr uint32_t kStPad = 1u << 17;   // padding slot, never processed

// process switches (match ECRIS_F_*)
constexpr uint32_t kFPush = 1u << 0;
constexpr uint32_t kFIonize = 1u << 1;
constexpr uint32_t kFCx = 1u << 2;
constexpr uint32_t kFEikick = 1u << 3;
constexpr uint32_t kFCoulomb = 1u << 4;
constexpr uint32_t kFRecycle = 1u << 5;
constexpr uint32_t kFIsoheat = 1u << 6;
constexpr uint32_t kFDouble = 1u << 7;
constexpr uint32_t kFElastic = 1u << 8;
constexpr uint32_t kFRecomb = 1u << 9;
constexpr uint32_t kFlagMask = 0x3FFu;
// processes whose code only the variant kernels carry (with the
// on-axis field table)
constexpr uint32_t kFVariants = kFDouble | kFElastic | kFRecomb;
constexpr uint32_t kFHasE = 1u << 16;   // internal: the run has a nonzero E grid (the push gathers it)

constexpr uint32_t kNoCell = 0xFFFFFFFFu;

// Nanbu A(s) table: ln A tabulated on a uniform grid in ln s over [1e-3, 6]
constexpr int kNanbuN = 2048;
constexpr double kNanbuSLo = 1e-3;
constexpr double kNanbuSHi = 6.0;

// words of RunDev::cword: the plan's planned cells and ranges; which of the two
// sets of a step's counts is in use (the ions' pass of a step sets it, the
// collision kernel clears the other set for the next step); the entries taken of
// the scratch of large cells, of their list and of overflow records; then the
// counts, two words each: the step's unplanned cells, their ions in one warp of
// kLooseEvery, and the overflow records; the ticket of the plan's kernels
constexpr int kCwPlanned = 0, kCwRanges = 1, kCwSet = 2, kCwHuge = 3, kCwBig = 4, kCwPast = 5, kCwUnplanned = 6,
              kCwLoose = 8, kCwOverflow = 10, kCwTicket = 12, kCwWords = 14;
constexpr uint32_t kLooseEvery = 8;
// Coulomb collisions: room (records) a range of cells spans; ions of several
// cells that a warp sorts in registers, of one cell that a warp ranks, and that a
// block ranks at a time; warps a block
constexpr uint32_t kRange = 128;
constexpr int kWarpIons = 128, kWarpCell = 512, kBlockIons = 1792, kCollideWarps = 4;

// Device parameter block of one run: FP32 constants of the kernels (built in
// FP64 on the host) and the run's device arrays.
struct alignas(16) RunDev {
    // geometry
    float R0, R0sq, L, r_ap_sq, eps_wall;
    float inlet_x, inlet_y, inlet_z;
    // fixed-point positions: x = X sxy, y = Y sxy, z = (Z + 2^31) sz for int32
    // X, Y, Z, a uniform grid of 2^32 points across [-R0, R0) and [0, L)
    float sxy, inv_sxy, sz, inv_sz;
    float dt_sxy, dt_sz;         // dt / sxy, dt / sz: displacement per unit velocity
    int32_t inlet_X, inlet_Y, inlet_Z;   // gas inlet in fixed point
    // FP64 geometry for the (rare) wall and aperture crossings
    double R0_d, L_d, r_ap_d, eps_wall_d, sxy_d, sz_d;
    // synthetic mirror B0(z): raised-cosine halves around z_m
    float B_min, aL, aR;         // half amplitudes (B_inj-B_min)/2, (B_ext-B_min)/2
    float zm, inv_zm, inv_zr;    // z_m, 1/z_m, 1/(L-z_m)
    float aLk, aLk2, aRk, aRk2;  // a k and a k^2 of each half (k = pi/z_m, pi/(L-z_m))
    float hex_c;                 // B_hex / R0^2
    // on-axis table instead of the mirror: per segment k of length h the cubic
    // B0 = a + t (b + t (c + t d)), t = z/h - k (nullptr: the mirror)
    const float4 *btab;
    int32_t nseg;
    float inv_h;
    float B_ecr;
    // mesh
    int32_t nx, ny, nz;
    float inv_dx, inv_dy, inv_dz;
    // species and push
    int32_t qmax;
    float qm_unit;               // e / (M amu)
    float dt, half_dt;
    // collisions
    uint32_t flags;
    float sig0;                  // sqrt(kT0/M): thermal speed of re-emitted atoms
    float n0s1;                  // n0 * sigma_1 (1/m)
    float vth2;                  // 8 kT0 / (pi M)
    float dv_cx;                 // kick of a Q>=3 charge exchange: sqrt(2 (E_cx/2) / M)
    float n0sel;                 // n0 * sigma_el1 (1/m): elastic ion-atom scattering
    float sig_refl;              // thermal speed of ions re-emitted after neutralisation at a wall
    float ei_coef[2];            // D^2 = ei_coef[zone] * n_e * Q^p (zone 0 cold, 1 warm)
    int32_t ei_pow;
    float ke_scale;              // (M/2) / e * 1e6: micro-eV per (m/s)^2
    uint32_t atom_gate;          // an atom whose ionisation word is >= atom_gate cannot ionise in
                                 // any cell (0xFFFFFFFF: no such bound); 0: read the gate the device
                                 // keeps after the rate table (set by a device update of n_e)
    float lnl_ii_coef;           // Nanbu s prefactor lnL/(4 pi) (e^2/(eps0 mu))^2 w / V_cell
    uint32_t seed_lo, seed_hi;
    // arrays
    int32_t *x, *y, *z;          // fixed-point positions (see sxy, sz)
    float *vx, *vy, *vz;
    uint32_t *meta;
    uint32_t *id;                // stable particle id (Philox counter word, output order)
    const float4 *cell;          // {n_e (m^-3), zone (0/1), delta_x, delta_y}
    const float4 *E;             // {E_x, E_y, E_z, 0} per cell centre
    const float *kdt;            // [zone * 64 + Q]: k dt with k = k1 (single ionisation) + k2 (double)
                                 // + k3 (triple) + kr (recombination) as switched on; then
                                 // [2 * 64 + ...] the share k1 / k, [4 * 64 + ...] the share
                                 // (k1 + k2) / k and [6 * 64 + ...] (k1 + k2 + k3) / k; then at
                                 // kGateWord the atom gate (uint32 bits): an atom whose ionisation
                                 // word is >= the gate cannot ionise in any cell (0xFFFFFFFF: no
                                 // such bound), and the largest n_e of the cold and warm cells
    unsigned long long *dep;     // packed deposit accumulator: count << 32 | charge
    unsigned long long *tally;   // kTallyWords
    uint4 *crec;                 // pool of 32-byte records of the step's Coulomb participants: (vx, vy, vz,
                                 // meta word as bits), (array slot, words 0, 1, 2 of the stream-1 Philox block); the
                                 // first cpool are the cells' buckets, the next cover the overflow
    uint32_t cpool, cover;
    uint2 *cnext;                // per link of overflow records in a row of one cell, at the first one's place: (place
                                 // of the next link of the cell's chain + 1, 0: none; records)
    uint32_t *chead;             // per cell: its chain (zero between steps)
    uint32_t *ccount;            // per cell without a plan: its participants (zero between steps)
    uint4 *cbkt;                 // per cell: its bucket (first record, room, planned place, 0); (kNoCell, 0, 0, 0):
                                 // not planned
    uint4 *pcell;                // planned cells by place: (first record, room, cell, participants where pcount is
                                 // nullptr)
    uint32_t *pcount;            // their participants (zero between steps; nullptr: see pcell)
    uint32_t *rstart;            // first planned place of each range
    uint32_t *xcell;             // unplanned cells with participants this step
    uint32_t *cidx, *cord;       // scratch, one word a participant each: the overflow records of each cell, the ions
                                 // in order of cells too large for shared memory
    uint4 *cbig;                 // cells that take a block: (first record, room, ions, see BigCell), (next + 1, 0, 0, 0)
    uint32_t *cword;             // counters (kCw*)
    const float *nanbu;          // ln A at ln s = nanbu_lnlo + i / nanbu_inv_dln, i < kNanbuN
    float nanbu_lnlo, nanbu_inv_dln;
    uint32_t *step;              // device step counter of the run
    uint32_t *leave;             // the window's listed particles by slot: ions from the front, atoms from the
                                 // back (of 4 n4 entries)
    uint32_t *nleave;            // [0], [1] their numbers (zero between windows), [2] with collisions between
                                 // ions, the steps left in the window
    uint32_t *birth;             // by particle id: step of the last ionisation from Q = 0 (~0: unknown)
    unsigned long long *fptd;    // [Q][kFptdBins] extraction counts by age bin, [Q] summed ages (steps),
                                 // [Q] summed extraction radii (nm)
    uint32_t n;                  // particles
    uint32_t n4;                 // float4 groups = ceil(n/4)
    uint32_t ncells;
};

// ----------------------------------------------------------------------------
// Philox4x32-10 (Salmon et al., SC'11), counter (c0, 0, c2, 0), key (k0, k1).
// ----------------------------------------------------------------------------
struct Words { uint32_t w0, w1, w2, w3; };

__device__ __forceinline__ Words philox(uint32_t c0, uint32_t c2, uint32_t k0, uint32_t k1)
{
    uint32_t c1 = 0u, c3 = 0u;
#pragma unroll
    for (int r = 0; r < 10; ++r) {
        // one 32x32 -> 64-bit product gives both halves
        const unsigned long long p0 = (unsigned long long)0xD2511F53u * c0;
        const unsigned long long p1 = (unsigned long long)0xCD9E8D57u * c2;
        const uint32_t lo0 = (uint32_t)p0, hi0 = (uint32_t)(p0 >> 32);
        const uint32_t lo1 = (uint32_t)p1, hi1 = (uint32_t)(p1 >> 32);
        const uint32_t n0 = hi1 ^ c1 ^ k0;
        const uint32_t n2 = hi0 ^ c3 ^ k1;
        c0 = n0; c1 = lo1; c2 = n2; c3 = lo0;
        k0 += 0x9E3779B9u;
        k1 += 0xBB67AE85u;
    }
    return Words{c0, c1, c2, c3};
}

// words of particle pid at step s, stream st: counter (pid, 0, 4 s + st, 0)
__device__ __forceinline__ Words rng_words(const RunDev& R, uint32_t pid, uint32_t step, uint32_t st)
{
    return philox(pid, step * 4u + st, R.seed_lo, R.seed_hi);
}

// the block's copy of a run's parameter block (all threads call it)
__device__ __forceinline__ void stage_run(RunDev& rs, const RunDev* src)
{
    const uint32_t* from = reinterpret_cast<const uint32_t*>(src);
    uint32_t* to = reinterpret_cast<uint32_t*>(&rs);
    for (uint32_t k = threadIdx.x; k < sizeof(RunDev) / 4; k += blockDim.x) to[k] = from[k];
}

// Programmatic dependent launch: a kernel launched with launch_pdl may be
// scheduled while the kernel before it in the stream finishes (that kernel's
// blocks signal with pdl_trigger, or by exiting); it calls pdl_wait before it
// touches memory, which waits until the kernel before it has completed and
// its writes are visible.  This hides the launch latency between the
// dependent kernels of a step.  What the kernel before it writes is read through
// plain pointers: a read-only load (const __restrict__, __ldg) says that the
// memory does not change while the kernel lives, so the compiler could move it
// above the wait; a load in inline assembly is volatile, which keeps it below.
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void pdl_trigger() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

// early: whether it may.
template <typename... KArgs, typename... Args>
inline cudaError_t launch_early(bool early, void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem,
                                cudaStream_t s, Args&&... args)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = early ? 1 : 0;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kernel, std::forward<Args>(args)...);
}

template <typename... KArgs, typename... Args>
inline cudaError_t launch_pdl(void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t s,
                              Args&&... args)
{
    return launch_early(true, kernel, grid, block, smem, s, std::forward<Args>(args)...);
}

// last block of a grid (after every block's work is visible): ticket reset
__device__ __forceinline__ bool last_block(unsigned int* ticket)
{
    __shared__ int last;
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();
        last = atomicAdd(ticket, 1u) == gridDim.x - 1 ? 1 : 0;
        if (last) *ticket = 0u;
    }
    __syncthreads();
    return last != 0;
}

// square root through the approximate hardware instruction (relative error
// of a few units in the last place): for quantities that only set a
// probability, the size of a random kick or a scattering geometry, where that
// error is far below the parity tolerance; the push itself uses no square root
__device__ __forceinline__ float sqrt_approx(float x)
{
    float r;
    asm("sqrt.approx.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}

// (cos, sin)(2 pi u) for u in (0, 1] through the fast intrinsic, its argument
// kept inside [-pi, pi] where the absolute error is below 2^-21:
// (cos, sin)(2 pi u) = -(cos, sin)(pi (2u - 1))
__device__ __forceinline__ void sincos_2pi(float u, float* s, float* c)
{
    float sp, cp;
    __sincosf(3.14159265358979f * (2.0f * u - 1.0f), &sp, &cp);
    *s = -sp;
    *c = -cp;
}

// uniform in (0, 1]: (top 24 bits + 1) * 2^-24, exact in FP32
__device__ __forceinline__ float unit01(uint32_t w)
{
    return (float)((w >> 8) + 1u) * (1.0f / 16777216.0f);
}

// event test: fires when the word is below floor(p * 2^32)
__device__ __forceinline__ bool fires(uint32_t w, float p)
{
    const float t = p * 4294967296.0f;
    if (t >= 4294967296.0f) return true;
    return w < __float2uint_rz(t);
}

// ----------------------------------------------------------------------------
// Static magnetic field: synthetic mirror, paraxial off axis, plus the
// hexapole B_H (2xy, x^2 - y^2) / R0^2 (the printed sin/cos(2 theta) R^2 form).
// ----------------------------------------------------------------------------
__device__ __forceinline__ void bfield(const RunDev& R, float x, float y, float z,
                                       float& Bx, float& By, float& Bz)
{
    float b0, b1, b2, s, c;
    if (z <= R.zm) {
        __sincosf(3.14159265358979f * (z * R.inv_zm), &s, &c);   // argument in [0, pi]
        b0 = fmaf(R.aL, 1.0f + c, R.B_min);
        b1 = -R.aLk * s;
        b2 = -R.aLk2 * c;
    } else {
        __sincosf(3.14159265358979f * ((z - R.zm) * R.inv_zr), &s, &c);
        b0 = fmaf(R.aR, 1.0f - c, R.B_min);
        b1 = R.aRk * s;
        b2 = R.aRk2 * c;
    }
    // (FMAs written out: the kernels that step are compiled without contraction)
    const float hx = -0.5f * b1, hz = -0.25f * b2;
    const float r2 = fmaf(x, x, y * y);
    Bx = fmaf(hx, x, R.hex_c * (2.0f * x * y));
    By = fmaf(hx, y, R.hex_c * fmaf(x, x, -y * y));
    Bz = fmaf(hz, r2, b0);
}

// the same from the on-axis table: the segment's cubic in t and its
// derivatives in z
__device__ __forceinline__ void bfield_table(const RunDev& R, float x, float y, float z,
                                             float& Bx, float& By, float& Bz)
{
    const float u = z * R.inv_h;
    int k = (int)u;
    k = k < 0 ? 0 : (k > R.nseg - 1 ? R.nseg - 1 : k);
    const float t = u - (float)k;
    const float4 cf = __ldg(R.btab + k);
    const float b0 = cf.x + t * (cf.y + t * (cf.z + t * cf.w));
    const float b1 = (cf.y + t * (2.0f * cf.z + 3.0f * t * cf.w)) * R.inv_h;
    const float b2 = (2.0f * cf.z + 6.0f * t * cf.w) * (R.inv_h * R.inv_h);
    const float r2 = x * x + y * y;
    Bx = -0.5f * x * b1 + R.hex_c * (2.0f * x * y);
    By = -0.5f * y * b1 + R.hex_c * (x * x - y * y);
    Bz = b0 - 0.25f * r2 * b2;
}

// one axis of the trilinear gather between cell centres, clamped at the faces
__device__ __forceinline__ void tri_axis(float g, int n, int& i0, float& f)
{
    const float gc = g - 0.5f;
    const float fl = floorf(gc);
    int i = (int)fl;
    if (i < 0) { i0 = 0; f = 0.0f; }
    else if (i > n - 2) { i0 = n - 2; f = 1.0f; }
    else { i0 = i; f = gc - fl; }
}

__device__ __forceinline__ void efield(const RunDev& R, float x, float y, float z,
                                       float& Ex, float& Ey, float& Ez)
{
    int ix, iy, iz;
    float fx, fy, fz;
    tri_axis((x + R.R0) * R.inv_dx, R.nx, ix, fx);
    tri_axis((y + R.R0) * R.inv_dy, R.ny, iy, fy);
    tri_axis(z * R.inv_dz, R.nz, iz, fz);
    const int sx = 1, sy = R.nx, sz = R.nx * R.ny;
    const float4* e = R.E + ((iz * R.ny + iy) * R.nx + ix);
    const float4 a000 = __ldg(e), a100 = __ldg(e + sx), a010 = __ldg(e + sy), a110 = __ldg(e + sy + sx);
    const float4 a001 = __ldg(e + sz), a101 = __ldg(e + sz + sx), a011 = __ldg(e + sz + sy),
                 a111 = __ldg(e + sz + sy + sx);
    const float gx = 1.0f - fx, gy = 1.0f - fy, gz = 1.0f - fz;
    const float w000 = gx * gy * gz, w100 = fx * gy * gz, w010 = gx * fy * gz, w110 = fx * fy * gz;
    const float w001 = gx * gy * fz, w101 = fx * gy * fz, w011 = gx * fy * fz, w111 = fx * fy * fz;
    Ex = w000 * a000.x + w100 * a100.x + w010 * a010.x + w110 * a110.x +
         w001 * a001.x + w101 * a101.x + w011 * a011.x + w111 * a111.x;
    Ey = w000 * a000.y + w100 * a100.y + w010 * a010.y + w110 * a110.y +
         w001 * a001.y + w101 * a101.y + w011 * a011.y + w111 * a111.y;
    Ez = w000 * a000.z + w100 * a100.z + w010 * a010.z + w110 * a110.z +
         w001 * a001.z + w101 * a101.z + w011 * a011.z + w111 * a111.z;
}

// fixed point <-> metres
__device__ __forceinline__ float fx_xy(const RunDev& R, int32_t X) { return (float)X * R.sxy; }
__device__ __forceinline__ float fx_z(const RunDev& R, int32_t Z) { return ((float)Z + 2147483648.0f) * R.sz; }
__device__ __forceinline__ int32_t to_fx_xy(const RunDev& R, float x) { return __float2int_rn(x * R.inv_sxy); }
__device__ __forceinline__ int32_t to_fx_z(const RunDev& R, float z)
{
    return (int32_t)(__float2uint_rn(z * R.inv_sz) ^ 0x80000000u);
}

// nearest-grid-point cell of a fixed-point position: with U = X + 2^31 the
// cell is floor(U n / 2^32), the high word of a 32x32-bit product (exact)
template <class Mesh>
__device__ __forceinline__ uint32_t ngp_cell(const Mesh& R, int32_t X, int32_t Y, int32_t Z)
{
    const uint32_t ix = __umulhi((uint32_t)X ^ 0x80000000u, (uint32_t)R.nx);
    const uint32_t iy = __umulhi((uint32_t)Y ^ 0x80000000u, (uint32_t)R.ny);
    const uint32_t iz = __umulhi((uint32_t)Z ^ 0x80000000u, (uint32_t)R.nz);
    return (iz * (uint32_t)R.ny + iy) * (uint32_t)R.nx + ix;
}

// moment probes and screens (probe.cu)
constexpr int kMaxScreens = ECRIS_MAX_SCREENS;
struct ProbeDev {
    const int32_t* slot;          // per cell: its probe slot, or -1 (nullptr: no probed cells)
    double* mom;                  // [slot][qs][7]: count, sums of v and of v^2 per component
    unsigned long long* screen;   // [screen][qs][pixels^2] hit counts
    uint32_t ulo[kMaxScreens];    // slab of each screen in U = Z + 2^31: ulo <= U <= uhi
    uint32_t uhi[kMaxScreens];
    int32_t nscreens;
    int32_t pix_log2;             // pixels = 2^pix_log2
    int32_t qs;                   // qmax + 1
};

// ----------------------------------------------------------------------------
// Launch wrappers (defined in step_kernel.cu / coulomb.cu)
// ----------------------------------------------------------------------------
// A window of up to kMaxWindow steps: launch_quiet takes the atoms that neither
// leave nor ionise in it and lists every other particle (R.leave, R.nleave);
// then launch_active takes the listed ones through all K steps and advances
// the step counter by K (ticket: a zeroed device word, left zero), or, with
// collisions between ions, each step is launch_ions and launch_coulomb, whose
// last kernel advances the counter and, at the window's end, clears the list.
constexpr uint32_t kMaxWindow = 32;
constexpr uint32_t kActiveTile = 128;   // threads a block of the passes over one run's list
cudaError_t launch_quiet(const RunDev& R, uint32_t K, int sm_count, cudaStream_t s);
cudaError_t launch_active(const RunDev& R, uint32_t K, unsigned int* ticket, int sm_count, cudaStream_t s);
cudaError_t launch_ions(const RunDev& R, int sm_count, cudaStream_t s);
// instead of launch_quiet and what follows it, a window of one step (with
// collisions between ions launch_coulomb follows, else the counter is advanced)
cudaError_t launch_one(const RunDev& R, unsigned int* ticket, int sm_count, cudaStream_t s);
// the same for every run of a batch: items are the (run, tile) work list of
// `tile` particles a tile, pref 2 (nruns + 1) words of scratch, grid the
// blocks; entries of runs with step == NULL are skipped.  variants: some run
// has one of kFVariants or an on-axis table
cudaError_t launch_quiet_batch(const RunDev* runs, uint32_t nruns, const uint2* items, uint32_t nitems, uint32_t tile,
                               int threads, int grid, uint32_t K, uint32_t* pref, unsigned int* ticket,
                               cudaStream_t s);
cudaError_t launch_active_batch(const RunDev* runs, uint32_t nruns, int threads, int grid, bool variants, uint32_t K,
                                const uint32_t* pref, unsigned int* ticket, cudaStream_t s);
cudaError_t launch_ions_batch(const RunDev* runs, uint32_t nruns, int threads, int grid, bool variants,
                              const uint32_t* pref, cudaStream_t s);
cudaError_t launch_one_batch(const RunDev* runs, uint32_t nruns, const uint2* items, uint32_t nitems, uint32_t tile,
                             int threads, int grid, bool variants, unsigned int* ticket, cudaStream_t s);
// resident blocks per SM of the batch's passes
struct WindowBlocks { int quiet, active, ions, one; };
WindowBlocks window_blocks_per_sm(int threads);
cudaError_t launch_fold(const RunDev& R, uint32_t ncells, unsigned long long* count,
                        unsigned long long* charge, cudaStream_t s);
// words of the rate table after its 8 kQSlots rates and shares: the atom gate and the
// FP32 bits of the largest n_e of the cold and the warm cells
constexpr int kGateWord = 8 * kQSlots;
constexpr int kKdtWords = kGateWord + 4;
// the atom gate from the rate table's k_0 dt and the stored largest n_e of
// each zone (ne_update.cu)
cudaError_t launch_atom_gate(float* kdt, cudaStream_t s);
// self-consistent n_e: every cell's n_e from the charge deposited since the
// mark over steps_vol = steps V_cell, the mark moved on, the records {n_e,
// zone, delta} rebuilt (rl_coef = 2.38e-6 sqrt(T_e)/(B dX) per cell) and the
// atom gate recomputed; ne (Nc doubles) is scratch
cudaError_t launch_ne_update(const unsigned long long* charge, unsigned long long* mark, double* ne,
                             const double* rl_coef, float4* cell, float* kdt, int nx, int ny, uint32_t ncells,
                             double weight, double steps_vol, bool isoheat, int sm_count, cudaStream_t s);
// validity limits and padding point for ecris_load_ions
struct LoadCheck {
    float R0sq, L;
    uint32_t qmax;
    float inlet_x, inlet_y, inlet_z;
    float inv_sxy_hi, inv_sxy_lo;   // metres -> fixed point, as an unevaluated FP32 sum
    float inv_sz_hi, inv_sz_lo;
    int32_t nx, ny, nz;
    uint32_t* count;                // ions per cell, added up for the first plan (nullptr: no collisions)
};
// check the positions and charge states of particles [0, n), convert the
// positions (metres, float) in place to fixed point, build the meta words from
// q8 and the ids, fill pads [n, cap); and the velocities, now or in
// launch_load_check.  bad[0] counts invalid particles, ~bad[1] is the lowest invalid
// index (bad zeroed before)
cudaError_t launch_load_init(const LoadCheck& lc, float* const soa[6], const uint8_t* q8, uint32_t* meta,
                             uint32_t* id, uint32_t n, uint32_t cap, unsigned int* bad, bool velocities,
                             cudaStream_t s);
cudaError_t launch_load_check(float* const soa[6], const uint32_t* meta, uint32_t n, uint32_t cap, unsigned int* bad,
                              cudaStream_t s);

// One set of particle arrays (the sort moves particles between two sets).
struct ParticleSet {
    int32_t *x, *y, *z;
    float *vx, *vy, *vz;
    uint32_t *meta, *id;
};
// Counting sort of the run's particles (in R) by (ion/atom, cell) into `dst`:
// live ions first, then live atoms, each by cell; frozen and padding slots
// last.  hist (2 Nc + 2 words: the bins and a ticket) must be zero and is left
// zero; off (2 Nc + 1) and blk (scan block totals) are scratch.  plan (plan_blocks words, or
// NULL): also plan the collisions' buckets from the counts.  aos (the memory of `dst` as cap
// 32-byte records, or NULL): for input in arbitrary order (the first sort
// after a load), move records there and unpack them back into the arrays of
// R, which then hold the sorted particles; NULL writes `dst` directly.
cudaError_t launch_sort(const RunDev& R, uint32_t cap, const ParticleSet& dst, uint32_t* hist, uint32_t* off,
                        uint32_t* blk, unsigned long long* plan, uint4* aos, cudaStream_t s);
// the collisions' buckets planned anew without a sort (hist as above)
cudaError_t launch_replan(const RunDev& R, uint32_t cap, uint32_t* hist, unsigned long long* plan, cudaStream_t s);
int sort_scan_blocks(uint32_t nbins);
// state in load order: out[id[slot]] = state[slot] for id < n (positions to
// metres), into device arrays; rec: scratch of n 32-byte records (not `out`),
// or NULL
cudaError_t launch_export_ordered(const RunDev& R, uint32_t n, uint32_t cap, float* const out[6], uint32_t* meta_out,
                                  double sxy, double sz, uint4* rec, cudaStream_t s);
cudaError_t launch_census(const RunDev& R, uint32_t n4, unsigned long long* census, cudaStream_t s);
// add the current particles to the probes' sums (probe.cu)
cudaError_t launch_probe(const RunDev& R, const ProbeDev& P, uint32_t n4, int sm_count, cudaStream_t s);

// Launch shapes of a batch's passes by their names in ecris_tuning, threads per
// block x particles per thread x stages: tiles of threads x particles of the atoms'
// pass and of single steps, blocks of at most 256 threads; no kernel has stages.
constexpr int kStepShapes = 12;
constexpr int kDefaultShape = 11;
constexpr int kShapeThreads[kStepShapes] = {128, 128, 128, 256, 256, 256, 512, 512, 512, 128, 256, 256};
constexpr int kShapeVec[kStepShapes] = {1, 2, 4, 1, 2, 4, 1, 2, 4, 2, 1, 2};
constexpr int kShapeStages[kStepShapes] = {2, 2, 2, 2, 2, 2, 2, 2, 2, 3, 3, 3};
inline int shape_block(int k) { return kShapeThreads[k] < 256 ? kShapeThreads[k] : 256; }   // threads of its blocks
inline uint32_t shape_tile(int k) { return (uint32_t)(kShapeThreads[k] * kShapeVec[k]); }
// does a shape before it launch the same?
inline bool shape_repeats(int k)
{
    for (int j = 0; j < k; ++j)
        if (shape_block(j) == shape_block(k) && shape_tile(j) == shape_tile(k)) return true;
    return false;
}
// message returned by ecris_last_error(NULL) on the calling thread
void ecris_internal_set_thread_error(const char* msg);
// host: ln A(s) of Nanbu's scattering law on kNanbuN points uniform in ln s
// over [kNanbuSLo, kNanbuSHi], built in FP64 once per process (api.cu)
const float* nanbu_table();
// host: the prefactor of Nanbu's s = coef Qa^2 Qb^2 m g^-3 dt for m ions of
// one cell: lnL/(4 pi) (e^2/(eps0 mu))^2 w / V_cell, mu = M/2 (api.cu)
float coulomb_s_coef(double lnL_ii, double mass_amu, double weight, double cell_volume_m3);

// Hooks of the served form (defined in api.cu, used by server.cu).  A tally
// snapshot is a run's tally words, copied in stream order into pinned host
// memory at a step boundary; the served loop reads it a tick later, while the
// batch keeps stepping.
struct TallySnapshot {
    unsigned long long tally[kTallyWords];
};
// enqueue the copies of run `run`'s tallies into *dst (pinned) on the batch stream
ecris_status batch_snapshot(ecris_batch* b, int32_t run, TallySnapshot* dst);
cudaStream_t batch_stream(const ecris_batch* b);
// the batch autotuner (ecris_batch_autotune); without `cadence` it keeps the
// sort cadence and times launch shapes and resident blocks only
ecris_status batch_autotune(ecris_batch* b, uint32_t trial_steps, bool cadence, ecris_tuning* chosen);
// fill out (extracted, lost, currents, power, wall energy, collisions) from a
// snapshot taken after `steps` steps of the run (time steps * dt)
void batch_snapshot_diag(const ecris_batch* b, int32_t run, const TallySnapshot& snap, uint64_t steps,
                         ecris_diag_out* out);

// Coulomb collisions (coulomb.cu).  launch_plan: the buckets of every cell
// from `count` ions per cell (blk: plan_blocks words of scratch; zero: count is
// left zero).  Any plan is valid, one of
// the present counts is fast.  launch_coulomb: the collisions of one step
// after its ions' pass, in a kernel that also advances the step counter and,
// at the window's end, clears the list; n: the run's particles (all runs' in a
// batch).
uint32_t plan_blocks(uint32_t ncells);
cudaError_t launch_plan(const RunDev& R, uint32_t* count, bool zero, unsigned long long* blk, cudaStream_t s);
int collide_blocks(int sm_count);    // most blocks of the collision kernel
cudaError_t launch_coulomb(const RunDev& R, uint32_t n, int most, cudaStream_t s);
cudaError_t launch_coulomb_batch(const RunDev* runs, uint32_t nruns, uint32_t n, int most, cudaStream_t s);

__device__ __forceinline__ unsigned long long warp_incl64(unsigned long long v)
{
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const unsigned long long t = __shfl_up_sync(0xFFFFFFFFu, v, o);
        if ((int)(threadIdx.x & 31) >= o) v += t;
    }
    return v;
}

// exclusive scan over the block of v; *total: the block's sum (kT threads)
template <int kT>
__device__ __forceinline__ unsigned long long block_excl64(unsigned long long v, unsigned long long* total)
{
    __shared__ unsigned long long ws[kT / 32 + 1];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const unsigned long long incl = warp_incl64(v);
    if (lane == 31) ws[warp] = incl;
    __syncthreads();
    if (warp == 0) {
        const unsigned long long w = lane < kT / 32 ? ws[lane] : 0ull;
        const unsigned long long wi = warp_incl64(w);
        if (lane < kT / 32) ws[lane] = wi - w;
        if (lane == kT / 32 - 1) ws[kT / 32] = wi;
    }
    __syncthreads();
    *total = ws[kT / 32];
    return ws[warp] + incl - v;
}

// the ranges that start in or just after the room of planned place k
__device__ __forceinline__ void mark_ranges(const RunDev& R, uint32_t k, uint32_t at, uint32_t room)
{
    for (uint32_t b = at / kRange + 1u; b * kRange < at + room; ++b) R.rstart[b] = k + 1u;
    // a range that starts just where the next cell's room does
    if ((at + room) % kRange == 0u) R.rstart[(at + room) / kRange] = k + 1u;
}

// a 32-byte record in one store: one full sector, one request to L2
__device__ __forceinline__ void store_record(uint4* rec, size_t d, const uint4& a, const uint4& b)
{
    asm volatile("st.global.v8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(rec + 2 * d), "r"(a.x), "r"(a.y),
                 "r"(a.z), "r"(a.w), "r"(b.x), "r"(b.y), "r"(b.z), "r"(b.w)
                 : "memory");
}

// Record this lane's Coulomb participant (ck != kNoCell) in its cell's bucket or,
// when that is full, in the overflow, chained to the cell (one record after the other:
// at their slots' places each took a line of the cache to itself, and 6 served requests
// 78 ms, 70 so); the whole warp
// calls this.  One returning atomic per run of neighbouring lanes in the same
// cell.
__device__ __forceinline__ void place_warp(const RunDev& R, uint32_t slot, uint32_t ck, uint32_t id, uint32_t step,
                                           float vx, float vy, float vz, uint32_t meta)
{
    const uint32_t lane = threadIdx.x & 31;
    const bool in = ck != kNoCell;
    if (!__any_sync(0xFFFFFFFFu, in)) return;
    const uint32_t prev = __shfl_up_sync(0xFFFFFFFFu, ck, 1);
    const uint32_t heads = __ballot_sync(0xFFFFFFFFu, lane == 0 || prev != ck);
    const uint32_t upto = 0xFFFFFFFFu >> (31u - lane);              // lanes 0..lane
    const uint32_t after = heads & ~upto;                            // run heads above this lane
    const uint32_t tl = after ? (uint32_t)(__ffs(after) - 2) : 31u;  // last lane of this lane's run
    const uint32_t h = 31u - (uint32_t)__clz(heads & upto);           // first lane of this lane's run
    uint4 bk = make_uint4(0u, 0u, 0u, 0u);
    if (in) bk = R.cbkt[ck];
    uint32_t k = 0u;
    if (in && lane == h) k = atomicAdd(bk.x == kNoCell ? R.ccount + ck : R.pcount + bk.z, tl - h + 1u);
    const Words w = rng_words(R, id, step, 1u);
    k = __shfl_sync(0xFFFFFFFFu, k, h) + (lane - h);
    const bool over = in && k >= bk.y;
    uint32_t p = bk.x + k;
    const uint32_t om = __ballot_sync(0xFFFFFFFFu, over);
    if (om) {
        uint32_t o = 0u;
        if (lane == 0) o = atomicAdd(R.cword + kCwOverflow + (step & 1u), (uint32_t)__popc(om));
        o = __shfl_sync(0xFFFFFFFFu, o, 0) + (uint32_t)__popc(om & (upto >> 1));
        if (over) {   // the lanes of a cell are one link
            p = R.cpool + o;
            if (lane == h || !((om >> (lane - 1u)) & 1u))
                R.cnext[o] = make_uint2(atomicExch(R.chead + ck, o + 1u), tl - lane + 1u);
        }
        const uint32_t loose = __ballot_sync(0xFFFFFFFFu, over && bk.x == kNoCell);
        if (loose && lane == 0 && (slot >> 5) % kLooseEvery == 0u)
            atomicAdd(R.cword + kCwLoose + (step & 1u), (uint32_t)__popc(loose));
        // the first ion of a cell without a bucket lists it
        const bool lists = over && bk.x == kNoCell && k == 0u;
        const uint32_t lm = __ballot_sync(0xFFFFFFFFu, lists);
        if (lm) {
            uint32_t o = 0u;
            const uint32_t first = (uint32_t)(__ffs(lm) - 1);
            if (lane == first) o = atomicAdd(R.cword + kCwUnplanned + (step & 1u), (uint32_t)__popc(lm));
            o = __shfl_sync(0xFFFFFFFFu, o, first) + (uint32_t)__popc(lm & (upto >> 1));
            if (lists) R.xcell[o] = ck;
        }
    }
    if (in)
        store_record(R.crec, p, make_uint4(__float_as_uint(vx), __float_as_uint(vy), __float_as_uint(vz), meta),
                     make_uint4(slot, w.w0, w.w1, w.w2));
}

}  // namespace ecris
