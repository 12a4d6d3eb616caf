// ecris_coulomb_collide_noalloc: one ion-ion Coulomb collision step (the same
// Takizawa-Abe pairing and Nanbu scattering kernels ecris_step runs) for a
// caller that cannot allocate device memory.
//
// Some callers cannot call cudaMalloc at the moment they need a collision
// step: code inside a region where the CUDA caching or stream-ordered
// allocators are off limits, embedded or real-time hosts that reserve all
// device memory up front and forbid allocation afterwards, and plug-ins
// running inside a larger simulation whose memory manager owns the device.
// cudaMalloc can also synchronise the device, which such callers must avoid.
// This entry point therefore keeps all its working memory (per-cell counts,
// participant records, the Nanbu table, counters) in one
// file-scope device array of fixed size, and allocates nothing.
//
// Limits: at most kNaMaxIons particles and kNaMaxCells cells per call; larger
// sizes are rejected with ECRIS_EINVAL.  The array (kNaScratchBytes, about
// 5 MB) is held by every GPU that loads the library until the process exits.
// Every call shares it and finds the last call's contents there; what must
// start at zero is cleared at the start of each call.  Calls whose GPU work
// overlaps (different streams, or several host threads) race on the array
// and must be serialised by the caller.  The first call on each device sets up
// that device (symbol address, Nanbu table upload, a synchronous copy); make
// that first call before any stream capture begins.  That set-up is kept for
// the life of the process: a device reset (cudaDeviceReset) is not supported,
// and the entry point must not be called on a device after one.
// There is no plan of the cells' buckets: the bucket records are shared out
// evenly among the call's cells, and what does not fit overflows.
#include <cmath>
#include <cstring>
#include <mutex>
#include <string>
#include <vector>

#include "../../include/ecris.h"
#include "ecris_internal.cuh"

using namespace ecris;

namespace {

constexpr uint32_t kNaMaxIons = 65536;
constexpr uint32_t kNaMaxCells = 65536;
constexpr uint32_t kNaPool = 49152;    // bucket records, shared out evenly among the call's cells
constexpr size_t align256(size_t b) { return (b + 255) & ~(size_t)255; }

// byte offsets of the sub-buffers inside the scratch array
constexpr size_t kOffRec = 0;
constexpr size_t kOffNext = kOffRec + align256(2 * sizeof(uint4) * (kNaPool + kNaMaxIons));
constexpr size_t kOffHead = kOffNext + align256(sizeof(uint32_t) * kNaMaxIons);
constexpr size_t kOffCcount = kOffHead + align256(sizeof(uint32_t) * kNaMaxCells);
constexpr size_t kOffIdx = kOffCcount + align256(sizeof(uint32_t) * kNaMaxCells);
constexpr size_t kOffOrd = kOffIdx + align256(sizeof(uint32_t) * kNaMaxIons);
constexpr size_t kOffNanbu = kOffOrd + align256(sizeof(uint32_t) * kNaMaxIons);
constexpr size_t kOffWords = kOffNanbu + align256(sizeof(float) * kNanbuN);
// words: step; from word 16 the collisions' counters; then the tally block
constexpr size_t kOffTally = kOffWords + 256;
constexpr size_t kNaScratchBytes = kOffTally + align256(sizeof(unsigned long long) * kTallyWords);

static __device__ __align__(256) unsigned char g_noalloc_scratch[kNaScratchBytes];

struct DeviceSetup {
    bool ready = false;
    unsigned char* base = nullptr;   // device address of g_noalloc_scratch
    int grid = 0;
};

std::mutex g_setup_mutex;
DeviceSetup g_setup[64];

// clear the per-call counters and store the step index
__global__ void k_na_init(unsigned char* base, uint32_t ncells, uint32_t step)
{
    uint32_t* ccount = reinterpret_cast<uint32_t*>(base + kOffCcount);
    uint32_t* chead = reinterpret_cast<uint32_t*>(base + kOffHead);
    uint32_t* words = reinterpret_cast<uint32_t*>(base + kOffWords);
    unsigned long long* tally = reinterpret_cast<unsigned long long*>(base + kOffTally);
    const uint32_t stride = gridDim.x * blockDim.x;
    for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < ncells; i += stride) ccount[i] = chead[i] = 0u;
    // (the collisions' counters: the set of this step)
    if (blockIdx.x == 0 && threadIdx.x < 16 + kCwWords)
        words[threadIdx.x] = threadIdx.x == 0 ? step : (threadIdx.x == 16 + kCwSet ? 2u * (step & 1u) : 0u);
    for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < (uint32_t)kTallyWords; i += stride) tally[i] = 0ull;
}

// record the participants (cell < ncells, Q >= 1) in their cells' buckets, as
// the ions' pass does for ecris_step (whole warps: n rounded up)
__global__ void k_na_pack(const __grid_constant__ RunDev R, uint32_t n, const uint32_t* __restrict__ cell,
                          const uint8_t* __restrict__ q)
{
    pdl_wait();
    pdl_trigger();
    const uint32_t end = (n + 31u) & ~31u;
    for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < end; i += gridDim.x * blockDim.x) {
        uint32_t c = kNoCell, Q = 0u;
        float vx = 0.0f, vy = 0.0f, vz = 0.0f;
        if (i < n) {
            c = cell[i];
            Q = q[i];
            if (c >= R.ncells || Q == 0u || Q > 63u) c = kNoCell;
            vx = R.vx[i];
            vy = R.vy[i];
            vz = R.vz[i];
        }
        place_warp(R, i, c, i, *R.step, vx, vy, vz, Q);   // slot and id are both the array index
    }
}

ecris_status na_fail(const std::string& msg)
{
    ecris_internal_set_thread_error(msg.c_str());
    return ECRIS_EINVAL;
}

ecris_status na_cuda(cudaError_t e, const char* what)
{
    ecris_internal_set_thread_error((std::string("coulomb_collide_noalloc: ") + what + ": " +
                                     cudaGetErrorString(e)).c_str());
    return ECRIS_ECUDA;
}

}  // namespace

extern "C" ecris_status ecris_coulomb_collide_noalloc(size_t n, const uint32_t* cell, const uint8_t* q, float* vx,
                                                      float* vy, float* vz, uint32_t* events, uint32_t ncells,
                                                      double mass_amu, double weight, double cell_volume_m3,
                                                      double lnL_ii, double dt, uint64_t seed, uint32_t step,
                                                      void* cuda_stream, int64_t* collisions_out)
{
    if (n > kNaMaxIons || ncells > kNaMaxCells || ncells == 0)
        return na_fail("coulomb_collide_noalloc: need n <= " + std::to_string(kNaMaxIons) + " and 1 <= ncells <= " +
                       std::to_string(kNaMaxCells) + " (fixed scratch size)");
    if (n > 0 && (!cell || !q || !vx || !vy || !vz || !events))
        return na_fail("coulomb_collide_noalloc: NULL array");
    if (!(mass_amu > 0.0) || !(weight > 0.0) || !(cell_volume_m3 > 0.0) || !(lnL_ii >= 0.0) || !(dt > 0.0) ||
        !std::isfinite(mass_amu) || !std::isfinite(weight) || !std::isfinite(cell_volume_m3) ||
        !std::isfinite(lnL_ii) || !std::isfinite(dt))
        return na_fail("coulomb_collide_noalloc: mass, weight, cell volume and dt must be finite and > 0");
    if ((uint64_t)step * 4u + 3u > 0xFFFFFFFFull) return na_fail("coulomb_collide_noalloc: step must be < 2^30");
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return na_cuda(e, "cudaGetDevice");
    if (dev < 0 || dev >= 64) return na_fail("coulomb_collide_noalloc: device index above 63");
    DeviceSetup setup;
    {
        std::lock_guard<std::mutex> lock(g_setup_mutex);
        DeviceSetup& d = g_setup[dev];
        if (!d.ready) {
            void* p = nullptr;
            e = cudaGetSymbolAddress(&p, g_noalloc_scratch);
            if (e != cudaSuccess) return na_cuda(e, "cudaGetSymbolAddress");
            // the same FP64-built table ecris_init_fields uploads for ecris_step
            e = cudaMemcpy(static_cast<unsigned char*>(p) + kOffNanbu, nanbu_table(), kNanbuN * sizeof(float),
                           cudaMemcpyHostToDevice);
            if (e != cudaSuccess) return na_cuda(e, "Nanbu table upload");
            int sms = 0;
            e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
            if (e != cudaSuccess) return na_cuda(e, "cudaDeviceGetAttribute");
            d.base = static_cast<unsigned char*>(p);
            d.grid = collide_blocks(sms);
            d.ready = true;
        }
        setup = d;
    }
    cudaStream_t s = (cudaStream_t)cuda_stream;
    unsigned char* base = setup.base;

    // the parameter block the collision kernels read, pointing into the scratch
    RunDev R;
    std::memset(&R, 0, sizeof R);
    R.lnl_ii_coef = coulomb_s_coef(lnL_ii, mass_amu, weight, cell_volume_m3);
    R.dt = (float)dt;
    R.seed_lo = (uint32_t)seed;
    R.seed_hi = (uint32_t)(seed >> 32);
    R.vx = vx;
    R.vy = vy;
    R.vz = vz;
    R.meta = events;
    R.ncells = ncells;
    R.crec = reinterpret_cast<uint4*>(base + kOffRec);
    R.cpool = kNaPool;
    R.cover = kNaMaxIons;
    R.cnext = reinterpret_cast<uint32_t*>(base + kOffNext);
    R.chead = reinterpret_cast<uint32_t*>(base + kOffHead);
    R.pcount = reinterpret_cast<uint32_t*>(base + kOffCcount);
    R.uroom = kNaPool / ncells;
    R.ucells = R.uroom > kRange ? 1u : (R.uroom < kRange / 32u ? 32u : kRange / R.uroom);
    R.cidx = reinterpret_cast<uint32_t*>(base + kOffIdx);
    R.cord = reinterpret_cast<uint32_t*>(base + kOffOrd);
    R.cword = reinterpret_cast<uint32_t*>(base + kOffWords) + 16;
    R.nanbu = reinterpret_cast<const float*>(base + kOffNanbu);
    R.nanbu_lnlo = (float)std::log(kNanbuSLo);
    R.nanbu_inv_dln = (float)((kNanbuN - 1) / std::log(kNanbuSHi / kNanbuSLo));
    R.step = reinterpret_cast<uint32_t*>(base + kOffWords);
    R.tally = reinterpret_cast<unsigned long long*>(base + kOffTally);

    k_na_init<<<(ncells + 255) / 256, 256, 0, s>>>(base, ncells, step);
    e = cudaGetLastError();
    if (e == cudaSuccess && n > 0)
        e = launch_pdl(k_na_pack, dim3((uint32_t)((n + 255) / 256)), dim3(256), 0, s, R, (uint32_t)n, cell, q);
    if (e != cudaSuccess) return na_cuda(e, "launch");
    e = launch_coulomb(R, (uint32_t)n, setup.grid, s);
    if (e != cudaSuccess) return na_cuda(e, "launch_coulomb");
    if (collisions_out) {
        // the call synchronises: read the collision count
        unsigned long long c = 0;
        e = cudaMemcpyAsync(&c, R.tally + kTallyCoulomb, sizeof c, cudaMemcpyDeviceToHost, s);
        if (e == cudaSuccess) e = cudaStreamSynchronize(s);
        if (e != cudaSuccess) return na_cuda(e, "collision count");
        *collisions_out = (int64_t)c;
    }
    return ECRIS_OK;
}
