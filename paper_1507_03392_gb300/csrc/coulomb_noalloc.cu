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
// 6 MB) is held by every GPU that loads the library until the process exits.
// Every call shares it and finds the last call's contents there; what must
// start at zero is cleared at the start of each call.  Calls whose GPU work
// overlaps (different streams, or several host threads) race on the array
// and must be serialised by the caller.  The first call on each device sets up
// that device (symbol address, Nanbu table upload, a synchronous copy); make
// that first call before any stream capture begins.  That set-up is kept for
// the life of the process: a device reset (cudaDeviceReset) is not supported,
// and the entry point must not be called on a device after one.
// A call knows its ions only when it is made, so it counts them by cell, plans
// exact buckets (k_na_plan) and places the records; nothing overflows, however
// the ions are spread.  (A pool shared out evenly among the cells needs neither
// count nor plan, two launches less, but its time hung on the spread: 65521 ions
// evenly in 65536 cells took 23 us a call and in 4096 cells 37, 60000 ions in 400 of
// 65536 cells 5559; 30, 36 and 33 so.)
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
constexpr uint32_t kNaPool = 2 * kNaMaxIons;   // bucket records: a cell that collides takes at most 2 an ion
constexpr size_t align256(size_t b) { return (b + 255) & ~(size_t)255; }

// byte offsets of the sub-buffers inside the scratch array
constexpr size_t kOffRec = 0;
constexpr size_t kOffCcount = kOffRec + align256(2 * sizeof(uint4) * kNaPool);
constexpr size_t kOffFirst = kOffCcount + align256(sizeof(uint32_t) * kNaMaxCells);
constexpr size_t kOffRank = kOffFirst + align256(sizeof(uint32_t) * kNaMaxCells);
constexpr size_t kOffPcell = kOffRank + align256(sizeof(uint32_t) * kNaMaxIons);
constexpr size_t kOffRstart = kOffPcell + align256(sizeof(uint4) * (kNaPool / 4));
constexpr size_t kOffOrd = kOffRstart + align256(sizeof(uint32_t) * (kNaPool / kRange + 1));
constexpr size_t kOffBig = kOffOrd + align256(sizeof(uint32_t) * kNaMaxIons);
constexpr size_t kOffNanbu = kOffBig + align256(2 * sizeof(uint4) * (kNaMaxIons / kWarpIons + 1));
constexpr size_t kOffWords = kOffNanbu + align256(sizeof(float) * kNanbuN);
// words: step; from word 16 the collisions' counters; from word 32 the plan's cursor; then the tally block
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

constexpr int kNaThreads = 256;
constexpr int kNaSmallThreads = 1024;
constexpr int kNaPer = 8;               // cells a thread of the plan

// clear the per-call counters and store the step index
__device__ __forceinline__ void na_clear(unsigned char* base, uint32_t ncells, uint32_t step)
{
    uint32_t* ccount = reinterpret_cast<uint32_t*>(base + kOffCcount);
    uint32_t* words = reinterpret_cast<uint32_t*>(base + kOffWords);
    unsigned long long* tally = reinterpret_cast<unsigned long long*>(base + kOffTally);
    const uint32_t stride = gridDim.x * blockDim.x;
    for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < ncells; i += stride) ccount[i] = 0u;
    // (the collisions' counters: this step's)
    if (blockIdx.x == 0 && threadIdx.x < 34)
        words[threadIdx.x] = threadIdx.x == 0 ? step : (threadIdx.x == 16 + kCwSet ? step & 1u : 0u);
    for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < (uint32_t)kTallyWords; i += stride) tally[i] = 0ull;
}

// cell of particle i if it takes part (cell < ncells, 1 <= Q <= 63)
__device__ __forceinline__ uint32_t na_cell(const RunDev& R, uint32_t i, const uint32_t* cell, const uint8_t* q)
{
    if (i >= R.n) return kNoCell;
    const uint32_t c = cell[i], Q = q[i];
    return c >= R.ncells || Q == 0u || Q > 63u ? kNoCell : c;
}

// count the participants by cell; rank: each one's arrival in its cell (one atomic per
// group of lanes in the same cell; the whole warp calls it)
__device__ __forceinline__ void na_count(const RunDev& R, uint32_t i, const uint32_t* cell, const uint8_t* q,
                                         uint32_t* count, uint32_t* rank)
{
    const uint32_t lane = threadIdx.x & 31u, c = na_cell(R, i, cell, q);
    const uint32_t grp = __match_any_sync(0xFFFFFFFFu, c);
    const int leader = __ffs(grp) - 1;
    uint32_t k = 0u;
    if (c != kNoCell && lane == (uint32_t)leader) k = atomicAdd(count + c, (uint32_t)__popc(grp));
    k = __shfl_sync(0xFFFFFFFFu, k, leader) + (uint32_t)__popc(grp & ((1u << lane) - 1u));
    if (i < R.n) rank[i] = k;
}

// Room of a cell of h ions whose bucket holds them for this step: at least 4, so
// that a range has at most 32 cells; none where nothing collides.  So n ions take at most
// 2 n records and n / 2 places.
__device__ __forceinline__ uint32_t na_room(uint32_t h) { return h < 2u ? 0u : max(h, 4u); }

// The plan: first[c] is cell c's first record (kNoCell: nothing to collide).  Any order
// of the cells' buckets will do, so a block takes the places and the records of kT kNaPer
// cells from one cursor (places << 32 | records) instead of a scan over the
// blocks.  (Two calls that share the working memory and overlap, which they must not, get
// no bucket past the pool.)
template <int kT>
__device__ __forceinline__ void na_plan(const RunDev& R, const uint32_t* count, uint32_t* first,
                                        unsigned long long* cursor)
{
    __shared__ unsigned long long s_start;
    const uint32_t base = (blockIdx.x * kT + threadIdx.x) * kNaPer;
    uint32_t h[kNaPer];
    unsigned long long v = 0ull, total;
#pragma unroll
    for (int j = 0; j < kNaPer; ++j) {
        h[j] = base + j < R.ncells ? __ldcg(count + base + j) : 0u;
        const uint32_t room = na_room(h[j]);
        v += ((unsigned long long)(room ? 1u : 0u) << 32) + room;
    }
    unsigned long long o = block_excl64<kT>(v, &total);
    if (threadIdx.x == 0) s_start = atomicAdd(cursor, total);
    __syncthreads();
    o += s_start;
#pragma unroll
    for (int j = 0; j < kNaPer; ++j) {
        const uint32_t c = base + j;
        if (c >= R.ncells) break;
        const uint32_t room = na_room(h[j]), k = (uint32_t)(o >> 32), at = (uint32_t)o;
        const bool in = room && at < R.cpool && room <= R.cpool - at;
        first[c] = in ? at : kNoCell;
        if (!in) continue;
        R.pcell[k] = make_uint4(at, room, c, h[j]);
        mark_ranges(R, k, at, room);
        o += (1ull << 32) + room;
    }
}

// its words, by one thread after all blocks
__device__ __forceinline__ void na_plan_end(const RunDev& R, const unsigned long long* cursor)
{
    const unsigned long long end = __ldcg(cursor);
    const uint32_t nr = min(((uint32_t)end + kRange - 1u) / kRange, R.cpool / kRange);
    const uint32_t np = min((uint32_t)(end >> 32), R.cpool / 4u);
    R.cword[kCwPlanned] = np;
    R.cword[kCwRanges] = nr;
    R.rstart[0] = 0u;
    R.rstart[nr] = np;
}

// record a participant in its cell's bucket, as the ions' pass does for ecris_step; slot
// and id are both the array index
__device__ __forceinline__ void na_pack(const RunDev& R, uint32_t i, const uint32_t* cell, const uint8_t* q,
                                        const uint32_t* first, const uint32_t* rank, uint32_t step)
{
    const uint32_t c = na_cell(R, i, cell, q);
    if (c == kNoCell) return;
    const uint32_t at = first[c], k = rank[i];
    if (at == kNoCell || k >= R.cpool - at) return;   // (alone in its cell)
    const Words w = rng_words(R, i, step, 1u);
    store_record(R.crec, at + k, make_uint4(__float_as_uint(R.vx[i]), __float_as_uint(R.vy[i]), __float_as_uint(R.vz[i]),
                                            (uint32_t)q[i]),
                 make_uint4(i, w.w0, w.w1, w.w2));
}

// what the passes before the collision kernel share
struct Front {
    unsigned char* base;
    const uint32_t* cell;
    const uint8_t* q;
    uint32_t *count, *first, *rank;
    unsigned long long* cursor;
    uint32_t step;
};

__global__ void k_na_init(Front f, uint32_t ncells)
{
    pdl_wait();
    pdl_trigger();
    na_clear(f.base, ncells, f.step);
}

__global__ void k_na_count(const __grid_constant__ RunDev R, Front f)
{
    pdl_wait();
    pdl_trigger();
    na_count(R, blockIdx.x * blockDim.x + threadIdx.x, f.cell, f.q, f.count, f.rank);
}

__global__ void __launch_bounds__(kNaThreads) k_na_plan(const __grid_constant__ RunDev R, Front f)
{
    pdl_wait();
    pdl_trigger();
    na_plan<kNaThreads>(R, f.count, f.first, f.cursor);
    if (last_block(R.cword + kCwTicket) && threadIdx.x == 0) na_plan_end(R, f.cursor);
}

__global__ void k_na_pack(const __grid_constant__ RunDev R, Front f)
{
    pdl_wait();
    pdl_trigger();
    na_pack(R, blockIdx.x * blockDim.x + threadIdx.x, f.cell, f.q, f.first, f.rank, f.step);
}

// All of it by one block, up to kNaSmallIons particles and as many cells as it plans in one
// round: the four launches cost more there than their work.  us a call alone, with them and
// so: 1001 particles in 4096 cells 67 and 63; 8001 70 and 74; 1001 in 32768 cells, four
// rounds of the plan, 61 and 80.
constexpr uint32_t kNaSmallIons = 4096, kNaSmallCells = kNaSmallThreads * kNaPer;
__global__ void __launch_bounds__(kNaSmallThreads) k_na_small(const __grid_constant__ RunDev R, Front f)
{
    pdl_wait();
    pdl_trigger();
    const uint32_t end = (R.n + 31u) & ~31u;
    na_clear(f.base, R.ncells, f.step);
    __syncthreads();
    for (uint32_t i = threadIdx.x; i < end; i += kNaSmallThreads) na_count(R, i, f.cell, f.q, f.count, f.rank);
    __syncthreads();
    na_plan<kNaSmallThreads>(R, f.count, f.first, f.cursor);
    __syncthreads();
    if (threadIdx.x == 0) na_plan_end(R, f.cursor);
    for (uint32_t i = threadIdx.x; i < end; i += kNaSmallThreads)
        na_pack(R, i, f.cell, f.q, f.first, f.rank, f.step);
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
    R.n = (uint32_t)n;
    Front f{};
    f.base = base;
    f.cell = cell;
    f.q = q;
    f.count = reinterpret_cast<uint32_t*>(base + kOffCcount);
    f.first = reinterpret_cast<uint32_t*>(base + kOffFirst);
    f.rank = reinterpret_cast<uint32_t*>(base + kOffRank);
    f.step = step;
    R.pcell = reinterpret_cast<uint4*>(base + kOffPcell);
    R.rstart = reinterpret_cast<uint32_t*>(base + kOffRstart);
    R.cord = reinterpret_cast<uint32_t*>(base + kOffOrd);
    R.cbig = reinterpret_cast<uint4*>(base + kOffBig);
    R.cword = reinterpret_cast<uint32_t*>(base + kOffWords) + 16;
    R.nanbu = reinterpret_cast<const float*>(base + kOffNanbu);
    R.nanbu_lnlo = (float)std::log(kNanbuSLo);
    R.nanbu_inv_dln = (float)((kNanbuN - 1) / std::log(kNanbuSHi / kNanbuSLo));
    R.step = reinterpret_cast<uint32_t*>(base + kOffWords);
    R.tally = reinterpret_cast<unsigned long long*>(base + kOffTally);

    f.cursor = reinterpret_cast<unsigned long long*>(R.cword + 16);
    if (n <= kNaSmallIons && ncells <= kNaSmallCells) {
        e = launch_pdl(k_na_small, dim3(1), dim3(kNaSmallThreads), 0, s, R, f);
    } else {
        const dim3 block(kNaThreads), grid((uint32_t)((n + kNaThreads - 1) / kNaThreads));
        e = launch_pdl(k_na_init, dim3((ncells + kNaThreads - 1) / kNaThreads), block, 0, s, f, ncells);
        if (n > 0) {
            if (e == cudaSuccess) e = launch_pdl(k_na_count, grid, block, 0, s, R, f);
            if (e == cudaSuccess)
                e = launch_pdl(k_na_plan, dim3((ncells + kNaThreads * kNaPer - 1) / (kNaThreads * kNaPer)), block, 0, s, R, f);
            if (e == cudaSuccess) e = launch_pdl(k_na_pack, grid, block, 0, s, R, f);
        }
    }
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
