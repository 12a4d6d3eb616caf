// Particle layout maintenance: a counting sort of a run's particles by
// (ion/atom, cell), and the export of the state in load order.
//
// The sort is a layout choice, not part of the model: every particle carries
// its stable id (the Philox counter word), and every result of the step is
// independent of where a particle sits in the arrays.  Keeping the particles
// grouped lets a warp's lanes take the same branch (ions and atoms run
// different code), share cell records and field samples in L1, add their
// deposits with one reduction per cell, and keeps a cell's ions close together
// for the collision kernels.
//
// Passes: count keys into a histogram (2 Nc + 1 bins: ions by cell, atoms by
// cell, one bin for frozen and padding slots); exclusive scan of it by blocks,
// whose totals the last block scans; move every particle to its key's place in
// the block, the block's offset and (histogram counted down by one), which
// leaves the histogram zero for the next sort.  A small run's sort is the
// latency of its launches: three, each free to start while the one before it
// ends (1000 steps of 1e4 particles with 31 sorts over 65536 cells take 1.63 ms;
// with the scan in three launches and no overlap 2.10).  Order inside a bin follows the atomics
// and does not matter.  The move writes the destination arrays directly when
// the input is mostly in key order already (every sort but the first after a
// load), since a warp's lanes then land on consecutive places and the eight
// arrays' writes coalesce.  For input in arbitrary order it writes one
// 32-byte record per particle, a full sector for a random destination instead
// of eight partial ones, and a second pass unpacks the records coalesced.  The
// records go to the memory of the set not in use and come back to the set
// they came from, so the sort takes no memory of its own.  The export in load
// order has a random destination too and goes the same way.
#include "ecris_internal.cuh"

namespace ecris {

namespace {

constexpr int kSortThreads = 256;
constexpr int kSortPerThread = 8;
constexpr int kSortScanBlock = kSortThreads * kSortPerThread;

__device__ __forceinline__ uint32_t key_of(const RunDev& R, int32_t x, int32_t y, int32_t z, uint32_t m)
{
    const uint32_t nc = R.ncells;
    if (m & (kStFrozen | kStPad)) return 2u * nc;
    return ((m & kQMask) ? 0u : nc) + ngp_cell(R, x, y, z);
}

__device__ __forceinline__ uint32_t sort_key(const RunDev& R, uint32_t i)
{
    return key_of(R, R.x[i], R.y[i], R.z[i], R.meta[i]);
}

// lanes with equal keys add once per group (input already in order makes
// whole warps share a key); kIons: the ions alone
template <bool kIons>
__global__ void k_sort_count(const __grid_constant__ RunDev R, uint32_t cap, uint32_t* __restrict__ hist)
{
    pdl_wait();
    pdl_trigger();
    const uint32_t stride = gridDim.x * blockDim.x;
    const uint32_t end = (cap + 31u) & ~31u;   // whole warps iterate together
    for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < end; i += stride) {
        uint32_t key = i < cap ? sort_key(R, i) : 0xFFFFFFFFu;
        if (kIons && key >= R.ncells) key = 0xFFFFFFFFu;
        const bool in = key != 0xFFFFFFFFu;
        const uint32_t act = __ballot_sync(0xFFFFFFFFu, in);
        if (!in) continue;
        const uint32_t grp = __match_any_sync(act, key);
        if ((threadIdx.x & 31) == (uint32_t)(__ffs(grp) - 1)) atomicAdd(hist + key, (uint32_t)__popc(grp));
    }
}

__device__ __forceinline__ uint32_t warp_incl(uint32_t v)
{
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t t = __shfl_up_sync(0xFFFFFFFFu, v, o);
        if (lane >= o) v += t;
    }
    return v;
}

// exclusive scan over the block's kSortThreads threads; *total: the sum
__device__ __forceinline__ uint32_t block_excl(uint32_t v, uint32_t* total)
{
    __shared__ uint32_t ws[kSortThreads / 32 + 1];
    const uint32_t incl = warp_incl(v);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (lane == 31) ws[warp] = incl;
    __syncthreads();
    if (warp == 0) {
        const uint32_t w = lane < kSortThreads / 32 ? ws[lane] : 0u;
        const uint32_t wi = warp_incl(w);
        if (lane < kSortThreads / 32) ws[lane] = wi - w;
        if (lane == kSortThreads / 32 - 1) ws[kSortThreads / 32] = wi;
    }
    __syncthreads();
    *total = ws[kSortThreads / 32];
    return ws[warp] + incl - v;
}

// exclusive scan of in[0, n) into out within blocks of kSortScanBlock; blk: the
// blocks' offsets (ticket: a zero word, left zero)
__global__ void __launch_bounds__(kSortThreads) k_sort_scan(const uint32_t* in, uint32_t* __restrict__ out,
                                                            uint32_t* blk, uint32_t n, uint32_t* ticket)
{
    pdl_wait();
    pdl_trigger();
    const uint32_t base = blockIdx.x * kSortScanBlock + threadIdx.x * kSortPerThread, nb = gridDim.x;
    uint32_t v[kSortPerThread], sum = 0, total;
#pragma unroll
    for (int j = 0; j < kSortPerThread; ++j) {
        v[j] = base + j < n ? in[base + j] : 0u;
        sum += v[j];
    }
    uint32_t o = block_excl(sum, &total);
#pragma unroll
    for (int j = 0; j < kSortPerThread; ++j) {
        if (base + j < n) out[base + j] = o;
        o += v[j];
    }
    if (threadIdx.x == 0) blk[blockIdx.x] = total;
    if (!last_block(ticket)) return;
    uint32_t carry = 0;
    for (uint32_t b0 = 0; b0 < nb; b0 += kSortThreads) {
        const uint32_t b = b0 + threadIdx.x;
        const uint32_t t = b < nb ? __ldcg(blk + b) : 0u;
        __syncthreads();   // (the scan's shared memory is used again)
        const uint32_t at = carry + block_excl(t, &total);
        if (b < nb) blk[b] = at;
        carry += total;
    }
}

// kRecords: write 32-byte records to aos (unpacked by k_sort_unpack), else
// the destination arrays
template <bool kRecords>
__global__ void k_sort_move(const __grid_constant__ RunDev R, uint32_t cap, ParticleSet dst, uint4* __restrict__ aos,
                            uint32_t* __restrict__ hist, const uint32_t* off, const uint32_t* blk)
{
    pdl_wait();
    pdl_trigger();
    const uint32_t stride = gridDim.x * blockDim.x;
    const uint32_t end = (cap + 31u) & ~31u;
    const uint32_t lane = threadIdx.x & 31;
    for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < end; i += stride) {
        const bool in = i < cap;
        // the particle's words and its bin's offset are loaded before the
        // atomic below, so their round trips overlap instead of following it
        int32_t x = 0, y = 0, z = 0;
        float vx = 0.0f, vy = 0.0f, vz = 0.0f;
        uint32_t meta = 0u, id = 0u, key = 0xFFFFFFFFu;
        if (in) {
            x = R.x[i];
            y = R.y[i];
            z = R.z[i];
            meta = R.meta[i];
            vx = R.vx[i];
            vy = R.vy[i];
            vz = R.vz[i];
            id = R.id[i];
            key = key_of(R, x, y, z, meta);
        }
        const uint32_t act = __ballot_sync(0xFFFFFFFFu, in);
        if (!in) continue;
        const uint32_t base = off[key] + blk[key / kSortScanBlock];
        // one atomic per group of lanes with the same key; lanes take
        // consecutive places below the group's previous count
        const uint32_t grp = __match_any_sync(act, key);
        const uint32_t leader = (uint32_t)(__ffs(grp) - 1);
        uint32_t top = 0;
        if (lane == leader) top = atomicSub(hist + key, (uint32_t)__popc(grp));
        top = __shfl_sync(grp, top, leader);
        const uint32_t rank = (uint32_t)__popc(grp & ((1u << lane) - 1u));
        const uint32_t d = base + top - 1u - rank;
        if (kRecords) {
            store_record(aos, d, make_uint4((uint32_t)x, (uint32_t)y, (uint32_t)z, __float_as_uint(vx)),
                         make_uint4(__float_as_uint(vy), __float_as_uint(vz), meta, id));
        } else {
            dst.x[d] = x;
            dst.y[d] = y;
            dst.z[d] = z;
            dst.vx[d] = vx;
            dst.vy[d] = vy;
            dst.vz[d] = vz;
            dst.meta[d] = meta;
            dst.id[d] = id;
        }
    }
}

// records in sorted order -> the destination arrays, coalesced both ways
__global__ void k_sort_unpack(const uint4* aos, uint32_t cap, ParticleSet dst)
{
    pdl_wait();
    pdl_trigger();
    for (uint32_t d = blockIdx.x * blockDim.x + threadIdx.x; d < cap; d += gridDim.x * blockDim.x) {
        const uint4 a = aos[2 * (size_t)d], b = aos[2 * (size_t)d + 1];
        dst.x[d] = (int32_t)a.x;
        dst.y[d] = (int32_t)a.y;
        dst.z[d] = (int32_t)a.z;
        dst.vx[d] = __uint_as_float(a.w);
        dst.vy[d] = __uint_as_float(b.x);
        dst.vz[d] = __uint_as_float(b.y);
        dst.meta[d] = b.z;
        dst.id[d] = b.w;
    }
}

// Fixed point to metres, (float)((double)k s) for the whole number k = hi + lo
// (both exact in FP32) and s = s_hi + s_lo + what 2^-49 s bounds.  The GPU has
// few FP64 units, and ten FP64 instructions a particle and loads waiting for
// stores bound the whole export (4e6 particles in load order 100 us, 40 so).  Here the product is formed as an unevaluated FP32 sum, h = fl(hi s_hi)
// with its exact error (an FMA) and the cross terms, to 2^-44.8 of its size: terms
// of 2^-22 and less, rounded twice, and lo s_lo <= 2^-47 left out.  Its rounding to
// FP32 is that of the FP64 product unless the sum lies within that of the middle
// between two FP32 numbers (or r is a power of two, below which they lie
// closer); those few, one in 2^17, take the FP64 product itself.
struct Scale {
    double s;
    float hi, lo;
};

Scale make_scale(double s) { return Scale{s, (float)s, (float)(s - (double)(float)s)}; }

// (out of line: inlined, its instructions are issued for every particle)
__device__ __noinline__ float to_metres_fp64(float hi, float lo, double s)
{
    return (float)(((double)hi + (double)lo) * s);
}

__device__ __forceinline__ float to_metres(float hi, float lo, const Scale& c)
{
    const float h = __fmul_rn(hi, c.hi);
    const float t = __fmaf_rn(lo, c.hi, __fmaf_rn(hi, c.lo, __fmaf_rn(hi, c.hi, -h)));
    const float r = __fadd_rn(h, t);
    const float d = fabsf(__fsub_rn(t, __fsub_rn(r, h)));   // (exact: |t| < |h|, or both are 0)
    const uint32_t bits = __float_as_uint(r);
    const float half = __uint_as_float((bits & 0x7F800000u) - (24u << 23));   // half the spacing above |r|
    if (fabsf(__fsub_rn(d, half)) <= half * 3.8146973e-6f || !(bits & 0x007FFFFFu))
        return to_metres_fp64(hi, lo, c.s);
    return r;
}

// a signed and an unsigned coordinate (see fx_xy, fx_z), truncated to FP32 and
// the rest
__device__ __forceinline__ float metres_xy(int32_t X, const Scale& c)
{
    const float hi = __int2float_rz(X);
    return to_metres(hi, (float)(X - __float2int_rz(hi)), c);
}

__device__ __forceinline__ float metres_z(int32_t Z, const Scale& c)
{
    const uint32_t U = (uint32_t)Z ^ 0x80000000u;
    const float hi = __uint2float_rz(U);
    return to_metres(hi, (float)(U - __float2uint_rz(hi)), c);
}

// a particle's words as the export writes them, all loaded at once (a load
// behind the store of the word before it waits for each in turn)
struct Exported {
    uint32_t d, meta;
    float v[6];
};

__device__ __forceinline__ Exported exported(const RunDev& R, uint32_t i, const Scale& sxy, const Scale& sz)
{
    Exported e;
    e.d = R.id[i];
    const int32_t X = R.x[i], Y = R.y[i], Z = R.z[i];
    e.v[3] = R.vx[i];
    e.v[4] = R.vy[i];
    e.v[5] = R.vz[i];
    e.meta = R.meta[i];
    e.v[0] = metres_xy(X, sxy);
    e.v[1] = metres_xy(Y, sxy);
    e.v[2] = metres_z(Z, sz);
    return e;
}

struct OutPtrs { float* p[6]; };

// Export of a large run, first pass: the particle's 32-byte record to place
// id.  Scattering the seven arrays one by one costs seven partial sectors a
// particle (393 us at 4e6 particles, 1636 at 8e6, where the outputs no longer
// fit in L2); the records cost one full sector, and the second pass is
// coalesced.
__global__ void k_export_records(const __grid_constant__ RunDev R, uint32_t n, uint32_t cap, uint4* __restrict__ rec,
                                 Scale sxy, Scale sz)
{
    pdl_wait();
    pdl_trigger();
    for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < cap; i += gridDim.x * blockDim.x) {
        const Exported e = exported(R, i, sxy, sz);
        if (e.d >= n) continue;   // padding
        store_record(rec, e.d, make_uint4(__float_as_uint(e.v[0]), __float_as_uint(e.v[1]), __float_as_uint(e.v[2]),
                                          __float_as_uint(e.v[3])),
                     make_uint4(__float_as_uint(e.v[4]), __float_as_uint(e.v[5]), e.meta, 0u));
    }
}

__global__ void k_export_unpack(const uint4* rec, uint32_t n, OutPtrs out, uint32_t* __restrict__ meta_out)
{
    pdl_wait();
    pdl_trigger();
    for (uint32_t d = blockIdx.x * blockDim.x + threadIdx.x; d < n; d += gridDim.x * blockDim.x) {
        const uint4 a = rec[2 * (size_t)d], b = rec[2 * (size_t)d + 1];
        if (out.p[0]) out.p[0][d] = __uint_as_float(a.x);
        if (out.p[1]) out.p[1][d] = __uint_as_float(a.y);
        if (out.p[2]) out.p[2][d] = __uint_as_float(a.z);
        if (out.p[3]) out.p[3][d] = __uint_as_float(a.w);
        if (out.p[4]) out.p[4][d] = __uint_as_float(b.x);
        if (out.p[5]) out.p[5][d] = __uint_as_float(b.y);
        if (meta_out) meta_out[d] = b.z;
    }
}

__global__ void k_export_ordered(const __grid_constant__ RunDev R, uint32_t n, uint32_t cap, OutPtrs out,
                                 uint32_t* __restrict__ meta_out, Scale sxy, Scale sz)
{
    pdl_wait();
    pdl_trigger();
    for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < cap; i += gridDim.x * blockDim.x) {
        const Exported e = exported(R, i, sxy, sz);
        if (e.d >= n) continue;   // padding
#pragma unroll
        for (int k = 0; k < 6; ++k)
            if (out.p[k]) out.p[k][e.d] = e.v[k];
        if (meta_out) meta_out[e.d] = e.meta;
    }
}

// particles from which the export goes through records
constexpr uint32_t kExportRecords = 1u << 18;

int grid_for(uint32_t n, int threads, int cap_blocks)
{
    int b = (int)((n + threads - 1) / threads);
    if (b > cap_blocks) b = cap_blocks;
    return b < 1 ? 1 : b;
}

}  // namespace

int sort_scan_blocks(uint32_t nbins) { return (int)((nbins + kSortScanBlock - 1) / kSortScanBlock); }

cudaError_t launch_sort(const RunDev& R, uint32_t cap, const ParticleSet& dst, uint32_t* hist, uint32_t* off,
                        uint32_t* blk, unsigned long long* plan, uint4* aos, cudaStream_t s)
{
    const uint32_t nbins = 2u * R.ncells + 1u;
    const dim3 grid(grid_for(cap, 256, 8192)), block(256);
    cudaError_t e = launch_pdl(k_sort_count<false>, grid, block, 0, s, R, cap, hist);
    if (e == cudaSuccess)
        e = launch_pdl(k_sort_scan, dim3(sort_scan_blocks(nbins)), dim3(kSortThreads), 0, s, (const uint32_t*)hist, off,
                       blk, nbins, hist + nbins);
    if (e == cudaSuccess && plan) e = launch_plan(R, hist, false, plan, s);
    if (e == cudaSuccess)
        e = launch_pdl(aos ? k_sort_move<true> : k_sort_move<false>, grid, block, 0, s, R, cap, dst, aos, hist,
                       (const uint32_t*)off, (const uint32_t*)blk);
    const ParticleSet src{R.x, R.y, R.z, R.vx, R.vy, R.vz, R.meta, R.id};
    if (e == cudaSuccess && aos) e = launch_pdl(k_sort_unpack, grid, block, 0, s, (const uint4*)aos, cap, src);
    return e;
}

cudaError_t launch_replan(const RunDev& R, uint32_t cap, uint32_t* hist, unsigned long long* plan, cudaStream_t s)
{
    const cudaError_t e = launch_pdl(k_sort_count<true>, dim3(grid_for(cap, 256, 8192)), dim3(256), 0, s, R, cap, hist);
    return e == cudaSuccess ? launch_plan(R, hist, true, plan, s) : e;
}

cudaError_t launch_export_ordered(const RunDev& R, uint32_t n, uint32_t cap, float* const out[6], uint32_t* meta_out,
                                  double sxy, double sz, uint4* rec, cudaStream_t s)
{
    OutPtrs o;
    for (int k = 0; k < 6; ++k) o.p[k] = out ? out[k] : nullptr;
    const dim3 grid(grid_for(cap, 256, 8192)), block(256);
    if (!rec || n < kExportRecords)
        return launch_pdl(k_export_ordered, grid, block, 0, s, R, n, cap, o, meta_out, make_scale(sxy), make_scale(sz));
    const cudaError_t e = launch_pdl(k_export_records, grid, block, 0, s, R, n, cap, rec, make_scale(sxy), make_scale(sz));
    if (e != cudaSuccess) return e;
    return launch_pdl(k_export_unpack, dim3(grid_for(n, 256, 8192)), block, 0, s, (const uint4*)rec, n, o, meta_out);
}

}  // namespace ecris
