// Ion-ion Coulomb collisions of the ECRIS model (arXiv:1507.03392, Sec. II
// collision block): Takizawa-Abe pairing of the ions of each cell and Nanbu's
// scattering angle, Coulomb logarithm lnL_ii.
//
// The ions' pass of a step leaves a 32-byte record of every ion that stayed
// inside, (v, Q) and (array slot, its three words of the stream-1 Philox
// block), in its cell's bucket (place_warp in step_kernel.cu):
//   - buckets are planned from the cells' ion counts at every load and layout
//     sort, and in between where plan_due in api.cu says so: a cell of h ions gets
//     room for h + h/8 + 4 (k_plan*), cells without ions none;
//   - an ion that finds its cell's bucket full, or a cell without one, goes to
//     the overflow part of the pool, where a warp's run of ions of one cell is
//     chained to the cell as one link.
// So a cell's records lie together without a count, a scan and a scatter in
// every step.  Then k_collide orders each cell's ions by (first word, particle
// id), which is independent of the order of arrival, pairs consecutive ones and
// collides them; a cell with an odd count puts ranks 0, 1, 2 in a triplet that
// collides (0,1), (1,2), (2,0) over dt/2 each:
//   - a warp takes a range of planned cells (kRange records' room) or up to 32
//     unplanned ones.  It sorts up to kWarpIons ions of several cells at once in
//     registers, by cell, the first word's high 20 bits and the ion's place (a
//     bitonic network over 32 lanes x 4); words that tie in those bits are put in
//     order afterwards;
//   - it ranks a cell of up to kWarpCell ions by counting into word buckets: ion j
//     of a cell of m goes to bucket floor(word m / 2^32) of m, the counts are
//     scanned, and the few ions that share a bucket compare their words, and
//     their ids if the words tie;
//   - triplets, three collisions in a row, and larger cells are put by for the
//     block, whose threads take a triplet each and a large cell together (ranked
//     the same way, above kBlockIons ions in windows of their words).
//
// A collision of ions a, b (same mass M, charges Qa, Qb) over time dt_c uses
//   s = lnL/(4 pi) (Qa Qb e^2 / (eps0 mu))^2 n g^-3 dt_c,  mu = M/2,
// n = w m / V_cell for the cell's m ions; A(s) from coth A - 1/A = e^-s
// (tabulated in FP64 on the host, s >= 1e-3; 1/(1 - e^-s) below, where coth A
// is 1 to working precision; isotropic for s > 6);
//   cos chi = 1 + ln(U + (1-U) e^-2A) / A,  eps = 2 pi U'
// (the logarithm's argument formed without cancellation in FP32, see collide);
// the relative velocity g is turned by (chi, eps) and the change is shared
// equally, which conserves momentum and energy of the pair.
#include <algorithm>

#include "ecris_internal.cuh"

namespace ecris {

namespace {

// ---------------------------------------------------------------------------
// The plan of the buckets
// ---------------------------------------------------------------------------
constexpr int kPlanThreads = 256;
constexpr int kPlanPer = 8;
constexpr uint32_t kPlanBlock = kPlanThreads * kPlanPer;

// room of a cell of h ions
__device__ __forceinline__ uint32_t bucket_room(uint32_t h) { return h ? h + (h >> 3) + 4u : 0u; }

// (planned cells, room) of the blocks of kPlanBlock cells, packed (<< 32 |);
// count: ions per cell.  The last block makes that the exclusive scan, and the
// plan's words.
__global__ void __launch_bounds__(kPlanThreads) k_plan_sum(const __grid_constant__ RunDev R,
                                                           const uint32_t* count, unsigned long long* blk)
{
    pdl_wait();
    pdl_trigger();
    const uint32_t base = blockIdx.x * kPlanBlock + threadIdx.x, nb = gridDim.x;
    unsigned long long v = 0ull, total;
#pragma unroll
    for (int j = 0; j < kPlanPer; ++j) {
        const uint32_t c = base + j * kPlanThreads;
        const uint32_t h = c < R.ncells ? count[c] : 0u;
        v += ((unsigned long long)(h ? 1u : 0u) << 32) + bucket_room(h);
    }
    block_excl64<kPlanThreads>(v, &total);
    if (threadIdx.x == 0) blk[blockIdx.x] = total;
    if (!last_block(R.cword + kCwTicket)) return;
    unsigned long long carry = 0ull;
    for (uint32_t b0 = 0; b0 < nb; b0 += kPlanThreads) {
        const uint32_t b = b0 + threadIdx.x;
        const unsigned long long t = b < nb ? __ldcg(blk + b) : 0ull;
        __syncthreads();   // (the scan's shared memory is used again)
        const unsigned long long o = carry + block_excl64<kPlanThreads>(t, &total);
        if (b < nb) blk[b] = o;
        carry += total;
    }
    if (threadIdx.x == 0) {
        const uint32_t np = (uint32_t)(carry >> 32), room = (uint32_t)carry;
        R.cword[kCwPlanned] = np;
        R.cword[kCwRanges] = (room + kRange - 1u) / kRange;
        R.rstart[0] = 0u;
        R.rstart[(room + kRange - 1u) / kRange] = np;
    }
}

// every cell's bucket, the compact list of planned cells, and the ranges: range
// b holds the planned cells whose room starts in [b kRange, (b + 1) kRange)
__global__ void __launch_bounds__(kPlanThreads) k_plan_cells(const __grid_constant__ RunDev R,
                                                             uint32_t* __restrict__ count,
                                                             const unsigned long long* blk, int zero)
{
    pdl_wait();
    pdl_trigger();
    const uint32_t base = blockIdx.x * kPlanBlock + threadIdx.x * kPlanPer;
    uint32_t h[kPlanPer];
    unsigned long long v = 0ull, total;
#pragma unroll
    for (int j = 0; j < kPlanPer; ++j) {
        h[j] = base + j < R.ncells ? count[base + j] : 0u;
        if (zero && h[j]) count[base + j] = 0u;
        v += ((unsigned long long)(h[j] ? 1u : 0u) << 32) + bucket_room(h[j]);
    }
    unsigned long long o = blk[blockIdx.x] + block_excl64<kPlanThreads>(v, &total);
#pragma unroll
    for (int j = 0; j < kPlanPer; ++j) {
        const uint32_t c = base + j;
        if (c >= R.ncells) break;
        const uint32_t room = bucket_room(h[j]), k = (uint32_t)(o >> 32), at = (uint32_t)o;
        // (a bucket past the pool's bucket part is cut short; its ions overflow)
        const uint32_t fits = at < R.cpool ? min(room, R.cpool - at) : 0u;
        R.cbkt[c] = room ? make_uint4(at, fits, k, 0u) : make_uint4(kNoCell, 0u, 0u, 0u);
        if (!room) continue;
        R.pcell[k] = make_uint4(at, fits, c, 0u);
        mark_ranges(R, k, at, room);
        o += (1ull << 32) + room;
    }
}

// ---------------------------------------------------------------------------
// One collision
// ---------------------------------------------------------------------------
// A(s) for 1e-3 <= s <= 6 from the table of ln A, linear in ln s.  The
// logarithm that indexes the table and the exponential of the interpolated
// ln A use the fast intrinsics: their errors (below 1e-6 in ln s and a few
// units in the last place of A) move A by far less than the table's own
// interpolation error.
__device__ __forceinline__ float nanbu_A(const RunDev& R, float s)
{
    if (s < (float)kNanbuSLo) return 1.0f / (-expm1f(-s));
    float t = (__logf(s) - R.nanbu_lnlo) * R.nanbu_inv_dln;
    t = fminf(fmaxf(t, 0.0f), (float)(kNanbuN - 1));
    int i = (int)t;
    if (i > kNanbuN - 2) i = kNanbuN - 2;
    const float f = t - (float)i;
    const float a0 = __ldg(R.nanbu + i);
    const float la = fmaf(f, __ldg(R.nanbu + i + 1) - a0, a0);
    return __expf(la);
}

// One collision over time dtc of the records ra, rb (vx, vy, vz, Q bits),
// with w1, w2 the stream-1 words 1 and 2 of the pair's first particle (the
// angles); updates the records in place.
__device__ __forceinline__ void collide(const RunDev& R, float4& ra, float4& rb, float dtc, float m_cell, uint32_t w1,
                                        uint32_t w2)
{
    // (FMAs written out: this file is compiled without contraction, so that
    // every inlined copy of this code rounds the same way, whichever kernel
    // takes a cell)
    const float gx = ra.x - rb.x, gy = ra.y - rb.y, gz = ra.z - rb.z;
    const float g2 = fmaf(gx, gx, fmaf(gy, gy, gz * gz));
    if (!(g2 > 0.0f)) return;
    // 1/g through the approximate reciprocal square root (a few units in the
    // last place): it sets s and the scattering geometry, not the angle's
    // small-angle digits (those come from eps below)
    const float rg = rsqrtf(g2);
    const float g = g2 * rg;
    const float qq = (float)((__float_as_uint(ra.w) & 63u) * (__float_as_uint(rb.w) & 63u));
    const float s = R.lnl_ii_coef * (qq * qq) * m_cell * dtc * (rg * rg * rg);
    const float U = unit01(w1);
    // eps = 1 - cos chi and epc = 1 + cos chi, each formed without
    // cancellation: in a small-angle collision cos chi lies within FP32
    // rounding of 1, so sin chi = sqrt(1 - cos^2 chi) would lose most of its
    // digits, while sin chi = sqrt(eps epc) keeps them
    float eps, epc;
    if (!(s <= (float)kNanbuSHi)) {
        eps = 2.0f * (1.0f - U);   // isotropic: cos chi = 2U - 1 (both exact in FP32)
        epc = 2.0f * U;
    } else {
        const float A = nanbu_A(R, s);
        // ln(U + (1-U) e^-2A): for small A the sum is close to 1 and log1p of
        // (1-U)(e^-2A - 1) keeps its precision; for larger A the two positive
        // terms are formed directly, since e^-2A can lie below the FP32
        // spacing of expm1 near -1 while U is small as well
        const float lnarg = A < 0.5f ? log1pf((1.0f - U) * expm1f(-2.0f * A))
                                     : logf(fmaf(1.0f - U, expf(-2.0f * A), U));
        eps = fminf(fmaxf(__fdividef(-lnarg, A), 0.0f), 2.0f);
        epc = 2.0f - eps;
    }
    const float schi = sqrt_approx(eps * epc);
    float se, ce;
    sincos_2pi(unit01(w2), &se, &ce);
    const float gp2 = fmaf(gy, gy, gz * gz);
    float hx, hy, hz;
    if (gp2 > 0.0f) {
        const float rgp = rsqrtf(gp2);
        hx = gp2 * rgp * ce;
        hy = -fmaf(gx * gy, ce, g * gz * se) * rgp;
        hz = -fmaf(gx * gz, ce, -(g * gy * se)) * rgp;
    } else {
        hx = 0.0f;
        hy = g * ce;
        hz = g * se;
    }
    const float dgx = 0.5f * fmaf(hx, schi, -(gx * eps));
    const float dgy = 0.5f * fmaf(hy, schi, -(gy * eps));
    const float dgz = 0.5f * fmaf(hz, schi, -(gz * eps));
    ra.x += dgx; ra.y += dgy; ra.z += dgz;
    rb.x -= dgx; rb.y -= dgy; rb.z -= dgz;
}

__device__ __forceinline__ void write_back(const RunDev& R, uint32_t slot, const float4& r)
{
    // (no ids: a caller's arrays, whose event words are not the records' meta
    // words; a slot past them is another call's that overlaps this one, which
    // it must not)
    if (!R.id && slot >= R.n) return;
    R.vx[slot] = r.x;
    R.vy[slot] = r.y;
    R.vz[slot] = r.z;
    if (R.id) R.meta[slot] = __float_as_uint(r.w) | kEvCoulomb;
    else R.meta[slot] |= kEvCoulomb;
}

// kind of sorted place r in a cell of m: 1 starts a pair, 2 starts a triplet
__device__ __forceinline__ uint32_t start_kind(uint32_t r, uint32_t m)
{
    if (m < 2u) return 0u;
    if (m & 1u) {
        if (r == 0u) return 2u;
        return (r >= 3u && !((r - 3u) & 1u)) ? 1u : 0u;
    }
    return (r & 1u) ? 0u : 1u;
}

struct Record {
    float4 v;      // vx, vy, vz, Q as bits
    uint4 w;       // array slot, words 0, 1, 2
};

__device__ __forceinline__ Record load_record(const RunDev& R, uint32_t p)
{
    uint32_t a[8];
    asm volatile("ld.global.v8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                 : "=r"(a[0]), "=r"(a[1]), "=r"(a[2]), "=r"(a[3]), "=r"(a[4]), "=r"(a[5]), "=r"(a[6]), "=r"(a[7])
                 : "l"(R.crec + 2 * (size_t)p));
    return Record{make_float4(__uint_as_float(a[0]), __uint_as_float(a[1]), __uint_as_float(a[2]),
                              __uint_as_float(a[3])),
                  make_uint4(a[4], a[5], a[6], a[7])};
}

// collide the records ia, ib of the pool as a pair, m ions in the cell
__device__ __forceinline__ void collide_pair(const RunDev& R, uint32_t ia, uint32_t ib, float m)
{
    Record a = load_record(R, ia), b = load_record(R, ib);
    collide(R, a.v, b.v, R.dt, m, a.w.z, a.w.w);
    write_back(R, a.w.x, a.v);
    write_back(R, b.w.x, b.v);
}

// ranks 0, 1, 2: (0,1), (1,2), (2,0) over dt/2 each
__device__ __forceinline__ void collide_triplet(const RunDev& R, uint32_t ia, uint32_t ib, uint32_t ic, float m)
{
    Record a = load_record(R, ia), b = load_record(R, ib), c = load_record(R, ic);
    const float dtc = 0.5f * R.dt;
#pragma unroll 1
    for (int k = 0; k < 3; ++k) {
        collide(R, a.v, b.v, dtc, m, a.w.z, a.w.w);
        const Record t = a;   // the next pair to the front
        a = b;
        b = c;
        c = t;
    }
    write_back(R, a.w.x, a.v);
    write_back(R, b.w.x, b.v);
    write_back(R, c.w.x, c.v);
}

// ---------------------------------------------------------------------------
// The cells
// ---------------------------------------------------------------------------
// Shared memory of a block that ranks up to kBlockIons ions of one cell
struct CellSmem {
    uint32_t word[kBlockIons];            // first words
    uint32_t rec[kBlockIons];             // the ions' places in the cell
    uint32_t cnt2[kBlockIons / 2 + 1];    // ions per word bucket, then their exclusive scan, two 16-bit counts a word
    uint16_t pos[kBlockIons];             // arrival in the word bucket
    uint16_t arr[kBlockIons];             // ions by word bucket
    uint32_t n;
};

// particle id at an array slot (the slot where there are no ids)
__device__ __forceinline__ uint32_t slot_id(const RunDev& R, uint32_t slot) { return R.id ? R.id[slot] : slot; }

__device__ __forceinline__ uint32_t record_id(const RunDev& R, uint32_t p)
{
    return slot_id(R, R.crec[2 * (size_t)p + 1].x);
}

// a cell that takes a block: (first record, room, ions, where in cidx the records
// past its bucket are, less the room)
using BigCell = uint4;

// the record of ion j of a cell
__device__ __forceinline__ uint32_t cell_record(const RunDev& R, const BigCell& b, uint32_t j)
{
    return j < b.y ? b.x + j : R.cidx[b.w + j];
}

// Order and collide the ions of one cell by the block.  The words are uniform,
// so a cell of more ions than the shared memory holds is ranked in windows of
// equal word ranges, each of them holding 7/8 of kBlockIons on average (a window
// that is too full all the same is halved); the order goes to global scratch.
__device__ __forceinline__ void collide_cell(const RunDev& R, CellSmem& S, const BigCell& b, uint32_t* s_off)
{
    constexpr uint32_t T = 32 * kCollideWarps;
    const uint32_t g = threadIdx.x, M = b.z;
    if (g == 0) *s_off = atomicAdd(R.cword + kCwHuge, M);
    __syncthreads();
    const uint32_t off = *s_off;
    if (off + M > R.cover) return;   // (the scratch holds every participant)
    uint32_t* const ord = R.cord + off;
    unsigned long long width = (1ull << 32) / ((M + kBlockIons * 7u / 8u - 1u) / (kBlockIons * 7u / 8u)) + 1ull;
    if (M <= (uint32_t)kBlockIons) width = 1ull << 32;
    uint32_t done = 0u;
    for (unsigned long long lo = 0ull; lo < (1ull << 32);) {
        // the window's ions
        __syncthreads();
        if (g == 0) S.n = 0u;
        for (uint32_t k = g; k < (uint32_t)kBlockIons / 2u + 1u; k += T) S.cnt2[k] = 0u;
        __syncthreads();
        for (uint32_t j = g; j < M; j += T) {
            const uint32_t w = R.crec[2 * (size_t)cell_record(R, b, j) + 1].y;
            if (w < lo || w - lo >= width) continue;
            const uint32_t at = atomicAdd(&S.n, 1u);
            if (at < (uint32_t)kBlockIons) {
                S.word[at] = w;
                S.rec[at] = j;
            }
        }
        __syncthreads();
        const uint32_t n = S.n;
        if (n > (uint32_t)kBlockIons && width > 1ull) {
            width = (width + 1ull) / 2ull;
            continue;
        }
        if (n > (uint32_t)kBlockIons) {   // one word for so many ions: in the order of their ids
            for (uint32_t j = g; j < M; j += T) {
                const uint32_t p = cell_record(R, b, j), id = record_id(R, p);
                if (R.crec[2 * (size_t)p + 1].y != (uint32_t)lo) continue;
                uint32_t r = 0u;
                for (uint32_t i = 0; i < M; ++i) {
                    const uint32_t pi = cell_record(R, b, i);
                    if (R.crec[2 * (size_t)pi + 1].y == (uint32_t)lo && record_id(R, pi) < id) ++r;
                }
                ord[done + r] = p;
            }
            done += n;
            lo += 1ull;
            continue;
        }
        // ranked by counting into n buckets of its range
        const float scale = (float)n / (float)width;   // (any monotone rule will do)
        const uint16_t* const cnt = reinterpret_cast<const uint16_t*>(S.cnt2);
        auto bucket = [&](uint32_t w) { return min((uint32_t)((float)(w - (uint32_t)lo) * scale), n - 1u); };
        for (uint32_t j = g; j < n; j += T) {
            const uint32_t k = bucket(S.word[j]), sh = 16u * (k & 1u);
            S.pos[j] = (uint16_t)(atomicAdd(&S.cnt2[k >> 1], 1u << sh) >> sh);
        }
        __syncthreads();
        {
            constexpr int kPer = kBlockIons / 2 / (int)T;
            uint32_t v[kPer], sum = 0u;
#pragma unroll
            for (int k = 0; k < kPer; ++k) {
                v[k] = S.cnt2[g * kPer + k];
                sum += (v[k] & 0xFFFFu) + (v[k] >> 16);
            }
            unsigned long long total;
            uint32_t o = (uint32_t)block_excl64<T>(sum, &total);
#pragma unroll
            for (int k = 0; k < kPer; ++k) {
                const uint32_t c = v[k] & 0xFFFFu;
                S.cnt2[g * kPer + k] = o | ((o + c) << 16);
                o += c + (v[k] >> 16);
            }
            if (g == 0) S.cnt2[kBlockIons / 2] = n;
        }
        __syncthreads();
        for (uint32_t j = g; j < n; j += T) S.arr[cnt[bucket(S.word[j])] + S.pos[j]] = (uint16_t)j;
        __syncthreads();
        for (uint32_t j = g; j < n; j += T) {
            const uint32_t w = S.word[j], k = bucket(w);
            const uint32_t first = cnt[k], end = cnt[k + 1];
            uint32_t r = first;
            for (uint32_t t = first; t < end; ++t) {
                const uint32_t i = S.arr[t], wi = S.word[i];
                if (wi < w || (wi == w && i != j && record_id(R, cell_record(R, b, S.rec[i])) <
                                                        record_id(R, cell_record(R, b, S.rec[j]))))
                    ++r;
            }
            ord[done + r] = cell_record(R, b, S.rec[j]);
        }
        done += n;
        lo += width;
    }
    __syncthreads();
    // the triplet to the last thread, the pairs from the first
    const uint32_t first = (M & 1u) ? 3u : 0u, np = (M - first) / 2u;
    if (first && g == T - 1u) collide_triplet(R, ord[0], ord[1], ord[2], (float)M);
    for (uint32_t e = g; e < np; e += T) collide_pair(R, ord[first + 2u * e], ord[first + 2u * e + 1u], (float)M);
    __syncthreads();   // the shared memory is used again
}

// collisions of a cell of m >= 2 ions
__device__ __forceinline__ uint32_t collisions_of(uint32_t m) { return (m & 1u) ? 3u + (m - 3u) / 2u : m / 2u; }

// Shared memory of a warp: up to kWarpIons ions of up to 32 cells
struct PackSmem {
    float4 v[kWarpIons];             // the ions' records, cell after cell
    uint4 w[kWarpIons];
    uint4 cell[32];                  // (first record - first place, places in the bucket end, first place, ions)
    uint32_t pidx[kWarpIons];        // where the records are in the pool
    uint32_t list[kWarpIons];        // pairs; or the keys while ties are put in order
};

// or one cell of up to kWarpCell
struct RankSmem {
    uint32_t word[kWarpCell];        // first words
    uint32_t cnt2[kWarpCell / 2 + 1];   // ions per word bucket, then their exclusive scan, two 16-bit counts a word
    uint16_t pos[kWarpCell];         // arrival in the word bucket, then the ions in order
    uint16_t arr[kWarpCell];         // ions by word bucket
};

union WarpSmem {
    PackSmem pack;
    RankSmem rank;
};

// what a block's warps put by for the block: triplets (three records, the cell's
// ions) and, in a list in R.cbig, large cells (big: the first + 1, 0: none)
constexpr uint32_t kTrips = 128;
struct WarpsSmem {
    WarpSmem warp[kCollideWarps];
    uint32_t past[kCollideWarps][32];   // of a warp's item: see item_overflow
    uint4 trip[kTrips];
};
union AnySmem {
    WarpsSmem w;
    CellSmem cell;
};
struct BlockSmem {
    AnySmem a;
    uint32_t ntrip, big, off;
};

// element exchange of the bitonic network: keep the smaller or the larger
__device__ __forceinline__ uint32_t keep(uint32_t a, uint32_t b, bool small) { return small ? min(a, b) : max(a, b); }

// sort 128 keys, key r of lane l at place 4 l + r, ascending
__device__ __forceinline__ void sort128(uint32_t (&k)[4])
{
    const uint32_t lane = threadIdx.x & 31;
#pragma unroll
    for (uint32_t size = 2; size <= 128u; size <<= 1) {
#pragma unroll
        for (uint32_t d = size >> 1; d > 0u; d >>= 1) {
            if (d >= 4u) {
                // partner 4 (lane ^ d/4) + r: the lower place keeps the smaller if its group ascends
                const bool up = ((4u * lane) & size) == 0u, low = ((4u * lane) & d) == 0u;
                const bool small = up == low;
#pragma unroll
                for (int r = 0; r < 4; ++r) k[r] = keep(k[r], __shfl_xor_sync(0xFFFFFFFFu, k[r], d / 4u), small);
            } else {
#pragma unroll
                for (int r = 0; r < 4; ++r) {
                    if (r & (int)d) continue;
                    const bool up = size >= 4u ? ((4u * lane) & size) == 0u || size > 64u : (r & 2) == 0;
                    const uint32_t lo = min(k[r], k[r | (int)d]), hi = max(k[r], k[r | (int)d]);
                    k[r] = up ? lo : hi;
                    k[r | (int)d] = up ? hi : lo;
                }
            }
        }
    }
}

// Order and collide the nq cells described in S.cell (M <= kWarpIons ions in
// all; starts: a bit at each cell's first place) by a warp.  Triplets go to
// the block's list while there is room.  Returns the collisions.
__device__ __forceinline__ uint32_t collide_warp(const RunDev& R, PackSmem& S, BlockSmem& B, uint32_t M,
                                                 const uint32_t (&starts)[4])
{
    const uint32_t lane = threadIdx.x & 31, le = 0xFFFFFFFFu >> (31u - lane);
    // the records, two a lane in flight (a lane past the last ion takes that one)
    uint32_t key[4], before[4];
    before[0] = 0u;
#pragma unroll
    for (int r = 0; r < 3; ++r) before[r + 1] = before[r] + (uint32_t)__popc(starts[r]);
#pragma unroll
    for (int h = 0; h < 4; h += 2) {
        uint32_t p[2], q[2];
        Record rec[2];
        if (h && M <= 64u) {
            key[2] = key[3] = 0xFFFFFFFFu;
            break;
        }
#pragma unroll
        for (int k = 0; k < 2; ++k) {
            const uint32_t at = 32u * (h + k) + lane, j = min(at, M - 1u);
            const uint32_t word = at < M ? (uint32_t)(h + k) : j >> 5;
            const uint32_t st = word == 0u ? starts[0] : word == 1u ? starts[1] : word == 2u ? starts[2] : starts[3];
            const uint32_t bf = word == 0u ? before[0] : word == 1u ? before[1] : word == 2u ? before[2] : before[3];
            q[k] = bf + (uint32_t)__popc(st & (0xFFFFFFFFu >> (31u - (j & 31u)))) - 1u;
            const uint4 c = S.cell[q[k]];
            p[k] = j < c.y ? c.x + j : S.pidx[j];
        }
#pragma unroll
        for (int k = 0; k < 2; ++k) rec[k] = load_record(R, p[k]);
#pragma unroll
        for (int k = 0; k < 2; ++k) {
            const uint32_t j = 32u * (h + k) + lane;
            key[h + k] = 0xFFFFFFFFu;
            if (j < M) {
                S.pidx[j] = p[k];
                S.v[j] = rec[k].v;
                S.w[j] = rec[k].w;
                key[h + k] = (q[k] << 27) | ((rec[k].w.y >> 12) << 7) | j;
            }
        }
    }
    sort128(key);
    // words of a cell that tie in their high bits: one lane puts them in order
    uint32_t next = __shfl_down_sync(0xFFFFFFFFu, key[0], 1);
    const uint32_t p0 = 4u * lane;
    const bool tie = (p0 + 1u < M && (key[0] >> 7) == (key[1] >> 7)) ||
                     (p0 + 2u < M && (key[1] >> 7) == (key[2] >> 7)) ||
                     (p0 + 3u < M && (key[2] >> 7) == (key[3] >> 7)) || (p0 + 4u < M && (key[3] >> 7) == (next >> 7));
    __syncwarp();
    if (__any_sync(0xFFFFFFFFu, tie)) {
#pragma unroll
        for (int r = 0; r < 4; ++r) S.list[4u * lane + r] = key[r];
        __syncwarp();
        if (lane == 0) {
            for (uint32_t i = 1; i < M; ++i)
                for (uint32_t t = i; t > 0u && (S.list[t - 1] >> 7) == (S.list[t] >> 7); --t) {
                    const uint32_t ka = S.list[t - 1], kb = S.list[t];
                    const uint4 wa = S.w[ka & 127u], wb = S.w[kb & 127u];
                    if (wa.y < wb.y || (wa.y == wb.y && slot_id(R, wa.x) < slot_id(R, wb.x))) break;
                    S.list[t - 1] = kb;
                    S.list[t] = ka;
                }
        }
        __syncwarp();
#pragma unroll
        for (int r = 0; r < 4; ++r) key[r] = S.list[4u * lane + r];
        next = __shfl_down_sync(0xFFFFFFFFu, key[0], 1);
        __syncwarp();
    }
    const uint32_t next2 = __shfl_down_sync(0xFFFFFFFFu, key[1], 1);
    uint32_t np = 0u, nt = 0u;
#pragma unroll
    for (int r = 0; r < 4; ++r) {
        const uint32_t p = 4u * lane + r, q = key[r] >> 27;
        const uint32_t kb = r < 3 ? key[r < 3 ? r + 1 : 0] : next;
        const uint32_t kc = r < 2 ? key[r < 2 ? r + 2 : 0] : (r == 2 ? next : next2);
        uint32_t kind = 0u, m = 0u;
        if (p < M) {
            const uint4 c = S.cell[q];
            m = c.w;
            kind = start_kind(p - c.z, m);
        }
        if (kind == 2u) {
            const uint32_t ia = S.pidx[key[r] & 127u], ib = S.pidx[kb & 127u], ic = S.pidx[kc & 127u];
            const uint32_t at = atomicAdd(&B.ntrip, 1u);
            if (at < kTrips) B.a.w.trip[at] = make_uint4(ia, ib, ic, m);
            else collide_triplet(R, ia, ib, ic, (float)m);
            S.w[key[r] & 127u].x = S.w[kb & 127u].x = S.w[kc & 127u].x = kNoCell;   // written back there
        }
        const uint32_t pairs = __ballot_sync(0xFFFFFFFFu, kind == 1u);
        nt += (uint32_t)__popc(__ballot_sync(0xFFFFFFFFu, kind == 2u));
        if (kind == 1u) S.list[np + (uint32_t)__popc(pairs & (le >> 1))] = (key[r] & 127u) | ((kb & 127u) << 7) | (q << 14);
        np += (uint32_t)__popc(pairs);
    }
    __syncwarp();
    for (uint32_t e = lane; e < np; e += 32u) {
        const uint32_t l = S.list[e], ja = l & 127u, jb = (l >> 7) & 127u;
        float4 a = S.v[ja], b = S.v[jb];
        const uint4 wa = S.w[ja];
        collide(R, a, b, R.dt, (float)S.cell[l >> 14].w, wa.z, wa.w);
        S.v[ja] = a;
        S.v[jb] = b;
    }
    __syncwarp();
    // back to the arrays in the records' order, in which neighbours mostly are
    // neighbours there too
    for (uint32_t j = lane; j < M; j += 32u) {
        const uint32_t slot = S.w[j].x;
        if (slot != kNoCell) write_back(R, slot, S.v[j]);
    }
    __syncwarp();   // the shared memory is used again
    return np + 3u * nt;
}

// Unplanned cells an item (log2), of n of them: 32, or fewer if they have so many
// ions that a warp would take these in several turns.  (One a warp, as long as the
// grid had warps, cost 6 runs at dt 1e-7 s 45.3 ms a 256 steps, and 41.2 so; 32
// always, a run with 156 ions in each of its cells a multiple.)
__device__ __forceinline__ uint32_t unplanned_lanes(const RunDev& R, uint32_t n)
{
    const unsigned long long ions = (unsigned long long)R.cword[kCwLoose + R.cword[kCwSet]] * kLooseEvery;
    uint32_t lw = 0u;
    while (lw < 5u && (ions << (lw + 1u)) <= (unsigned long long)n * kWarpIons) ++lw;
    return lw;
}

// ranges and groups of unplanned cells of a run
__device__ __forceinline__ uint32_t collide_items(const RunDev& R)
{
    const uint32_t n = R.cword[kCwUnplanned + R.cword[kCwSet]], lw = unplanned_lanes(R, n);
    return R.cword[kCwRanges] + ((n + (1u << lw) - 1u) >> lw);
}

// Order and collide one cell of kWarpIons to kWarpCell ions that all lie in its
// bucket, by a warp
__device__ __forceinline__ uint32_t collide_warp_cell(const RunDev& R, RankSmem& S, BlockSmem& B, uint32_t base,
                                                      uint32_t M)
{
    const uint32_t lane = threadIdx.x & 31;
    uint32_t* const cnt2 = S.cnt2;
    const uint16_t* const cnt = reinterpret_cast<const uint16_t*>(S.cnt2);
    for (uint32_t j = lane; j < (M + 2u) / 2u; j += 32u) cnt2[j] = 0u;
    __syncwarp();
#pragma unroll 4
    for (uint32_t j = lane; j < M; j += 32u) {
        const uint32_t w = R.crec[2 * (size_t)(base + j) + 1].y, k = __umulhi(w, M);
        S.word[j] = w;
        S.pos[j] = (uint16_t)(atomicAdd(cnt2 + (k >> 1), 1u << (16u * (k & 1u))) >> (16u * (k & 1u)));
    }
    __syncwarp();
    // exclusive scan, 16 counts a lane
    {
        constexpr int kPer = kWarpCell / 32 / 2;
        uint32_t v[kPer], sum = 0u;
#pragma unroll
        for (int k = 0; k < kPer; ++k) {
            const uint32_t i = lane * kPer + k;
            v[k] = 2u * i < M ? cnt2[i] : 0u;
            sum += (v[k] & 0xFFFFu) + (v[k] >> 16);
        }
        uint32_t incl = sum;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t t = __shfl_up_sync(0xFFFFFFFFu, incl, o);
            if (lane >= (uint32_t)o) incl += t;
        }
        uint32_t o = incl - sum;
        __syncwarp();
#pragma unroll
        for (int k = 0; k < kPer; ++k) {
            const uint32_t i = lane * kPer + k, lo = v[k] & 0xFFFFu;
            if (2u * i < M) cnt2[i] = o | ((o + lo) << 16);
            o += lo + (v[k] >> 16);
        }
        __syncwarp();
        if (lane == 0) {   // the end: the high half of a word, or a word of its own
            if (M & 1u) cnt2[M >> 1] = (cnt2[M >> 1] & 0xFFFFu) | (M << 16);
            else cnt2[M >> 1] = M;
        }
    }
    __syncwarp();
    for (uint32_t j = lane; j < M; j += 32u) S.arr[cnt[__umulhi(S.word[j], M)] + S.pos[j]] = (uint16_t)j;
    __syncwarp();
    for (uint32_t j = lane; j < M; j += 32u) {
        const uint32_t w = S.word[j], k = __umulhi(w, M);
        const uint32_t lo = cnt[k], hi = cnt[k + 1];
        uint32_t r = lo;
        for (uint32_t t = lo; t < hi; ++t) {
            const uint32_t i = S.arr[t], wi = S.word[i];
            if (wi < w || (wi == w && i != j && record_id(R, base + i) < record_id(R, base + j))) ++r;
        }
        S.pos[r] = (uint16_t)j;   // (the arrivals are done with)
    }
    __syncwarp();
    const uint32_t first = (M & 1u) ? 3u : 0u, np = (M - first) / 2u;
    if (first && lane == 0) {
        const uint32_t ia = base + S.pos[0], ib = base + S.pos[1], ic = base + S.pos[2];
        const uint32_t at = atomicAdd(&B.ntrip, 1u);
        if (at < kTrips) B.a.w.trip[at] = make_uint4(ia, ib, ic, M);
        else collide_triplet(R, ia, ib, ic, (float)M);
    }
    for (uint32_t e = lane; e < np; e += 32u)
        collide_pair(R, base + S.pos[first + 2u * e], base + S.pos[first + 2u * e + 1u], (float)M);
    __syncwarp();   // the shared memory is used again
    return np + (first ? 3u : 0u);
}

// a lane's cell of an item: its bucket, its participants and chain
struct ItemCell { uint32_t base, room, m, head; };

// The cells of an item of a run, a lane each; their counts (and chains) are
// taken and left zero for the next step
__device__ __forceinline__ ItemCell item_cell(const RunDev& R, uint32_t item)
{
    const uint32_t lane = threadIdx.x & 31;
    const uint32_t nr = R.cword[kCwRanges];
    uint32_t c = kNoCell;
    uint32_t* count = nullptr;
    ItemCell ic{0u, 0u, 0u, 0u};
    if (item < nr) {
        const uint32_t k = R.rstart[item] + lane;
        if (k < R.rstart[item + 1]) {
            const uint4 p = R.pcell[k];
            ic.base = p.x;
            ic.room = p.y;
            ic.m = p.w;
            c = p.z;
            if (R.pcount) count = R.pcount + k;
        }
    } else {
        const uint32_t n = R.cword[kCwUnplanned + R.cword[kCwSet]], lw = unplanned_lanes(R, n);
        const uint32_t k = ((item - nr) << lw) + lane;
        if (!(lane >> lw) && k < n) {
            c = R.xcell[k];
            count = R.ccount + c;
        }
    }
    if (count) {
        ic.m = *count;
        if (ic.m) *count = 0u;
        if (ic.m > ic.room) {
            ic.head = R.chead[c];
            R.chead[c] = 0u;
        }
    }
    if (ic.m < 2u) ic.m = 0u;   // nothing to collide with
    return ic;
}

// does a cell that takes a block have records past its bucket?
__device__ __forceinline__ bool past_large(const ItemCell& ic) { return ic.m > ic.room && ic.m > (uint32_t)kWarpIons; }

// The records past the buckets of an item with such a cell, written to cidx: each
// lane walks its cell's chain, all of them at once.  past: the lanes' places there
// less their rooms.  (Out of line: its registers are not the others'.)
__device__ __noinline__ void item_overflow(const RunDev& R, const ItemCell ic, uint32_t* past)
{
    const uint32_t lane = threadIdx.x & 31, n = ic.m > ic.room ? ic.m - ic.room : 0u;
    uint32_t incl = n;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t t = __shfl_up_sync(0xFFFFFFFFu, incl, o);
        if (lane >= (uint32_t)o) incl += t;
    }
    uint32_t first = 0u;
    if (lane == 31u) first = atomicAdd(R.cword + kCwPast, incl);   // (all of a step's are at most cover)
    first = __shfl_sync(0xFFFFFFFFu, first, 31) + incl - n;
    uint32_t at = ic.head;
    for (uint32_t i = 0; i < n && at;) {   // (a chain holds as many as the count says)
        const uint32_t p = R.cpool + at - 1u;
        const uint2 run = R.cnext[at - 1u];
        for (uint32_t k = 0; k < run.y && i < n; ++k, ++i) R.cidx[first + i] = p + k;
        at = run.x;
    }
    past[lane] = first - ic.room;
    __syncwarp();
}

// One item of a run by a warp.  Returns the collisions.
__device__ __forceinline__ uint32_t collide_item(const RunDev& R, WarpSmem& S, BlockSmem& B, const ItemCell& ic)
{
    const uint32_t lane = threadIdx.x & 31;
    const uint32_t m = ic.m;
    uint32_t ncoll = 0u;
    // (else the records past a cell's bucket are found as it is taken: 1.7e7 particles in
    // 12 runs, 32 steps, 12.7 ms with all of them through cidx, 12.2 so)
    uint32_t* const past = B.a.w.past[threadIdx.x >> 5];
    const bool many = __any_sync(0xFFFFFFFFu, past_large(ic));
    if (many) item_overflow(R, ic, past);
    uint32_t left = __ballot_sync(0xFFFFFFFFu, m > 0u);
    while (left) {
        // the next cells that fit together
        const bool mine = (left >> lane) & 1u;
        uint32_t incl = mine ? m : 0u;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t t = __shfl_up_sync(0xFFFFFFFFu, incl, o);
            if (lane >= (uint32_t)o) incl += t;
        }
        const uint32_t take = __ballot_sync(0xFFFFFFFFu, mine && incl <= (uint32_t)kWarpIons);
        if (!take) {   // the first of them goes alone
            const int src = __ffs(left) - 1;
            left &= left - 1u;
            const uint32_t cm = __shfl_sync(0xFFFFFFFFu, m, src), room = __shfl_sync(0xFFFFFFFFu, ic.room, src);
            const uint32_t base = __shfl_sync(0xFFFFFFFFu, ic.base, src);
            if (cm <= (uint32_t)kWarpCell && cm <= room) {
                ncoll += collide_warp_cell(R, S.rank, B, base, cm);
                continue;
            }
            const BigCell big = make_uint4(base, room, cm, past[src]);
            if (lane == 0) {
                const uint32_t at = atomicAdd(R.cword + kCwBig, 1u);
                R.cbig[2 * at] = big;
                R.cbig[2 * at + 1].x = atomicExch(&B.big, at + 1u);
            }
            continue;
        }
        left &= ~take;
        const bool taken = (take >> lane) & 1u;
        const uint32_t seg = incl - m;
        if (taken)
            S.pack.cell[__popc(take & ((1u << lane) - 1u))] = make_uint4(ic.base - seg, seg + min(ic.room, m), seg, m);
        const uint32_t M = __shfl_sync(0xFFFFFFFFu, incl, 31 - __clz((int)take));
        uint32_t starts[4];
#pragma unroll
        for (uint32_t r = 0; r < 4u; ++r)
            starts[r] = __reduce_or_sync(0xFFFFFFFFu, taken && (seg >> 5) == r ? 1u << (seg & 31u) : 0u);
        if (taken && m > ic.room) {   // the ions past the bucket
            uint32_t at = ic.head, i = ic.room;
            if (many)
                for (; i < m; ++i) S.pack.pidx[seg + i] = R.cidx[past[lane] + i];
            while (i < m && at) {   // (a chain holds as many as the count says)
                const uint2 link = R.cnext[at - 1u];
                for (uint32_t k = 0; k < link.y && i < m; ++k, ++i) S.pack.pidx[seg + i] = R.cpool + at - 1u + k;
                at = link.x;
            }
        }
        __syncwarp();
        ncoll += collide_warp(R, S.pack, B, M, starts);
    }
    return ncoll;
}

// a large cell, by the block
__device__ __forceinline__ void collide_big(const RunDev& R, BlockSmem& B, const BigCell& b)
{
    collide_cell(R, B.a.cell, b, &B.off);
    if (threadIdx.x == 0) atomicAdd(R.tally + kTallyCoulomb, (unsigned long long)collisions_of(b.z));
}

// what the block's warps have put by (all threads call it, at the same point)
__device__ __forceinline__ void collide_rest(const RunDev& R, BlockSmem& B)
{
    __syncthreads();
    const uint32_t nt = min(B.ntrip, kTrips);
    static_assert(kTrips == 32 * kCollideWarps, "a triplet a thread");
    if (threadIdx.x < nt) {
        const uint4 t = B.a.w.trip[threadIdx.x];
        collide_triplet(R, t.x, t.y, t.z, (float)t.w);
    }
    __syncthreads();   // the list's memory is the large cells' too
    for (uint32_t e = B.big; e;) {
        const BigCell b = R.cbig[2 * (e - 1u)];
        e = R.cbig[2 * (e - 1u) + 1].x;
        collide_big(R, B, b);
    }
    __syncthreads();
    if (threadIdx.x == 0) B.ntrip = B.big = 0u;
    __syncthreads();
}

// End of a run's step, by one thread at the start of the collision kernel: it
// touches only what this kernel does not read (the step number, the window's
// list and the counters of the next step)
__device__ __forceinline__ void step_done(const RunDev& R)
{
    *R.step += 1u;
    const uint32_t other = 1u - R.cword[kCwSet];
    R.cword[kCwUnplanned + other] = 0u;
    R.cword[kCwLoose + other] = 0u;
    R.cword[kCwOverflow + other] = 0u;
    if (R.nleave && --R.nleave[2] == 0u) R.nleave[0] = R.nleave[1] = 0u;   // the window's list is done with
}

// items of each of up to kRunChunk runs at a time, and which run item v belongs to
constexpr uint32_t kRunChunk = 128;

// the runs' item counts (f(run)) as an exclusive prefix in s_pref[0..nr]; all
// threads of the block call it
template <class F>
__device__ __forceinline__ void run_prefix(const RunDev* runs, uint32_t nr, uint32_t* s_pref, F f)
{
    __syncthreads();
    for (uint32_t r = threadIdx.x; r < nr; r += blockDim.x)
        s_pref[r + 1] = runs[r].step && (runs[r].flags & kFCoulomb) ? f(runs[r]) : 0u;
    if (threadIdx.x == 0) s_pref[0] = 0u;
    __syncthreads();
    if (threadIdx.x < 32) {
        uint32_t carry = 0u;
        for (uint32_t r0 = 0; r0 < nr; r0 += 32u) {
            uint32_t v = r0 + threadIdx.x < nr ? s_pref[r0 + threadIdx.x + 1] : 0u;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const uint32_t t = __shfl_up_sync(0xFFFFFFFFu, v, o);
                if ((threadIdx.x & 31u) >= (uint32_t)o) v += t;
            }
            if (r0 + threadIdx.x < nr) s_pref[r0 + threadIdx.x + 1] = carry + v;
            carry += __shfl_sync(0xFFFFFFFFu, v, 31);
        }
    }
    __syncthreads();
}

__device__ __forceinline__ uint32_t run_of(const uint32_t* s_pref, uint32_t nr, uint32_t v)
{
    uint32_t lo = 0, hi = nr;   // s_pref[lo] <= v < s_pref[hi]
    while (hi - lo > 1u) {
        const uint32_t mid = (lo + hi) >> 1;
        if (s_pref[mid] <= v) lo = mid;
        else hi = mid;
    }
    return lo;
}

// items a warp takes between two visits of the block to what was put by
constexpr uint32_t kVisit = 4;

// The block's share of a run's items: its warps take one each of every
// kCollideWarps, from v0, then go on stride items further.  The next item's
// cells are read while this one's collide.
__device__ __forceinline__ void collide_share(const RunDev& R, BlockSmem& B, uint32_t v0, uint32_t end, uint32_t stride)
{
    const uint32_t warp = threadIdx.x >> 5;
    uint32_t n = 0u, ncoll = 0u;
    ItemCell next{0u, 0u, 0u, 0u};
    if (v0 + warp < end) next = item_cell(R, v0 + warp);
    for (; v0 < end; v0 += stride) {
        const ItemCell ic = next;
        next = ItemCell{0u, 0u, 0u, 0u};
        if (v0 + stride + warp < end) next = item_cell(R, v0 + stride + warp);
        ncoll += collide_item(R, B.a.w.warp[warp], B, ic);
        if (++n % kVisit == 0u) collide_rest(R, B);
    }
    if ((threadIdx.x & 31u) == 0u && ncoll) atomicAdd(R.tally + kTallyCoulomb, (unsigned long long)ncoll);
    collide_rest(R, B);
}

__global__ void __launch_bounds__(32 * kCollideWarps, 8) k_collide(const __grid_constant__ RunDev R)
{
    __shared__ BlockSmem B;
    pdl_wait();
    pdl_trigger();
    if (threadIdx.x == 0) B.ntrip = B.big = 0u;
    if (blockIdx.x == 0 && threadIdx.x == 32) step_done(R);
    __syncthreads();
    collide_share(R, B, blockIdx.x * kCollideWarps, collide_items(R), gridDim.x * kCollideWarps);
}

// Every run of a batch.  A block takes one stretch of the runs' items, so that
// it has a run's parameter block in shared memory for many items, and reads
// ahead as above (4.2e6 ions in 12 runs: 205 us with the items dealt out in turn
// and the parameters read from global memory, 180 so).
__global__ void __launch_bounds__(32 * kCollideWarps, 8) k_collide_batch(const RunDev* __restrict__ runs,
                                                                        uint32_t nruns)
{
    __shared__ BlockSmem B;
    __shared__ RunDev rs;
    __shared__ uint32_t s_pref[kRunChunk + 1];
    pdl_wait();
    pdl_trigger();
    if (threadIdx.x == 0) B.ntrip = B.big = 0u;
    if (blockIdx.x == 0)
        for (uint32_t r = threadIdx.x; r < nruns; r += blockDim.x)
            if (runs[r].step && (runs[r].flags & kFCoulomb)) step_done(runs[r]);
    for (uint32_t r0 = 0; r0 < nruns; r0 += kRunChunk) {
        const uint32_t nr = min(kRunChunk, nruns - r0);
        run_prefix(runs + r0, nr, s_pref, [](const RunDev& R) { return collide_items(R); });
        const uint32_t total = s_pref[nr];
        // whole rounds of the block's warps
        const uint32_t rounds = (total + kCollideWarps - 1u) / kCollideWarps;
        uint32_t v = (uint32_t)((unsigned long long)rounds * blockIdx.x / gridDim.x) * kCollideWarps;
        const uint32_t end = min(total, (uint32_t)((unsigned long long)rounds * (blockIdx.x + 1u) / gridDim.x) * kCollideWarps);
        while (v < end) {
            const uint32_t r = run_of(s_pref, nr, v), first = s_pref[r], stop = min(end, s_pref[r + 1]);
            stage_run(rs, runs + r0 + r);
            __syncthreads();
            collide_share(rs, B, v - first, stop - first, kCollideWarps);
            v = stop;
        }
    }
}

template <class K>
int resident(K kernel, int threads)
{
    int b = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, kernel, threads, 0) != cudaSuccess || b < 1) b = 1;
    return b;
}

}  // namespace

uint32_t plan_blocks(uint32_t ncells) { return (ncells + kPlanBlock - 1u) / kPlanBlock; }

cudaError_t launch_plan(const RunDev& R, uint32_t* count, bool zero, unsigned long long* blk, cudaStream_t s)
{
    const uint32_t nb = plan_blocks(R.ncells);
    cudaError_t e = launch_pdl(k_plan_sum, dim3(nb), dim3(kPlanThreads), 0, s, R, (const uint32_t*)count, blk);
    if (e == cudaSuccess)
        e = launch_pdl(k_plan_cells, dim3(nb), dim3(kPlanThreads), 0, s, R, count, (const unsigned long long*)blk,
                       zero ? 1 : 0);
    return e;
}

int collide_blocks(int sm_count)
{
    return sm_count * std::min(resident(k_collide, 32 * kCollideWarps), resident(k_collide_batch, 32 * kCollideWarps));
}

// no more blocks than n particles can give work (an item holds two colliding
// ions or more, few items hold fewer than 32)
static int grid_for(int most, uint32_t n) { return (int)std::min((uint32_t)most, n / (kCollideWarps * 32u) + 2u); }

cudaError_t launch_coulomb(const RunDev& R, uint32_t n, int most, cudaStream_t s)
{
    return launch_pdl(k_collide, dim3(grid_for(most, n)), dim3(32 * kCollideWarps), 0, s, R);
}

cudaError_t launch_coulomb_batch(const RunDev* runs, uint32_t nruns, uint32_t n, int most, cudaStream_t s)
{
    return launch_pdl(k_collide_batch, dim3(grid_for(most, n)), dim3(32 * kCollideWarps), 0, s, runs, nruns);
}

}  // namespace ecris
