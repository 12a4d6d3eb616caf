// Per-macroparticle time step (push -> boundary test -> MCC -> NGP
// deposition) of the ECRIS model of Mironov et al. (arXiv:1507.03392, Sec.
// II), the wall and aperture bookkeeping of the particles that leave the
// chamber, the deposit fold and the charge-state census used by the
// diagnostics.
//
// Data layout: each run's particles are SoA arrays x, y, z (fixed point), vx,
// vy, vz, a u32 meta word and a u32 stable id, padded to a multiple of 4.
// Per-cell data (n_e, zone, delta) and the E grid are float4 records read
// through L1/L2; the rate table is read through L1.  The deposit is one packed
// 64-bit reduction per run of lanes in the same cell (count in the high word,
// charge in the low word).  The rare crossing geometry of a leaver (FP64) is
// out of line, so the step itself carries no FP64 registers.
#include <algorithm>

#include "ecris_internal.cuh"

namespace ecris {

namespace {

// Cosine-law re-emission at temperature T0 (full accommodation): normal speed
// sigma sqrt(-2 ln U0) along the inward normal n, tangential components one
// Box-Muller pair along e1, e2.
__device__ __forceinline__ void emit(float sigma, float nx, float ny, float nz, float e1x, float e1y,
                                     float e1z, float e2x, float e2y, float e2z, const Words& w,
                                     float& vx, float& vy, float& vz)
{
    const float vn = sigma * sqrtf(-2.0f * logf(unit01(w.w0)));
    const float rt = sigma * sqrtf(-2.0f * logf(unit01(w.w1)));
    float s, c;
    sincospif(2.0f * unit01(w.w2), &s, &c);
    const float t1 = rt * c, t2 = rt * s;
    vx = vn * nx + t1 * e1x + t2 * e2x;
    vy = vn * ny + t1 * e1y + t2 * e2y;
    vz = vn * nz + t1 * e1z + t2 * e2z;
}

// |v|^2 + a, contraction written out
__device__ __forceinline__ float norm2_plus(float vx, float vy, float vz, float a)
{
    return fmaf(vx, vx, fmaf(vy, vy, fmaf(vz, vz, a)));
}

// probability 1 - exp(-lam) of at least one event in a step; for small lam
// the cubic Taylor polynomial is exact to FP32 rounding (error < lam^4 / 24)
__device__ __forceinline__ float event_prob(float lam)
{
    if (lam < 1e-3f) return lam * fmaf(-lam, fmaf(-lam, 1.0f / 6.0f, 0.5f), 1.0f);
    return -expm1f(-lam);
}

// 64-bit displacement for the rare step longer than 2^30 fixed-point units
// (kept out of line: the common path converts in 32 bits)
struct Disp { long long x, y, z; };

__device__ __noinline__ Disp far_displacement(float dx, float dy, float dz)
{
    return Disp{__float2ll_rn(fminf(fmaxf(dx, -1e12f), 1e12f)), __float2ll_rn(fminf(fmaxf(dy, -1e12f), 1e12f)),
                __float2ll_rn(fminf(fmaxf(dz, -1e12f), 1e12f))};
}

// Position after the step's straight move with the (already pushed)
// velocity, in 64-bit fixed point, for a particle that left the chamber; move
// below gets the same integers.  The displacement is rounded to
// nearest; below 2^30 units a 32-bit conversion gives the same integer,
// larger (or non-finite) ones take the bounded 64-bit conversion.
__device__ __forceinline__ void displace(const RunDev& R, int32_t X, int32_t Y, int32_t Z, float vx, float vy,
                                         float vz, long long& xn, long long& yn, long long& zn)
{
    xn = X;
    yn = Y;
    zn = Z;
    if (!(R.flags & kFPush)) return;
    const float dx = vx * R.dt_sxy, dy = vy * R.dt_sxy, dz = vz * R.dt_sz;
    if (fmaxf(fabsf(dx), fmaxf(fabsf(dy), fabsf(dz))) < 1.0e9f) {
        xn += __float2int_rn(dx);
        yn += __float2int_rn(dy);
        zn += __float2int_rn(dz);
    } else {
        const Disp d = far_displacement(dx, dy, dz);
        xn += d.x;
        yn += d.y;
        zn += d.z;
    }
}

constexpr long long kLim = 2147483648ll;   // 2^31: the fixed-point range

// Boundary test on the new position, exact in fixed point: outside the
// cylinder wall (r > R0), behind the injection plane (z < 0), past the
// extraction plane (z >= L).
__device__ __forceinline__ void outside(long long xn, long long yn, long long zn, bool& out_r, bool& out_0,
                                        bool& out_L)
{
    const bool out_xy = xn < -kLim || xn >= kLim || yn < -kLim || yn >= kLim;
    out_r = out_xy || (long long)(int32_t)xn * (int32_t)xn + (long long)(int32_t)yn * (int32_t)yn > (1ll << 62);
    out_0 = zn < -kLim;
    out_L = zn >= kLim;
}

__device__ __forceinline__ int32_t clamp_fx(long long v) { return (int32_t)max(min(v, kLim - 1), -kLim); }

// a + b in 32 bits, and whether the exact sum left the 32-bit range
__device__ __forceinline__ int32_t add_wrap(int32_t a, int32_t b, bool& over)
{
    const int32_t s = (int32_t)((uint32_t)a + (uint32_t)b);
    over = ((a ^ s) & (b ^ s)) < 0;
    return s;
}

// The straight move of the step and the boundary test, as displace() and
// outside() give them, but in 32-bit arithmetic for the common step shorter
// than 2^30 units: the fixed-point range is the chamber's bounding box, so a
// sum that leaves the 32-bit range has left the chamber.  On return X, Y, Z
// hold the new position (clamped into the range for a leaver); true if the
// particle left.
template <bool kPush>
__device__ __forceinline__ bool move(const RunDev& R, int32_t& X, int32_t& Y, int32_t& Z, float vx, float vy,
                                     float vz)
{
    const bool push = kPush || (R.flags & kFPush) != 0;
    const float dx = push ? vx * R.dt_sxy : 0.0f, dy = push ? vy * R.dt_sxy : 0.0f, dz = push ? vz * R.dt_sz : 0.0f;
    if (fmaxf(fabsf(dx), fmaxf(fabsf(dy), fabsf(dz))) < 1.0e9f) {
        bool ox, oy, oz;
        const int32_t xn = add_wrap(X, __float2int_rn(dx), ox);
        const int32_t yn = add_wrap(Y, __float2int_rn(dy), oy);
        const int32_t zn = add_wrap(Z, __float2int_rn(dz), oz);
        const bool leave = ox | oy | oz ||
                           (long long)xn * xn + (long long)yn * yn > (1ll << 62);
        if (!leave) {
            X = xn;
            Y = yn;
            Z = zn;
        }
        return leave;
    }
    long long xn, yn, zn;
    displace(R, X, Y, Z, vx, vy, vz, xn, yn, zn);
    bool out_r, out_0, out_L;
    outside(xn, yn, zn, out_r, out_0, out_L);
    if (out_r | out_0 | out_L) return true;
    X = clamp_fx(xn);
    Y = clamp_fx(yn);
    Z = clamp_fx(zn);
    return false;
}

// Elastic ion-atom scattering (a rare event, kept out of line so that the
// per-particle code's registers do not carry it): isotropic in the
// centre-of-mass frame with a background atom drawn at T0 from the stream-3
// words u; the new direction of the relative velocity from the wall stream,
// unused by a particle that stays inside
__device__ __noinline__ void elastic_scatter(const RunDev& R, const Words& u, uint32_t pid, uint32_t step, float& vx,
                                             float& vy, float& vz)
{
    const Words d = rng_words(R, pid, step, 2u);
    float s1, c1, s2, c2;
    const float r1 = R.sig0 * sqrtf(-2.0f * logf(unit01(u.w0)));
    sincospif(2.0f * unit01(u.w1), &s1, &c1);
    const float r2 = R.sig0 * sqrtf(-2.0f * logf(unit01(u.w2)));
    sincospif(2.0f * unit01(u.w3), &s2, &c2);
    const float ax = r1 * c1, ay = r1 * s1, az = r2 * c2;
    const float gx = vx - ax, gy = vy - ay, gz = vz - az;
    const float gm = sqrtf(gx * gx + gy * gy + gz * gz);
    const float ct = 2.0f * unit01(d.w0) - 1.0f;
    const float st = sqrtf(fmaxf(0.0f, 1.0f - ct * ct));
    float sp, cp;
    sincospif(2.0f * unit01(d.w1), &sp, &cp);
    vx = 0.5f * (vx + ax) + 0.5f * gm * (st * cp);
    vy = 0.5f * (vy + ay) + 0.5f * gm * (st * sp);
    vz = 0.5f * (vz + az) + 0.5f * gm * ct;
}

// false if no cell can ionise an atom whose ionisation word is w0: the gate
// bounds the threshold of every cell.  It comes with the parameter block
// while the host knows the densest cell, else from the word the device keeps
// after the rate table (a gate of 0 reads the same either way)
__device__ __forceinline__ bool atom_may_ionize(const RunDev& R, uint32_t w0)
{
    uint32_t gate = R.atom_gate;
    if (gate == 0u) gate = __ldg(reinterpret_cast<const uint32_t*>(R.kdt) + kGateWord);
    return w0 < gate || gate == 0xFFFFFFFFu;
}

// Is the run one for the step without tests: every process on, neutrals there,
// no E grid, the kick quadratic in Q?  Testing them for every particle took one
// instruction in eight.
__device__ __forceinline__ bool plain_run(const RunDev& R)
{
    constexpr uint32_t all = kFPush | kFIonize | kFCx | kFEikick;
    return (R.flags & (all | kFHasE)) == all && R.n0s1 > 0.0f && R.ei_pow == 2;
}

// What a particle carries from step to step of a window: its cell's record and
// what follows from it and the charge state, so that a particle that stays in
// its cell reads nothing and forms neither again.
struct Carry {
    uint32_t cell = kNoCell;   // the cell at X, Y, Z (kNoCell: not known)
    float4 cr;                 // its record
    uint32_t qthr = kNoCell;   // charge state that thr holds for (kNoCell: none)
    uint32_t thr, always;      // the ionisation word fires below thr, or always (~0)
    uint32_t qD = kNoCell;     // charge state that D holds for
    float D;                   // the kick's size
};

// Advance one particle by one step.  pid is its stable id (the Philox counter
// word).  On return dep_cell is the cell it deposits in and ckey the cell
// where it can take part in Coulomb collisions (kNoCell: no ion, or it left).  A
// particle that left the chamber keeps its old position and returns true
// with its pushed velocity: leave_particle finishes its step.
// kVar: with the code of the opt-in processes (double ionisation, elastic
// ion-atom scattering); without it the kernels carry none of their branches.
// kCarry: c holds the particle's cell from its last step.  kPlain: every process
// is on and there is no E grid (plain_run), so nothing is left to test
template <bool kVar, bool kCarry, bool kPlain>
__device__ __forceinline__ bool step_particle(const RunDev& R, uint32_t pid, uint32_t step, int32_t& X,
                                              int32_t& Y, int32_t& Z, float& vx, float& vy, float& vz,
                                              uint32_t& meta, uint32_t& ckey, uint32_t& dep_cell, Carry& c)
{
    ckey = kNoCell;
    dep_cell = kNoCell;
    const uint32_t status = meta & 0xFFFF0000u;
    if (status & (kStFrozen | kStPad)) {
        meta = status | (meta & kQMask);   // events of a frozen particle are cleared
        return false;
    }
    uint32_t Q = meta & kQMask;
    uint32_t ev = 0;

    // ---- push: Boris rotation for ions, straight line for atoms ----
    // an ion's cell record is fetched with its field gather, at the old
    // position; the push moves it far less than a cell, so it is reused
    // unless the particle crossed into another cell
    if (!kCarry) c.cell = kNoCell;
    if (Q > 0 && c.cell == kNoCell) {
        c.cell = ngp_cell(R, X, Y, Z);
        c.cr = __ldg(R.cell + c.cell);
        if (kCarry) c.qthr = c.qD = kNoCell;
    }
    if ((kPlain || (R.flags & kFPush)) && Q > 0) {
        const float x0 = fx_xy(R, X), y0 = fx_xy(R, Y), z0 = fx_z(R, Z);
        float Bx, By, Bz, Ex, Ey, Ez;
        if (kVar && R.btab) bfield_table(R, x0, y0, z0, Bx, By, Bz);
        else bfield(R, x0, y0, z0, Bx, By, Bz);
        if (!kPlain && (R.flags & kFHasE)) {
            efield(R, x0, y0, z0, Ex, Ey, Ez);
        } else {
            Ex = 0.0f;   // no E grid: the gather would return zeros
            Ey = 0.0f;
            Ez = 0.0f;
        }
        // (FMAs written out: this file is compiled without contraction)
        const float h = (float)Q * R.qm_unit * R.half_dt;
        float mx = fmaf(h, Ex, vx), my = fmaf(h, Ey, vy), mz = fmaf(h, Ez, vz);
        const float tx = h * Bx, ty = h * By, tz = h * Bz;
        const float sf = __fdividef(2.0f, fmaf(tx, tx, fmaf(ty, ty, fmaf(tz, tz, 1.0f))));
        const float px = mx + fmaf(my, tz, -mz * ty);
        const float py = my + fmaf(mz, tx, -mx * tz);
        const float pz = mz + fmaf(mx, ty, -my * tx);
        mx = fmaf(fmaf(py, tz, -pz * ty), sf, mx);
        my = fmaf(fmaf(pz, tx, -px * tz), sf, my);
        mz = fmaf(fmaf(px, ty, -py * tx), sf, mz);
        vx = fmaf(h, Ex, mx);
        vy = fmaf(h, Ey, my);
        vz = fmaf(h, Ez, mz);
    }
    const int32_t X0 = X, Y0 = Y, Z0 = Z;
    if (move<kPlain>(R, X, Y, Z, vx, vy, vz)) {
        X = X0;   // leave_particle redoes the move from the old position
        Y = Y0;
        Z = Z0;
        meta = status | Q;
        if (kCarry) c.cell = kNoCell;   // it goes on elsewhere
        return true;
    }

    // ---- MCC in the particle's cell ----
    const uint32_t cell = ngp_cell(R, X, Y, Z);
    const Words w = rng_words(R, pid, step, 0u);
    // an atom needs its cell only if its ionisation word could fire in
    // the densest cell; otherwise no cell can ionise it this step
    const bool ionize = (kPlain || (R.flags & kFIonize)) && (int)Q < R.qmax;
    const bool need = Q > 0 || (ionize && atom_may_ionize(R, w.w0));
    if (need && cell != c.cell) {
        c.cr = __ldg(R.cell + cell);   // n_e, zone, delta_x, delta_y
        if (kCarry) c.qthr = c.qD = kNoCell;
    }
    // (an atom that needed no record has none to carry)
    if (kCarry) c.cell = need ? cell : kNoCell;
    const float4 cr = c.cr;
    const int zone = cr.y > 0.5f ? 1 : 0;
    const bool recomb = kVar && (R.flags & kFRecomb) && Q >= 1;
    if ((ionize && need) || recomb) {
        if (!kCarry || c.qthr != Q) {
            const float t = event_prob(cr.x * __ldg(R.kdt + zone * kQSlots + Q)) * 4294967296.0f;
            c.always = t >= 4294967296.0f ? 0xFFFFFFFFu : 0u;   // (as fires())
            c.thr = __float2uint_rz(t);
            if (kCarry) c.qthr = Q;
        }
        if (w.w0 < c.thr || c.always) {
            if constexpr (kVar) {
                // single, double, triple and recombination share [0, p) in
                // proportion to their rates: below p k1/k one electron goes,
                // below p (k1+k2)/k two, below p (k1+k2+k3)/k three, above
                // that one is captured
                const float p = event_prob(cr.x * __ldg(R.kdt + zone * kQSlots + Q));
                int up = 1;
                if (R.flags & (kFDouble | kFRecomb)) {
                    if (!fires(w.w0, p * __ldg(R.kdt + 2 * kQSlots + zone * kQSlots + Q))) {
                        if (fires(w.w0, p * __ldg(R.kdt + 4 * kQSlots + zone * kQSlots + Q))) up = 2;
                        else up = fires(w.w0, p * __ldg(R.kdt + 6 * kQSlots + zone * kQSlots + Q)) ? 3 : -1;
                    }
                }
                if (up > 0) {
                    if (Q == 0) R.birth[pid] = step;   // an ion is born (first-passage clock)
                    Q += (uint32_t)up;
                    ev |= kEvIonize;
                } else {
                    Q -= 1u;
                    ev |= kEvRecomb;
                }
            } else {
                if (Q == 0) R.birth[pid] = step;   // an ion is born (first-passage clock)
                Q += 1;
                ev |= kEvIonize;
            }
        }
    }
    // collisions with the neutral background: 1 charge exchange, 2 elastic
    uint32_t coll = 0u;
    if (kVar && (R.flags & kFElastic) && R.n0sel > 0.0f) {
        if (Q >= 1) {
            // either process with probability 1 - exp(-n0 (sigma_cx + sigma_el)
            // v_rel dt), shared in proportion to the cross sections
            const float vrel = sqrt_approx(norm2_plus(vx, vy, vz, R.vth2));
            const float scx = ((R.flags & kFCx) && Q != 2) ? R.n0s1 * (float)Q : 0.0f;
            const float sel = R.n0sel * (float)Q;
            const float pt = event_prob((scx + sel) * vrel * R.dt);
            if (fires(w.w1, pt)) coll = fires(w.w1, pt * (scx / (scx + sel))) ? 1u : 2u;
        }
    } else if ((kPlain || ((R.flags & kFCx) && R.n0s1 > 0.0f)) && Q >= 1 && Q != 2) {
        const float vrel = sqrt_approx(norm2_plus(vx, vy, vz, R.vth2));
        const float p = event_prob(R.n0s1 * (float)Q * vrel * R.dt);
        if (fires(w.w1, p)) coll = 1u;
    }
    if (coll) {
        const Words u = rng_words(R, pid, step, 3u);
        if (kVar && coll == 2u) {
            elastic_scatter(R, u, pid, step, vx, vy, vz);
            ev |= kEvElastic;
        } else {
            ev |= kEvCx;
            if (Q == 1) {
                float s1, c1, s2, c2;
                const float r1 = R.sig0 * sqrtf(-2.0f * logf(unit01(u.w0)));
                sincospif(2.0f * unit01(u.w1), &s1, &c1);
                const float r2 = R.sig0 * sqrtf(-2.0f * logf(unit01(u.w2)));
                sincospif(2.0f * unit01(u.w3), &s2, &c2);
                vx = r1 * c1; vy = r1 * s1; vz = r2 * c2;
            } else {
                const float ct = 2.0f * unit01(u.w0) - 1.0f;
                const float st = sqrtf(fmaxf(0.0f, 1.0f - ct * ct));
                float sp, cp;
                sincospif(2.0f * unit01(u.w1), &sp, &cp);
                vx += R.dv_cx * st * cp;
                vy += R.dv_cx * st * sp;
                vz += R.dv_cx * ct;
                Q -= 1;
            }
        }
    }
    if ((kPlain || (R.flags & kFEikick)) && Q >= 1) {
        if (!kCarry || c.qD != Q) {
            const float qp = !kPlain && R.ei_pow == 1 ? (float)Q : (float)(Q * Q);
            c.D = sqrt_approx((zone ? R.ei_coef[1] : R.ei_coef[0]) * cr.x * qp);
            if (kCarry) c.qD = Q;
        }
        const float D = c.D;
        const float ct = fmaf(2.0f, unit01(w.w2), -1.0f);
        const float st = sqrt_approx(fmaxf(0.0f, fmaf(-ct, ct, 1.0f)));
        float sp, cp;
        sincos_2pi(unit01(w.w3), &sp, &cp);   // azimuth
        const float dxv = fmaf(st, cp, cr.z), dyv = fmaf(st, sp, cr.w), dzv = ct;
        const float m2 = norm2_plus(dxv, dyv, dzv, 0.0f);
        if (m2 > 0.0f) {
            const float k = D * rsqrtf(m2);
            vx = fmaf(k, dxv, vx);
            vy = fmaf(k, dyv, vy);
            vz = fmaf(k, dzv, vz);
        }
    }
    if (Q >= 1) ckey = cell;
    dep_cell = cell;   // NGP deposition at the final position (aggregated over the warp by the caller)
    meta = status | ev | Q;
    return false;
}

// first-passage time of an extracted ion, age in steps (>= 1 for an ion born
// in an earlier step): 4 log bins per octave, and the age summed by Q
__device__ __forceinline__ void fptd_record(const RunDev& R, uint32_t Q, uint32_t age)
{
    if (age == 0u) return;
    const int e = 31 - __clz(age);
    const uint32_t m = e >= 2 ? (age >> (e - 2)) & 3u : (age << (2 - e)) & 3u;
    atomicAdd(R.fptd + Q * kFptdBins + 4 * e + m, 1ull);
    atomicAdd(R.fptd + kFptdAgeSum + Q, (unsigned long long)age);
}

// Finish the step of a particle that left the chamber (step_particle kept
// its old position X, Y, Z and its pushed velocity): the first crossing of
// the straight segment with the wall, the injection plane or the extraction
// plane, in FP64 from the exact fixed-point coordinates; the extracted / lost
// tallies and the energy carried to the wall; then re-emission (cosine law at
// T0 from the crossing point, or from the inlet after extraction) or, without
// recycling, freezing.  Returns the cell it deposits in (kNoCell if frozen).
__device__ __forceinline__ uint32_t leave_particle(const RunDev& R, uint32_t pid, uint32_t step, int32_t& X,
                                                   int32_t& Y, int32_t& Z, float& vx, float& vy, float& vz,
                                                   uint32_t& meta)
{
    const uint32_t status = meta & 0xFFFF0000u;
    const uint32_t Q = meta & kQMask;
    long long xn, yn, zn;
    displace(R, X, Y, Z, vx, vy, vz, xn, yn, zn);
    bool out_r, out_0, out_L;
    outside(xn, yn, zn, out_r, out_0, out_L);

    const double sxy = R.sxy_d, szd = R.sz_d;
    const double dx0 = (double)X * sxy, dy0 = (double)Y * sxy, dz0 = ((double)Z + 2147483648.0) * szd;
    const double ddx = (double)(xn - X) * sxy, ddy = (double)(yn - Y) * sxy, ddz = (double)(zn - Z) * szd;
    double fbest = 2.0;
    int kind = 0;
    if (out_r) {
        // |p0 + f d|^2 = R0^2 with c = |p0|^2 - R0^2 <= 0, taken exactly in fixed point
        const double a = ddx * ddx + ddy * ddy, b = dx0 * ddx + dy0 * ddy;
        const double c = (double)((long long)X * X + (long long)Y * Y - (1ll << 62)) * sxy * sxy;
        const double disc = sqrt(fmax(0.0, b * b - a * c));
        double f = (b + disc > 0.0) ? -c / (b + disc) : 0.0;
        f = fmax(f, 0.0);
        fbest = f;
        kind = 1;
    }
    if (out_0) {
        const double f = (double)((long long)Z + kLim) / (double)((long long)Z - zn);
        if (f < fbest) { fbest = f; kind = 2; }
    }
    if (out_L) {
        const double f = (double)(kLim - (long long)Z) / (double)(zn - (long long)Z);
        if (f < fbest) { fbest = f; kind = 3; }
    }
    const double cxd = dx0 + fbest * ddx, cyd = dy0 + fbest * ddy, czd = dz0 + fbest * ddz;
    if (kind == 3 && cxd * cxd + cyd * cyd < R.r_ap_d * R.r_ap_d) kind = 4;

    // ---- wall / aperture bookkeeping ----
    if (Q >= 1) atomicAdd(R.tally + kTallyKe, __float2ull_rn(R.ke_scale * (vx * vx + vy * vy + vz * vz)));
    uint32_t ev;
    if (kind == 4) {
        atomicAdd(R.tally + kTallyExtracted + Q, 1ull);
        ev = kEvExtract;
        const uint32_t born = Q >= 1 ? R.birth[pid] : 0xFFFFFFFFu;
        if (born <= step) fptd_record(R, Q, step - born);
        // radius at the aperture plane (mean radial displacement by Q), in nm
        atomicAdd(R.fptd + kFptdRadius + Q, (unsigned long long)rint(sqrt(cxd * cxd + cyd * cyd) * 1e9));
    } else {
        atomicAdd(R.tally + kTallyLost + Q, 1ull);
        ev = kEvWall;
    }
    if (!(R.flags & kFRecycle)) {
        // frozen at its last position, clamped into the fixed-point range
        X = clamp_fx(xn);
        Y = clamp_fx(yn);
        Z = clamp_fx(zn);
        meta = status | kStFrozen | ev;
        return kNoCell;
    }
    const Words u = rng_words(R, pid, step, 2u);
    // an ion neutralised at a wall comes back at T_refl; atoms and the gas
    // reinjected at the inlet at T0
    const float sig = Q >= 1 ? R.sig_refl : R.sig0;
    if (kind == 4) {
        X = R.inlet_X; Y = R.inlet_Y; Z = R.inlet_Z;
        emit(R.sig0, 0.f, 0.f, 1.f, 1.f, 0.f, 0.f, 0.f, 1.f, 0.f, u, vx, vy, vz);
    } else if (kind == 1) {
        const double rc = sqrt(cxd * cxd + cyd * cyd);
        const float ux = (float)(cxd / rc), uy = (float)(cyd / rc);
        const double sc = (R.R0_d - R.eps_wall_d) / rc;
        X = (int32_t)rint(cxd * sc / sxy);
        Y = (int32_t)rint(cyd * sc / sxy);
        Z = (int32_t)(long long)rint(czd / szd - 2147483648.0);
        emit(sig, -ux, -uy, 0.f, -uy, ux, 0.f, 0.f, 0.f, 1.f, u, vx, vy, vz);
    } else if (kind == 2) {
        X = (int32_t)rint(cxd / sxy);
        Y = (int32_t)rint(cyd / sxy);
        Z = (int32_t)(long long)rint(R.eps_wall_d / szd - 2147483648.0);
        emit(sig, 0.f, 0.f, 1.f, 1.f, 0.f, 0.f, 0.f, 1.f, 0.f, u, vx, vy, vz);
    } else {
        X = (int32_t)rint(cxd / sxy);
        Y = (int32_t)rint(cyd / sxy);
        Z = (int32_t)(long long)rint((R.L_d - R.eps_wall_d) / szd - 2147483648.0);
        emit(sig, 0.f, 0.f, -1.f, 1.f, 0.f, 0.f, 0.f, 1.f, 0.f, u, vx, vy, vz);
    }
    meta = status | ev;   // Q = 0: the particle comes back as an atom
    return ngp_cell(R, X, Y, Z);
}

// NGP deposition of one particle per lane (the whole warp calls it), summed
// over runs of neighbouring lanes in the same cell (particles are kept sorted
// by cell, so neighbours mostly are): a segmented inclusive scan of the charge
// over each run's lanes (shuffles that stay inside the run), and the last lane
// of the run adds count << 32 | charge for it.
__device__ __forceinline__ void deposit_warp(const RunDev& R, uint32_t cell, uint32_t Q)
{
    const uint32_t lane = threadIdx.x & 31;
    const uint32_t prev = __shfl_up_sync(0xFFFFFFFFu, cell, 1);
    const uint32_t heads = __ballot_sync(0xFFFFFFFFu, lane == 0 || prev != cell);
    const uint32_t h = 31u - (uint32_t)__clz(heads & (0xFFFFFFFFu >> (31u - lane)));   // first lane of the run
    uint32_t q = Q;
    if (__any_sync(0xFFFFFFFFu, Q != 0u)) {   // a warp of atoms deposits counts only
#pragma unroll
        for (uint32_t d = 1; d < 32u; d <<= 1) {
            const uint32_t o = __shfl_up_sync(0xFFFFFFFFu, q, d);
            if (lane >= h + d) q += o;   // lane - d lies in the same run
        }
    }
    const bool last = lane == 31u || ((heads >> (lane + 1u)) & 1u);
    if (last && cell != kNoCell)
        atomicAdd(R.dep + cell, ((unsigned long long)(lane - h + 1u) << 32) | (unsigned long long)q);
}

// ---------------------------------------------------------------------------
// Windows of steps.  A call's steps run in windows of up to kMaxWindow: an
// atom's step depends on no other particle, and without collisions between
// ions neither does an ion's, so their state is read once, stepped through the
// window in registers and written once.
//
// k_quiet takes the atoms.  An atom moves on a straight line by the same whole
// number of grid units every step, so its place after the window is one
// multiply away; it stays in the chamber throughout if it is inside at the
// window's start and end (the chamber is convex, and the box and r <= R0 tests
// are exact in the integers).  A load tests r <= R0 in FP32 and lets an atom
// in up to some hundred grid units outside, so the start is tested, too.  What is left of its steps is the ionisation word: one Philox
// block a step, of which the first two rounds hardly depend on both the
// particle and the step (see QuietAtom), compared with the atom gate.  An atom
// that neither leaves nor ionises in the window is done: moved, its deposits
// added, its events cleared.  All other particles (ions, and atoms with an
// event to come) are listed by slot.
//
// k_active takes the listed particles through step_particle and, for those
// that leave the chamber, leave_particle, step by step.  Ions are listed from
// the front of the list and atoms from its back, so that a warp has one kind.
//
// With collisions between ions the listed particles take one step at a time
// (k_ions), which also records the ions for the collision kernel; the list
// holds for the window.  A window of one step takes all particles in place
// (k_one).
//
// Against a step kernel and a leaver pass a step, which read and wrote every
// particle each time and were bound by instruction issue: 32 steps of the 32
// oxygen runs of a gas-flow scan (2.6e7 particles, dt 1 ns) took 11.8 ms and
// take 4.3 (k_quiet 1.6, k_active 2.7); 1000 steps of 1e4 particles, bound by
// the latency of two launches a step, 9.1 ms and 1.6.
// ---------------------------------------------------------------------------

// The part of an atom's Philox blocks in a window that does not depend on the
// step, and a step's part that does not depend on the particle.  With the
// counter (pid, 0, c, 0), c = 4 step, the first round leaves (hi(M1 c) ^ k0,
// lo(M1 c), hi(M0 pid) ^ k1, lo(M0 pid)): two words of the step and two of
// the particle.  The second multiplies word 0 (the step's) and word 2 (the
// particle's), so its products need no particle-and-step multiply either.
struct QuietAtom { uint32_t p0, p1, p2; };

__device__ __forceinline__ QuietAtom quiet_atom(const RunDev& R, uint32_t pid)
{
    const uint32_t a = __umulhi(0xD2511F53u, pid) ^ R.seed_hi, b = 0xD2511F53u * pid;
    return QuietAtom{__umulhi(0xCD9E8D57u, a), 0xCD9E8D57u * a, b};
}

// a step's words after two rounds: to be xored into words 0 and 2, and word 3
__device__ __forceinline__ uint4 quiet_step(const RunDev& R, uint32_t step)
{
    const uint32_t c = 4u * step;
    const uint32_t u0 = __umulhi(0xCD9E8D57u, c) ^ R.seed_lo, lo1 = 0xCD9E8D57u * c;
    return make_uint4(lo1 ^ (R.seed_lo + 0x9E3779B9u), __umulhi(0xD2511F53u, u0) ^ (R.seed_hi + 0xBB67AE85u),
                      0xD2511F53u * u0, 0u);
}

// The round keys of rounds 3 to 10.  The empty asm keeps them in registers: left
// to itself the compiler forms each one anew from the run's key wherever it is
// used, one instruction in three of the words' arithmetic.
struct QuietKeys { uint32_t a[8], b[8]; };

__device__ __forceinline__ QuietKeys quiet_keys(const RunDev& R)
{
    QuietKeys k;
#pragma unroll
    for (int r = 0; r < 8; ++r) {
        k.a[r] = R.seed_lo + (uint32_t)(r + 2) * 0x9E3779B9u;
        k.b[r] = R.seed_hi + (uint32_t)(r + 2) * 0xBB67AE85u;
        asm("" : "+r"(k.a[r]), "+r"(k.b[r]));
    }
    return k;
}

// word 0 of the block: rounds 3 to 10
__device__ __forceinline__ uint32_t quiet_word0(const QuietKeys& k, const QuietAtom& a, const uint4& st)
{
    uint32_t c0 = a.p0 ^ st.x, c1 = a.p1, c2 = a.p2 ^ st.y, c3 = st.z;
#pragma unroll
    for (int r = 0; r < 8; ++r) {
        const unsigned long long p0 = (unsigned long long)0xD2511F53u * c0;
        const unsigned long long p1 = (unsigned long long)0xCD9E8D57u * c2;
        const uint32_t n0 = (uint32_t)(p1 >> 32) ^ c1 ^ k.a[r];
        const uint32_t n2 = (uint32_t)(p0 >> 32) ^ c3 ^ k.b[r];
        c0 = n0; c1 = (uint32_t)p1; c2 = n2; c3 = (uint32_t)p0;
    }
    return c0;
}

// What a warp of the quiet pass puts by: slots for the run's lists (written 128
// at a time, one atomic each: many warps adding to one word queue for it), and
// atoms whose steps must be looked at one by one (taken 32 at a time)
constexpr uint32_t kQuietFlush = 128;
struct QuietWarp {
    uint32_t slots[2][kQuietFlush + 32];   // ions, atoms
    uint32_t detail[64];                   // slot << 1 | hit
};
struct QuietSteps { uint4 rng[kMaxWindow]; };   // quiet_step of the window's steps
struct QuietCount { uint32_t n[2], detail; };   // of the warp's three lists

__device__ __forceinline__ void atom_words(const RunDev& R, uint32_t i, int32_t& X, int32_t& Y, int32_t& Z,
                                           uint32_t& id, float3& v)
{
    X = R.x[i]; Y = R.y[i]; Z = R.z[i];
    id = R.id[i];
    v = make_float3(R.vx[i], R.vy[i], R.vz[i]);
}

// An atom's straight way through the window: its displacement a step and its
// end; false if it may leave the chamber within the window (it ends outside, or
// starts outside the cylinder) or moves too far in it for 32-bit arithmetic
struct Way { int32_t DX, DY, DZ, XE, YE, ZE; };

__device__ __forceinline__ bool quiet_way(const RunDev& R, const float3& v, int32_t X, int32_t Y, int32_t Z,
                                          uint32_t K, Way& w)
{
    const bool push = (R.flags & kFPush) != 0;
    const float dx = push ? v.x * R.dt_sxy : 0.0f, dy = push ? v.y * R.dt_sxy : 0.0f, dz = push ? v.z * R.dt_sz : 0.0f;
    if (!(fmaxf(fabsf(dx), fmaxf(fabsf(dy), fabsf(dz))) * (float)K < 1.0e9f)) return false;
    if (K > 1u && (long long)X * X + (long long)Y * Y > (1ll << 62)) return false;
    w.DX = __float2int_rn(dx);
    w.DY = __float2int_rn(dy);
    w.DZ = __float2int_rn(dz);
    bool ox, oy, oz;
    w.XE = add_wrap(X, (int32_t)K * w.DX, ox);
    w.YE = add_wrap(Y, (int32_t)K * w.DY, oy);
    w.ZE = add_wrap(Z, (int32_t)K * w.DZ, oz);
    return !(ox | oy | oz || (long long)w.XE * w.XE + (long long)w.YE * w.YE > (1ll << 62));
}

// Deposit of the whole warp's particles: each lane `count` visits and `charge`
// in all to `cell` (kNoCell: none), one reduction per run of neighbouring lanes
// in the same cell
__device__ __forceinline__ void deposit_sums(const RunDev& R, uint32_t cell, uint32_t count, uint32_t charge)
{
    const uint32_t lane = threadIdx.x & 31;
    const uint32_t prev = __shfl_up_sync(0xFFFFFFFFu, cell, 1);
    const uint32_t heads = __ballot_sync(0xFFFFFFFFu, lane == 0 || prev != cell);
    const uint32_t h = 31u - (uint32_t)__clz(heads & (0xFFFFFFFFu >> (31u - lane)));   // first lane of the run
    uint32_t n = count, q = charge;
    const uint32_t any_q = __any_sync(0xFFFFFFFFu, charge != 0u);
#pragma unroll
    for (uint32_t d = 1; d < 32u; d <<= 1) {
        const uint32_t on = __shfl_up_sync(0xFFFFFFFFu, n, d);
        const bool in = lane >= h + d;   // lane - d lies in the same run
        if (in) n += on;
        if (any_q) {
            const uint32_t oq = __shfl_up_sync(0xFFFFFFFFu, q, d);
            if (in) q += oq;
        }
    }
    const bool last = lane == 31u || ((heads >> (lane + 1u)) & 1u);
    if (last && cell != kNoCell) atomicAdd(R.dep + cell, ((unsigned long long)n << 32) | (unsigned long long)q);
}

// write the first m of the warp's listed slots (which: 0 ions, 1 atoms) to the
// run's list
__device__ __forceinline__ void quiet_flush(const RunDev& R, QuietWarp& W, uint32_t which, uint32_t m)
{
    const uint32_t lane = threadIdx.x & 31;
    uint32_t base = 0u;
    if (lane == 0) base = atomicAdd(R.nleave + which, m);
    base = __shfl_sync(0xFFFFFFFFu, base, 0);
    for (uint32_t k = lane; k < m; k += 32u)
        R.leave[which ? 4u * R.n4 - 1u - (base + k) : base + k] = W.slots[which][k];
}

// list the lanes' slots
__device__ __forceinline__ void quiet_list(const RunDev& R, QuietWarp& W, QuietCount& n, uint32_t which, bool listed,
                                           uint32_t slot)
{
    const uint32_t m = __ballot_sync(0xFFFFFFFFu, listed);
    if (!m) return;
    const uint32_t lane = threadIdx.x & 31;
    if (listed) W.slots[which][n.n[which] + (uint32_t)__popc(m & ((1u << lane) - 1u))] = slot;
    n.n[which] += (uint32_t)__popc(m);
    __syncwarp();
    if (n.n[which] < kQuietFlush) return;
    quiet_flush(R, W, which, kQuietFlush);
    n.n[which] -= kQuietFlush;
    const uint32_t rest = W.slots[which][kQuietFlush + lane];
    __syncwarp();
    W.slots[which][lane] = rest;
    __syncwarp();
}

// An atom that crosses cells in the window, or one of whose words lies below
// the atom gate (hit): true if it ionises in one of its steps (the decision of
// step_particle in the cell it is in then); else its deposits are added
__device__ __forceinline__ bool quiet_detail(const RunDev& R, const QuietSteps& S, uint32_t id, uint32_t K, int32_t X,
                                             int32_t Y, int32_t Z, const Way& w, bool hit)
{
    if (hit) {
        const QuietAtom a = quiet_atom(R, id);
        for (uint32_t s = 0; s < K; ++s) {
            const uint32_t w0 = quiet_word0(quiet_keys(R), a, S.rng[s]);
            if (!atom_may_ionize(R, w0)) continue;
            const int32_t n = (int32_t)s + 1;
            const float4 cr = __ldg(R.cell + ngp_cell(R, X + n * w.DX, Y + n * w.DY, Z + n * w.DZ));
            const int zone = cr.y > 0.5f ? 1 : 0;
            if (fires(w0, event_prob(cr.x * __ldg(R.kdt + zone * kQSlots)))) return true;
        }
    }
    uint32_t at = kNoCell, n = 0u;
    for (uint32_t s = 0; s < K; ++s) {
        X += w.DX;
        Y += w.DY;
        Z += w.DZ;
        const uint32_t c = ngp_cell(R, X, Y, Z);
        if (c != at) {
            if (n) atomicAdd(R.dep + at, (unsigned long long)n << 32);
            at = c;
            n = 0u;
        }
        ++n;
    }
    atomicAdd(R.dep + at, (unsigned long long)n << 32);
    return false;
}

// the first m (<= 32) atoms that were put by
__device__ __forceinline__ void quiet_details(const RunDev& R, const QuietSteps& S, QuietWarp& W, QuietCount& n,
                                              uint32_t m, uint32_t K)
{
    const uint32_t lane = threadIdx.x & 31;
    bool listed = false;
    uint32_t i = 0u;
    if (lane < m) {
        const uint32_t d = W.detail[lane];
        i = d >> 1;
        int32_t X, Y, Z;
        uint32_t id;
        float3 v;
        atom_words(R, i, X, Y, Z, id, v);
        Way w;
        quiet_way(R, v, X, Y, Z, K, w);
        listed = quiet_detail(R, S, id, K, X, Y, Z, w, d & 1u);
        if (!listed) {
            R.x[i] = w.XE;
            R.y[i] = w.YE;
            R.z[i] = w.ZE;
            const uint32_t meta = R.meta[i];
            if (meta & 0xFFFFu) R.meta[i] = meta & 0xFFFF0000u;   // its events are over
        }
    }
    quiet_list(R, W, n, 1u, listed, i);
    n.detail -= m;
    const uint32_t rest = lane < n.detail ? W.detail[m + lane] : 0u;
    __syncwarp();
    W.detail[lane] = rest;
    __syncwarp();
}

// Deposit of the whole warp's atoms: each lane K visits to `cell` (kNoCell: none)
__device__ __forceinline__ void deposit_atoms(const RunDev& R, uint32_t cell, uint32_t K)
{
    const uint32_t lane = threadIdx.x & 31;
    const uint32_t prev = __shfl_up_sync(0xFFFFFFFFu, cell, 1);
    const uint32_t heads = __ballot_sync(0xFFFFFFFFu, lane == 0 || prev != cell);
    const bool last = lane == 31u || ((heads >> (lane + 1u)) & 1u);
    const uint32_t h = 31u - (uint32_t)__clz(heads & (0xFFFFFFFFu >> (31u - lane)));   // first lane of the run
    if (last && cell != kNoCell) atomicAdd(R.dep + cell, (unsigned long long)((lane - h + 1u) * K) << 32);
}

// 32 particles from slot i0 by a warp.  The few atoms that need their steps
// looked at one by one are put by and taken 32 at a time: in place they would
// keep whole warps waiting (at dt 1 ns, 3 % of the atoms were on two thirds of
// the warps).
__device__ __forceinline__ void quiet_group(const RunDev& R, const QuietSteps& S, QuietWarp& W, QuietCount& n,
                                            uint32_t i0, uint32_t K)
{
    const uint32_t lane = threadIdx.x & 31, i = i0 + lane, nslot = 4u * R.n4;
    const uint32_t meta = i < nslot ? R.meta[i] : kStPad;
    int32_t X = 0, Y = 0, Z = 0;
    uint32_t id = 0u;
    float3 v = make_float3(0.f, 0.f, 0.f);
    const uint32_t status = meta & 0xFFFF0000u, Q = meta & kQMask;
    const bool live = !(status & (kStFrozen | kStPad));
    bool listed = false, detail = false, hit = false;
    uint32_t dep_cell = kNoCell;
    if (live && Q == 0u) {
        atom_words(R, i, X, Y, Z, id, v);
        Way w;
        listed = !quiet_way(R, v, X, Y, Z, K, w);
        if (!listed && (R.flags & kFIonize)) {
            const QuietAtom a = quiet_atom(R, id);
            const QuietKeys key = quiet_keys(R);
            uint32_t lo = 0xFFFFFFFFu, s = 0;
            for (; s + 4u <= K; s += 4u)   // four steps' blocks side by side
                lo = min(lo, min(min(quiet_word0(key, a, S.rng[s]), quiet_word0(key, a, S.rng[s + 1u])),
                                 min(quiet_word0(key, a, S.rng[s + 2u]), quiet_word0(key, a, S.rng[s + 3u]))));
            for (; s < K; ++s) lo = min(lo, quiet_word0(key, a, S.rng[s]));
            hit = atom_may_ionize(R, lo);
        }
        if (!listed) {
            // the cells it visits: the same one throughout if the first and
            // the last step share it (each coordinate is monotone)
            dep_cell = ngp_cell(R, w.XE, w.YE, w.ZE);
            detail = hit || ngp_cell(R, X + w.DX, Y + w.DY, Z + w.DZ) != dep_cell;
            if (detail) {
                dep_cell = kNoCell;
            } else {
                R.x[i] = w.XE;
                R.y[i] = w.YE;
                R.z[i] = w.ZE;
            }
        }
    }
    const bool ion = live && Q > 0u;
    if (!listed && !detail && !ion && i < nslot && meta != (status | Q)) R.meta[i] = status | Q;   // its events are over
    // the deposits of the atoms that kept their cell
    if (__any_sync(0xFFFFFFFFu, dep_cell != kNoCell)) deposit_atoms(R, dep_cell, K);
    quiet_list(R, W, n, 0u, ion, i);
    quiet_list(R, W, n, 1u, listed, i);
    const uint32_t md = __ballot_sync(0xFFFFFFFFu, detail);
    if (!md) return;
    if (detail) W.detail[n.detail + (uint32_t)__popc(md & ((1u << lane) - 1u))] = i << 1 | (hit ? 1u : 0u);
    n.detail += (uint32_t)__popc(md);
    __syncwarp();
    if (n.detail >= 32u) quiet_details(R, S, W, n, 32u, K);
}

// what the warp still holds
__device__ __forceinline__ void quiet_end(const RunDev& R, const QuietSteps& S, QuietWarp& W, QuietCount& n,
                                          uint32_t K)
{
    if (n.detail) quiet_details(R, S, W, n, n.detail, K);
    for (uint32_t which = 0; which < 2u; ++which) {
        if (n.n[which]) quiet_flush(R, W, which, n.n[which]);
        n.n[which] = 0u;
    }
    __syncwarp();
}

// the window's steps (all threads of the block call it, after *R.step is final)
__device__ __forceinline__ void quiet_start(const RunDev& R, QuietSteps& S, uint32_t K)
{
    if (threadIdx.x < K) S.rng[threadIdx.x] = quiet_step(R, *R.step + threadIdx.x);
    __syncthreads();
}

// groups: 32-particle groups a warp takes in a row (they stay together in the
// list).  Fewer resident blocks with four steps' words side by side did better
// than more with two: 240 us a 32-step window of 3e6 atoms with 6 blocks and
// four, 257 and 261 with 10 or 8 and two.
constexpr int kQuietBlocks = 6;
__global__ void __launch_bounds__(128, kQuietBlocks) k_quiet(const __grid_constant__ RunDev R, uint32_t K,
                                                                          uint32_t groups)
{
    __shared__ QuietSteps S;
    __shared__ QuietWarp warps[4];
    pdl_wait();
    pdl_trigger();
    quiet_start(R, S, K);
    if (blockIdx.x == 0 && threadIdx.x == 0) R.nleave[2] = K;
    QuietWarp& W = warps[threadIdx.x >> 5];
    QuietCount n{{0u, 0u}, 0u};
    const uint32_t nslot = 4u * R.n4, run = 32u * groups, nw = gridDim.x * 4u;
    for (uint32_t g = blockIdx.x * 4u + (threadIdx.x >> 5); g * run < nslot; g += nw)
#pragma unroll 1
        for (uint32_t k = 0; k < run; k += 32u) quiet_group(R, S, W, n, g * run + k, K);
    quiet_end(R, S, W, n, K);
}

// entries of a run's list: its ions, padded to whole warps, then its atoms
__device__ __forceinline__ uint32_t list_entries(uint32_t ni, uint32_t na) { return ((ni + 31u) & ~31u) + na; }

// Entries a warp takes (log2): 32, or fewer if the run's list is so short that
// the grid has warps to spare.  The lanes of a warp of atoms leave the chamber in
// different steps, and each one that does takes the whole warp through its FP64
// geometry (k_active, 1e4 particles x 32 steps: 33 us with 32 a warp, 30 so).
// Not in k_ions: in one step few do, and more warps add to the deposit and the
// buckets more often (2e4 and 2e5 particles 2 and 4 % slower).
__device__ __forceinline__ uint32_t list_lanes(uint32_t entries)
{
    uint32_t lw = 5u;
    while (lw > 0u && (entries >> (lw - 1u)) <= gridDim.x * (blockDim.x >> 5)) --lw;
    return lw;
}

// tiles of a run's list
__device__ __forceinline__ uint32_t list_tiles(uint32_t entries, uint32_t lw)
{
    const uint32_t warps = (entries + (1u << lw) - 1u) >> lw, per = blockDim.x >> 5;
    return (warps + per - 1u) / per;
}

// this lane's entry of tile t (none: past every list)
__device__ __forceinline__ uint32_t list_entry(uint32_t t, uint32_t lw)
{
    const uint32_t lane = threadIdx.x & 31u, w = t * (blockDim.x >> 5) + (threadIdx.x >> 5);
    return lane >> lw ? 0xFFFFFFFFu : (w << lw) + lane;
}

// every run of a batch; the last block works out where each run's tiles of
// listed particles start in the passes over them: pref[r] for the runs without
// collisions between ions (k_active_batch), pref[nruns + 1 + r] for those with
// (k_ions_batch), nruns + 1 entries each
__global__ void __launch_bounds__(256, 4) k_quiet_batch(const RunDev* __restrict__ runs,
                                                                   const uint2* __restrict__ items, uint32_t nitems,
                                                                   uint32_t tile, uint32_t K, uint32_t nruns,
                                                                   uint32_t* __restrict__ pref, unsigned int* ticket)
{
    __shared__ QuietSteps S;
    extern __shared__ QuietWarp warps[];
    __shared__ RunDev rs;
    __shared__ uint2 s_sum[256];
    pdl_wait();
    pdl_trigger();
    QuietWarp& W = warps[threadIdx.x >> 5];
    QuietCount n{{0u, 0u}, 0u};
    uint32_t cur = 0xFFFFFFFFu;
    for (uint32_t i = blockIdx.x; i < nitems; i += gridDim.x) {
        const uint2 it = items[i];
        if (it.x != cur) {
            if (cur != 0xFFFFFFFFu) quiet_end(rs, S, W, n, K);
            __syncthreads();
            cur = it.x;
            stage_run(rs, runs + cur);
            __syncthreads();
            quiet_start(rs, S, K);
        }
        // the tile's particles, a stretch of them a warp
        const uint32_t per = tile / (blockDim.x >> 5), i0 = it.y * tile + (threadIdx.x >> 5) * per;
#pragma unroll 1
        for (uint32_t k = 0; k < per; k += 32u) quiet_group(rs, S, W, n, i0 + k, K);
    }
    if (cur != 0xFFFFFFFFu) quiet_end(rs, S, W, n, K);
    if (!last_block(ticket)) return;
    const uint32_t tid = threadIdx.x, T = blockDim.x;
    uint2 carry = make_uint2(0u, 0u);
    for (uint32_t r0 = 0; r0 < nruns; r0 += T) {
        const uint32_t r = r0 + tid;
        uint2 v = make_uint2(0u, 0u);
        if (r < nruns && runs[r].step) {
            volatile uint32_t* nl = runs[r].nleave;
            const uint32_t nt = (list_entries(nl[0], nl[1]) + T - 1u) / T;
            if (runs[r].flags & kFCoulomb) v.y = nt;
            else v.x = nt;
            nl[2] = K;
        }
        s_sum[tid] = v;
        __syncthreads();
        for (uint32_t d = 1; d < T; d <<= 1) {
            const uint2 o = tid >= d ? s_sum[tid - d] : make_uint2(0u, 0u);
            __syncthreads();
            s_sum[tid].x += o.x;
            s_sum[tid].y += o.y;
            __syncthreads();
        }
        if (r < nruns) {
            pref[r] = carry.x + s_sum[tid].x - v.x;
            pref[nruns + 1u + r] = carry.y + s_sum[tid].y - v.y;
        }
        carry.x += s_sum[T - 1u].x;
        carry.y += s_sum[T - 1u].y;
        __syncthreads();
    }
    if (tid == 0) {
        pref[nruns] = carry.x;
        pref[2u * nruns + 1u] = carry.y;
    }
}

// a particle that left the chamber, out of line: its FP64 geometry's registers
// are not the step's
struct Left {
    int32_t X, Y, Z;
    float vx, vy, vz;
    uint32_t meta, cell;
};

__device__ __noinline__ Left leave_call(const RunDev& R, uint32_t pid, uint32_t step, int32_t X, int32_t Y, int32_t Z,
                                        float vx, float vy, float vz, uint32_t meta)
{
    Left l{X, Y, Z, vx, vy, vz, meta, kNoCell};
    l.cell = leave_particle(R, pid, step, l.X, l.Y, l.Z, l.vx, l.vy, l.vz, l.meta);
    return l;
}

// One tile of k_active: entries [t T, (t + 1) T) of the run's list, one a thread
// of the block of T, K steps each
template <bool kVar, bool kPlain>
__device__ __forceinline__ void active_tile(const RunDev& R, uint32_t t, uint32_t K, uint32_t ni, uint32_t na,
                                            uint32_t lw = 5u)
{
    const uint32_t step0 = *R.step, ni32 = (ni + 31u) & ~31u, nslot = 4u * R.n4;
    const uint32_t e = list_entry(t, lw);
    const bool in = e < ni || (e >= ni32 && e - ni32 < na);
    if (!__any_sync(0xFFFFFFFFu, in)) return;
    uint32_t i = 0u, id = 0u, meta = kStPad;
    int32_t x = 0, y = 0, z = 0;
    float vx = 0.0f, vy = 0.0f, vz = 0.0f;
    if (in) {
        i = R.leave[e < ni ? e : nslot - 1u - (e - ni32)];
        meta = R.meta[i];
        id = R.id[i];
        x = R.x[i]; y = R.y[i]; z = R.z[i];
        vx = R.vx[i]; vy = R.vy[i]; vz = R.vz[i];
    }
    // deposits: summed while the particle stays in a cell
    uint32_t at = kNoCell, n = 0u, q = 0u;
    Carry carry;
#pragma unroll 1
    for (uint32_t s = 0; s < K; ++s) {
        uint32_t ck, dc;
        if (step_particle<kVar, true, kPlain>(R, id, step0 + s, x, y, z, vx, vy, vz, meta, ck, dc, carry)) {
            const Left l = leave_call(R, id, step0 + s, x, y, z, vx, vy, vz, meta);
            x = l.X; y = l.Y; z = l.Z;
            vx = l.vx; vy = l.vy; vz = l.vz;
            meta = l.meta;
            dc = l.cell;   // (as an atom: no charge)
        }
        if (dc != at) {
            if (n) atomicAdd(R.dep + at, ((unsigned long long)n << 32) | (unsigned long long)q);
            at = dc;
            n = q = 0u;
        }
        if (dc != kNoCell) {
            ++n;
            q += meta & kQMask;
        }
    }
    deposit_sums(R, at, n, q);
    if (in) {
        R.x[i] = x; R.y[i] = y; R.z[i] = z;
        R.vx[i] = vx; R.vy[i] = vy; R.vz[i] = vz;
        R.meta[i] = meta;
    }
}

// Resident blocks an SM that the passes over the lists are compiled for.  They
// wait on gathers and long chains, so more warps hide more, until the spilled
// registers cost more than that gives.  Times with 3/4/5 blocks of 256 threads
// (or twice as many of 128), in us: k_ions, 1.0e6 ions 32.2/30.0/30.9; k_active,
// 1e4 particles x 32 steps 32.5/34.9/38.1, with variants 1e6 x 32 284/260/273;
// k_active_batch, 7e6 ions x 32 2711/2744/2864; k_ions_batch, 4.2e6 ions
// 167/145/135.
constexpr int kListBlocks = 8;   // the most, of kActiveTile threads
constexpr int kActiveBatchBlocks = 3, kIonsBatchBlocks = 5;   // of 256

// the last block clears the lists and advances the step counter
template <bool kVar>
__global__ void __launch_bounds__(kActiveTile, kVar ? 8 : 6) k_active(const __grid_constant__ RunDev R, uint32_t K,
                                                                      unsigned int* ticket)
{
    pdl_wait();
    pdl_trigger();
    const uint32_t ni = R.nleave[0], na = R.nleave[1];
    const uint32_t lw = list_lanes(list_entries(ni, na)), nt = list_tiles(list_entries(ni, na), lw);
    const bool plain = !kVar && plain_run(R);
    for (uint32_t t = blockIdx.x; t < nt; t += gridDim.x) {
        if (!kVar && plain) active_tile<false, true>(R, t, K, ni, na, lw);
        else active_tile<kVar, false>(R, t, K, ni, na, lw);
    }
    if (last_block(ticket) && threadIdx.x == 0) {
        R.nleave[0] = 0u;
        R.nleave[1] = 0u;
        *R.step += K;
    }
}

// the run whose listed tiles hold tile v of a batch pass, and v less the run's
// first tile: staged in rs, with *s_at = (run, first tile) (all threads call it)
__device__ __forceinline__ uint32_t batch_tile(const RunDev* __restrict__ runs, uint32_t nruns,
                                               const uint32_t* pref, uint32_t v, RunDev& rs, uint2& s_at,
                                               uint32_t& cur)
{
    for (uint32_t r = threadIdx.x; r < nruns; r += blockDim.x) {
        const uint32_t lo = pref[r];
        if (lo <= v && v < pref[r + 1]) s_at = make_uint2(r, lo);
    }
    __syncthreads();
    const uint2 at = s_at;
    if (at.x != cur) {
        cur = at.x;
        stage_run(rs, runs + cur);
    }
    __syncthreads();
    return v - at.y;
}

template <bool kVar>
__global__ void __launch_bounds__(256, kActiveBatchBlocks) k_active_batch(const RunDev* __restrict__ runs, uint32_t nruns,
                                                         const uint32_t* pref, uint32_t K,
                                                         unsigned int* ticket)
{
    __shared__ RunDev rs;
    __shared__ uint2 s_at;
    pdl_wait();
    pdl_trigger();
    const uint32_t nt = pref[nruns];
    uint32_t cur = 0xFFFFFFFFu;
    for (uint32_t v = blockIdx.x; v < nt; v += gridDim.x) {
        const uint32_t t = batch_tile(runs, nruns, pref, v, rs, s_at, cur);
        if (!kVar && plain_run(rs)) active_tile<false, true>(rs, t, K, rs.nleave[0], rs.nleave[1]);
        else active_tile<kVar, false>(rs, t, K, rs.nleave[0], rs.nleave[1]);
        __syncthreads();
    }
    if (last_block(ticket))
        for (uint32_t r = threadIdx.x; r < nruns; r += blockDim.x)
            if (runs[r].step && !(runs[r].flags & kFCoulomb)) {
                runs[r].nleave[0] = 0u;
                runs[r].nleave[1] = 0u;
                *runs[r].step += K;
            }
}

// One step of a tile of listed particles of a run with collisions between
// ions; the ions that stay are recorded in their cells' buckets
template <bool kVar, bool kPlain>
__device__ __forceinline__ void ions_tile(const RunDev& R, uint32_t t, uint32_t ni, uint32_t na)
{
    const uint32_t step = *R.step, ni32 = (ni + 31u) & ~31u, nslot = 4u * R.n4;
    const uint32_t e = t * blockDim.x + threadIdx.x;
    const bool in = e < ni || (e >= ni32 && e - ni32 < na);
    if (!__any_sync(0xFFFFFFFFu, in)) return;
    uint32_t i = 0u, id = 0u, meta = kStPad;
    int32_t x = 0, y = 0, z = 0;
    float vx = 0.0f, vy = 0.0f, vz = 0.0f;
    if (in) {
        i = R.leave[e < ni ? e : nslot - 1u - (e - ni32)];
        meta = R.meta[i];
        id = R.id[i];
        x = R.x[i]; y = R.y[i]; z = R.z[i];
        vx = R.vx[i]; vy = R.vy[i]; vz = R.vz[i];
    }
    uint32_t ck, dc;
    Carry carry;
    if (step_particle<kVar, false, kPlain>(R, id, step, x, y, z, vx, vy, vz, meta, ck, dc, carry)) {
        const Left l = leave_call(R, id, step, x, y, z, vx, vy, vz, meta);
        x = l.X; y = l.Y; z = l.Z;
        vx = l.vx; vy = l.vy; vz = l.vz;
        meta = l.meta;
        dc = l.cell;   // (as an atom: no charge)
    }
    if (in) {
        R.x[i] = x; R.y[i] = y; R.z[i] = z;
        R.vx[i] = vx; R.vy[i] = vy; R.vz[i] = vz;
        R.meta[i] = meta;
    }
    deposit_warp(R, dc, meta & kQMask);
    place_warp(R, i, ck, id, step, vx, vy, vz, meta);
}

// what the collision kernel of the step finds set (by one thread)
__device__ __forceinline__ void begin_collisions(const RunDev& R)
{
    R.cword[kCwSet] = *R.step & 1u;
    R.cword[kCwHuge] = 0u;
    R.cword[kCwBig] = 0u;
    R.cword[kCwPast] = 0u;
}

template <bool kVar>
__global__ void __launch_bounds__(kActiveTile, 8) k_ions(const __grid_constant__ RunDev R)
{
    pdl_wait();
    pdl_trigger();
    if (blockIdx.x == 0 && threadIdx.x == 0) begin_collisions(R);
    const uint32_t ni = R.nleave[0], na = R.nleave[1];
    const uint32_t nt = (list_entries(ni, na) + blockDim.x - 1u) / blockDim.x;
    const bool plain = !kVar && plain_run(R);
    for (uint32_t t = blockIdx.x; t < nt; t += gridDim.x) {
        if (!kVar && plain) ions_tile<false, true>(R, t, ni, na);
        else ions_tile<kVar, false>(R, t, ni, na);
    }
}

template <bool kVar>
__global__ void __launch_bounds__(256, kIonsBatchBlocks) k_ions_batch(const RunDev* __restrict__ runs, uint32_t nruns,
                                                       const uint32_t* pref)
{
    __shared__ RunDev rs;
    __shared__ uint2 s_at;
    pdl_wait();
    pdl_trigger();
    if (blockIdx.x == 0)
        for (uint32_t r = threadIdx.x; r < nruns; r += blockDim.x)
            if (runs[r].step && runs[r].cword) begin_collisions(runs[r]);
    const uint32_t nt = pref[nruns];
    uint32_t cur = 0xFFFFFFFFu;
    for (uint32_t v = blockIdx.x; v < nt; v += gridDim.x) {
        const uint32_t t = batch_tile(runs, nruns, pref, v, rs, s_at, cur);
        if (!kVar && plain_run(rs)) ions_tile<false, true>(rs, t, rs.nleave[0], rs.nleave[1]);
        else ions_tile<kVar, false>(rs, t, rs.nleave[0], rs.nleave[1]);
        __syncthreads();
    }
}

// A window of one step (a call of one step, a timed one, the step up to a sort):
// every particle in its place, in one pass over the arrays.  Listing the ions
// and the atoms with an event to come, and gathering them again, costs more
// than it saves here (4e6 particles with collisions, cold caches: k_quiet and
// k_ions 100 us, this 78; 4.8e7 without: k_quiet and k_active 1030 us, this 712,
// with four blocks of 256 threads an SM instead of five 741).
template <bool kVar, bool kPlain>
__device__ __forceinline__ void one_group(const RunDev& R, uint32_t i, uint32_t step)
{
    const bool in = i < 4u * R.n4;
    uint32_t id = 0u, meta = kStPad;
    int32_t x = 0, y = 0, z = 0;
    float vx = 0.0f, vy = 0.0f, vz = 0.0f;
    if (in) {
        meta = R.meta[i];
        id = R.id[i];
        x = R.x[i]; y = R.y[i]; z = R.z[i];
        vx = R.vx[i]; vy = R.vy[i]; vz = R.vz[i];
    }
    const uint32_t was = meta;
    uint32_t ck = kNoCell, dc = kNoCell;
    bool left = false;
    // nearly all atoms: those that neither leave nor can ionise, as in the quiet
    // pass.  In a mixed warp they would wait for the ions all the same (4e6
    // particles in load order 2 % slower from 24 atoms a warp on, the same from 29
    // on; sorted 3 % faster with either).
    bool quick = false;
    if (__popc(__ballot_sync(0xFFFFFFFFu, (was & kQMask) == 0u)) >= 29 && !(was & (kStFrozen | kStPad | kQMask))) {
        Way w;
        quick = quiet_way(R, make_float3(vx, vy, vz), x, y, z, 1u, w);
        if (quick && (R.flags & kFIonize))
            quick = !atom_may_ionize(R, quiet_word0(quiet_keys(R), quiet_atom(R, id), quiet_step(R, step)));
        if (quick) {
            x = w.XE; y = w.YE; z = w.ZE;
            meta = was & 0xFFFF0000u;   // its events are over
            dc = ngp_cell(R, x, y, z);
        }
    }
    // a warp of such atoms is done here, past no test of the others (32 runs of 2.5e7
    // particles in a batch 402 us a step, 385 so)
    if (__all_sync(0xFFFFFFFFu, quick)) {
        R.x[i] = x; R.y[i] = y; R.z[i] = z;
        if (meta != was) R.meta[i] = meta;
        deposit_atoms(R, dc, 1u);
        return;
    }
    if (!quick) {
        Carry carry;
        left = step_particle<kVar, false, kPlain>(R, id, step, x, y, z, vx, vy, vz, meta, ck, dc, carry);
    }
    if (left) {
        const Left l = leave_call(R, id, step, x, y, z, vx, vy, vz, meta);
        x = l.X; y = l.Y; z = l.Z;
        vx = l.vx; vy = l.vy; vz = l.vz;
        meta = l.meta;
        dc = l.cell;   // (as an atom: no charge)
    }
    if (in) {
        if (!(was & (kStFrozen | kStPad))) {
            R.x[i] = x; R.y[i] = y; R.z[i] = z;
            if (((was | meta) & kQMask) || left) {   // (an atom keeps its velocity)
                R.vx[i] = vx; R.vy[i] = vy; R.vz[i] = vz;
            }
        }
        if (meta != was) R.meta[i] = meta;
    }
    deposit_warp(R, dc, meta & kQMask);
    if (R.flags & kFCoulomb) place_warp(R, i, ck, id, step, vx, vy, vz, meta);
}

// what the collision kernel of a window of one step finds set (by one thread)
__device__ __forceinline__ void begin_one(const RunDev& R)
{
    begin_collisions(R);
    R.nleave[2] = 1u;
}

template <bool kVar>
__global__ void __launch_bounds__(kActiveTile, 8) k_one(const __grid_constant__ RunDev R, unsigned int* ticket)
{
    pdl_wait();
    pdl_trigger();
    const bool plain = !kVar && plain_run(R), coulomb = (R.flags & kFCoulomb) != 0;
    if (coulomb && blockIdx.x == 0 && threadIdx.x == 0) begin_one(R);
    const uint32_t end = 4u * R.n4, step = *R.step;
    for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; (i & ~31u) < end; i += gridDim.x * blockDim.x) {
        if (!kVar && plain) one_group<false, true>(R, i, step);
        else one_group<kVar, false>(R, i, step);
    }
    if (!coulomb && last_block(ticket) && threadIdx.x == 0) *R.step += 1u;
}

template <bool kVar>
__global__ void __launch_bounds__(256, 5) k_one_batch(const RunDev* __restrict__ runs, uint32_t nruns,
                                                      const uint2* __restrict__ items, uint32_t nitems, uint32_t tile,
                                                      unsigned int* ticket)
{
    __shared__ RunDev rs;
    pdl_wait();
    pdl_trigger();
    uint32_t cur = 0xFFFFFFFFu;
    for (uint32_t k = blockIdx.x; k < nitems; k += gridDim.x) {
        const uint2 it = items[k];
        if (it.x != cur) {
            __syncthreads();
            cur = it.x;
            stage_run(rs, runs + cur);
            __syncthreads();
        }
        const uint32_t step = *rs.step;
        for (uint32_t j = threadIdx.x; j < tile; j += blockDim.x) {
            if (!kVar && plain_run(rs)) one_group<false, true>(rs, it.y * tile + j, step);
            else one_group<kVar, false>(rs, it.y * tile + j, step);
        }
    }
    if (!last_block(ticket)) return;
    for (uint32_t r = threadIdx.x; r < nruns; r += blockDim.x) {
        if (!runs[r].step) continue;
        if (runs[r].flags & kFCoulomb) begin_one(runs[r]);
        else *runs[r].step += 1u;
    }
}

// Fold the packed per-step deposit into the time-summed count and charge
// grids and clear it.
__global__ void k_fold(const __grid_constant__ RunDev R, uint32_t ncells,
                       unsigned long long* __restrict__ count, unsigned long long* __restrict__ charge)
{
    for (uint32_t c = blockIdx.x * blockDim.x + threadIdx.x; c < ncells; c += gridDim.x * blockDim.x) {
        const unsigned long long v = R.dep[c];
        if (v) {
            count[c] += v >> 32;
            charge[c] += v & 0xFFFFFFFFull;
            R.dep[c] = 0ull;
        }
    }
}

// Number of particles in the chamber per charge state.
__global__ void k_census(const __grid_constant__ RunDev R, uint32_t n4,
                         unsigned long long* __restrict__ census)
{
    __shared__ unsigned int h[kQSlots];
    for (int i = threadIdx.x; i < kQSlots; i += blockDim.x) h[i] = 0u;
    __syncthreads();
    for (uint32_t g = blockIdx.x * blockDim.x + threadIdx.x; g < n4; g += gridDim.x * blockDim.x) {
        const uint4 m = reinterpret_cast<const uint4*>(R.meta)[g];
        const uint32_t mm[4] = {m.x, m.y, m.z, m.w};
#pragma unroll
        for (int j = 0; j < 4; ++j)
            if (!(mm[j] & (kStFrozen | kStPad))) atomicAdd(&h[mm[j] & kQMask], 1u);
    }
    __syncthreads();
    for (int i = threadIdx.x; i < kQSlots; i += blockDim.x)
        if (h[i]) atomicAdd(census + i, (unsigned long long)h[i]);
}

struct SoaPtrs { float* p[6]; };

// v * (hi + lo) rounded to the nearest integer: the FP32 product p = v hi is
// an integer once |p| >= 2^24, and its rounding error (exact by FMA) plus
// v lo is added as a small correction.  Float-to-64-bit conversions run on
// the narrow FP64 pipe, so values inside the signed or unsigned 32-bit range
// (every position but the chamber's outermost points) convert in 32 bits, to
// the same integers
__device__ __forceinline__ long long scale_round(float v, float hi, float lo)
{
    const float p = v * hi;
    const float e = fmaf(v, hi, -p) + v * lo;
    const float r = rintf(p);
    long long P;
    if (fabsf(r) < 2147483648.0f) P = (long long)__float2int_rn(r);
    else if (r >= 0.0f && r < 4294967296.0f) P = (long long)__float2uint_rn(r);
    else P = (long long)r;
    return P + (long long)__float2int_rn(e + (p - r));
}

// metres -> fixed point, rounded to nearest, saturated
__device__ __forceinline__ int3 to_fx(float x, float y, float z, const LoadCheck& lc)
{
    const long long lim = 2147483647ll;
    const long long X = max(min(scale_round(x, lc.inv_sxy_hi, lc.inv_sxy_lo), lim), -lim - 1);
    const long long Y = max(min(scale_round(y, lc.inv_sxy_hi, lc.inv_sxy_lo), lim), -lim - 1);
    const long long Z = max(min(scale_round(z, lc.inv_sz_hi, lc.inv_sz_lo) - 2147483648ll, lim), -lim - 1);
    return make_int3((int32_t)X, (int32_t)Y, (int32_t)Z);
}

__device__ __forceinline__ void store_fx(SoaPtrs soa, uint32_t i, const int3& p)
{
    reinterpret_cast<int32_t*>(soa.p[0])[i] = p.x;
    reinterpret_cast<int32_t*>(soa.p[1])[i] = p.y;
    reinterpret_cast<int32_t*>(soa.p[2])[i] = p.z;
}

__device__ __forceinline__ bool velocity_ok(const SoaPtrs& soa, uint32_t i)
{
    const float vx = soa.p[3][i], vy = soa.p[4][i], vz = soa.p[5][i];
    return isfinite(vx) & isfinite(vy) & isfinite(vz);   // (three loads at once)
}

__device__ __forceinline__ void pad_velocity(const SoaPtrs& soa, uint32_t i)
{
    soa.p[3][i] = soa.p[4][i] = soa.p[5][i] = 0.0f;
}

__global__ void k_load_init(LoadCheck lc, SoaPtrs soa, const uint8_t* __restrict__ q8,
                            uint32_t* __restrict__ meta, uint32_t* __restrict__ id, uint32_t n, uint32_t cap,
                            unsigned int* __restrict__ bad, int velocities)
{
    for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < cap; i += gridDim.x * blockDim.x) {
        id[i] = i;
        if (i < n) {
            const float x = soa.p[0][i], y = soa.p[1][i], z = soa.p[2][i];
            const uint32_t q = q8[i];
            bool ok = (x * x + y * y <= lc.R0sq) && (z >= 0.0f) && (z <= lc.L) && q <= lc.qmax;
            if (velocities) ok = ok && velocity_ok(soa, i);
            if (!ok) {
                atomicAdd(bad, 1u);
                atomicMax(bad + 1, ~i);
            }
            meta[i] = ok ? q : kStPad;   // (counted: the velocity check leaves it out)
            const int3 p = to_fx(x, y, z, lc);
            store_fx(soa, i, p);
            if (lc.count && q > 0u) atomicAdd(lc.count + ngp_cell(lc, p.x, p.y, p.z), 1u);
        } else {
            store_fx(soa, i, to_fx(lc.inlet_x, lc.inlet_y, lc.inlet_z, lc));
            meta[i] = kStPad;
            if (velocities) pad_velocity(soa, i);
        }
    }
}

// the velocities alone
__global__ void k_load_check(SoaPtrs soa, const uint32_t* meta, uint32_t n, uint32_t cap,
                             unsigned int* __restrict__ bad)
{
    pdl_wait();
    pdl_trigger();
    for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < cap; i += gridDim.x * blockDim.x) {
        if (i >= n) {
            pad_velocity(soa, i);
        } else if (!velocity_ok(soa, i) && meta[i] != kStPad) {
            atomicAdd(bad, 1u);
            atomicMax(bad + 1, ~i);
        }
    }
}

}  // namespace

cudaError_t launch_load_init(const LoadCheck& lc, float* const soa[6], const uint8_t* q8, uint32_t* meta,
                             uint32_t* id, uint32_t n, uint32_t cap, unsigned int* bad, bool velocities,
                             cudaStream_t s)
{
    SoaPtrs p;
    for (int k = 0; k < 6; ++k) p.p[k] = soa[k];
    const int threads = 256;
    int blocks = (int)((cap + threads - 1) / threads);
    if (blocks > 8192) blocks = 8192;
    k_load_init<<<blocks, threads, 0, s>>>(lc, p, q8, meta, id, n, cap, bad, velocities ? 1 : 0);
    return cudaGetLastError();
}

cudaError_t launch_load_check(float* const soa[6], const uint32_t* meta, uint32_t n, uint32_t cap, unsigned int* bad,
                              cudaStream_t s)
{
    SoaPtrs p;
    for (int k = 0; k < 6; ++k) p.p[k] = soa[k];
    return launch_pdl(k_load_check, dim3(std::min((cap + 255u) / 256u, 8192u)), dim3(256), 0, s, p, meta, n, cap, bad);
}

template <class K>
static int blocks_per_sm(K kernel, int threads, int smem)
{
    int b = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, kernel, threads, smem) != cudaSuccess || b < 1) b = 1;
    return b;
}

WindowBlocks window_blocks_per_sm(int threads)
{
    const int smem = (threads / 32) * (int)sizeof(QuietWarp);
    WindowBlocks b;
    b.quiet = blocks_per_sm(k_quiet_batch, threads, smem);
    b.active = std::min(blocks_per_sm(k_active_batch<false>, threads, 0), blocks_per_sm(k_active_batch<true>, threads, 0));
    b.ions = std::min(blocks_per_sm(k_ions_batch<false>, threads, 0), blocks_per_sm(k_ions_batch<true>, threads, 0));
    b.one = std::min(blocks_per_sm(k_one_batch<false>, threads, 0), blocks_per_sm(k_one_batch<true>, threads, 0));
    return b;
}

cudaError_t launch_quiet(const RunDev& R, uint32_t K, int sm_count, cudaStream_t s)
{
    // at most one wave of blocks; four groups in a row once every warp has some
    const uint32_t most = (uint32_t)(kQuietBlocks * sm_count), slots = 4u * R.n4;
    const uint32_t groups = slots >= most * 4u * 128u * 2u ? 4u : 1u;
    const uint32_t need = (slots + 128u * groups - 1u) / (128u * groups);
    return launch_pdl(k_quiet, dim3(std::max(1u, std::min(need, most))), dim3(128), 0, s, R, K, groups);
}

// as many blocks as the list could need, at most kListBlocks an SM: one wave, but of
// k_active<false> a third more than the six it holds at a time
static dim3 list_grid(const RunDev& R, int sm_count)
{
    return dim3(std::min(4u * R.n4 / kActiveTile + 2u, (uint32_t)(kListBlocks * sm_count)));
}

static bool variants(const RunDev& R) { return (R.flags & kFVariants) || R.btab; }

cudaError_t launch_active(const RunDev& R, uint32_t K, unsigned int* ticket, int sm_count, cudaStream_t s)
{
    return launch_pdl(variants(R) ? k_active<true> : k_active<false>, list_grid(R, sm_count), dim3(kActiveTile), 0, s,
                      R, K, ticket);
}

// Blocks that start while the collision kernel before them ends get an SM
// whose memory that kernel has split for its shared memory, with little left
// for the cache that the gathers live on.  Up to about three blocks' work a
// resident block the early start gives more than that costs: us a step with
// and without, 2e5 particles 27.7 and 32.4, 4e5 35.5 and 38.7, 5e5 42.4 and
// 39.8, 1e6 53.7 and 49.8, 4e6 92.4 and 88.9.
static bool small_list(const RunDev& R, int sm_count)
{
    return 4u * R.n4 <= 3u * kListBlocks * kActiveTile * (uint32_t)sm_count;
}

cudaError_t launch_ions(const RunDev& R, int sm_count, cudaStream_t s)
{
    return launch_early(small_list(R, sm_count), variants(R) ? k_ions<true> : k_ions<false>, list_grid(R, sm_count), dim3(kActiveTile), 0,
                        s, R);
}

cudaError_t launch_one(const RunDev& R, unsigned int* ticket, int sm_count, cudaStream_t s)
{
    const uint32_t need = (4u * R.n4 + kActiveTile - 1u) / kActiveTile, most = (uint32_t)(8 * sm_count);
    return launch_early(small_list(R, sm_count), variants(R) ? k_one<true> : k_one<false>,
                        dim3(std::max(1u, std::min(need, most))), dim3(kActiveTile), 0, s, R, ticket);
}

cudaError_t launch_one_batch(const RunDev* runs, uint32_t nruns, const uint2* items, uint32_t nitems, uint32_t tile,
                             int threads, int grid, bool variants, unsigned int* ticket, cudaStream_t s)
{
    return launch_early(false, variants ? k_one_batch<true> : k_one_batch<false>,
                        dim3(std::max(1u, std::min(nitems, (uint32_t)grid))), dim3(threads), 0, s, runs, nruns, items,
                        nitems, tile, ticket);
}

cudaError_t launch_quiet_batch(const RunDev* runs, uint32_t nruns, const uint2* items, uint32_t nitems, uint32_t tile,
                               int threads, int grid, uint32_t K, uint32_t* pref, unsigned int* ticket,
                               cudaStream_t s)
{
    const uint32_t g = std::max(1u, std::min(nitems, (uint32_t)grid));
    return launch_pdl(k_quiet_batch, dim3(g), dim3(threads),
                      (threads / 32) * sizeof(QuietWarp), s, runs, items, nitems, tile, K, nruns, pref, ticket);
}

cudaError_t launch_active_batch(const RunDev* runs, uint32_t nruns, int threads, int grid, bool variants, uint32_t K,
                                const uint32_t* pref, unsigned int* ticket, cudaStream_t s)
{
    return launch_pdl(variants ? k_active_batch<true> : k_active_batch<false>, dim3(grid), dim3(threads), 0, s, runs,
                      nruns, pref, K, ticket);
}

cudaError_t launch_ions_batch(const RunDev* runs, uint32_t nruns, int threads, int grid, bool variants,
                              const uint32_t* pref, cudaStream_t s)
{
    // (no early start, as for one large run: 1.7e7 particles in 12 runs 14.2 ms
    // with it, 12.3 without)
    return launch_early(false, variants ? k_ions_batch<true> : k_ions_batch<false>, dim3(grid), dim3(threads), 0, s, runs,
                      nruns, pref + nruns + 1u);
}

cudaError_t launch_fold(const RunDev& R, uint32_t ncells, unsigned long long* count, unsigned long long* charge,
                        cudaStream_t s)
{
    const int threads = 256;
    int blocks = (int)((ncells + threads - 1) / threads);
    if (blocks > 4096) blocks = 4096;
    if (blocks < 1) blocks = 1;
    k_fold<<<blocks, threads, 0, s>>>(R, ncells, count, charge);
    return cudaGetLastError();
}

cudaError_t launch_census(const RunDev& R, uint32_t n4, unsigned long long* census, cudaStream_t s)
{
    const int threads = 256;
    int blocks = (int)((n4 + threads - 1) / threads);
    if (blocks > 2048) blocks = 2048;
    if (blocks < 1) blocks = 1;
    k_census<<<blocks, threads, 0, s>>>(R, n4, census);
    return cudaGetLastError();
}

}  // namespace ecris
