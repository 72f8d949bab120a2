// The FP64 pair-once force kernel in 64-bit fixed point (forces without
// energies, plain or energy-shifted truncation; slotted cells, lj_slots.cuh).
//
// The method is that of lj_force_w64.cu: a warp per home cell stages its
// half stencil, lists the pairs within rc by FP32 filters (Phase A), and
// evaluates the listed pairs at full precision, each once (Phase B).  What
// differs is Phase B's arithmetic.  GB300's FP64 pipe takes a warp
// instruction every 16 cycles per SM, and the pair term needs 20 of them:
// 320 cycles, in which the SM could issue 1,280 other instructions.  The
// same term in integers takes about 200.
//
//  * Coordinates are x 2^S mod 2^64, 2^-S being 2^-63 of 1.5 cell sides (the
//    reach of the half stencil from the home cell's centre): exact for x >=
//    2^(53-S) (a double has 53 bits), and so are the differences of particles
//    within rc, whatever the box; a periodic image adds +-L 2^S, an integer.  So d = x_i - x_j carries no
//    rounding at all; FP64 coordinates relative to cell centres carried the
//    centres' (the forces' error at N = 131,072 was 2.5e-14 of their norm).
//  * r^2: the upper 64 bits of the squares, 2^-57 relative at r = 0.4 rc.
//  * u = sigma^2 / r^2: a float reciprocal of the normalised r^2 (error e <
//    2^-22, formed exactly in integers) and the series 1 + e + e^2 (e^3 <
//    2^-66), then u^2, u^3, u^4 by high products and |F(r)| / r = 24 eps /
//    sigma^2 u^4 |2 u^3 - 1|.
//  * The sums are 64-bit integers, added by integer atomics: exact, so they
//    do not depend on the order (the forces repeat from run to run).  One
//    unit cannot hold them all: a pair at 2.45 sigma is 1/3,300 of the
//    largest one taken here, and in that one's unit it had 43 bits.  So there
//    are three sums per component, of units q = 2^-52 24 eps / sigma at
//    sigma = 1 (fx_tsh), q / 32 and q / 256, for the repulsive pairs, the
//    attractive ones and those beyond 1.8 sigma, the products rounded to
//    nearest in magnitude.  With |F| <= 6.35, 0.1 and 0.0155 of 24 eps /
//    sigma in the three, their ranges hold 320, 590 and 480 pairs that all
//    pull one way, more than cells of 32 slots can place so; sums that leave
//    the range on the way come back.  A home particle's partial sums become
//    one number in units of q / 256, which is added as its upper bits, to the
//    first sum, and its lowest 8, which the three components share a word
//    for: four atomics, not nine.
//    Emulated in exact integers for single pairs, RMS error relative to the
//    force (FP64 coordinates and term: L = 7.6, 13, 27, 54; one unit for all
//    pairs): r = 1.0 2.5e-16 (1e-15 to 2e-14), 1.2 5e-17 (3e-16 to 6e-15; one
//    unit 2.4e-15), 1.7 1.6e-16 (4e-16 to 5e-15; 9e-15), 2.45 2.4e-16 (4e-16
//    to 5e-15; 1.1e-13), 2.65 4.0e-16 (4.2e-16 at L = 9); 2.9 7.7e-16
//    (4.1e-16): hence rc <= 2.6 sigma in uses_fx.
//  * Pairs closer than sqrt(0.8) sigma, where u > 1.25 and the force has no
//    bound, and cells that take the plain path are evaluated in FP64 as
//    before (pair64_nf) and added to f itself; the readers of the sums add
//    the two (fx_force, lj_slots.cu).
// Bound by instruction issue and the latencies that 15 warps per SM leave (60
// % of issue slots; ALU pipe 47 %).  Step in FP64: 257 -> 105 us at 131,072
// particles (the force kernel 220 -> 95), 174 -> 35 at 32,000, 1,309 -> 655 at
// 10^6.  Forces against the oracle: 4.9e-15 of their norm at 131,072 particles
// (2.8e-14 with lj_force_w64.cu), 3.0e-15 at 2,048 (1.0e-14), 4.7e-15 for a gas
// of 100,003 at density 0.3 (2.1e-14).
#include <math.h>
#include <string.h>

#include "lj_force_n3.cuh"
#include "lj_slots.cuh"

namespace {

constexpr int kFxThreads = 32;    // one warp per CTA, as the FP64 kernel
constexpr int kFxPMax = 32;       // home particles of a staged cell
constexpr int kFxList = 1024;     // list entries per batch

struct FxParams {
    int nc, cap, scap, nslots, last;
    float inv_nc, to_f;                    // to_f = 2^(32 - S)
    float rc2_box, rc2_pair;
    unsigned *work;
    int64_t ncell;
    const int2 *cellq;
    int2 *cellq_next;
    unsigned *octr_next, *last_par;
    unsigned par;
    const int32_t *onext;
    const long long *cfix;                 // cell centres, fixed point
    int kappa_e, tsh;                           // u = K / 2^63 2^kappa_e 2^lz RI 2^-62
    long long Lfix;
    unsigned long long K, r2c, r2min, r2far;
    // FP64 pairs
    double to_d;                           // 2^-S
    double rc2, a12, b6;
};

// Byte layout of a warp's slice (cap a multiple of 2).
struct FxLayout {
    int x64, x32, iw, sh, spre, off, list, bytes;
    __host__ __device__ explicit FxLayout(int cap)
    {
        x64 = 0;                                   // int64[3][cap]
        sh = x64 + 24 * cap;                       // int64[3][kN3Half], then int start[kN3Half]
        x32 = (sh + 28 * kN3Half + 15) & ~15;      // float[3][cap]
        iw = x32 + 12 * cap;                       // int[cap] particle index
        spre = (iw + 4 * cap + 15) & ~15;          // int[16]
        off = spre + 64;                           // int[kFxPMax + 4]
        list = off + 4 * (kFxPMax + 4);            // uint16[kFxList]
        bytes = (list + 2 * kFxList + 15) & ~15;
    }
};

// The FP64 pair term of lj_force_w64.cu (pair64_nf) for truncation without a
// force shift: -F(r) / r, 0 outside rc or for r = 0.
__device__ __forceinline__ double fx_pair64(double dx, double dy, double dz, const FxParams &k)
{
    const double r2 = fma(dz, dz, fma(dy, dy, dx * dx));
    const bool in = r2 < k.rc2 && r2 != 0.0;
    const double ri = in ? 1.0 / r2 : 0.0;
    const double r6 = ri * ri * ri;
    return ri * r6 * fma(-k.a12, r6, k.b6);
}

__device__ __forceinline__ void fx_add64(double4_16a *f, int i, double x, double y, double z)
{
    atomicAdd(&f[i].x, x);
    atomicAdd(&f[i].y, y);
    atomicAdd(&f[i].z, z);
}

__device__ __forceinline__ void fx_red(unsigned long long *o, long long v) { atomicAdd(o, (unsigned long long)v); }

// A home particle's partial sums (of at most 32 pairs): r, m, f in units of q,
// q / 32, q / 256.  v = 8 m + f: |m| < 2^59, |f| < 2^59.
__device__ __forceinline__ long long fx_split(long long r, long long m, long long f, int sh, unsigned long long &lo)
{
    const long long v = (m << 3) + f;
    lo += (unsigned long long)(v & 255) << sh;
    return r + (v >> 8);
}

__device__ __forceinline__ unsigned long long fx_abs(long long d) { return (unsigned long long)(d < 0 ? -d : d); }

// |F(r)| / r in units of 24 eps / sigma^2 2^-(58 + 4 cls) for r2min <= R2 <
// r2c; cls: 0 repulsive, 1 attractive, 2 beyond 1.8 sigma.  u^2 is shifted up
// by 2 cls bits (u^2 < 1.5, 0.631, 0.096), so that u^4 and the result keep 58 bits.
__device__ __forceinline__ unsigned long long fx_term(unsigned long long R2, const FxParams &k, int &cls)
{
    const int lz = __clzll((long long)R2);
    const unsigned long long M = R2 << lz;   // m = M 2^-64 in [1/2, 1)
    const float y = rcp_approx(__uint_as_float(0x3f000000u | ((unsigned)(M >> 40) & 0x7fffffu)));
    const unsigned y0 = __float_as_uint(y) - 0x3f800000u + 0x800000u;   // y 2^23, in (2^23, 2^24]
    // e = 1 - m y in units of 2^-63
    const unsigned long long plo = (unsigned long long)(unsigned)M * y0;
    const unsigned long long phi = (M >> 32) * y0;
    const long long E = (long long)(0x8000000000000000ull - ((phi << 8) + (plo >> 24)));
    const int eh = (int)(E >> 11);
    const long long G = E + (((long long)eh * eh) >> 41);
    // 1 / m in units of 2^-62
    const unsigned long long RI = ((unsigned long long)y0 << 39) + (unsigned long long)(((long long)y0 * (G >> 3)) >> 21);
    const unsigned long long h = __umul64hi(RI, k.K);
    const int s = k.kappa_e + lz + 2;
    const unsigned long long U = s >= 0 ? h << s : (s > -64 ? h >> -s : 0ull);   // u 2^63
    const unsigned long long U2 = __umul64hi(U, U);                              // 2^62
    const unsigned long long U3 = __umul64hi(U2, U);                             // 2^61
    const long long T = (long long)U3 - (1ll << 60);                             // (2 u^3 - 1) 2^60
    cls = R2 >= k.r2far ? 2 : T < 0 ? 1 : 0;
    const unsigned long long V2 = U2 << (2 * cls);                               // 2^(62 + 2 cls)
    const unsigned long long V4 = __umul64hi(V2, V2);                            // u^4 2^(60 + 4 cls)
    return __umul64hi(V4, fx_abs(T)) << 2;
}

// t a 2^-64, rounded to nearest at bit sh >= 1: in magnitude, so that a pair's
// force does not depend on which of the two is home.
__device__ __forceinline__ long long fx_mul(unsigned long long t, unsigned long long a, int sh)
{
    return (long long)((__umul64hi(t, a) + (1ull << (sh - 1))) >> sh);
}

// Plain path: lanes own home particles, FP64 over the half stencil's slots
// and overflow lists.
__device__ void fx_plain(const FxParams &k, const longlong4_16a *pos, double4_16a *f,
                         const long long *sh, const int *st, const int *spre, int c, int n_home)
{
    const int lane = threadIdx.x & 31;
    for (int p0 = 0; p0 < n_home; p0 += 32) {
        const int i = p0 + lane;
        const bool vi = i < n_home;
        int si = st[0] + (vi ? i : 0);
        if (vi && i >= k.scap) {
            int o = k.cellq[c].y;
            for (int m = k.scap; m < i && o > 0; m++) o = k.onext[o - 1];
            if (o > 0) si = k.nslots + o - 1;
        }
        const longlong4_16a pi = pos[si];
        // coordinates relative to the home cell's centre (their differences
        // may leave the range of 64 bits here: formed in FP64)
        const double xi = (double)(pi.x + sh[0]), yi = (double)(pi.y + sh[kN3Half]), zi = (double)(pi.z + sh[2 * kN3Half]);
        double fx = 0.0, fy = 0.0, fz = 0.0;
        for (int kk = 0; kk < kN3Half; kk++) {
            const int nn = spre[kk + 1] - spre[kk];
            int o = 0;
            for (int j = 0; j < nn; j++) {
                int sj = st[kk] + j;
                if (j >= k.scap) {
                    o = j == k.scap ? k.cellq[half_cell(c, kk, k.nc, k.inv_nc)].y : k.onext[o - 1];
                    if (o <= 0) break;
                    sj = k.nslots + o - 1;
                }
                if (!vi || (kk == 0 && j <= i)) continue;
                const longlong4_16a q = pos[sj];
                const double dx = (xi - (double)(q.x + sh[kk])) * k.to_d,
                             dy = (yi - (double)(q.y + sh[kN3Half + kk])) * k.to_d,
                             dz = (zi - (double)(q.z + sh[2 * kN3Half + kk])) * k.to_d;
                const double nf = fx_pair64(dx, dy, dz, k);
                if (nf == 0.0) continue;
                fx -= nf * dx;
                fy -= nf * dy;
                fz -= nf * dz;
                fx_add64(f, (int)q.w, nf * dx, nf * dy, nf * dz);
            }
        }
        if (vi) fx_add64(f, (int)pi.w, fx, fy, fz);
    }
}

// Staging: the half stencil's candidates within rc of the home box, home
// particles first; returns their number, or -1 when they and 64 entries of
// padding would not fit.  PART: as many as fit of those from `next` on, after
// the T that are there already (none, or the home particles); next is then the
// next part's first.  A part takes at least 32 candidates (cap >= 128).
// tmp: int[kN3Half].
template <bool PART>
__device__ __forceinline__ int fx_stage(const FxParams &k, const longlong4_16a *pos, int &next, int T, long long *X64,
                                        float *X, int *iw, int *tmp, const long long *sh, const int *st,
                                        const int *spre, int tot, int n_home)
{
    const int lane = threadIdx.x & 31;
    if (!PART) T = 0;
    const unsigned lt = (1u << lane) - 1u, le = (2u << lane) - 1u;
    float bxl = 3.4e38f, byl = 3.4e38f, bzl = 3.4e38f, bxh = -3.4e38f, byh = -3.4e38f, bzh = -3.4e38f;
    // warp-vote entry lookup, as n3_stage
    const int s_e = lane < kN3Half ? spre[lane] : 0x7fffffff;
    const bool ne = lane < kN3Half && spre[lane + 1] > s_e;
    const unsigned nem = __ballot_sync(0xffffffffu, ne);
    if (ne) tmp[__popc(nem & lt)] = lane;
    __syncwarp();
    const int j_entry = lane < __popc(nem) ? tmp[lane] : 0;
    __syncwarp();
    if (PART && T > 0) {
        if (lane < n_home) {
            bxl = bxh = X[lane];
            byl = byh = X[k.cap + lane];
            bzl = bzh = X[2 * k.cap + lane];
        }
        box_reduce(bxl, byl, bzl, bxh, byh, bzh);
    }
    constexpr int kB = 2;   // rounds whose loads are in flight together
    int t0 = PART ? next : 0, end = tot;
    for (; t0 < end; t0 += 32 * kB) {
        longlong2 qa[kB], qb[kB];
        int kcs[kB];
#pragma unroll
        for (int u = 0; u < kB; u++) {
            const int tb = t0 + 32 * u, t = tb + lane;
            const int o = s_e - tb;
            const unsigned inside = __reduce_or_sync(0xffffffffu, (ne && o >= 1 && o <= 31) ? (1u << o) : 0u);
            const int jc = __popc(__ballot_sync(0xffffffffu, ne && o <= 0)) - 1 + __popc(inside & le);
            const int kc = __shfl_sync(0xffffffffu, j_entry, jc & 31);
            const int kb = __shfl_sync(0xffffffffu, s_e, kc);
            kcs[u] = kc;
            const longlong2 *p = reinterpret_cast<const longlong2 *>(pos + min(st[kc] + (t - kb), k.last));
            qa[u] = p[0];
            qb[u] = p[1];
        }
#pragma unroll
        for (int u = 0; u < kB; u++) {
            const int t = t0 + 32 * u + lane;
            const int kc = kcs[u];
            const long long x = qa[u].x + sh[kc], y = qa[u].y + sh[kN3Half + kc], z = qb[u].x + sh[2 * kN3Half + kc];
            const float cx = (float)(int)(x >> 32) * k.to_f, cy = (float)(int)(y >> 32) * k.to_f,
                        cz = (float)(int)(z >> 32) * k.to_f;
            if (u == 0 && t0 == 0) {   // the home particles are the first n_home <= 32 candidates
                if (lane < n_home) {
                    bxl = bxh = cx;
                    byl = byh = cy;
                    bzl = bzh = cz;
                }
                box_reduce(bxl, byl, bzl, bxh, byh, bzh);
            }
            const float dx = fmaxf(fmaxf(bxl - cx, cx - bxh), 0.f);
            const float dy = fmaxf(fmaxf(byl - cy, cy - byh), 0.f);
            const float dz = fmaxf(fmaxf(bzl - cz, cz - bzh), 0.f);
            const bool keep = t < tot && dx * dx + dy * dy + dz * dz < k.rc2_box;
            const unsigned kept = __ballot_sync(0xffffffffu, keep);
            if (T + __popc(kept) + 64 > k.cap) {   // the next part's
                if (!PART) {
                    __syncwarp();
                    return -1;
                }
                end = t0 + 32 * u;
                break;
            }
            if (keep) {
                const int s = T + __popc(kept & lt);
                X[s] = cx;
                X[k.cap + s] = cy;
                X[2 * k.cap + s] = cz;
                X64[s] = x;
                X64[k.cap + s] = y;
                X64[2 * k.cap + s] = z;
                iw[s] = (int)qb[u].y;
            }
            T += __popc(kept);
        }
    }
    for (int u = 0; u < 64; u += 32) X[T + u + lane] = X[k.cap + T + u + lane] = X[2 * k.cap + T + u + lane] = kFar;
    __syncwarp();
    if (PART) next = end;
    return T;
}

// Phase B over one batch: the entries [0, E) of the list, home particles pb
// .. pb + P - 1; every lane takes an equal contiguous range.
__device__ __forceinline__ void fx_pairs(const FxParams &k, long long *acc, double4_16a *f,
                                         const long long *X64, const int *iw, const uint16_t *list, const int *off,
                                         int E, int P, int pb)
{
    const int lane = threadIdx.x & 31;
    const int lo = (lane * E) >> 5, hi = ((lane + 1) * E) >> 5;
    const long long *Y64 = X64 + k.cap, *Z64 = Y64 + k.cap;
    if (lo < hi) {
        int q = 0;
#pragma unroll
        for (int step = kFxPMax / 2; step > 0; step >>= 1)
            if (q + step < P && off[q + step] <= lo) q += step;
        int nxt = off[q + 1];
        long long xp = X64[pb + q], yp = Y64[pb + q], zp = Z64[pb + q];
        long long sx[3] = {0, 0, 0}, sy[3] = {0, 0, 0}, sz[3] = {0, 0, 0};   // per class
        auto flush = [&](int i) {
            unsigned long long *o = reinterpret_cast<unsigned long long *>(acc) + kFxAcc * (int64_t)i;
            unsigned long long lo = 0;
            fx_red(o, fx_split(sx[0], sx[1], sx[2], 0, lo));
            fx_red(o + 1, fx_split(sy[0], sy[1], sy[2], kFxLow, lo));
            fx_red(o + 2, fx_split(sz[0], sz[1], sz[2], 2 * kFxLow, lo));
            fx_red(o + 9, (long long)lo);
        };
        for (int e = lo; e < hi; e++) {
            if (e == nxt) {
                flush(iw[pb + q]);
                do {
                    q++;
                    nxt = off[q + 1];
                } while (nxt == e);
                xp = X64[pb + q];
                yp = Y64[pb + q];
                zp = Z64[pb + q];
#pragma unroll
                for (int u = 0; u < 3; u++) sx[u] = sy[u] = sz[u] = 0;
            }
            const int j = list[e];
            const long long dx = xp - X64[j], dy = yp - Y64[j], dz = zp - Z64[j];
            const unsigned long long bx = fx_abs(dx), by = fx_abs(dy), bz = fx_abs(dz);
            const unsigned long long R2 = __umul64hi(bx, bx) + __umul64hi(by, by) + __umul64hi(bz, bz);
            if (R2 >= k.r2c) continue;
            if (R2 < k.r2min) {   // too close for the fixed-point range
                const double ex = (double)dx * k.to_d, ey = (double)dy * k.to_d, ez = (double)dz * k.to_d;
                const double nf = fx_pair64(ex, ey, ez, k);
                fx_add64(f, iw[pb + q], -nf * ex, -nf * ey, -nf * ez);
                fx_add64(f, iw[j], nf * ex, nf * ey, nf * ez);
                continue;
            }
            int cls;
            const unsigned long long t = fx_term(R2, k, cls);
            const int sh = k.tsh + (cls == 1 ? 1 : 2);
            long long gx = fx_mul(t, bx, sh), gy = fx_mul(t, by, sh), gz = fx_mul(t, bz, sh);
            const long long at = cls == 0 ? 0 : -1;   // attractive: F against d
            const long long mx = (dx >> 63) ^ at, my = (dy >> 63) ^ at, mz = (dz >> 63) ^ at;
            gx = (gx ^ mx) - mx;
            gy = (gy ^ my) - my;
            gz = (gz ^ mz) - mz;
            unsigned long long *o = reinterpret_cast<unsigned long long *>(acc) + (kFxAcc * (int64_t)iw[j] + 3 * cls);
            fx_red(o, -gx);
            fx_red(o + 1, -gy);
            fx_red(o + 2, -gz);
#pragma unroll
            for (int u = 0; u < 3; u++)
                if (cls == u) {
                    sx[u] += gx;
                    sy[u] += gy;
                    sz[u] += gz;
                }
        }
        flush(iw[pb + q]);
    }
    __syncwarp();   // list and off are rewritten by the next batch
}

// Phases A and B for T staged candidates, of which those from `done` on are
// taken (and home pairs only if done = 0).
__device__ __forceinline__ void fx_compute(const FxParams &k, long long *acc, double4_16a *f, const long long *X64,
                                           const float *X, const int *iw, uint16_t *list, int *off, int T, int done,
                                           int n_home)
{
    const int lane = threadIdx.x & 31;
    const unsigned lt = (1u << lane) - 1u;
    const float2 *X2 = reinterpret_cast<const float2 *>(X);
    const float2 *Y2 = reinterpret_cast<const float2 *>(X + k.cap);
    const float2 *Z2 = reinterpret_cast<const float2 *>(X + 2 * k.cap);
    int p = 0;
    while (p < n_home) {
        // Phase A: the lists of the batch's particles (candidates j > p)
        const int pb = p;
        int E = 0;
        if (lane == 0) off[0] = 0;
        while (p < n_home && E + T <= kFxList) {
            const float2 xs = f2(X[p]), ys = f2(X[k.cap + p]), zs = f2(X[2 * k.cap + p]);
            const int jlo = max(p + 1, done);
            for (int j0 = 0; j0 < T; j0 += 64) {
                const int jx = j0 + 2 * lane;
                const float2 qx = X2[(j0 >> 1) + lane], qy = Y2[(j0 >> 1) + lane], qz = Z2[(j0 >> 1) + lane];
                const float2 dx = __ffma2_rn(qx, f2(-1.0f), xs);
                const float2 dy = __ffma2_rn(qy, f2(-1.0f), ys);
                const float2 dz = __ffma2_rn(qz, f2(-1.0f), zs);
                float2 r2 = __fmul2_rn(dx, dx);
                r2 = __ffma2_rn(dy, dy, r2);
                r2 = __ffma2_rn(dz, dz, r2);
                const bool ina = r2.x < k.rc2_pair && jx >= jlo;
                const bool inb = r2.y < k.rc2_pair && jx + 1 >= jlo;
                const unsigned ba = __ballot_sync(0xffffffffu, ina);
                const unsigned bb = __ballot_sync(0xffffffffu, inb);
                if (ina) list[E + __popc(ba & lt)] = (uint16_t)jx;
                if (inb) list[E + __popc(ba) + __popc(bb & lt)] = (uint16_t)(jx + 1);
                E += __popc(ba) + __popc(bb);
            }
            if (lane == 0) off[p - pb + 1] = E;
            p++;
        }
        __syncwarp();
        fx_pairs(k, acc, f, X64, iw, list, off, E, p - pb, pb);
    }
}

// The slice of a warp.
struct FxSlice {
    long long *X64, *sh;
    int *st, *iw, *spre, *off;
    float *X;
    uint16_t *list;
    __device__ FxSlice(unsigned char *smem, int cap)
    {
        const FxLayout L(cap);
        X64 = reinterpret_cast<long long *>(smem + L.x64);
        sh = reinterpret_cast<long long *>(smem + L.sh);
        st = reinterpret_cast<int *>(sh + 3 * kN3Half);
        X = reinterpret_cast<float *>(smem + L.x32);
        iw = reinterpret_cast<int *>(smem + L.iw);
        spre = reinterpret_cast<int *>(smem + L.spre);
        off = reinterpret_cast<int *>(smem + L.off);
        list = reinterpret_cast<uint16_t *>(smem + L.list);
    }
};

// The pairs of home cell c.  A cell whose candidates do not fit the slice, or
// with more than 32 home particles or a cell of its half stencil beyond its
// slots, takes the plain path (FITS); is left, the result being false; or, ANY,
// is taken in parts, the home particles with some of the candidates at a time,
// or by the plain path if it must.
template <bool FITS, bool ANY>
__device__ __forceinline__ bool fx_cell(const FxParams &k, const longlong4_16a *pos, long long *acc, double4_16a *f,
                                        const FxSlice &w, int c)
{
    const int lane = threadIdx.x & 31;
    if (lane == 31) k.cellq_next[c] = make_int2(0, 0);
    __syncwarp();   // the slice still holds the previous cell's data
    // half-stencil table: first slot, prefix sums, image shift minus the
    // home cell's centre
    const HalfLoad tl = half_load<true, true>(reinterpret_cast<const int32_t *>(k.cellq), c, k.nc, k.inv_nc, 0, k.scap);
    const int nn = tl.e - tl.s;
    if (lane < kN3Half) {
        int cx, cy, cz, dx, dy, dz;
        lj_cell_decode(c, k.nc, k.inv_nc, cx, cy, cz);
        half_delta(lane, dx, dy, dz);
        const int ux = cx + dx, uy = cy + dy, uz = cz + dz;
        w.sh[lane] = (ux < 0 ? -k.Lfix : ux >= k.nc ? k.Lfix : 0ll) - __ldg(k.cfix + cx);
        w.sh[kN3Half + lane] = (uy < 0 ? -k.Lfix : uy >= k.nc ? k.Lfix : 0ll) - __ldg(k.cfix + cy);
        w.sh[2 * kN3Half + lane] = (uz < 0 ? -k.Lfix : uz >= k.nc ? k.Lfix : 0ll) - __ldg(k.cfix + cz);
        w.st[lane] = tl.s;
    }
    int Pf = nn;
#pragma unroll
    for (int o = 1; o < 16; o <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, Pf, o);
        if (lane >= o) Pf += y;
    }
    if (lane < kN3Half) w.spre[lane] = Pf - nn;
    if (lane == kN3Half - 1) w.spre[kN3Half] = Pf;
    __syncwarp();
    const int tot = w.spre[kN3Half], n_home = w.spre[1];
    if (n_home == 0) return true;
    const bool plain = __any_sync(0xffffffffu, nn > k.scap) || n_home > 32;
    int next = 0;
    if constexpr (ANY) {
        if (plain)
            fx_plain(k, pos, f, w.sh, w.st, w.spre, c, n_home);
        else
            for (int done = 0; next < tot; done = n_home) {
                const int T =
                    fx_stage<true>(k, pos, next, done, w.X64, w.X, w.iw, w.off, w.sh, w.st, w.spre, tot, n_home);
                fx_compute(k, acc, f, w.X64, w.X, w.iw, w.list, w.off, T, done, n_home);
            }
    } else {
        const int T = plain || tot > 4 * k.cap
                          ? -1 : fx_stage<false>(k, pos, next, 0, w.X64, w.X, w.iw, w.off, w.sh, w.st, w.spre, tot, n_home);
        if (T >= 0)
            fx_compute(k, acc, f, w.X64, w.X, w.iw, w.list, w.off, T, 0, n_home);
        else if (FITS)
            fx_plain(k, pos, f, w.sh, w.st, w.spre, c, n_home);
        else
            return false;
    }
    return true;
}

// The next cell (asked for when a cell is done, as k_force_n3's single pulls).
__device__ __forceinline__ int fx_next(const FxParams &k)
{
    unsigned nx = 0;
    if ((threadIdx.x & 31) == 0) nx = gridDim.x + atomicAdd(k.work, 1u);
    return (int)__shfl_sync(0xffffffffu, nx, 0);
}

// FITS: the slice has room for a liquid's cells (fx_fits), and the few that do
// not fit take the plain path.  Otherwise a warp that meets one (a droplet's
// in a box sized for its vapour) takes all further cells by the general form,
// in a loop of its own: a droplet of 97,556 particles at a mean density of 0.1
// 2,210 -> 116 us, at 0.5 1,850 -> 100.  The second loop costs the first one 2
// to 4 % by itself (500,000 particles of liquid 363 -> 372 us); as the only
// loop, for its registers, it costs 7 % (a gas of density 0.1 84 -> 90).
template <bool FITS>
__global__ void __launch_bounds__(kFxThreads, 26) k_force_fx(FxParams k, const longlong4_16a *pos,
                                                         long long *acc, double4_16a *f)
{
    extern __shared__ __align__(16) unsigned char fxsmem[];
    const FxSlice w(fxsmem, k.cap);
    pdl_wait();
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        k.cellq_next[k.ncell] = make_int2(0, 0);
        *k.octr_next = 0u;
        *k.last_par = k.par;
    }
    int c = blockIdx.x;
    for (; c < k.ncell; c = fx_next(k))
        if (!fx_cell<FITS, false>(k, pos, acc, f, w, c)) break;
    if constexpr (!FITS)
        for (; c < k.ncell; c = fx_next(k)) fx_cell<false, true>(k, pos, acc, f, w, c);
}

}  // namespace

int fx_shift(const lj_ctx *c) { return (int)floor(62.95 - log2(1.5 * c->cw)); }

// The first sums' unit is 24 eps / sigma^2 2^-(S - 8 - tsh); tsh makes that
// 2^-52 24 eps / sigma at sigma = 1, and elsewhere so much that the range is
// 2,040 to 4,080 of 24 eps / sigma (with rc <= 2.6 sigma S - 8 - tsh is never
// below it: cells are less than 4/3 rc wide).
static int fx_tsh(const lj_ctx *c)
{
    const int fb = (int)floor(63.0 - log2(2040.0 * c->p.sigma));
    const int t = fx_shift(c) - 8 - fb;
    return t > 0 ? t : 0;
}

double fx_scale(const lj_ctx *c)
{
    return ldexp(24.0 * c->p.eps / (c->p.sigma * c->p.sigma), 8 + fx_tsh(c) - fx_shift(c));
}

cudaError_t fx_configure(lj_ctx *c)
{
    const double mean = (double)c->p.n / (double)c->ncell;
    // ~0.63 m of the m = 14 n_cell raw candidates survive the box test; room
    // for 2.5 sqrt(m) more and the padding.  Slots cost resident warps (12 KB
    // a warp at liquid density, 18 warps per SM): with 4 sqrt(m) + 96 the step
    // at 10^6 particles took 6 % longer, with 2.5 sqrt(m) + 96 3 %.
    const double m = kN3Half * mean;
    int cap = ((int)(0.65 * m + 2.5 * sqrt(m)) + 64 + 7) & ~7;
    cap = cap < 128 ? 128 : (cap > kFxList ? kFxList : cap);
    c->fx_cap = cap;
    c->fx_smem = FxLayout(cap).bytes;
    int nb = 1 << 30;
    for (const void *kern : {(const void *)k_force_fx<true>, (const void *)k_force_fx<false>}) {
        int b = 0;
        cudaError_t e = raise_dyn_smem(kern, c->fx_smem);
        if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, kern, kFxThreads, c->fx_smem);
        if (e != cudaSuccess) return e;
        nb = b < nb ? b : nb;
    }
    const int64_t grid = (int64_t)(nb > 0 ? nb : 1) * c->nsm;
    c->fx_grid = (int)(grid < c->ncell ? grid : c->ncell);
    return cudaSuccess;
}

// The slice holds what is left of a liquid's half stencil (density 0.85) and
// the padding: mean densities of 0.6 and above at rc = 2.5 sigma.
static bool fx_fits(const lj_ctx *c)
{
    const double cw = c->cw / c->p.sigma;
    return 0.63 * kN3Half * 0.85 * cw * cw * cw + 64.0 <= (double)c->fx_cap;
}

cudaError_t launch_force_fx(lj_ctx *c, double4_16a *f)
{
    FxParams k;
    memset(&k, 0, sizeof(k));
    const double rc = c->p.rc, sg = c->p.sigma;
    const int S = fx_shift(c);
    k.nc = c->nc;
    k.cap = c->fx_cap;
    k.scap = c->scap;
    k.nslots = c->nslots;
    k.last = c->nslots + (int)c->p.n - 1;
    k.inv_nc = c->inv_nc_f;
    k.to_f = (float)ldexp(1.0, 32 - S);
    k.rc2_box = (float)(rc * rc) * 1.0001f;
    k.rc2_pair = (float)(rc * rc * (1.0 + 1e-4));
    k.work = c->work;
    k.ncell = c->ncell;
    k.cellq = c->cellq[c->slot_par];
    k.cellq_next = c->cellq[c->slot_par ^ 1];
    k.octr_next = c->octr + (c->slot_par ^ 1);
    k.last_par = c->octr + 2;
    k.par = (unsigned)c->slot_par;
    k.onext = c->onext;
    k.cfix = c->cfix;
    k.tsh = fx_tsh(c);
    k.Lfix = lj_fix64(c->p.box, S);
    int ex = 0;
    const double s2 = sg * sg, mant = frexp(s2, &ex);   // sigma^2 to 64 bits: the product and its rounding error
    k.K = (unsigned long long)ldexp(mant, 64) + (unsigned long long)(long long)ldexp(fma(sg, sg, -s2), 64 - ex);
    k.kappa_e = ex + 2 * S - 129;
    k.r2c = (unsigned long long)ldexp(rc * rc, 2 * S - 64);
    const double rmin = ldexp(0.8 * sg * sg, 2 * S - 64);
    k.r2min = rmin < (double)k.r2c ? (unsigned long long)rmin : k.r2c;
    const double rfar = ldexp(3.24 * sg * sg, 2 * S - 64);   // none beyond it if rc is not
    k.r2far = rfar < (double)k.r2c ? (unsigned long long)rfar : ~0ull;
    k.to_d = ldexp(1.0, -S);
    const double s6 = sg * sg * sg * sg * sg * sg;
    k.rc2 = rc * rc;
    k.a12 = 48.0 * c->p.eps * s6 * s6;
    k.b6 = 24.0 * c->p.eps * s6;
    const longlong4_16a *pos = (const longlong4_16a *)c->spos;
    long long *acc = c->fx_acc;
    void *args[] = {&k, (void *)&pos, &acc, &f};
    if (c->timing && c->ev_used + 2 <= c->nev) cudaEventRecord(c->ev[c->ev_used], c->stream);
    const cudaError_t e = launch_pdl(fx_fits(c) ? (const void *)k_force_fx<true> : (const void *)k_force_fx<false>, c->fx_grid, kFxThreads, args, (size_t)c->fx_smem, c->stream,
                                     !c->timing);
    if (c->timing && c->ev_used + 2 <= c->nev) {
        cudaEventRecord(c->ev[c->ev_used + 1], c->stream);
        c->ev_used += 2;
    }
    c->kernel_launches++;
    if (e != cudaSuccess) return e;
    slots_consumed(c);
    return cudaGetLastError();
}
