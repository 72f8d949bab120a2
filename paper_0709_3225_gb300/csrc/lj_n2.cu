// All-pairs forces (Section 2, Eq. n2_force): every particle against every
// other at the minimum image, with the cutoff and the shift of the context.
// This is the paper's first GPU algorithm, kept as the GPU brute-force
// cross-check of the cell list and for the N^2-versus-cells break-even study.
//
// Organisation on GB300:
//  * A CTA of kN2Threads threads; thread t owns particle
//    i = blockIdx.x * kN2Threads + t.
//  * The j particles stream through shared memory in tiles,
//    copied by cp.async.bulk (issued by thread 0, completing on an mbarrier,
//    two buffers, bounded waits).  This is the paper's "load a block of
//    particles into shared memory, synchronise, compute", with the copy
//    engine doing the loads while the threads compute on the other buffer.
//  * The grid is i-blocks x j-splits: split s takes tiles s, s + nsplit, ...,
//    so that small systems still fill the SMs.  The per-split partial forces
//    are summed in split order by k_n2_sum (deterministic).
//  * Coordinates are the wrapped positions minus L/2 (|x| <= L/2) in the
//    context's precision: absolute coordinates, as in the paper's N^2 code.
//    The minimum image is d -= L rint(d / L).
#include "lj_pair.cuh"

namespace {

constexpr int kN2Threads = 128;
constexpr int kN2Tile = 512;    // j particles per shared-memory tile, FP64
constexpr int kN2TileF = 128;   // FP32: at most (a multiple of 32; 256 measured 48 us against 46 at 8,788)

struct N2Params {
    int n, ntiles;
    double L, invL;
    double rc2, rc, a12, b6, c12, c6, uc, fc;
};

// pos[i] = (wrap(x_i) - L/2, i); non-finite coordinates latch LJ_ENONFINITE.
template <typename T>
__global__ void k_n2_prep(const double *__restrict__ x, int n, double L, double whi, double wlo,
                          typename Vec4<T>::type *__restrict__ pos, int32_t *err)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const double px = x[3 * (int64_t)i], py = x[3 * (int64_t)i + 1], pz = x[3 * (int64_t)i + 2];
    if (!(isfinite(px) && isfinite(py) && isfinite(pz))) atomicOr(err, LJ_ERRBIT_NONFINITE);
    const double h = 0.5 * L;
    typename Vec4<T>::type q;
    q.x = (T)(lj_wrap_fast(px, L, whi, wlo) - h);
    q.y = (T)(lj_wrap_fast(py, L, whi, wlo) - h);
    q.z = (T)(lj_wrap_fast(pz, L, whi, wlo) - h);
    if constexpr (sizeof(T) == 4) {
        q.w = __int_as_float(i);
    } else {
        q.w = (double)i;
    }
    pos[i] = q;
}

// FP32: coordinates in three arrays of npad (a multiple of 32) floats; the
// padding is far away (its squared distance is inf, the image included).
// After them, for each group of 32 consecutive particles, its bounding box as
// two float4: the centre, and the half extents (with the rounding of both, and
// 1e30 for a group with a non-finite coordinate, which is never left out).
__global__ void k_n2_prep_f32(const double *__restrict__ x, int n, int npad, double L, double whi, double wlo,
                              float *__restrict__ soa, int32_t *err)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= npad) return;
    float q[3] = {1.0e30f, 1.0e30f, 1.0e30f};
    if (i < n) {
        const double px = x[3 * (int64_t)i], py = x[3 * (int64_t)i + 1], pz = x[3 * (int64_t)i + 2];
        if (!(finite64(px) && finite64(py) && finite64(pz))) atomicOr(err, LJ_ERRBIT_NONFINITE);
        const double h = 0.5 * L;
        q[0] = (float)(lj_wrap_fast(px, L, whi, wlo) - h);
        q[1] = (float)(lj_wrap_fast(py, L, whi, wlo) - h);
        q[2] = (float)(lj_wrap_fast(pz, L, whi, wlo) - h);
    }
    soa[i] = q[0];
    soa[(size_t)npad + i] = q[1];
    soa[2 * (size_t)npad + i] = q[2];
    const bool real = i < n;
    const bool fin = !real || (fabsf(q[0]) < 1.0e30f && fabsf(q[1]) < 1.0e30f && fabsf(q[2]) < 1.0e30f);
    const bool all = __all_sync(0xffffffffu, fin);
    float c[3], h[3];
#pragma unroll
    for (int d = 0; d < 3; d++) {
        float lo = real && fin ? q[d] : 3.0e38f, hi = real && fin ? q[d] : -3.0e38f;
        for (int o = 16; o > 0; o >>= 1) {
            lo = fminf(lo, __shfl_xor_sync(0xffffffffu, lo, o));
            hi = fmaxf(hi, __shfl_xor_sync(0xffffffffu, hi, o));
        }
        c[d] = all ? 0.5f * (lo + hi) : 0.0f;
        h[d] = all ? 0.5f * (hi - lo) + 1.0e-6f * (float)L : 1.0e30f;
    }
    if ((i & 31) == 0) {
        float4 *box = reinterpret_cast<float4 *>(soa + 3 * (size_t)npad) + 2 * (i >> 5);
        box[0] = make_float4(c[0], c[1], c[2], 0.0f);
        box[1] = make_float4(h[0], h[1], h[2], 0.0f);
    }
}

// A lower bound of the squared minimum-image distance between the particles
// of two boxes.
__device__ __forceinline__ float n2_gap2(float4 ca, float4 ha, float4 cb, float4 hb, float L)
{
    const float dx = fabsf(ca.x - cb.x), dy = fabsf(ca.y - cb.y), dz = fabsf(ca.z - cb.z);
    const float gx = fmaxf(fminf(dx, L - dx) - (ha.x + hb.x), 0.0f);
    const float gy = fmaxf(fminf(dy, L - dy) - (ha.y + hb.y), 0.0f);
    const float gz = fmaxf(fminf(dz, L - dz) - (ha.z + hb.z), 0.0f);
    return gx * gx + gy * gy + gz * gz;
}

template <typename V>
__device__ __forceinline__ V load_shared(const V *p)
{
    return *p;
}

template <typename T>
__device__ __forceinline__ T rint_t(T v)
{
    if constexpr (sizeof(T) == 4) {
        return rintf(v);
    } else {
        return rint(v);
    }
}

// part[split * n + i] = (sum over this split's j of the pair force on i,
// half the pair energies of i); epart[cta] = (sum of half energies, half
// virials) of this CTA's particles, FP64.
template <typename T, int MODE, bool ENERGY>
__global__ void __launch_bounds__(kN2Threads) k_n2_force(N2Params p, const typename Vec4<T>::type *__restrict__ pos,
                                                         typename Vec4<T>::type *__restrict__ part,
                                                         double *__restrict__ epart, int32_t *err)
{
    using V = typename Vec4<T>::type;
    extern __shared__ __align__(128) unsigned char n2_smem[];
    V *buf0 = reinterpret_cast<V *>(n2_smem);
    V *buf1 = buf0 + kN2Tile;
    uint64_t *bars = reinterpret_cast<uint64_t *>(buf1 + kN2Tile);
    __shared__ int s_abort;
    __shared__ double red[2 * (kN2Threads / 32)];

    const int i = blockIdx.x * kN2Threads + threadIdx.x;
    const bool vi = i < p.n;
    V pi;
    if (vi) {
        pi = pos[i];
    } else {
        pi.x = pi.y = pi.z = (T)0;
        pi.w = (T)0;
    }
    const int split = blockIdx.y, nsplit = gridDim.y;
    const int mine = p.ntiles > split ? (p.ntiles - split + nsplit - 1) / nsplit : 0;
    auto issue = [&](int k, V *dst, uint64_t *bar) {
        const int t = split + k * nsplit;
        const int cnt = min(kN2Tile, p.n - t * kN2Tile);
        mbar_arrive_expect_tx(bar, (uint32_t)(cnt * sizeof(V)));
        bulk_g2s(dst, pos + (size_t)t * kN2Tile, (uint32_t)(cnt * sizeof(V)), bar);
    };
    if (threadIdx.x == 0) {
        s_abort = 0;
        mbar_init(&bars[0], 1);
        mbar_init(&bars[1], 1);
        fence_mbar_init();
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        if (mine > 0) issue(0, buf0, &bars[0]);
        if (mine > 1) issue(1, buf1, &bars[1]);
    }
    const Coef<T> kc(p);
    const T L = (T)p.L, invL = (T)p.invL;
    T fx = 0, fy = 0, fz = 0, e = 0, w = 0;
    int k = 0;
    for (; k < mine; k++) {
        const int b = k & 1;
        V *buf = b ? buf1 : buf0;
        const int t = split + k * nsplit;
        const int cnt = min(kN2Tile, p.n - t * kN2Tile);
        if (!mbar_wait_bounded(&bars[b], (uint32_t)((k >> 1) & 1), err)) s_abort = 1;
        __syncthreads();
        if (s_abort) break;
        for (int j = 0; j < cnt; j++) {
            const V q = load_shared(buf + j);
            T dx = pi.x - q.x, dy = pi.y - q.y, dz = pi.z - q.z;
            dx -= L * rint_t(dx * invL);
            dy -= L * rint_t(dy * invL);
            dz -= L * rint_t(dz * invL);
            pair_accum<T, MODE, ENERGY>(dx, dy, dz, kc, fx, fy, fz, e, w);
        }
        __syncthreads();   // everyone is done with buffer b
        if (threadIdx.x == 0 && k + 2 < mine) {
            fence_proxy_async_smem();
            issue(k + 2, buf, &bars[b]);
        }
    }
    if (s_abort && threadIdx.x == 0) {
        // a wait gave up: wait once more (bounded) for the copies that may
        // still be in flight, tile k and tile k + 1, before the CTA's shared
        // memory goes away
        mbar_wait_bounded(&bars[k & 1], (uint32_t)((k >> 1) & 1), err);
        if (k + 1 < mine) mbar_wait_bounded(&bars[(k + 1) & 1], (uint32_t)(((k + 1) >> 1) & 1), err);
    }
    if (vi) {
        V o;
        o.x = fx;
        o.y = fy;
        o.z = fz;
        o.w = ENERGY ? (T)0.5 * e : (T)0;
        part[(size_t)split * p.n + i] = o;
    }
    if constexpr (ENERGY) {
        double de = vi ? 0.5 * (double)e : 0.0, dw = vi ? 0.5 * (double)w : 0.0;
        for (int o = 16; o > 0; o >>= 1) {
            de += __shfl_xor_sync(0xffffffffu, de, o);
            dw += __shfl_xor_sync(0xffffffffu, dw, o);
        }
        const int warp = threadIdx.x >> 5;
        if ((threadIdx.x & 31) == 0) {
            red[2 * warp] = de;
            red[2 * warp + 1] = dw;
        }
        __syncthreads();
        if (threadIdx.x == 0) {
            double es = 0.0, ws = 0.0;
            for (int q = 0; q < kN2Threads / 32; q++) {
                es += red[2 * q];
                ws += red[2 * q + 1];
            }
            const size_t cta = (size_t)blockIdx.y * gridDim.x + blockIdx.x;
            epart[2 * cta] = es;
            epart[2 * cta + 1] = ws;
        }
    }
}

// The squared minimum-image distances of two j to one i, for the cutoff
// test only: per component min(|d|, L - |d|), the magnitude of d - L rint(d /
// L) for every pair within L / 2, bit for bit, without the rounding
// instruction (a quarter-rate one) and the two multiplications around it.
__device__ __forceinline__ float2 n2_r2(float2 xi, float2 yi, float2 zi, float2 xj, float2 yj, float2 zj, float L)
{
    const float2 m1 = make_float2(-1.0f, -1.0f);
    float2 dx = __ffma2_rn(xj, m1, xi);
    float2 dy = __ffma2_rn(yj, m1, yi);
    float2 dz = __ffma2_rn(zj, m1, zi);
    dx.x = fminf(fabsf(dx.x), L - fabsf(dx.x));
    dx.y = fminf(fabsf(dx.y), L - fabsf(dx.y));
    dy.x = fminf(fabsf(dy.x), L - fabsf(dy.x));
    dy.y = fminf(fabsf(dy.y), L - fabsf(dy.y));
    dz.x = fminf(fabsf(dz.x), L - fabsf(dz.x));
    dz.y = fminf(fabsf(dz.y), L - fabsf(dz.y));
    float2 r2 = __fmul2_rn(dx, dx);
    r2 = __ffma2_rn(dy, dy, r2);
    return __ffma2_rn(dz, dz, r2);
}

// FP32 form of k_n2_force.  Only some 55 of the n - 1 pairs of a particle
// are within rc, so all pairs go through the distance test alone and the
// few that pass through the pair term: a thread takes its particle against
// 32 j at a time, collects the passing ones in a bit mask (the sign of r^2 -
// rc^2 (1 + 1e-5), shifted in), and then evaluates those with the exact
// cutoff and minimum image of pair_accum, in the order of j.  Bound by
// instruction issue: ~13 instructions per pair (six for the three
// components' images, 1.5 each for r^2 and the mask) against ~30 with three
// quarter-rate roundings before.  At 8,788
// particles a call took 137 us, then 46.
// A warp's 32 particles leave out a group of 32 j whose bounding box is
// further than rc from theirs: no pair of the two is in range, so the sums
// stay the same bits.  Particles that are stored near their neighbours (grown
// on a lattice, read from a file written by cells) leave out most groups (46
// -> 27 us, 120 -> 40 at 16,000); where the order is random the boxes fill the
// system and the test's cost does not show (46 us).
template <int MODE, bool ENERGY>
__global__ void __launch_bounds__(kN2Threads) k_n2_force_f32(N2Params p, int npad, int tile, const float *soa,
                                                             float4 *part, double *epart,
                                                             int32_t *err)
{
    __shared__ __align__(128) float sm[2][3][kN2TileF];
    __shared__ __align__(8) uint64_t bars[2];
    __shared__ int s_abort;
    __shared__ double red[2 * (kN2Threads / 32)];
    pdl_wait();
    const int i = blockIdx.x * kN2Threads + threadIdx.x;
    const bool vi = i < p.n;
    const float pix = soa[vi ? i : 0], piy = soa[(size_t)npad + (vi ? i : 0)], piz = soa[2 * (size_t)npad + (vi ? i : 0)];
    const int split = blockIdx.y, nsplit = gridDim.y;
    const int mine = p.ntiles > split ? (p.ntiles - split + nsplit - 1) / nsplit : 0;
    auto issue = [&](int k) {
        const int t0 = (split + k * nsplit) * tile;
        const uint32_t bytes = (uint32_t)min(tile, npad - t0) * 4u;   // a multiple of 128
        const int b = k & 1;
        mbar_arrive_expect_tx(&bars[b], 3 * bytes);
        for (int d = 0; d < 3; d++) bulk_g2s(sm[b][d], soa + (size_t)d * npad + t0, bytes, &bars[b]);
    };
    if (threadIdx.x == 0) {
        s_abort = 0;
        mbar_init(&bars[0], 1);
        mbar_init(&bars[1], 1);
        fence_mbar_init();
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        if (mine > 0) issue(0);
        if (mine > 1) issue(1);
    }
    const Coef<float> kc(p);
    const float L = (float)p.L, invL = (float)p.invL;
    const float thr = -(float)p.rc2 * 1.00001f;
    const float2 xi = make_float2(pix, pix), yi = make_float2(piy, piy), zi = make_float2(piz, piz);
    const float4 *box = reinterpret_cast<const float4 *>(soa + 3 * (size_t)npad);
    const int lane = threadIdx.x & 31, gi = i >> 5;
    const bool wi = 32 * gi < p.n;   // the warp has particles
    const float4 ci = box[wi ? 2 * gi : 0], hi = box[wi ? 2 * gi + 1 : 1];
    const float far2 = (float)p.rc2 * 1.0001f;
    float fx = 0, fy = 0, fz = 0, e = 0, w = 0;
    int k = 0;
    for (; k < mine; k++) {
        const int b = k & 1;
        const int cnt = min(tile, npad - (split + k * nsplit) * tile);   // a multiple of 32
        bool near = false;   // group lane of the tile (cnt / 32 of at most 4)
        if (wi && lane < cnt / 32) {
            const int gj = (split + k * nsplit) * (tile / 32) + lane;
            near = n2_gap2(ci, hi, box[2 * gj], box[2 * gj + 1], L) < far2;
        }
        const unsigned live = __ballot_sync(0xffffffffu, near);
        if (!mbar_wait_bounded(&bars[b], (uint32_t)((k >> 1) & 1), err)) s_abort = 1;
        __syncthreads();
        if (s_abort) break;
        const float *X = sm[b][0], *Y = sm[b][1], *Z = sm[b][2];
        for (int j0 = 0; j0 < cnt; j0 += 32) {
            if (!((live >> (j0 / 32)) & 1u)) continue;
            unsigned mask = 0;
#pragma unroll
            for (int u = 0; u < 32; u += 4) {
                const float4 qx = *reinterpret_cast<const float4 *>(X + j0 + u);
                const float4 qy = *reinterpret_cast<const float4 *>(Y + j0 + u);
                const float4 qz = *reinterpret_cast<const float4 *>(Z + j0 + u);
                const float2 t = make_float2(thr, thr);
                const float2 a = __fadd2_rn(n2_r2(xi, yi, zi, make_float2(qx.x, qx.y), make_float2(qy.x, qy.y),
                                                  make_float2(qz.x, qz.y), L), t);
                const float2 c = __fadd2_rn(n2_r2(xi, yi, zi, make_float2(qx.z, qx.w), make_float2(qy.z, qy.w),
                                                  make_float2(qz.z, qz.w), L), t);
                mask = __funnelshift_l(__float_as_uint(a.x), mask, 1);   // j0 ends in the top bit
                mask = __funnelshift_l(__float_as_uint(a.y), mask, 1);
                mask = __funnelshift_l(__float_as_uint(c.x), mask, 1);
                mask = __funnelshift_l(__float_as_uint(c.y), mask, 1);
            }
            while (mask) {
                const int u = __clz((int)mask);
                mask &= ~(0x80000000u >> u);
                float dx = pix - X[j0 + u], dy = piy - Y[j0 + u], dz = piz - Z[j0 + u];
                dx -= L * rint_t(dx * invL);
                dy -= L * rint_t(dy * invL);
                dz -= L * rint_t(dz * invL);
                pair_accum<float, MODE, ENERGY>(dx, dy, dz, kc, fx, fy, fz, e, w);
            }
        }
        __syncthreads();   // everyone is done with buffer b
        if (threadIdx.x == 0 && k + 2 < mine) {
            fence_proxy_async_smem();
            issue(k + 2);
        }
    }
    if (s_abort && threadIdx.x == 0) {   // as k_n2_force: the copies that may still be in flight
        mbar_wait_bounded(&bars[k & 1], (uint32_t)((k >> 1) & 1), err);
        if (k + 1 < mine) mbar_wait_bounded(&bars[(k + 1) & 1], (uint32_t)(((k + 1) >> 1) & 1), err);
    }
    if (vi) part[(size_t)split * p.n + i] = make_float4(fx, fy, fz, ENERGY ? 0.5f * e : 0.0f);
    if constexpr (ENERGY) {
        double de = vi ? 0.5 * (double)e : 0.0, dw = vi ? 0.5 * (double)w : 0.0;
        for (int o = 16; o > 0; o >>= 1) {
            de += __shfl_xor_sync(0xffffffffu, de, o);
            dw += __shfl_xor_sync(0xffffffffu, dw, o);
        }
        const int warp = threadIdx.x >> 5;
        if ((threadIdx.x & 31) == 0) {
            red[2 * warp] = de;
            red[2 * warp + 1] = dw;
        }
        __syncthreads();
        if (threadIdx.x == 0) {
            double es = 0.0, ws = 0.0;
            for (int q = 0; q < kN2Threads / 32; q++) {
                es += red[2 * q];
                ws += red[2 * q + 1];
            }
            const size_t cta = (size_t)blockIdx.y * gridDim.x + blockIdx.x;
            epart[2 * cta] = es;
            epart[2 * cta + 1] = ws;
        }
    }
}

// f[i] = sum over splits s = 0 .. nsplit-1 (in order) of part[s * n + i].
// Latency, not bytes: small blocks, to reach more SMs, and the loads of
// several splits in flight (8,788 particles, 35 splits: 28.7 -> 27.3 us a call
// against blocks of 256; one load at a time 32.7).
constexpr int kN2SumThreads = 64;

template <typename T>
__global__ void __launch_bounds__(kN2SumThreads) k_n2_sum(const typename Vec4<T>::type *part, int nsplit, int n,
                         typename Vec4<T>::type *f)
{
    pdl_wait();
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    typename Vec4<T>::type a = part[i];
#pragma unroll 8
    for (int s = 1; s < nsplit; s++) {
        const typename Vec4<T>::type b = part[(size_t)s * n + i];
        a.x += b.x;
        a.y += b.y;
        a.z += b.z;
        a.w += b.w;
    }
    f[i] = a;
}

// scalars[0..1] = sums of the (energy, virial) pairs of epart, fixed order.
__global__ void k_n2_energy(const double *__restrict__ epart, int m, double *__restrict__ scalars)
{
    __shared__ double se[256], sw[256];
    double e = 0.0, w = 0.0;
    for (int k = threadIdx.x; k < m; k += 256) {
        e += epart[2 * k];
        w += epart[2 * k + 1];
    }
    se[threadIdx.x] = e;
    sw[threadIdx.x] = w;
    __syncthreads();
    for (int s = 128; s > 0; s >>= 1) {
        if (threadIdx.x < s) {
            se[threadIdx.x] += se[threadIdx.x + s];
            sw[threadIdx.x] += sw[threadIdx.x + s];
        }
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        scalars[0] = se[0];
        scalars[1] = sw[0];
    }
}

void *n2_kernel(bool fp64, int mode, bool energy)
{
    switch ((fp64 ? 6 : 0) + mode * 2 + (energy ? 1 : 0)) {
        case 0: return (void *)k_n2_force_f32<0, false>;
        case 1: return (void *)k_n2_force_f32<0, true>;
        case 2: return (void *)k_n2_force_f32<1, false>;
        case 3: return (void *)k_n2_force_f32<1, true>;
        case 4: return (void *)k_n2_force_f32<2, false>;
        case 5: return (void *)k_n2_force_f32<2, true>;
        case 6: return (void *)k_n2_force<double, 0, false>;
        case 7: return (void *)k_n2_force<double, 0, true>;
        case 8: return (void *)k_n2_force<double, 1, false>;
        case 9: return (void *)k_n2_force<double, 1, true>;
        case 10: return (void *)k_n2_force<double, 2, false>;
        default: return (void *)k_n2_force<double, 2, true>;
    }
}

template <typename T>
cudaError_t run_n2(lj_ctx *c, const double *x, void *f, bool energy)
{
    using V = typename Vec4<T>::type;
    const int n = (int)c->p.n;
    const int iblocks = (n + kN2Threads - 1) / kN2Threads;
    constexpr bool fp64 = sizeof(T) == 8;
    // FP32: smaller tiles while they give fewer than 8 CTAs per SM, and j
    // splits up to 16 per SM: with 2 per SM (of 4 warps) the SMs were unevenly
    // loaded and the distance tests' latency showed.
    int tile = fp64 ? kN2Tile : kN2TileF;
    while (!fp64 && tile > 32 && (int64_t)iblocks * ((n + tile - 1) / tile) < 8 * c->nsm) tile /= 2;
    int ntiles = (n + tile - 1) / tile;
    int nsplit = ((fp64 ? 2 : 16) * c->nsm + iblocks - 1) / iblocks;
    nsplit = nsplit < 1 ? 1 : (nsplit > ntiles ? ntiles : nsplit);
    nsplit = nsplit > 64 ? 64 : nsplit;
    int npad = (n + 31) & ~31;
    // scratch: sorted-free positions, per-split partials, per-CTA energy pairs
    const size_t need = (size_t)npad * sizeof(V) * (size_t)(1 + nsplit) + 2 * sizeof(double) * (size_t)iblocks * nsplit;
    if (need > c->n2_bytes) {
        cudaFree(c->n2_scratch);
        c->n2_scratch = nullptr;
        c->n2_bytes = 0;
        cudaError_t e = cudaMalloc(&c->n2_scratch, need);
        if (e != cudaSuccess) return e;
        c->n2_bytes = need;
    }
    V *pos = reinterpret_cast<V *>(c->n2_scratch);
    V *part = pos + npad;
    double *epart = reinterpret_cast<double *>(part + (size_t)n * nsplit);
    V *fo = reinterpret_cast<V *>(f);
    if constexpr (fp64)
        k_n2_prep<T><<<(n + 255) / 256, 256, 0, c->stream>>>(x, n, c->p.box, c->wrap_hi, c->wrap_lo, pos, c->err);
    else   // three arrays of npad floats
        k_n2_prep_f32<<<(npad + 255) / 256, 256, 0, c->stream>>>(x, n, npad, c->p.box, c->wrap_hi, c->wrap_lo,
                                                                 (float *)pos, c->err);
    N2Params p;
    p.n = n;
    p.ntiles = ntiles;
    p.L = c->p.box;
    p.invL = 1.0 / c->p.box;
    const double eps = c->p.eps, sg = c->p.sigma, rc = c->p.rc;
    const double s6 = sg * sg * sg * sg * sg * sg, s12 = s6 * s6;
    const double rci2 = 1.0 / (rc * rc), rci6 = rci2 * rci2 * rci2;
    p.rc2 = rc * rc;
    p.rc = rc;
    p.a12 = 48.0 * eps * s12;
    p.b6 = 24.0 * eps * s6;
    p.c12 = 4.0 * eps * s12;
    p.c6 = 4.0 * eps * s6;
    p.uc = rci6 * (p.c12 * rci6 - p.c6);
    p.fc = rc * rci2 * rci6 * (p.a12 * rci6 - p.b6);
    void *kern = n2_kernel(fp64, c->p.shift_mode, energy);
    V *dst = nsplit == 1 ? fo : part;
    int32_t *err = c->err;
    cudaError_t e;
    if constexpr (fp64) {
        const int smem = 2 * kN2Tile * (int)sizeof(V) + 2 * (int)sizeof(uint64_t);
        if ((e = raise_dyn_smem(kern, smem)) != cudaSuccess) return e;
        void *args[] = {&p, (void *)&pos, (void *)&dst, (void *)&epart, (void *)&err};
        e = cudaLaunchKernel(kern, dim3(iblocks, nsplit), dim3(kN2Threads), args, smem, c->stream);
    } else {
        void *args[] = {&p, &npad, &tile, (void *)&pos, (void *)&dst, (void *)&epart, (void *)&err};
        e = launch_pdl(kern, dim3(iblocks, nsplit), kN2Threads, args, 0, c->stream, true);
    }
    if (e != cudaSuccess) return e;
    c->kernel_launches += 2;
    if (nsplit > 1) {
        int np = nsplit, nn = n;
        void *args[] = {(void *)&part, &np, &nn, (void *)&fo};
        e = launch_pdl((const void *)k_n2_sum<T>, dim3((n + kN2SumThreads - 1) / kN2SumThreads), kN2SumThreads, args, 0,
                       c->stream, !fp64);
        if (e != cudaSuccess) return e;
        c->kernel_launches++;
    }
    if (energy) {
        k_n2_energy<<<1, 256, 0, c->stream>>>(epart, iblocks * nsplit, c->scalars);
        c->kernel_launches++;
    }
    return cudaGetLastError();
}

}  // namespace

cudaError_t launch_forces_n2(lj_ctx *c, const double *x, void *f, bool energy)
{
    if (c->p.n == 0) return cudaSuccess;
    if (c->p.precision == LJ_PREC_FP64) return run_n2<double>(c, x, f, energy);
    return run_n2<float>(c, x, f, energy);
}
