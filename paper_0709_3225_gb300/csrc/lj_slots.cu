// Slotted cells (lj_slots.cuh): set-up, the binning kernels, and the
// conversion to the sorted lists that lj_get_cells returns.
#include <math.h>

#include "lj_slots.cuh"

namespace {

constexpr size_t kSlotsTogether = (size_t)16 << 20;
constexpr int kSlotMax = 32;   // the pair-once kernels' limit on home particles

// Bin given positions (wrapped here), zero the array the force (VJP) kernel
// adds into, and copy the cotangents, if any, beside the positions.
__global__ void __launch_bounds__(256) k_bin_slots(SlotBin b, const double *__restrict__ x, int n,
                                                   float4 *__restrict__ zero, const double *__restrict__ g,
                                                   float4 *__restrict__ g4, int32_t *__restrict__ err)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i == 0) *b.work = 0u;
    const bool valid = i < n;
    double px = 0.0, py = 0.0, pz = 0.0;
    if (valid) {
        const int64_t o = 3 * (int64_t)i;
        px = x[o];
        py = x[o + 1];
        pz = x[o + 2];
        zero[i] = make_float4(0.f, 0.f, 0.f, 0.f);
        px = lj_wrap_fast(px, b.L, b.whi, b.wlo);
        py = lj_wrap_fast(py, b.L, b.whi, b.wlo);
        pz = lj_wrap_fast(pz, b.L, b.whi, b.wlo);
    }
    const int slot = slot_place(b, valid, i, px, py, pz, err);
    if (g && slot >= 0) {
        const int64_t o = 3 * (int64_t)i;
        g4[slot] = make_float4((float)g[o], (float)g[o + 1], (float)g[o + 2], 0.f);
    }
}

// The velocity-Verlet update of k_kick_drift_bin (nkick half kicks, drift,
// wrap; the same FP64 operations) with the slotted binning: x, v, f are read
// and written once (f zeroed for the force kernel, which adds into it) and
// the position goes to its slot.  Bound by HBM: 144 bytes per particle
// (x, v 96, f 32, slot 16), 99 us at 4M particles (5.3 TB/s of DRAM traffic).
// It takes the place of three kernels and a memset: k_kick_drift_bin (98 us),
// the scan of the counts (11 us, and 10 us of latency at 131,072 particles
// too), k_scatter (49 us) and the zeroing of f.  Per step: 815 -> 763 us at
// 4M, 57 -> 40 at 131,072, 26 -> 16.5 at 2,048.
// xo: where the new positions go, x itself or the next state of a trajectory.
__global__ void __launch_bounds__(256) k_kick_drift_slots(SlotBin b, const double *x, double *xo,
                                                          double *v, float4 *f, int i_begin,
                                                          int n, double hk, double dt, int32_t *err)
{
    pdl_wait();
    // the last particles first: what this kernel wrote last, and the force
    // kernel reads (adds into) first, is then still in L2
    const int t = (gridDim.x - 1 - blockIdx.x) * blockDim.x + threadIdx.x;
    if (t == 0) *b.work = 0u;
    const int i = i_begin + t;
    const bool valid = i < n;
    double px = 0.0, py = 0.0, pz = 0.0;
    if (valid) {
        const int64_t o = 3 * (int64_t)i;
        const float4 q = f[i];
        const double v0 = v[o], v1 = v[o + 1], v2 = v[o + 2];
        const double x0 = x[o], x1 = x[o + 1], x2 = x[o + 2];
        f[i] = make_float4(0.f, 0.f, 0.f, 0.f);
        const double vx = __fma_rn(hk, f64_of_f32(q.x), v0);
        const double vy = __fma_rn(hk, f64_of_f32(q.y), v1);
        const double vz = __fma_rn(hk, f64_of_f32(q.z), v2);
        px = lj_wrap_fast(__fma_rn(dt, vx, x0), b.L, b.whi, b.wlo);
        py = lj_wrap_fast(__fma_rn(dt, vy, x1), b.L, b.whi, b.wlo);
        pz = lj_wrap_fast(__fma_rn(dt, vz, x2), b.L, b.whi, b.wlo);
        v[o] = vx;
        v[o + 1] = vy;
        v[o + 2] = vz;
        xo[o] = px;
        xo[o + 1] = py;
        xo[o + 2] = pz;
    }
    slot_place(b, valid, i, px, py, pz, err);
}

// lj_step_host on pinned arrays: the first update reads x, v, f where they
// are, over the link, and the last half kick writes v and f there (small
// systems' x too).  The link is the bound, 205 GB/s in and 190 out here, by
// copy engine or by loads alike; twelve chunked copies and an update per chunk
// took 193 us for the 32 MB of 500,009 particles (156 at the link's rate), and
// the closing kick ran before its copies: a call of one step there 437 -> 369
// us.  The (n, 3) arrays go through shared memory, so that the link sees
// whole 16-byte accesses in order.
constexpr int kHostThreads = 256;

// The block's 3 kHostThreads doubles of an (n, 3) array, from element e0.
__device__ __forceinline__ void host_rows_in(const double *__restrict__ src, double2 *s, int64_t e0, int64_t end)
{
    for (int k = threadIdx.x; k < 3 * kHostThreads / 2; k += kHostThreads) {
        const int64_t e = e0 + 2 * k;
        double2 q = make_double2(0.0, 0.0);
        if (e + 1 < end) q = __ldg(reinterpret_cast<const double2 *>(src + e));
        else if (e < end) q.x = src[e];
        s[k] = q;
    }
}

__device__ __forceinline__ void host_rows_out(double *__restrict__ dst, const double2 *s, int64_t e0, int64_t end)
{
    for (int k = threadIdx.x; k < 3 * kHostThreads / 2; k += kHostThreads) {
        const int64_t e = e0 + 2 * k;
        if (e + 1 < end) *reinterpret_cast<double2 *>(dst + e) = s[k];
        else if (e < end) dst[e] = s[k].x;
    }
}

// k_kick_drift_slots from the host arrays hx, hv, hf to x, v and f (zeroed).
__global__ void __launch_bounds__(kHostThreads) k_host_in(SlotBin b, const double *__restrict__ hx,
                                                          const double *__restrict__ hv, const float4 *__restrict__ hf,
                                                          double *__restrict__ x, double *__restrict__ v,
                                                          float4 *__restrict__ f, int n, double hk, double dt,
                                                          int32_t *__restrict__ err)
{
    __shared__ double2 sx[3 * kHostThreads / 2], sv[3 * kHostThreads / 2];
    const int64_t i0 = (int64_t)blockIdx.x * kHostThreads;
    const int i = (int)i0 + threadIdx.x;
    if (i == 0) *b.work = 0u;
    const bool valid = i < n;
    float4 q = make_float4(0.f, 0.f, 0.f, 0.f);
    if (valid) q = __ldg(hf + i);
    host_rows_in(hx, sx, 3 * i0, 3 * (int64_t)n);
    host_rows_in(hv, sv, 3 * i0, 3 * (int64_t)n);
    __syncthreads();
    double *px3 = reinterpret_cast<double *>(sx) + 3 * threadIdx.x;
    double *pv3 = reinterpret_cast<double *>(sv) + 3 * threadIdx.x;
    double px = 0.0, py = 0.0, pz = 0.0;
    if (valid) {
        f[i] = make_float4(0.f, 0.f, 0.f, 0.f);
        const double vx = __fma_rn(hk, f64_of_f32(q.x), pv3[0]);
        const double vy = __fma_rn(hk, f64_of_f32(q.y), pv3[1]);
        const double vz = __fma_rn(hk, f64_of_f32(q.z), pv3[2]);
        px = lj_wrap_fast(__fma_rn(dt, vx, px3[0]), b.L, b.whi, b.wlo);
        py = lj_wrap_fast(__fma_rn(dt, vy, px3[1]), b.L, b.whi, b.wlo);
        pz = lj_wrap_fast(__fma_rn(dt, vz, px3[2]), b.L, b.whi, b.wlo);
        const int64_t o = 3 * (int64_t)i;
        v[o] = vx;
        v[o + 1] = vy;
        v[o + 2] = vz;
        x[o] = px;
        x[o + 1] = py;
        x[o + 2] = pz;
    }
    slot_place(b, valid, i, px, py, pz, err);
}

// The closing half kick v += h f into the host arrays, with f (and x, if hx)
// and the latched errors.
__global__ void __launch_bounds__(kHostThreads) k_host_out(const double *x, const double *v,
                                                           const float4 *f, int n, double h,
                                                           double *hx, double *hv,
                                                           float4 *hf, const int32_t *err,
                                                           int32_t *host_err)
{
    __shared__ double2 s[3 * kHostThreads / 2];
    pdl_wait();
    const int64_t i0 = (int64_t)blockIdx.x * kHostThreads, end = 3 * (int64_t)n;
    const int i = (int)i0 + threadIdx.x;
    if (i == 0) *host_err = *err;
    if (i < n) {
        const int64_t o = 3 * (int64_t)i;
        const float4 q = f[i];
        double *d = reinterpret_cast<double *>(s) + 3 * threadIdx.x;
        d[0] = __fma_rn(h, f64_of_f32(q.x), v[o]);
        d[1] = __fma_rn(h, f64_of_f32(q.y), v[o + 1]);
        d[2] = __fma_rn(h, f64_of_f32(q.z), v[o + 2]);
        hf[i] = q;
    }
    __syncthreads();
    host_rows_out(hv, s, 3 * i0, end);
    if (hx) {
        for (int k = threadIdx.x; k < 3 * kHostThreads; k += kHostThreads)
            if (3 * i0 + k < end) hx[3 * i0 + k] = x[3 * i0 + k];
    }
}

// The FP64 forms (lj_force_fx.cu): fixed-point coordinates; f holds the
// forces of the pairs taken in FP64 and acc those of all others.  Their three
// sums and the low part make one integer in units of q / 256, exactly, which
// is then rounded once.
__device__ __forceinline__ double fx_sum(long long r, long long m, long long f, unsigned long long lo, double q)
{
    const __int128 t = ((__int128)r << 8) + ((__int128)m << 3) + f + (long long)(lo & ((1ull << kFxLow) - 1));
    const long long v = (long long)t;
    if (t == v) return (double)v * (q * 0x1p-8);
    return (double)(long long)(t >> 8) * q;
}

__device__ __forceinline__ void fx_force(const double4_16a *f, const longlong2 *acc, int i, double q, double &fx,
                                         double &fy, double &fz)
{
    const double4_16a p = f[i];
    const longlong2 *o = acc + kFxAcc / 2 * (int64_t)i;
    const longlong2 a = o[0], b = o[1], c = o[2], d = o[3], e = o[4];
    const unsigned long long lo = (unsigned long long)e.y;
    fx = fx_sum(a.x, b.y, d.x, lo, q) + p.x;
    fy = fx_sum(a.y, c.x, d.y, lo >> kFxLow, q) + p.y;
    fz = fx_sum(b.x, c.y, e.x, lo >> (2 * kFxLow), q) + p.z;
}

__device__ __forceinline__ void fx_zero(double4_16a *f, longlong2 *acc, int i)
{
    double4_16a z;
    z.x = z.y = z.z = z.w = 0.0;
    f[i] = z;
#pragma unroll
    for (int u = 0; u < kFxAcc / 2; u++) acc[kFxAcc / 2 * (int64_t)i + u] = make_longlong2(0, 0);
}

__global__ void __launch_bounds__(256) k_bin_fx(SlotBin b, const double *__restrict__ x, int n, double4_16a *__restrict__ f,
                                                longlong2 *__restrict__ acc, int32_t *__restrict__ err)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i == 0) *b.work = 0u;
    const bool valid = i < n;
    double px = 0.0, py = 0.0, pz = 0.0;
    if (valid) {
        const int64_t o = 3 * (int64_t)i;
        px = lj_wrap_fast(x[o], b.L, b.whi, b.wlo);
        py = lj_wrap_fast(x[o + 1], b.L, b.whi, b.wlo);
        pz = lj_wrap_fast(x[o + 2], b.L, b.whi, b.wlo);
        fx_zero(f, acc, i);
    }
    slot_place<true>(b, valid, i, px, py, pz, err);
}

// k_kick_drift_slots in FP64; with_acc: f alone is not yet the force.
__global__ void __launch_bounds__(256) k_kick_drift_fx(SlotBin b, double *x, double *v,
                                                       double4_16a *f, longlong2 *acc,
                                                       int with_acc, double scale, int i_begin, int n, double hk,
                                                       double dt, int32_t *err)
{
    pdl_wait();
    const int t = (gridDim.x - 1 - blockIdx.x) * blockDim.x + threadIdx.x;
    if (t == 0) *b.work = 0u;
    const int i = i_begin + t;
    const bool valid = i < n;
    double px = 0.0, py = 0.0, pz = 0.0;
    if (valid) {
        const int64_t o = 3 * (int64_t)i;
        double fx, fy, fz;
        if (with_acc) {
            fx_force(f, acc, i, scale, fx, fy, fz);
        } else {
            const double4_16a q = f[i];
            fx = q.x;
            fy = q.y;
            fz = q.z;
        }
        fx_zero(f, acc, i);
        const double vx = __fma_rn(hk, fx, v[o]);
        const double vy = __fma_rn(hk, fy, v[o + 1]);
        const double vz = __fma_rn(hk, fz, v[o + 2]);
        px = lj_wrap_fast(__fma_rn(dt, vx, x[o]), b.L, b.whi, b.wlo);
        py = lj_wrap_fast(__fma_rn(dt, vy, x[o + 1]), b.L, b.whi, b.wlo);
        pz = lj_wrap_fast(__fma_rn(dt, vz, x[o + 2]), b.L, b.whi, b.wlo);
        v[o] = vx;
        v[o + 1] = vy;
        v[o + 2] = vz;
        x[o] = px;
        x[o + 1] = py;
        x[o + 2] = pz;
    }
    slot_place<true>(b, valid, i, px, py, pz, err);
}

// f := the force; with v also the closing half kick v += h f.
__global__ void __launch_bounds__(256) k_fx_finish(double *v, double4_16a *f,
                                                   const longlong2 *acc, int n, double scale, double h)
{
    pdl_wait();
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    double4_16a q;
    fx_force(f, acc, i, scale, q.x, q.y, q.z);
    q.w = 0.0;
    f[i] = q;
    if (v) {
        const int64_t o = 3 * (int64_t)i;
        v[o] = __fma_rn(h, q.x, v[o]);
        v[o + 1] = __fma_rn(h, q.y, v[o + 1]);
        v[o + 2] = __fma_rn(h, q.z, v[o + 2]);
    }
}

// Particle index of a slot.
template <bool FX>
__device__ __forceinline__ int slot_index(const void *pos, int64_t s)
{
    if constexpr (FX) return (int)reinterpret_cast<const longlong2 *>(pos)[2 * s + 1].y;
    return __float_as_int(reinterpret_cast<const float4 *>(pos)[s].w);
}

// The count buffers and which of them the last force launch read; its value
// -1: the sorted lists are newer and stay as they are.
struct SlotLast {
    const int2 *cellq[2];
    const int *last;
};

// Counts of every cell (the extra one included) for the scan of
// launch_slots_to_lists; cell_of starts as the extra cell everywhere.
__global__ void k_slot_counts(SlotLast l, int ncell1, const int32_t *__restrict__ start, int32_t *__restrict__ count,
                              int n, int32_t *__restrict__ cell_of)
{
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    const int q = *l.last;
    if (t < ncell1) count[t] = q < 0 ? start[t + 1] - start[t] : l.cellq[q][t].x;
    if (q >= 0 && t < n) cell_of[t] = ncell1 - 1;
}

// perm and cell_of of the particles in slots and overflow lists, one thread
// per cell.
template <bool FX>
__global__ void k_slot_lists(SlotLast l, const void *__restrict__ pos,
                             const int32_t *__restrict__ onext, int ncell, int cap, int nslots,
                             const int32_t *__restrict__ start, int32_t *__restrict__ perm,
                             int32_t *__restrict__ cell_of)
{
    const int c = blockIdx.x * blockDim.x + threadIdx.x;
    const int p = *l.last;
    if (c >= ncell || p < 0) return;
    const int2 q = l.cellq[p][c];
    const int s = start[c];
    int r = 0;
    for (; r < min(q.x, cap); r++) {
        const int i = slot_index<FX>(pos, (int64_t)c * cap + r);
        perm[s + r] = i;
        cell_of[i] = c;
    }
    for (int o = q.y; o > 0 && r < q.x; o = onext[o - 1], r++) {
        const int i = slot_index<FX>(pos, (int64_t)nslots + o - 1);
        perm[s + r] = i;
        cell_of[i] = c;
    }
}

// The particles left in the extra cell (non-finite positions), listed after
// the grid's; count[ncell] is the cursor, zero before and after (last block).
__global__ void k_slot_extra(SlotLast l, const int32_t *__restrict__ cell_of, int n, int ncell, const int32_t *__restrict__ start,
                             int32_t *__restrict__ perm, int32_t *__restrict__ cursor)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (*l.last >= 0 && i < n && cell_of[i] == ncell) perm[start[ncell] + atomicAdd(cursor, 1)] = i;
}

inline unsigned blocks_for(int64_t n, int threads) { return (unsigned)((n + threads - 1) / threads); }

}  // namespace

SlotBin slot_bin_of(const lj_ctx *c)
{
    SlotBin b;
    b.cellq = c->cellq[c->slot_par];
    b.pos = c->spos;
    b.onext = c->onext;
    b.octr = c->octr + c->slot_par;
    b.work = c->work;
    b.cfix = c->cfix;
    b.thb = c->thb;
    b.L = c->p.box;
    b.whi = c->wrap_hi;
    b.wlo = c->wrap_lo;
    b.s = c->inv_cw;
    b.sf = (float)c->inv_cw;
    b.nc = c->nc;
    b.ncell = (int)c->ncell;
    b.cap = c->scap;
    b.nslots = c->nslots;
    b.nover = (int)c->p.n;
    b.grow_at = slots_grow_at(c->scap, kSlotMax, c->p.n);
    b.grow = c->host_err + 1;
    b.cell0 = 0;
    b.S = c->p.precision == LJ_PREC_FP64 ? fx_shift(c) : rel_shift(c->cw);
    return b;
}

void slots_free(lj_ctx *c)
{
    cudaFree(c->slot_mem);
    if (!c->sg4_inside) cudaFree(c->sg4);
    c->slot_mem = nullptr;
    c->cellq[0] = c->cellq[1] = nullptr;
    c->octr = nullptr;
    c->spos = nullptr;
    c->sg4 = nullptr;
    c->sg4_inside = 0;
    c->onext = nullptr;
    c->fx_acc = nullptr;
    c->scap = c->nslots = 0;
    c->slot_par = c->slots_open = c->slots_last = 0;
}

cudaError_t slots_setup(lj_ctx *c, bool wide)
{
    slots_free(c);
    // (FP64: the fixed-point kernel has no force-shifted form)
    const bool fp64 = c->p.precision == LJ_PREC_FP64;
    if (c->p.cell_subdiv == 2 || c->p.n == 0 || (fp64 && c->p.shift_mode == LJ_SHIFT_FORCE)) return cudaSuccess;
    const double mean = (double)c->p.n / (double)c->ncell;
    const size_t bytes = fp64 ? sizeof(longlong4_16a) : sizeof(float4);
    const int cap = slots_per_cell(mean, c->cw / c->p.sigma, kSlotMax, c->ncell, c->p.n, bytes, wide);
    const int64_t nslots = c->ncell * cap;
    if (mean > 22.0 || cap == 0 || nslots + c->p.n >= ((int64_t)1 << 31)) return cudaSuccess;
    // One allocation: each costs a context's creation about 10 us, and one
    // above 1 MB some 90.  Small contexts get the cotangents' slots with it
    // (32,000 particles: the first gradient 143 us when it allocated them, now
    // 61); large ones with their first gradient (ensure_vjp_buffers), if any.
    const size_t m = (size_t)(nslots + c->p.n), n = (size_t)c->p.n;
    const size_t sb = m * bytes;
    c->sg4_inside = !fp64 && sb <= kSlotsTogether;
    const size_t qb = (size_t)(c->ncell + 1) * sizeof(int2);
    const size_t part[7] = {sb, c->sg4_inside ? sb : 0, fp64 ? n * kFxAcc * sizeof(long long) : 0,
                            qb, qb, n * sizeof(int32_t), 4 * sizeof(unsigned)};
    char *at[7];
    size_t total = 0;
    for (size_t p : part) total += (p + 255) & ~(size_t)255;
    cudaError_t e = cudaMalloc(&c->slot_mem, total);
    if (e == cudaErrorMemoryAllocation) {   // the sorted lists need less
        cudaGetLastError();
        slots_free(c);
        return cudaSuccess;
    }
    if (e != cudaSuccess) return e;
    total = 0;
    for (int k = 0; k < 7; k++) {
        at[k] = (char *)c->slot_mem + total;
        total += (part[k] + 255) & ~(size_t)255;
    }
    c->spos = at[0];
    c->sg4 = c->sg4_inside ? (float4 *)at[1] : nullptr;
    c->fx_acc = fp64 ? (long long *)at[2] : nullptr;
    c->cellq[0] = (int2 *)at[3];
    c->cellq[1] = (int2 *)at[4];
    c->onext = (int32_t *)at[5];
    c->octr = (unsigned *)at[6];
    e = cudaMemsetAsync(c->octr, 0xff, part[6], c->stream);
    if (e != cudaSuccess) return e;
    c->scap = cap;
    c->nslots = (int)nslots;
    c->slots_open = 2;
    return fp64 ? fx_configure(c) : cudaSuccess;
}

// Not while a caller's graph holds the old buffers, and not inside a capture.
cudaError_t slots_new_call(lj_ctx *c)
{
    c->new_call = 1;
    if (c->scap == 0 || *(volatile int32_t *)(c->host_err + 1) == 0) return cudaSuccess;
    if (c->captured || capture_id(c->stream)) return cudaSuccess;
    RelaxedCapture relaxed;
    cudaError_t e = cudaStreamSynchronize(c->stream);
    c->host_err[1] = 0;
    if (e != cudaSuccess) return e;
    c->gen++;   // captured steps hold the old buffers
    e = slots_setup(c, true);
    return e == cudaSuccess && c->scap == 0 ? slots_setup(c, false) : e;   // (no memory for the wide ones)
}

// Force evaluations take the slotted cells where the pair-once kernel runs
// and a cell beyond its slots is rare: cells so thinly filled that even a
// random gas overflows one in some 10^5, or a dense fluid (n sigma^3 / L^3
// >= 0.5), whose excluded volume keeps the occupancy near its mean.
static bool slots_suit(const lj_ctx *c)
{
    const double mean = (double)c->p.n / (double)c->ncell;
    const double sg = c->p.sigma / c->p.box;
    return mean + 4.5 * sqrt(mean) <= kSlotMax || (double)c->p.n * sg * sg * sg >= 0.5;
}

bool uses_slots(const lj_ctx *c)
{
    return c->scap > 0 && c->skin <= 0.0 && !c->fuse_update && uses_force_n3(c) && slots_suit(c);
}

// The fixed-point forces are the more exact ones, pair by pair, while rc <=
// 2.6 sigma (the file header of lj_force_fx.cu has the errors).
bool uses_fx(const lj_ctx *c)
{
    return c->scap > 0 && c->p.rc <= 2.6 * c->p.sigma && c->skin <= 0.0 && c->p.precision == LJ_PREC_FP64 && c->n3 &&
           !c->deterministic && !c->use_run_kernel && !c->use_aop && slots_suit(c);
}

cudaError_t launch_bin_fx(lj_ctx *c, const double *x, double4_16a *f)
{
    cudaError_t e = slots_begin(c, 0);
    if (e != cudaSuccess) return e;
    const int n = (int)c->p.n;
    k_bin_fx<<<blocks_for(n, 256), 256, 0, c->stream>>>(slot_bin_of(c), x, n, f, (longlong2 *)c->fx_acc, c->err);
    c->kernel_launches++;
    return cudaGetLastError();
}

cudaError_t launch_kick_drift_fx(lj_ctx *c, double *x, double *v, double4_16a *f, int nkick, bool with_acc,
                                 int64_t i_begin, int64_t i_end, bool after_force)
{
    const int n = (int)(i_end < 0 ? c->p.n : i_end);
    if (n <= (int)i_begin) return cudaSuccess;
    cudaError_t e = slots_begin(c, i_begin);
    if (e != cudaSuccess) return e;
    SlotBin b = slot_bin_of(c);
    int i0 = (int)i_begin, i1 = n, wa = with_acc ? 1 : 0;
    double h = nkick * (0.5 * c->p.dt / c->p.mass), dt = c->p.dt, scale = fx_scale(c);
    int32_t *err = c->err;
    void *args[] = {&b, &x, &v, &f, &c->fx_acc, &wa, &scale, &i0, &i1, &h, &dt, &err};
    e = launch_pdl((const void *)k_kick_drift_fx, (int)blocks_for(n - i_begin, 256), 256, args, 0, c->stream, after_force);
    c->kernel_launches++;
    return e != cudaSuccess ? e : cudaGetLastError();
}

cudaError_t launch_fx_finish(lj_ctx *c, double *v, double4_16a *f)
{
    int n = (int)c->p.n;
    double scale = fx_scale(c), h = 0.5 * c->p.dt / c->p.mass;
    void *args[] = {&v, &f, &c->fx_acc, &n, &scale, &h};
    const cudaError_t e = launch_pdl((const void *)k_fx_finish, (int)blocks_for(n, 256), 256, args, 0, c->stream,
                                     !c->timing);
    c->kernel_launches++;
    return e != cudaSuccess ? e : cudaGetLastError();
}

cudaError_t slots_begin(lj_ctx *c, int64_t i_begin)
{
    if (i_begin > 0) return cudaSuccess;
    cudaError_t e = cudaSuccess;
    bool zero = c->slots_open != 0;   // first use, or a binning that no kernel consumed
    if (!c->own_capture) {
        const unsigned long long id = capture_id(c->stream);
        if (id) {   // recorded: replays start from buffers in any state
            zero = zero || id != c->cap_id;
            c->cap_id = id;
            c->captured = 1;
        } else if (c->captured && c->new_call) {   // a replay may have come since the last call
            zero = true;
        }
        c->new_call = 0;
    }
    if (zero) {
        const size_t qb = (size_t)(c->ncell + 1) * sizeof(int2);
        e = cudaMemsetAsync(c->cellq[0], 0, qb, c->stream);
        if (e == cudaSuccess) e = cudaMemsetAsync(c->cellq[1], 0, qb, c->stream);
        if (e == cudaSuccess) e = cudaMemsetAsync(c->octr, 0, 2 * sizeof(unsigned), c->stream);
    }
    c->slots_open = 1;
    return e;
}

cudaError_t lists_begin(lj_ctx *c)
{
    c->slots_last = 0;
    if (c->scap == 0 || c->own_capture) return cudaSuccess;
    if (!c->captured && !capture_id(c->stream)) return cudaSuccess;
    c->captured = 1;
    return cudaMemsetAsync(c->octr + 2, 0xff, sizeof(unsigned), c->stream);
}

void slots_consumed(lj_ctx *c)
{
    c->slot_par ^= 1;
    c->slots_open = 0;
    c->slots_last = 1;
}

cudaError_t launch_bin_slots(lj_ctx *c, const double *x, float4 *zero, const double *g)
{
    cudaError_t e = slots_begin(c, 0);
    if (e != cudaSuccess) return e;
    const int n = (int)c->p.n;
    k_bin_slots<<<blocks_for(n, 256), 256, 0, c->stream>>>(slot_bin_of(c), x, n, zero, g, c->sg4, c->err);
    c->kernel_launches++;
    return cudaGetLastError();
}

cudaError_t launch_kick_drift_slots(lj_ctx *c, const double *x, double *xo, double *v, float4 *f, int nkick,
                                    int64_t i_begin, int64_t i_end, bool after_force)
{
    const int n = (int)(i_end < 0 ? c->p.n : i_end);
    if (n <= (int)i_begin) return cudaSuccess;
    cudaError_t e = slots_begin(c, i_begin);
    if (e != cudaSuccess) return e;
    const double hk = nkick * (0.5 * c->p.dt / c->p.mass);
    SlotBin b = slot_bin_of(c);
    int i0 = (int)i_begin, i1 = n;
    double h = hk, dt = c->p.dt;
    int32_t *err = c->err;
    void *args[] = {&b, (void *)&x, &xo, &v, &f, &i0, &i1, &h, &dt, &err};
    e = launch_pdl((const void *)k_kick_drift_slots, (int)blocks_for(n - i_begin, 256), 256, args, 0, c->stream, after_force);
    c->kernel_launches++;
    return e != cudaSuccess ? e : cudaGetLastError();
}

cudaError_t launch_host_in(lj_ctx *c, const double *hx, const double *hv, const float4 *hf, double *x, double *v, float4 *f)
{
    cudaError_t e = slots_begin(c, 0);
    if (e != cudaSuccess) return e;
    const int n = (int)c->p.n;
    k_host_in<<<blocks_for(n, kHostThreads), kHostThreads, 0, c->stream>>>(
        slot_bin_of(c), hx, hv, hf, x, v, f, n, 0.5 * c->p.dt / c->p.mass, c->p.dt, c->err);
    c->kernel_launches++;
    return cudaGetLastError();
}

cudaError_t launch_host_out(lj_ctx *c, const double *x, const double *v, const float4 *f, double *hx, double *hv,
                            float4 *hf)
{
    int n = (int)c->p.n;
    double h = 0.5 * c->p.dt / c->p.mass;
    const int32_t *err = c->err;
    void *args[] = {(void *)&x, (void *)&v, (void *)&f, &n, &h, &hx, &hv, &hf, (void *)&err, &c->host_err};
    c->kernel_launches++;
    return launch_pdl((const void *)k_host_out, blocks_for(n, kHostThreads), kHostThreads, args, 0, c->stream, !c->timing);
}

cudaError_t launch_slots_to_lists(lj_ctx *c)
{
    if (c->scap == 0) return cudaSuccess;
    if (capture_id(c->stream)) c->captured = 1;   // recorded, not run
    if (!c->slots_last && !c->captured) return cudaSuccess;
    const int n = (int)c->p.n, ncell = (int)c->ncell;
    const SlotLast q = {{c->cellq[0], c->cellq[1]}, reinterpret_cast<const int *>(c->octr + 2)};
    k_slot_counts<<<blocks_for(n > ncell + 1 ? n : ncell + 1, 256), 256, 0, c->stream>>>(q, ncell + 1, c->start,
                                                                                         c->count, n, c->cell_of);
    c->kernel_launches++;
    cudaError_t e = cudaGetLastError();
    if (e == cudaSuccess) e = launch_scan(c);   // start from the counts, which it zeroes
    if (e != cudaSuccess) return e;
    if (c->p.precision == LJ_PREC_FP64)
        k_slot_lists<true><<<blocks_for(ncell, 256), 256, 0, c->stream>>>(q, c->spos, c->onext, ncell, c->scap, c->nslots,
                                                                          c->start, c->perm, c->cell_of);
    else
        k_slot_lists<false><<<blocks_for(ncell, 256), 256, 0, c->stream>>>(q, c->spos, c->onext, ncell, c->scap,
                                                                           c->nslots, c->start, c->perm, c->cell_of);
    k_slot_extra<<<blocks_for(n, 256), 256, 0, c->stream>>>(q, c->cell_of, n, ncell, c->start, c->perm, c->count + ncell);
    c->kernel_launches += 2;
    e = cudaMemsetAsync(c->count + ncell, 0, sizeof(int32_t), c->stream);
    if (e != cudaSuccess) return e;
    c->slots_last = 0;   // cell_of, start and perm hold this binning now
    return cudaGetLastError();
}
