// Slotted cells (lj_slots.cuh): set-up, the binning kernels, and the
// conversion to the sorted lists that lj_get_cells returns.
#include <math.h>

#include "lj_slots.cuh"

namespace {

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
__global__ void __launch_bounds__(256) k_kick_drift_slots(SlotBin b, double *__restrict__ x, double *__restrict__ v,
                                                          float4 *__restrict__ f, int i_begin, int n, double hk,
                                                          double dt, int32_t *__restrict__ err)
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
        x[o] = px;
        x[o + 1] = py;
        x[o + 2] = pz;
    }
    slot_place(b, valid, i, px, py, pz, err);
}

// Counts of every cell (the extra one included) for the scan of
// launch_slots_to_lists; cell_of starts as the extra cell everywhere.
__global__ void k_slot_counts(const int2 *__restrict__ cellq, int ncell1, int32_t *__restrict__ count, int n,
                              int32_t *__restrict__ cell_of)
{
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t < ncell1) count[t] = cellq[t].x;
    if (t < n) cell_of[t] = ncell1 - 1;
}

// perm and cell_of of the particles in slots and overflow lists, one thread
// per cell.
__global__ void k_slot_lists(const int2 *__restrict__ cellq, const float4 *__restrict__ pos,
                             const int32_t *__restrict__ onext, int ncell, int cap, int nslots,
                             const int32_t *__restrict__ start, int32_t *__restrict__ perm,
                             int32_t *__restrict__ cell_of)
{
    const int c = blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= ncell) return;
    const int2 q = cellq[c];
    const int s = start[c];
    int r = 0;
    for (; r < min(q.x, cap); r++) {
        const int i = __float_as_int(pos[(int64_t)c * cap + r].w);
        perm[s + r] = i;
        cell_of[i] = c;
    }
    for (int o = q.y; o > 0; o = onext[o - 1], r++) {
        const int i = __float_as_int(pos[(int64_t)nslots + o - 1].w);
        perm[s + r] = i;
        cell_of[i] = c;
    }
}

// The particles left in the extra cell (non-finite positions), listed after
// the grid's; count[ncell] is the cursor, zero before and after (last block).
__global__ void k_slot_extra(const int32_t *__restrict__ cell_of, int n, int ncell, const int32_t *__restrict__ start,
                             int32_t *__restrict__ perm, int32_t *__restrict__ cursor)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n && cell_of[i] == ncell) perm[start[ncell] + atomicAdd(cursor, 1)] = i;
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
    b.centre = c->centre2;
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
    return b;
}

void slots_free(lj_ctx *c)
{
    cudaFree(c->cellq[0]);
    cudaFree(c->cellq[1]);
    cudaFree(c->octr);
    cudaFree(c->spos);
    cudaFree(c->sg4);
    cudaFree(c->onext);
    c->cellq[0] = c->cellq[1] = nullptr;
    c->octr = nullptr;
    c->spos = c->sg4 = nullptr;
    c->onext = nullptr;
    c->scap = c->nslots = 0;
    c->slot_par = c->slots_open = c->slots_last = 0;
}

cudaError_t slots_setup(lj_ctx *c)
{
    slots_free(c);
    if (c->p.precision != LJ_PREC_MIXED || c->p.cell_subdiv == 2 || c->p.n == 0) return cudaSuccess;
    // Slots per cell: the mean occupancy plus 7 standard deviations of a
    // random gas, a multiple of 8 (128 bytes), at most the 32 home particles
    // that the kernels' fast path takes.
    const double mean = (double)c->p.n / (double)c->ncell;
    int cap = ((int)ceil(mean + 7.0 * sqrt(mean) + 3.0) + 7) & ~7;
    cap = cap > kSlotMax ? kSlotMax : cap;
    const int64_t nslots = c->ncell * cap;
    // sparse boxes (far more slots than particles) keep the sorted lists
    if (mean > 22.0 || nslots + c->p.n >= ((int64_t)1 << 31) ||
        nslots > (int64_t)12 * c->p.n + ((int64_t)1 << 16))
        return cudaSuccess;
    cudaError_t e = cudaSuccess;
    const size_t qb = (size_t)(c->ncell + 1) * sizeof(int2);
    for (int k = 0; k < 2 && e == cudaSuccess; k++) e = cudaMalloc(&c->cellq[k], qb);
    if (e == cudaSuccess) e = cudaMalloc(&c->octr, 2 * sizeof(unsigned));
    if (e == cudaSuccess) e = cudaMalloc(&c->spos, (size_t)(nslots + c->p.n) * sizeof(float4));
    if (e == cudaSuccess) e = cudaMalloc(&c->onext, (size_t)c->p.n * sizeof(int32_t));
    if (e == cudaErrorMemoryAllocation) {   // the sorted lists need less
        cudaGetLastError();
        slots_free(c);
        return cudaSuccess;
    }
    if (e != cudaSuccess) return e;
    c->scap = cap;
    c->nslots = (int)nslots;
    c->slots_open = 2;
    return cudaSuccess;
}

// Force evaluations take the slotted cells where the pair-once kernel runs
// and a cell beyond its slots is rare: cells so thinly filled that even a
// random gas overflows one in some 10^5, or a dense fluid (n sigma^3 / L^3
// >= 0.5), whose excluded volume keeps the occupancy near its mean.
bool uses_slots(const lj_ctx *c)
{
    if (c->scap == 0 || c->skin > 0.0 || c->fuse_update || !uses_force_n3(c)) return false;
    const double mean = (double)c->p.n / (double)c->ncell;
    const double sg = c->p.sigma / c->p.box;
    return mean + 4.5 * sqrt(mean) <= kSlotMax || (double)c->p.n * sg * sg * sg >= 0.5;
}

cudaError_t slots_begin(lj_ctx *c, int64_t i_begin)
{
    if (i_begin > 0) return cudaSuccess;
    cudaError_t e = cudaSuccess;
    if (c->slots_open) {   // first use, or a binning that no kernel consumed
        const size_t qb = (size_t)(c->ncell + 1) * sizeof(int2);
        e = cudaMemsetAsync(c->cellq[0], 0, qb, c->stream);
        if (e == cudaSuccess) e = cudaMemsetAsync(c->cellq[1], 0, qb, c->stream);
        if (e == cudaSuccess) e = cudaMemsetAsync(c->octr, 0, 2 * sizeof(unsigned), c->stream);
    }
    c->slots_open = 1;
    return e;
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

cudaError_t launch_kick_drift_slots(lj_ctx *c, double *x, double *v, float4 *f, int nkick, int64_t i_begin,
                                    int64_t i_end, bool after_force)
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
    void *args[] = {&b, &x, &v, &f, &i0, &i1, &h, &dt, &err};
    e = launch_pdl((const void *)k_kick_drift_slots, (int)blocks_for(n - i_begin, 256), 256, args, 0, c->stream, after_force);
    c->kernel_launches++;
    return e != cudaSuccess ? e : cudaGetLastError();
}

cudaError_t launch_slots_to_lists(lj_ctx *c)
{
    const int n = (int)c->p.n, ncell = (int)c->ncell;
    const int2 *q = c->cellq[c->slot_par ^ 1];
    k_slot_counts<<<blocks_for(n > ncell + 1 ? n : ncell + 1, 256), 256, 0, c->stream>>>(q, ncell + 1, c->count, n,
                                                                                         c->cell_of);
    c->kernel_launches++;
    cudaError_t e = cudaGetLastError();
    if (e == cudaSuccess) e = launch_scan(c);   // start from the counts, which it zeroes
    if (e != cudaSuccess) return e;
    k_slot_lists<<<blocks_for(ncell, 256), 256, 0, c->stream>>>(q, c->spos, c->onext, ncell, c->scap, c->nslots,
                                                                c->start, c->perm, c->cell_of);
    k_slot_extra<<<blocks_for(n, 256), 256, 0, c->stream>>>(c->cell_of, n, ncell, c->start, c->perm, c->count + ncell);
    c->kernel_launches += 2;
    e = cudaMemsetAsync(c->count + ncell, 0, sizeof(int32_t), c->stream);
    if (e != cudaSuccess) return e;
    c->slots_last = 0;   // cell_of, start and perm hold this binning now
    return cudaGetLastError();
}
