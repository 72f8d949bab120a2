// The pair-once force kernel for single systems (FP32-mixed; the design and
// the device code are in lj_force_n3.cuh): configuration and launch.
#include <string.h>

#include "lj_force_n3.cuh"

namespace {

// SLOTS: slotted cells (start unused); the launch also zeroes the next
// binning's counts.  SPLIT: each cell is 2^k.lgw items.
template <int MODE, bool ENERGY, bool SLOTS, bool SPLIT>
__global__ void __launch_bounds__(kN3Threads, ENERGY ? 4 : 6) k_force_n3(WarpParams k, const float4 *pos,
                                                         const int32_t *start, float4 *fout,
                                                         double *partial)
{
    extern __shared__ __align__(16) float nsmem[];
    const int lane = threadIdx.x & 31;
    const int warp = threadIdx.x >> 5;
    float4 *S = reinterpret_cast<float4 *>(nsmem + (size_t)warp * n3_slice_words(k.cap));
    float4 *stab = S + k.cap;
    int *spre = reinterpret_cast<int *>(stab + kN3Half);
    float4 *H = reinterpret_cast<float4 *>(spre + 16);
    const int nc = k.nc;
    double eacc = 0.0, wacc = 0.0;
    if constexpr (SLOTS) {
        pdl_wait();
        start = reinterpret_cast<const int32_t *>(k.cellq);
        if (blockIdx.x == 0 && threadIdx.x == 0) {
            k.cellq_next[k.ncell] = make_int2(0, 0);
            *k.octr_next = 0u;
            *k.last_par = k.par;
        }
    }
    auto load = [&](int c) { return half_load<true, SLOTS>(start, c, nc, k.inv_nc, 0, k.scap); };
    auto one_cell = [&](HalfLoad tl, int c, int part) {
        if (SLOTS && lane == 31 && part == 0) k.cellq_next[c] = make_int2(0, 0);
        n3_cell<MODE, ENERGY, !SLOTS, SLOTS, SPLIT>(k, pos, fout, tl, c, 0, nc, k.inv_nc, part, k.lgw, k.cw, S, stab, spre, H,
                                                  eacc, wacc);
    };
    if constexpr (SPLIT) {
        // at most one item per resident warp: no pulls
        const int it = blockIdx.x * (kN3Threads / 32) + warp;
        const int c = it >> k.lgw;
        if (c < k.ncell) one_cell(load(c), c, it & ((1 << k.lgw) - 1));
    } else if (k.grab > 0) {
        // pulls of k.grab cells, then single cells over the last stretch (two
        // rounds of pulls of the whole grid), so that the warps finish closer
        // together
        const int64_t tail = 2 * (int64_t)k.grab * gridDim.x * (kN3Threads / 32);
        unsigned last = 0;
        for (;;) {
            const unsigned g = (int64_t)last + tail >= k.ncell ? 1u : (unsigned)k.grab;
            unsigned c0 = 0;
            if (lane == 0) c0 = atomicAdd(k.work, g);
            c0 = __shfl_sync(0xffffffffu, c0, 0);
            if ((int64_t)c0 >= k.ncell) break;
            last = c0;
            const int c1 = (int)min((int64_t)c0 + g, k.ncell);
            // the next cell's table loads are issued before this cell's work
            HalfLoad nxt = load((int)c0);
            for (int c = (int)c0; c < c1; c++) {
                const HalfLoad cur = nxt;
                if (c + 1 < c1) nxt = load(c + 1);
                one_cell(cur, c, 0);
            }
        }
    } else {
        const int nwarps = gridDim.x * (kN3Threads / 32);
        int c = blockIdx.x * (kN3Threads / 32) + warp;
        HalfLoad nxt = load(c < k.ncell ? c : 0);
        for (; c < k.ncell; c += nwarps) {
            const HalfLoad cur = nxt;
            if (c + nwarps < k.ncell) nxt = load(c + nwarps);
            one_cell(cur, c, 0);
        }
    }
    if constexpr (ENERGY) {
        __shared__ double red[2 * (kN3Threads / 32)];
        for (int o = 16; o > 0; o >>= 1) {
            eacc += __shfl_xor_sync(0xffffffffu, eacc, o);
            wacc += __shfl_xor_sync(0xffffffffu, wacc, o);
        }
        if (lane == 0) {
            red[2 * warp] = eacc;
            red[2 * warp + 1] = wacc;
        }
        __syncthreads();
        if (threadIdx.x == 0) {
            double es = 0.0, ws = 0.0;
            for (int q = 0; q < kN3Threads / 32; q++) {
                es += red[2 * q];
                ws += red[2 * q + 1];
            }
            partial[2 * blockIdx.x] = es;
            partial[2 * blockIdx.x + 1] = ws;
        }
    }
}

template <bool SLOTS, bool SPLIT>
void *n3_kernel_of(int mode, bool energy)
{
    switch (mode * 2 + (energy ? 1 : 0)) {
        case 0: return (void *)k_force_n3<0, false, SLOTS, SPLIT>;
        case 1: return (void *)k_force_n3<0, true, SLOTS, SPLIT>;
        case 2: return (void *)k_force_n3<1, false, SLOTS, SPLIT>;
        case 3: return (void *)k_force_n3<1, true, SLOTS, SPLIT>;
        case 4: return (void *)k_force_n3<2, false, SLOTS, SPLIT>;
        default: return (void *)k_force_n3<2, true, SLOTS, SPLIT>;
    }
}

// form: 0 sorted lists, 1 slotted cells, 2 slotted and split
void *n3_kernel(int mode, bool energy, int form)
{
    return form == 2 ? n3_kernel_of<true, true>(mode, energy)
                     : form == 1 ? n3_kernel_of<true, false>(mode, energy) : n3_kernel_of<false, false>(mode, energy);
}

}  // namespace

cudaError_t n3_force_configure(lj_ctx *c)
{
    // Staged candidates per warp: the pruned half stencil of a fluid cell
    // (~125 at rho 0.84) plus 32 padding, with room for a Poisson spread of
    // the raw half stencil m = 14 n_cell (4 sqrt(m) + 32), and at least the
    // home forces' transpose (kN3Home * 32), which reuses the same space.
    const double mean = c->ncell > 0 ? (double)c->p.n / (double)c->ncell : 0.0;
    const double m = kN3Half * mean;
    int cap = (int)(m + 4.0 * sqrt(m)) + 64;
    cap = cap < kN3Home * 32 ? kN3Home * 32 : cap;   // S also holds the home forces' transpose
    cap = (cap + 31) & ~31;
    const int max_cap = ((227 * 1024 - 2 * (kN3Threads / 32) * 8) / (4 * (kN3Threads / 32)) -
                         kN3FixedWords) / 4 & ~31;
    if (cap > max_cap) cap = max_cap;
    c->n3cap = cap;   // float4 slots
    c->n3_smem = (kN3Threads / 32) * n3_slice_words(cap) * (int)sizeof(float);
    int minblk = 1 << 30;
    for (int mode = 0; mode < 3; mode++)
        for (int en = 0; en < 6; en++) {
            void *kern = n3_kernel(mode, (en & 1) != 0, en >> 1);
            cudaError_t e = raise_dyn_smem(kern, c->n3_smem);
            if (e != cudaSuccess) return e;
            int nb = 0;
            e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, kern, kN3Threads, c->n3_smem);
            if (e != cudaSuccess) return e;
            if ((en & 1) == 0 && nb < minblk) minblk = nb;   // the energy kernels get the same grid
        }
    if (minblk < 1) minblk = 1;
    int64_t grid = (int64_t)minblk * c->nsm;
    // Cells so few that warps would stand idle are split over 2 or 4 warps
    // each, while that still gives every item a resident warp of its own: one
    // warp takes a cell's chain of loads, staging and compute in 6 us alone,
    // a share of it in 3 (step at 2,048 particles 16.5 -> 14.4 us, 10,007
    // 17.2 -> 16.2; from two cells per warp up the shares' common work, the
    // home particles' staging and the final sums, costs more than it gains).
    c->n3_lgw = 0;
    while (c->n3_lgw < 2 && (c->ncell << (c->n3_lgw + 1)) <= grid * (kN3Threads / 32)) c->n3_lgw++;
    const int64_t need = ((c->ncell << c->n3_lgw) + kN3Threads / 32 - 1) / (kN3Threads / 32);
    if (grid > need) grid = need;
    if (grid < 1) grid = 1;
    c->n3_grid = (int)grid;
    return cudaSuccess;
}

cudaError_t launch_force_n3(lj_ctx *c, void *f, bool energy)
{
    if (c->p.n == 0) return cudaSuccess;
    WarpParams k = warp_params_of(c);
    k.cap = c->n3cap;
    k.inv_nc = c->inv_nc_f;
    k.lgw = c->n3_lgw;
    // the slotted binning, when it was one, has zeroed f
    const bool slots = c->slots_open == 1;
    const float4 *pos = (const float4 *)(slots ? c->spos : c->pos);
    const int32_t *start = c->start;
    if (slots) {
        k.last = c->nslots + k.n - 1;
        k.scap = c->scap;
        k.nslots = c->nslots;
        k.cellq = c->cellq[c->slot_par];
        k.cellq_next = c->cellq[c->slot_par ^ 1];
        k.octr_next = c->octr + (c->slot_par ^ 1);
        k.last_par = c->octr + 2;
        k.par = (unsigned)c->slot_par;
        k.onext = c->onext;
    }
    double *partial = c->partial;
    void *args[] = {&k, (void *)&pos, (void *)&start, &f, &partial};
    if (c->timing && c->ev_used + 2 <= c->nev) cudaEventRecord(c->ev[c->ev_used], c->stream);
    // f must start at zero: zeroed here, unless the step zeroed it already
    // on its side stream
    cudaError_t e = cudaSuccess;
    if (!c->f_prezeroed && !slots) e = cudaMemsetAsync(f, 0, (size_t)c->p.n * sizeof(float4), c->stream);
    c->f_prezeroed = 0;
    if (e == cudaSuccess)
        e = launch_pdl(n3_kernel(c->p.shift_mode, energy, !slots ? 0 : c->n3_lgw > 0 ? 2 : 1), c->n3_grid, kN3Threads,
                       args, c->n3_smem, c->stream, slots && !c->timing);
    if (c->timing && c->ev_used + 2 <= c->nev) {
        cudaEventRecord(c->ev[c->ev_used + 1], c->stream);
        c->ev_used += 2;
    }
    c->npartial = c->n3_grid;
    c->kernel_launches++;
    if (e != cudaSuccess) return e;
    if (slots) slots_consumed(c);
    return cudaGetLastError();
}
