// Slotted cells: the cell lists of the FP32-mixed pair-once kernels, built in
// one pass over the particles.
//
// Section 3.1 of the paper keeps a cell's particles physically together in
// a fixed number of placeholders.  Here cell c owns `cap` slots of the
// sorted-position array, [c cap, (c + 1) cap), and a particle's slot is its
// rank in the cell, which the binning's atomic count returns anyway: the
// position goes straight to its slot, with no scan over the counts, no
// second pass over x, and no cell-id and rank arrays in between.  Particles
// beyond a cell's slots are not dropped: they go to an overflow region after
// the slots, chained per cell (a lock-free push on the cell's list head),
// which the kernels' plain path reads.  Non-finite particles are counted
// in the extra cell ncell and get no slot.
//
// The counts must be zero when a binning starts.  They are held twice; the
// force (or VJP) kernel that reads one buffer zeroes the other for the
// next binning.  Which buffer is next is the host's knowledge; calls that a
// caller records into a graph zero both first (slots_begin).
#pragma once

#include <math.h>

#include "lj_internal.cuh"

struct SlotBin {
    int2 *cellq;            // this binning's (count, list head + 1) per cell, zero before it
    void *pos;              // [nslots + n] float4, or longlong4 in FP64 contexts
    int32_t *onext;
    unsigned *octr, *work;  // overflow counter of this buffer; the force kernel's work counter, zeroed here
    const long long *cfix;  // cell centres (rel_f32)
    const long long *thb;
    double L, whi, wlo, s;
    float sf;               // (float)s
    int nc, ncell, cap, nslots, S;   // S: scale of the fixed-point coordinates (FP64: lj_force_fx.cu, else rel_shift)
    int nover;              // entries of the overflow region
    int grow_at;            // overflow particles that set *grow (pinned host memory)
    int32_t *grow;
    int cell0;              // id of the grid's first cell (a batch's replica; else 0); ncell counts all grids' cells
};

// Slots per cell of `cw` sigma a side in ncell cells of n particles, `bytes`
// each, a multiple of 8 (128 bytes) up to limit; 0: the box is too sparse (far
// more slots than particles) and keeps the sorted lists.  The mean occupancy
// plus 7 standard deviations of a random gas; and, where that makes up to 24
// MB of slots, room for a liquid or crystal (0.9 particles per sigma^3 and 16
// more: at 2.5 sigma a lattice can put 4 of its planes in a cell, 32
// particles).  A vapour may condense, a box hold both, and a cell beyond its
// slots takes all cells around it to the plain path (a droplet of 97,556
// particles at a mean density of 0.1, 16 slots by the gas alone: forces 288 us,
// VJP 383).  Larger boxes get the wide slots (limit) when they are seen to need
// them (slot_place, slots_new_call): 32 slots in place of 16 cost a gas of 10^6
// particles, whose positions then lie further apart in memory, 1 to 5 %.
inline int slots_per_cell(double mean, double cw, int limit, int64_t ncell, int64_t n, size_t bytes, bool wide)
{
    auto up8 = [limit](double m) { return m < (double)limit ? ((int)ceil(m) + 7) & ~7 : limit; };
    const int gas = up8(mean + 7.0 * sqrt(mean) + 3.0), liquid = up8(0.9 * cw * cw * cw + 16.0);
    if (ncell * gas > 12 * n + ((int64_t)1 << 16)) return 0;
    if (wide) return limit;
    return liquid > gas && (size_t)(ncell * liquid) * bytes <= ((size_t)24 << 20) ? liquid : gas;
}

// The wide slots are asked for when a binning has so many particles beyond
// their cells' slots.
inline int slots_grow_at(int cap, int limit, int64_t n)
{
    return cap < limit ? 32 + (int)(n / 2048) : 0x7fffffff;
}

#ifdef __CUDACC__
namespace {

// Cell of the wrapped position (px, py, pz); the guess comes from the FP32
// truncated coordinates (integer work: no FP64-pipe multiply or conversion)
// and lj_cell_from_guess makes it exact.
__device__ __forceinline__ int3 slot_cell(const SlotBin &b, double px, double py, double pz)
{
    int3 c;
    c.x = lj_cell_from_guess(px, __float2int_rz(f32_trunc(px) * b.sf), b.thb, b.s, b.nc);
    c.y = lj_cell_from_guess(py, __float2int_rz(f32_trunc(py) * b.sf), b.thb, b.s, b.nc);
    c.z = lj_cell_from_guess(pz, __float2int_rz(f32_trunc(pz) * b.sf), b.thb, b.s, b.nc);
    return c;
}

// Rank particle i in its cell and store its position, relative to the cell
// centre (FX: in fixed point, lj_force_fx.cu).  All 32 lanes call it; lanes
// with valid = false do nothing.  Returns the slot, or -1 when none was taken.
template <bool FX = false>
__device__ __forceinline__ int slot_place(const SlotBin &b, bool valid, int i, double px, double py, double pz,
                                          int32_t *err)
{
    int c = 0;
    int3 cc = make_int3(0, 0, 0);
    if (valid) {
        if (finite64(px) && finite64(py) && finite64(pz)) {
            cc = slot_cell(b, px, py, pz);
            c = b.cell0 + cc.x + b.nc * (cc.y + b.nc * cc.z);
        } else {
            atomicOr(err, LJ_ERRBIT_NONFINITE);
            c = b.ncell;
        }
    }
    const int r = lj_warp_rank(reinterpret_cast<int32_t *>(b.cellq), c, valid, 2);
    if (!valid || c >= b.ncell) return -1;
    int slot = c * b.cap + r;
    if (r >= b.cap) {   // overflow: the next free entry, pushed on the cell's list
        const int k = (int)atomicAdd(b.octr, 1u);
        if (k == b.grow_at) *b.grow = 1;
        if (k >= b.nover) {   // never with counts that were zero
            atomicOr(err, LJ_ERRBIT_OVERFLOW);
            return -1;
        }
        slot = b.nslots + k;
        b.onext[k] = atomicExch(&b.cellq[c].y, k + 1);
    }
    if constexpr (FX) {
        longlong2 *o = reinterpret_cast<longlong2 *>(b.pos) + 2 * (int64_t)slot;
        o[0] = make_longlong2(lj_fix64(px, b.S), lj_fix64(py, b.S));
        o[1] = make_longlong2(lj_fix64(pz, b.S), (long long)i);
    } else {
        reinterpret_cast<float4 *>(b.pos)[slot] =
            make_float4(rel_f32(px, __ldg(b.cfix + cc.x), b.S), rel_f32(py, __ldg(b.cfix + cc.y), b.S),
                        rel_f32(pz, __ldg(b.cfix + cc.z), b.S), __int_as_float(i));
    }
    return slot;
}

}  // namespace
#endif

SlotBin slot_bin_of(const lj_ctx *c);
