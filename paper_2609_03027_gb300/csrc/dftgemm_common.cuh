// What the tensor path's kernels share: bounded waits, FP16 packing, the layout of the grid
// tiles and the cuts of a launch's work between blocks.
#pragma once

#include <cuda_fp16.h>
#include <stdint.h>

#include <algorithm>

#include "tc_ptx.cuh"

namespace epic {

constexpr long long kWaitBudget = 4000000000LL;  // clock cycles before a wait gives up (~2 s)

__host__ __device__ inline int pad64(int k) { return (k + 63) & ~63; }

inline size_t align_up(size_t v, size_t a) { return (v + a - 1) / a * a; }

__device__ __forceinline__ uint32_t pack_h2(float a, float b)
{
    __half2 h = __floats2half2_rn(a, b);
    return *reinterpret_cast<uint32_t*>(&h);
}

// First unit of block b of G when a launch's units -- ipc items of each of n_ch channels from
// c0 in channel order, nt frames per item, item-major -- are cut into G ranges of equal cost,
// a unit costing its channel's weight (wcum: prefix sums of the weights over the plan's
// channels).  Without weights, G ranges of equal numbers of units.  Non-decreasing in b,
// 0 at b = 0 and every unit at b = G.
__device__ __forceinline__ long long split_start(const long long* wcum, int c0, int n_ch, int ipc, int nt, int b, int G)
{
    const long long per = (long long)ipc * nt;  // units of one channel
    if (!wcum) return (long long)n_ch * per * b / G;
    const long long base = wcum[c0];
    const long long s = per * (wcum[c0 + n_ch] - base) * b / G;  // cost position of the block's start
    int lo = 0, hi = n_ch;                                        // last channel whose units start at or before s
    while (hi - lo > 1) {
        const int mid = (lo + hi) >> 1;
        if (per * (wcum[c0 + mid] - base) <= s) lo = mid;
        else hi = mid;
    }
    const long long w = wcum[c0 + lo + 1] - wcum[c0 + lo];
    const long long u = min(per, (s - per * (wcum[c0 + lo] - base)) / w);
    return (long long)lo * per + u;
}

// Largest i of [lo, hi) with f(i) <= s, by a whole warp (f increasing, f(lo) <= s): two rounds of loads where one
// thread's search takes a chain of eight.
template <class F>
__device__ __forceinline__ int warp_find(int lo, int hi, int lane, long long s, F&& f)
{
    while (hi - lo > 1) {
        const int step = (hi - lo + 31) / 32, i = lo + lane * step;
        const int k = 31 - __clz(__ballot_sync(0xffffffffu, i < hi && f(i) <= s) | 1);
        lo += k * step;
        hi = min(hi, lo + step);
    }
    return lo;
}

// split_start (with weights) by a whole warp
__device__ __forceinline__ long long split_start_warp(const long long* wcum, int c0, int n_ch, int ipc, int nt, int b, int G,
                                                      int lane)
{
    const long long per = (long long)ipc * nt, base = __ldg(wcum + c0);
    const long long s = per * (__ldg(wcum + c0 + n_ch) - base) * b / G;
    const int lo = warp_find(0, n_ch, lane, s, [&](int c) { return per * (__ldg(wcum + c0 + c) - base); });
    const long long w = __ldg(wcum + c0 + lo + 1) - __ldg(wcum + c0 + lo);
    return (long long)lo * per + min(per, (s - per * (__ldg(wcum + c0 + lo) - base)) / w);
}

// K order of a grid tile's rows: the cell pair (x, x + 1), x even, takes K indices 2 x .. 2 x + 3 as
// (re x, re x+1, im x, im x+1), so that a thread with a pair's sums stores 8 bytes and the pairs of
// a row fill whole 32-byte sectors whatever the box width (with all real parts before the imaginary
// ones, boxes of an odd number of 8-cell chunks left half sectors: a 56 x 56 box's tiles took 1.6
// times as long to write as a 64 x 64 box's).  Box column and part of K index k:
__host__ __device__ __forceinline__ int tile_k_x(int k) { return 2 * (k >> 2) + (k & 1); }
__host__ __device__ __forceinline__ bool tile_k_im(int k) { return (k & 2) != 0; }

__host__ __device__ __forceinline__ uint32_t tile_half_off(int R, int k, int N1)
{
    return (uint32_t)((k >> 6) * (N1 * 128) + R * 128 + ((((k >> 3) & 7) ^ (R & 7)) << 4) + ((k & 7) << 1));
}

// Byte offset of the FP16 at (pol-X row y, K index k) of a grid tile cut into row parts of
// nyh rows: part h = y / nyh is an operand of its own (P nyh rows: pol X rows 0..nyh-1, pol
// Y rows nyh..2 nyh-1, so a pol-Y value sits nyh * 128 bytes after its pol-X value),
// part_bytes apart.  One part (nyh = box rows) is the plain layout.
__host__ __device__ __forceinline__ uint32_t tile_part_off(int y, int k, int nyh, int P, uint32_t part_bytes)
{
    const int h = y / nyh;
    return (uint32_t)h * part_bytes + tile_half_off(y - h * nyh, k, P * nyh);
}

// The same without padding of K, for k_dftgemm_grid_tc and k_dftgemm_ws3: whole panels of 64 K indices as
// above, then one of 32 (64-byte swizzle) and one of 16 (32-byte swizzle) as K1 = 2 nx needs them.  Padded,
// a 48-wide box's rows ended in half a 128-byte line, and such tiles took 1.5 times as long a byte
// to write as those of 64 or 96 columns.  tile_dense_row: bytes from a row to the next at K index k.
__host__ __device__ __forceinline__ uint32_t tile_dense_row(int k, int K1)
{
    if ((k >> 6) < (K1 >> 6)) return 128;
    return (K1 & 32) && (k & 63) < 32 ? 64 : 32;
}

__host__ __device__ __forceinline__ uint32_t tile_dense_off(int y, int k, int nyh, int P, int K1)
{
    const int h = y / nyh, R = y - h * nyh, N1 = P * nyh;
    const uint32_t part = (uint32_t)h * (uint32_t)(N1 * K1 * 2);
    if ((k >> 6) < (K1 >> 6)) return part + tile_half_off(R, k, N1);
    uint32_t base = part + (uint32_t)((K1 >> 6) * N1 * 128);
    if (K1 & 32) {
        if ((k & 63) < 32) return base + (uint32_t)(R * 64 + ((((k >> 3) ^ (R >> 1)) & 3) << 4) + ((k & 7) << 1));
        base += (uint32_t)N1 * 64;
    }
    return base + (uint32_t)(R * 32 + ((((k >> 3) ^ (R >> 2)) & 1) << 4) + ((k & 7) << 1));
}

// 8 consecutive 32-bit TMEM columns of this thread's lane
__device__ __forceinline__ void tmem_ld8(uint32_t taddr, uint32_t* r)
{
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
                 : "r"(taddr)
                 : "memory");
}

__device__ __forceinline__ void mbar_arrive(uint64_t* bar)
{
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(tc::smem_u32(bar)) : "memory");
}

}  // namespace epic
