// Gridding on the tensor cores: the FP16 grid tiles of the DFT-as-GEMM path (Eq. 1's bracket,
// G_p[cell] = sum_e w_e(cell) E_e^p) as a contraction over elements.  The box's cell pairs (two
// adjacent x; row-major, row-part padding included) come in M-tiles of 128 pairs; a tile's
// elements are those whose footprints reach it (about 60 of 256 for an LWA station), padded to
// K steps of 16.  Per tile and group of 128 / (2 P) frames
//   D_even[pair][n] = W_even[pair][e] . V[n][e]      n = (pol, re | im, frame): 128 columns
//   D_odd [pair][n] = W_odd [pair][e] . V[n][e]
// with the voltages exact in FP16 (4- and 8-bit samples times a power of two) and each weight
// split into FP16 w_hi + w_lo (what is left: up to 2^-23 of the weight, where FP32 rounds to 2^-24), both
// accumulated in FP32 in TMEM.  Polarisation-mixed voltages (FP32) are split the same way, and
// w_hi v_hi + w_lo v_hi + w_hi v_lo is summed (w_lo v_lo, up to 2^-22 of a product, is left out).  The
// tiles round to 2^-12: errors against 64 bits are those of the FP32 gather kernels to three digits.
// The gather kernels compute the same sums with FP32 FMAs and are bound by shared-memory gathers and list walks
// (7.5 k SM cycles a frame of a 96 x 96 box); here a frame takes its MMAs (64 cycles each, 4 a K step, 32
// frames) and its tile stores, which bound it (LWA block of 1000 samples: 0.46 ms for 2.4 GB, 0.28 with the stores of a group to one frame; 0.97 by gather).
// Work: units of one M-tile and one chunk of up to 4 (8) groups, channel by channel and chunk by chunk, cut
// into one range of equal modelled cost a block.  What bounds a unit is its tile stores (2.7 k
// cycles a group at the memory's write rate), so a finer cut matters more than the weights' reuse: ranges of whole
// channels' groups (SKA-Low: 4 or 5 of 33 tiles) left a fifth of the time to the longest.
// Roles of the 640-thread block (one per SM), all walking the block's range alike; all hand-offs are
// mbarriers with bounded waits:
//   warp 0      issues the MMAs of a K step: (even, odd) x (hi, lo), then frees its operands
//   warps 1-3   build weight steps in a shared-memory ring: zeros, then the step's non-zero
//               weights scattered (about 150 of 4096) -- far fewer bytes than reading the dense
//               operands from L2 (80 KB a tile).  A tile of at most RW steps is built once for all
//               the groups of a staged chunk, a denser one once per group.
//   warps 4-11  stage the raw voltages of up to 4 groups (row stride odd in words, so that lanes
//               = frames read without bank conflicts; 4-byte asynchronous copies, so that a whole
//               chunk is in flight) and expand them, a K step at a time, into FP16 operands: lanes
//               are frames, so a 16-byte chunk store of a warp is contiguous
//   warps 12-19 read D (a lane is a cell pair, a column a frame) and store a pair's real and
//               imaginary FP16 pairs as 8 bytes: 32 lanes fill whole sectors of the tile, no staging
// D is double buffered (2 x 256 TMEM columns), the operand rings hold 6 weight and 8 voltage steps.
#include <math.h>

#include <algorithm>
#include <cstring>
#include <vector>

#include "dftgemm_common.cuh"
#include "epic_internal.h"
#include "kcommon.cuh"
#include "tc_ptx.cuh"
#include "voltage_words.h"

namespace epic {

namespace {

constexpr int kGtThreads = 640;
constexpr int kGtRW = 6;               // weight steps in the ring (a multiple of the builder warps: a slot is one warp's)
constexpr int kGtRV = 8;               // voltage steps in the ring (a multiple of the expander warps)
constexpr int kGtEnt = 10;             // weights a lane loads ahead (320 a step: more than a 7 x 7 GCF's tile of 256 elements has)
constexpr int kGtBuilders = 3, kGtExpanders = 8;
constexpr unsigned kGtWBytes = 16384;  // one weight step: (hi, lo) x (even, odd) x 128 pairs x 16 halves
constexpr unsigned kGtVBytes = 4096;   // one voltage step: 128 columns x 16 halves (mixed: hi, then lo)

// where the staged voltage rows begin in shared memory
__host__ __device__ constexpr unsigned gt_raw_at(bool mix) { return kGtRW * kGtWBytes + kGtRV * kGtVBytes * (mix ? 2 : 1); }

struct GridTcArgs {
    const uint8_t* volt;
    int t0, c0, n_ch, nt, C, A;
    const int4* box;
    const int4* tbox;
    uint8_t* tiles;
    unsigned long long tile_stride;
    int* status;
    const int* tile0;       // [C + 1] first M-tile of each channel
    const int* unit0;       // [tiles + 1] first K step of each tile
    const int* ent0;        // [steps + 1] first weight of each K step
    const int2* ent;        // weights: byte offset in the step's hi half, value (scaled)
    const int* el;          // 16 (complex weights: 8) elements of each K step
    const long long* tcum;  // [tiles + 1] prefix sums of the tiles' costs per group
    int dense;              // the tiles' K is not padded (k_dftgemm_ws3 reads them)
    int ngr;                // frame groups of the launch
    int gc, nch;            // groups per staged chunk, chunks
    int raw_stride;         // bytes of a staged frame row (4 x odd)
    int shift;              // rows are staged shifted to a word boundary (samples at no multiple of their size)
    int edges;              // rows that do not begin and end at a word
    uint32_t vscale, vbias; // half2: 2^-s, and what the decode's offset becomes
    const float4* jones;    // MIX: [C][A][2] polarisation-mixing rows (conj J)
    float unscale;          // MIX: 2^-s of the results (the weights are scaled, the voltages are not)
};

__device__ __forceinline__ int gt_uni(int x) { return __shfl_sync(0xffffffffu, x, 0); }

// A whole warp's bounded wait for a barrier phase: the same answer for every lane.
__device__ __forceinline__ bool gt_wait(uint64_t* bar, uint32_t parity)
{
    if (__all_sync(0xffffffffu, tc::mbar_try_wait(bar, parity))) return true;
    const long long t0 = clock64();
    for (;;) {
        if (__all_sync(0xffffffffu, tc::mbar_try_wait(bar, parity))) return true;
        if (__any_sync(0xffffffffu, clock64() - t0 > kWaitBudget)) return false;
    }
}

__device__ __forceinline__ uint32_t hfma2_u(uint32_t a, uint32_t b, uint32_t c)
{
    uint32_t d;
    asm("fma.rn.f16x2 %0, %1, %2, %3;" : "=r"(d) : "r"(a), "r"(b), "r"(c));
    return d;
}

// Two samples' parts as integers u + offset in the low bits of each half (0 <= u < 1024) ->
// FP16 (u - offset) 2^-s: 0x6400 | u is 1024 + u, exact, and the fused multiply-add rounds once.
__device__ __forceinline__ uint32_t gt_dec(uint32_t u, uint32_t flip, const GridTcArgs& a)
{
    return hfma2_u((u ^ flip) | 0x64006400u, a.vscale, a.vbias);
}

// Raw sample words of element e of a staged frame row: P samples of BITS / 4 bytes.
template <int P, int BITS>
__device__ __forceinline__ uint32_t gt_raw(const uint8_t* row, int e)
{
    if (P * BITS == 16) return *reinterpret_cast<const uint32_t*>(row + 4 * e);
    if (P * BITS == 8) return *reinterpret_cast<const uint16_t*>(row + 2 * e);
    return row[e];
}

// The same part (pol p, q: 0 real, 1 imaginary) of two elements' raw words as FP16 pairs.
template <int P, int BITS>
__device__ __forceinline__ uint32_t gt_part(uint32_t w0, uint32_t w1, int p, int q, const GridTcArgs& a)
{
    if (BITS == 4) {  // byte p: real in the high nibble
        const uint32_t u = w0 | (w1 << 16);
        return gt_dec((u >> (8 * p + (q ? 0 : 4))) & 0x000F000Fu, 0x00080008u, a);
    }
    const int b = 2 * p + q;  // byte of the sample pair: real, imaginary
    return gt_dec(__byte_perm(w0, w1, b | 0x40 | ((4 + b) << 8) | 0x4000) & 0x00FF00FFu, 0x00800080u, a);
}

// MIX: a frame's polarisation-mixed samples of one element (FP32, as load_pair computes them),
// part by part (X re, X im, Y re, Y im).
template <int BITS>
__device__ __forceinline__ float4 gt_mix(uint32_t raw, const float4* jm)
{
    float2 x, y;
    if (BITS == 4) {
        x = unpack44(raw & 0xFFu);
        y = unpack44(raw >> 8);
    } else {
        x = make_float2((float)(int8_t)raw, (float)(int8_t)(raw >> 8));
        y = make_float2((float)(int8_t)(raw >> 16), (float)(int8_t)(raw >> 24));
    }
    const float4 r0 = __ldg(jm), r1 = __ldg(jm + 1);
    const float2 mx = cfma(make_float2(r0.z, r0.w), y, cmul(make_float2(r0.x, r0.y), x));
    const float2 my = cfma(make_float2(r1.z, r1.w), y, cmul(make_float2(r1.x, r1.y), x));
    return make_float4(mx.x, mx.y, my.x, my.y);
}

__device__ __forceinline__ void cp_async4(uint32_t dst, const void* src)
{
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(dst), "l"(src) : "memory");
}

// Stages rows that do not begin and end at a word: the aligned words that hold a byte of the row, whose samples keep
// their offset in the first, or (shift) those words shifted to a word boundary.  Words that reach outside the
// launch's voltages (of its first row and its last) are read by bytes.
__device__ __forceinline__ void gt_stage_edges(const uint8_t* lo, const uint8_t* hi, const uint8_t* src, size_t step, int FB, int nf,
                                            uint8_t* raw, int raw_stride, int shift, int xw, int lane)
{
    auto byte = [](const uint8_t* q) { return __ldg(q); };
    auto word = [&](const uint8_t* q) {
        return in_block(q, 4, lo, hi) ? __ldg(reinterpret_cast<const uint32_t*>(q)) : edge_word(q, lo, hi, byte);
    };
    if (!shift) {
        for (int f = xw; f < nf; f += kGtExpanders) {
            const uint8_t* r = src + f * step;
            const int o = (int)((uintptr_t)r & 3), nw = row_words(o, FB);
            const uint8_t* w = r - o;
            const uint32_t d = tc::smem_u32(raw) + f * raw_stride;
            if (in_block(w, 4 * nw, lo, hi)) {
                for (int j = lane; j < nw; j += 32) cp_async4(d + 4 * j, w + 4 * j);
            } else {
                for (int j = lane; j < nw; j += 32)
                    if (in_block(w + 4 * j, 4, lo, hi)) cp_async4(d + 4 * j, w + 4 * j);
                    else reinterpret_cast<uint32_t*>(raw + (size_t)f * raw_stride)[j] = edge_word(w + 4 * j, lo, hi, byte);
            }
        }
        asm volatile("cp.async.wait_all;" ::: "memory");
        return;
    }
    const int nw = (FB + 3) >> 2;
    for (int f = xw; f < nf; f += 4 * kGtExpanders)
        for (int j = lane; j < nw; j += 32) {
            uint32_t v[4];
#pragma unroll
            for (int k = 0; k < 4; ++k)
                if (f + kGtExpanders * k < nf) {
                    const uint8_t* r = src + (f + kGtExpanders * k) * step;
                    const int o = (int)((uintptr_t)r & 3);
                    const uint8_t* w = r - o + 4 * j;
                    v[k] = __funnelshift_r(word(w), 4 * j + 4 < o + FB ? word(w + 4) : 0u, 8 * o);
                }
#pragma unroll
            for (int k = 0; k < 4; ++k)
                if (f + kGtExpanders * k < nf)
                    reinterpret_cast<uint32_t*>(raw + (size_t)(f + kGtExpanders * k) * raw_stride)[j] = v[k];
        }
}

__device__ __forceinline__ float gt_lo(float v) { return v - __half2float(__float2half_rn(v)); }

// First unit (local channel, chunk, tile) of block b: the one at its share of the launch's cost.
__device__ __forceinline__ int4 gt_start(const GridTcArgs& a, int b, int lane)
{
    const int* t0 = a.tile0 + a.c0;
    const long long base = __ldg(a.tcum + __ldg(t0)), all = __ldg(a.tcum + __ldg(t0 + a.n_ch)) - base;
    if (b == (int)gridDim.x) return make_int4(a.n_ch, 0, __ldg(t0 + a.n_ch), 0);
    const long long s = all * a.nch * b / gridDim.x;
    const int cl = warp_find(0, a.n_ch, lane, s, [&](int c) { return (__ldg(a.tcum + __ldg(t0 + c)) - base) * a.nch; });
    const int ta = __ldg(t0 + cl), tb = __ldg(t0 + cl + 1);
    const long long cb = __ldg(a.tcum + ta), w = __ldg(a.tcum + tb) - cb, r = s - (cb - base) * a.nch;
    const int ch = (int)min((long long)(a.nch - 1), r / w);
    const int t = warp_find(ta, tb, lane, r - ch * w, [&](int i) { return __ldg(a.tcum + i) - cb; });
    return make_int4(cl, ch, t, 0);
}

template <int P, int BITS, bool CPLX, bool MIX>
__global__ void __launch_bounds__(kGtThreads, 1) k_dftgemm_grid_tc(GridTcArgs a)
{
    constexpr unsigned VB = kGtVBytes * (MIX ? 2 : 1);  // bytes of a voltage step
    constexpr int FG = 64 / P;                 // frames of a group
    constexpr int EL = CPLX ? 8 : 16;          // elements of a K step
    extern __shared__ __align__(1024) uint8_t smem[];
    __shared__ uint64_t w_full[kGtRW], w_free[kGtRW], v_full[kGtRV], v_free[kGtRV], d_full[2], d_empty[2], drain;
    __shared__ uint32_t tmem_sh;
    __shared__ int err_sh;
    __shared__ int4 range[2];  // first unit and the next block's
    const int tid = threadIdx.x, warp = gt_uni(tid >> 5), lane = tid & 31;
    if (warp == 0) {
        tc::tmem_alloc(&tmem_sh, 512);
        tc::tmem_relinquish();
    }
    if (tid == 32) {
        for (int i = 0; i < kGtRW; ++i) {
            tc::mbar_init(&w_full[i], 1);
            tc::mbar_init(&w_free[i], 1);
        }
        for (int i = 0; i < kGtRV; ++i) {
            tc::mbar_init(&v_full[i], 1);
            tc::mbar_init(&v_free[i], 1);
        }
        for (int i = 0; i < 2; ++i) {
            tc::mbar_init(&d_full[i], 1);
            tc::mbar_init(&d_empty[i], 8);
        }
        tc::mbar_init(&drain, 1);
        err_sh = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 2 || warp == 3) {
        const int4 r = gt_start(a, blockIdx.x + warp - 2, lane);
        if (lane == 0) range[warp - 2] = r;
    }
    tc::fence_before_sync();
    __syncthreads();
    tc::fence_after_sync();
    const uint32_t tmem = gt_uni(tmem_sh);
    uint8_t* sbase = smem + ((1024u - (tc::smem_u32(smem) & 1023u)) & 1023u);
    const uint32_t sW = tc::smem_u32(sbase), sV = sW + kGtRW * kGtWBytes;
    uint8_t* raw = sbase + gt_raw_at(MIX);
    if (tid == 0) tc::grid_launch_dependents();  // k_dftgemm_ws3, which waits for the tiles
    const int4 first = range[0], last = range[1];

    // Every role's walk through the block's units: f(channel, local channel, tiles [T0, T1), first
    // group, groups, end of the groups that follow for the same tiles' channel) per staged chunk.
    auto walk = [&](auto&& f) {
        int cl = gt_uni(first.x), ch = gt_uni(first.y), T0 = gt_uni(first.z);
        const int ecl = gt_uni(last.x), ech = gt_uni(last.y), eT = gt_uni(last.z);
        while (cl < ecl || (cl == ecl && (ch < ech || (ch == ech && T0 < eT)))) {
            const int c = a.c0 + cl, Tn = gt_uni(a.tile0[c + 1]);
            const int T1 = cl == ecl && ch == ech ? eT : Tn, gb = ch * a.gc, g1 = min(a.ngr, gb + a.gc);
            const bool more = ch + 1 < a.nch && (cl < ecl || ch < ech);
            if (T1 > T0) f(c, cl, T0, T1, gb, g1 - gb, more ? min(a.ngr, g1 + a.gc) : g1);
            if (++ch == a.nch) {
                ch = 0;
                ++cl;
                T0 = Tn;
            } else {
                T0 = gt_uni(a.tile0[c]);
            }
        }
    };
    bool good = true;  // a role whose wait ran out walks on without waiting or working

    if (warp == 0) {
        // ------------------------------------------------------------ MMAs
        const uint32_t lead = tc::elect_one();
        const uint32_t id = tc::idesc_f16_f32(128, 128);
        int ws = 0, vs = 0;                 // ring slots
        uint32_t ph_w = 0, ph_v = 0;        // parities, one bit a slot
        unsigned nd = 0;                    // D buffers filled so far
        walk([&](int, int, int T0, int T1, int, int ng, int) {
            for (int t = T0; t < T1 && good; ++t) {
                const int steps = gt_uni(a.unit0[t + 1] - a.unit0[t]);
                const bool keep = steps <= kGtRW;  // the tile's weights stay for every group
                const int wb = ws;
                for (int g = 0; g < ng && good; ++g, ++nd) {
                    const int b = nd & 1;
                    const uint32_t d = tmem + 256 * b;
                    if (nd >= 2) good = gt_wait(&d_empty[b], ((nd >> 1) - 1) & 1u);
                    if (keep) ws = wb;
                    for (int s = 0; s < steps && good; ++s) {
                        if (!keep || g == 0) {
                            good = gt_wait(&w_full[ws], (ph_w >> ws) & 1u);
                            ph_w ^= 1u << ws;
                        }
                        good = good && gt_wait(&v_full[vs], (ph_v >> vs) & 1u);
                        if (!good) break;
                        ph_v ^= 1u << vs;
                        tc::fence_after_sync();
                        const uint32_t wa = tc::desc_step_lo(sW + ws * kGtWBytes, 2048);
                        const uint32_t va = tc::desc_step_lo(sV + vs * VB, 2048);
                        tc::mma_f16_lead<tc::kDescStep128Hi>(d, wa, va, id, s > 0, lead);
                        tc::mma_f16_lead<tc::kDescStep128Hi>(d + 128, wa + (4096 >> 4), va, id, s > 0, lead);
                        tc::mma_f16_lead<tc::kDescStep128Hi>(d, wa + (8192 >> 4), va, id, 1, lead);
                        tc::mma_f16_lead<tc::kDescStep128Hi>(d + 128, wa + (12288 >> 4), va, id, 1, lead);
                        if (MIX) {  // w_hi v_lo (w_lo v_lo is far below the tiles' rounding)
                            tc::mma_f16_lead<tc::kDescStep128Hi>(d, wa, va + (kGtVBytes >> 4), id, 1, lead);
                            tc::mma_f16_lead<tc::kDescStep128Hi>(d + 128, wa + (4096 >> 4), va + (kGtVBytes >> 4), id, 1, lead);
                        }
                        tc::mma_commit_lead(&v_free[vs], lead);
                        if (!keep || g == ng - 1) tc::mma_commit_lead(&w_free[ws], lead);
                        if (++vs == kGtRV) vs = 0;
                        if (++ws == kGtRW) ws = 0;
                    }
                    if (good) tc::mma_commit_lead(&d_full[b], lead);
                }
            }
        });
        // every MMA of this block is complete before its memory goes (bounded)
        tc::mma_commit_lead(&drain, lead);
        if (!gt_wait(&drain, 0) || !good) err_sh = 1;
    } else if (warp < 4) {
        // ------------------------------------------------------------ weight steps
        unsigned q = 0;  // steps built so far by all builders
        walk([&](int, int, int T0, int T1, int, int ng, int) {
            for (int t = T0; t < T1; ++t) {
                const int ub = a.unit0[t], steps = gt_uni(a.unit0[t + 1] - ub);
                const int n = steps <= kGtRW ? steps : steps * ng;
                for (int i = 0; i < n && good; ++i, ++q) {
                    const int slot = q % kGtRW;
                    if (slot % kGtBuilders != warp - 1) continue;  // a slot is always the same warp's
                    const int u = ub + (steps <= kGtRW ? i : i % steps);
                    const int e0 = __ldg(a.ent0 + u) + lane, e1 = __ldg(a.ent0 + u + 1);
                    int2 en[kGtEnt];  // the weights' latency runs under the wait and the zeros
#pragma unroll
                    for (int k = 0; k < kGtEnt; ++k) en[k] = e0 + 32 * k < e1 ? __ldg(a.ent + e0 + 32 * k) : make_int2(-1, 0);
                    if (q >= kGtRW) good = gt_wait(&w_free[slot], (q / kGtRW - 1) & 1u);
                    if (!good) break;
                    const uint32_t dst = sW + slot * kGtWBytes;
#pragma unroll 8
                    for (int k = 0; k < (int)(kGtWBytes / 512); ++k) tc::st_shared_v4(dst + k * 512 + lane * 16, 0, 0, 0, 0);
                    __syncwarp();
                    auto put = [&](int2 w2) {
                        const float w = __int_as_float(w2.y);
                        const __half hi = __float2half_rn(w), lo = __float2half_rn(w - __half2float(hi));
                        uint8_t* o = sbase + slot * kGtWBytes + w2.x;
                        *reinterpret_cast<__half*>(o) = hi;
                        *reinterpret_cast<__half*>(o + 8192) = lo;
                    };
#pragma unroll
                    for (int k = 0; k < kGtEnt; ++k)
                        if (en[k].x >= 0) put(en[k]);
                    for (int k = e0 + 32 * kGtEnt; k < e1; k += 32) put(__ldg(a.ent + k));
                    tc::fence_proxy_async();
                    __syncwarp();
                    if (lane == 0) mbar_arrive(&w_full[slot]);
                }
            }
        });
        if (!good) err_sh = 1;
    } else if (warp < 4 + kGtExpanders) {
        // ------------------------------------------------------------ voltages
        const int FB = a.A * P * (BITS / 4);
        unsigned q = 0;  // steps expanded so far by all expanders
        walk([&](int c, int, int T0, int T1, int gb, int ng, int gend) {
            const int f0 = gb * FG, nf = min(a.nt - f0, ng * FG);
            asm volatile("bar.sync 1, %0;" ::"n"(32 * kGtExpanders) : "memory");  // the last chunk's rows are read
            const uint8_t* src = a.volt + ((size_t)(a.t0 + f0) * a.C + c) * (size_t)FB;
            const size_t step = (size_t)a.C * FB;
            const int xw = warp - 4;
            if (!a.edges) {  // rows of whole words
                for (int f = xw; f < nf; f += kGtExpanders) {
                    const uint8_t* r = src + f * step;
                    const uint32_t d = tc::smem_u32(raw) + f * a.raw_stride;
                    for (int j = lane; j < FB >> 2; j += 32) cp_async4(d + 4 * j, r + 4 * j);
                }
                asm volatile("cp.async.wait_all;" ::: "memory");
            } else {
                gt_stage_edges(a.volt, a.volt + (size_t)(a.t0 + a.nt) * step, src, step, FB, nf, raw, a.raw_stride, a.shift, xw, lane);
            }
            if (!a.shift) {
                // the next chunk's rows into L2
                const int more = min(a.nt - f0, (gend - gb) * FG), lines = (FB + 127) >> 7;
                for (int i = tid - 128; i < (more - nf) * lines && i < a.gc * FG * lines; i += 32 * kGtExpanders) {
                    const int f = i / lines;
                    asm volatile("prefetch.global.L2 [%0];" ::"l"(src + (nf + f) * step + 128 * (i - f * lines)));
                }
            }
            asm volatile("bar.sync 1, %0;" ::"n"(32 * kGtExpanders) : "memory");
            for (int t = T0; t < T1; ++t) {
                const int ub = a.unit0[t], steps = gt_uni(a.unit0[t + 1] - ub);
                for (int g = 0; g < ng; ++g)
                    for (int s = 0; s < steps && good; ++s, ++q) {
                        const int slot = q % kGtRV;
                        if (slot % kGtExpanders != warp - 4) continue;
                        int4 el[EL / 4];  // the step's elements
#pragma unroll
                        for (int k = 0; k < EL / 4; ++k)
                            el[k] = __ldg(reinterpret_cast<const int4*>(a.el + (size_t)(ub + s) * EL) + k);
                        if (q >= kGtRV) good = gt_wait(&v_free[slot], (q / kGtRV - 1) & 1u);
                        if (!good) break;
                        const uint32_t dst = sV + slot * VB + lane * 16;
                        const float4* jm = MIX ? a.jones + (size_t)c * a.A * 2 : nullptr;
                        for (int h = 0; h < 2 / P; ++h) {  // one pol: two sets of 32 frames
                            const int f = g * FG + 32 * h + lane;
                            const uint8_t* row = raw + (size_t)f * a.raw_stride;
                            if (!a.shift) row += ((uint32_t)(uintptr_t)src + (uint32_t)f * (uint32_t)step) & 3u;
#pragma unroll
                            for (int o = 0; o < 2; ++o) {  // 16-byte chunks (8 K positions)
                                constexpr int NE = EL / 2;
                                uint32_t rw[NE];
                                if (MIX) {  // mixed samples as FP16 hi and lo, pairs of K positions
                                    uint32_t h[4][4], l[4][4];  // [part][pair]
#pragma unroll
                                    for (int k = 0; k < NE; k += 2) {
                                        const int4 e = el[(o * NE + k) / 4];
                                        const int e0 = k & 2 ? e.z : e.x, e1 = k & 2 ? e.w : e.y;
                                        const float4 m0 = gt_mix<BITS>(gt_raw<P, BITS>(row, e0), jm + 2 * e0);
                                        const float4 m1 = gt_mix<BITS>(gt_raw<P, BITS>(row, e1), jm + 2 * e1);
                                        const float u0[4] = {m0.x, m0.y, m0.z, m0.w}, u1[4] = {m1.x, m1.y, m1.z, m1.w};
#pragma unroll
                                        for (int r = 0; r < 4; ++r) {
                                            if (!CPLX) {
                                                h[r][k / 2] = pack_h2(u0[r], u1[r]);
                                                l[r][k / 2] = pack_h2(gt_lo(u0[r]), gt_lo(u1[r]));
                                            } else {  // re row (vr, -vi), im row (vi, vr) of each element
                                                const float s0 = r & 1 ? u0[r - 1] : -u0[r + 1], s1 = r & 1 ? u1[r - 1] : -u1[r + 1];
                                                h[r][k] = pack_h2(u0[r], s0);
                                                h[r][k + 1] = pack_h2(u1[r], s1);
                                                l[r][k] = pack_h2(gt_lo(u0[r]), gt_lo(s0));
                                                l[r][k + 1] = pack_h2(gt_lo(u1[r]), gt_lo(s1));
                                            }
                                        }
                                    }
#pragma unroll
                                    for (int r = 0; r < 4; ++r) {
                                        const uint32_t at = dst + o * 2048 + r * 512;
                                        tc::st_shared_v4(at, h[r][0], h[r][1], h[r][2], h[r][3]);
                                        tc::st_shared_v4(at + kGtVBytes, l[r][0], l[r][1], l[r][2], l[r][3]);
                                    }
                                    continue;
                                }
#pragma unroll
                                for (int k = 0; k < NE; k += 4) {
                                    const int4 e = el[(o * NE + k) / 4];
                                    rw[k] = gt_raw<P, BITS>(row, e.x);
                                    rw[k + 1] = gt_raw<P, BITS>(row, e.y);
                                    rw[k + 2] = gt_raw<P, BITS>(row, e.z);
                                    rw[k + 3] = gt_raw<P, BITS>(row, e.w);
                                }
#pragma unroll
                                for (int p = 0; p < P; ++p) {
                                    uint32_t re[4], im[4];
                                    if (!CPLX) {
#pragma unroll
                                        for (int k = 0; k < 4; ++k) {
                                            re[k] = gt_part<P, BITS>(rw[(2 * k) % NE], rw[(2 * k + 1) % NE], p, 0, a);
                                            im[k] = gt_part<P, BITS>(rw[(2 * k) % NE], rw[(2 * k + 1) % NE], p, 1, a);
                                        }
                                    } else {  // K positions (w_re, w_im) of an element: re row (vr, -vi), im row (vi, vr)
#pragma unroll
                                        for (int k = 0; k < 4; k += 2) {
                                            const uint32_t vr = gt_part<P, BITS>(rw[k], rw[k + 1], p, 0, a);
                                            const uint32_t vi = gt_part<P, BITS>(rw[k], rw[k + 1], p, 1, a);
                                            im[k] = __byte_perm(vi, vr, 0x5410);      // (vi, vr) of the first
                                            im[k + 1] = __byte_perm(vi, vr, 0x7632);  // and of the second
                                            re[k] = __byte_perm(vr, vi, 0x5410) ^ 0x80000000u;
                                            re[k + 1] = __byte_perm(vr, vi, 0x7632) ^ 0x80000000u;
                                        }
                                    }
                                    const uint32_t at = dst + o * 2048 + (P == 2 ? p * 1024 : h * 512);
                                    tc::st_shared_v4(at, re[0], re[1], re[2], re[3]);
                                    tc::st_shared_v4(at + (P == 2 ? 512 : 1024), im[0], im[1], im[2], im[3]);
                                }
                            }
                        }
                        tc::fence_proxy_async();
                        __syncwarp();
                        if (lane == 0) mbar_arrive(&v_full[slot]);
                    }
            }
        });
        if (!good) err_sh = 1;
    } else {
        // ------------------------------------------------------------ tiles
        const int q4 = warp & 3, j = (warp >> 2) & 1;  // cell pairs; pol j, or half j of the one pol's frames
        constexpr int IM = P == 2 ? 32 : 64;            // columns from a frame's real part to its imaginary part
        const uint32_t lanes = tmem + ((uint32_t)(32 * q4) << 16) + (P == 2 ? 64 : 32) * j;
        const size_t frame_step = a.dense ? a.tile_stride : (size_t)a.n_ch * a.tile_stride;
        unsigned nd = 0;
        walk([&](int c, int cl, int T0, int T1, int gb, int ng, int) {
            if (!good) return;
            const int4 bx = a.box[c], tp = a.tbox[c];
            const int half = bx.z >> 1, pairs = tp.z * half;
            const int K1 = 2 * bx.z;
            const uint32_t part_bytes = (uint32_t)(P * tp.x) * pad64(K1) * 2;
            for (int t = T0; t < T1; ++t) {
                const int pr = (t - a.tile0[c]) * 128 + 32 * q4 + lane, y = pr / half, x = 2 * (pr - y * half);
                const bool live = pr < pairs;
                uint32_t off = 0;
                if (live) {
                    off = a.dense ? tile_dense_off(y, 2 * x, tp.x, P, K1) : tile_part_off(y, 2 * x, tp.x, P, part_bytes);
                    if (P == 2) off += j * tp.x * (a.dense ? tile_dense_row(2 * x, K1) : 128);
                }
                for (int g = 0; g < ng; ++g, ++nd) {
                    const int b = nd & 1, f0 = (gb + g) * FG + (P == 2 ? 0 : 32 * j), nf = min(32, a.nt - f0);
                    good = gt_wait(&d_full[b], (nd >> 1) & 1u);
                    if (!good) return;
                    tc::fence_after_sync();
                    uint8_t* q = a.tiles + (a.dense ? (size_t)cl * a.nt + f0 : (size_t)f0 * a.n_ch + cl) * a.tile_stride + off;
                    uint32_t d[4][8];  // real and imaginary parts of the even and the odd cell, 8 frames
                    auto load = [&](int k) {
                        const uint32_t at = lanes + 256 * b + 8 * k;
                        tmem_ld8(at, d[0]);
                        tmem_ld8(at + 128, d[1]);
                        tmem_ld8(at + IM, d[2]);
                        tmem_ld8(at + IM + 128, d[3]);
                    };
                    load(0);
#pragma unroll
                    for (int k = 0; k < 4; ++k) {
#pragma unroll
                        for (int i = 0; i < 4; ++i) tc::tmem_wait_ld(d[i]);
                        if (MIX) {
#pragma unroll
                            for (int i = 0; i < 32; ++i)
                                d[i >> 3][i & 7] = __float_as_uint(__uint_as_float(d[i >> 3][i & 7]) * a.unscale);
                        }
                        uint2 v[8];
#pragma unroll
                        for (int i = 0; i < 8; ++i)
                            v[i] = make_uint2(pack_h2(__uint_as_float(d[0][i]), __uint_as_float(d[1][i])),
                                              pack_h2(__uint_as_float(d[2][i]), __uint_as_float(d[3][i])));
                        if (k < 3) {
                            load(k + 1);
                        } else {  // this warp's part of D is in registers
                            tc::fence_before_sync();
                            __syncwarp();
                            if (lane == 0) mbar_arrive(&d_empty[b]);
                        }
                        if (live && 8 * k + 8 <= nf) {
#pragma unroll
                            for (int i = 0; i < 8; ++i, q += frame_step) *reinterpret_cast<uint2*>(q) = v[i];
                        } else if (live) {
#pragma unroll
                            for (int i = 0; i < 8; ++i, q += frame_step)
                                if (8 * k + i < nf) *reinterpret_cast<uint2*>(q) = v[i];
                        }
                    }
                }
            }
        });
        if (!good) err_sh = 1;
    }
    tc::fence_before_sync();
    __syncthreads();
    if (warp == 0) tc::tmem_dealloc(tmem, 512);
    if (err_sh && tid == 0) atomicExch(a.status, 1);
}

using GridTcFn = void (*)(GridTcArgs);

GridTcFn grid_tc_fn(const epic_plan_s* p)
{
    const bool cplx = p->gcf.kind != EPIC_GCF_GAUSSIAN, four = p->bits == 4;
    if (!p->jones.empty()) {  // two pols
        if (four) return cplx ? k_dftgemm_grid_tc<2, 4, true, true> : k_dftgemm_grid_tc<2, 4, false, true>;
        return cplx ? k_dftgemm_grid_tc<2, 8, true, true> : k_dftgemm_grid_tc<2, 8, false, true>;
    }
    if (p->P == 2) {
        if (four) return cplx ? k_dftgemm_grid_tc<2, 4, true, false> : k_dftgemm_grid_tc<2, 4, false, false>;
        return cplx ? k_dftgemm_grid_tc<2, 8, true, false> : k_dftgemm_grid_tc<2, 8, false, false>;
    }
    if (four) return cplx ? k_dftgemm_grid_tc<1, 4, true, false> : k_dftgemm_grid_tc<1, 4, false, false>;
    return cplx ? k_dftgemm_grid_tc<1, 8, true, false> : k_dftgemm_grid_tc<1, 8, false, false>;
}

template <class T>
cudaError_t put(T** dst, const std::vector<T>& v, size_t* bytes)
{
    cudaError_t e = cudaMalloc(reinterpret_cast<void**>(dst), std::max<size_t>(1, v.size()) * sizeof(T));
    if (e == cudaSuccess && !v.empty()) e = cudaMemcpy(*dst, v.data(), v.size() * sizeof(T), cudaMemcpyHostToDevice);
    *bytes += v.size() * sizeof(T);
    return e;
}

// bytes of a staged frame row: the words that hold a byte of it, wherever it begins (rows of whole
// words: at a word), an odd number of them
int raw_stride(const epic_plan_s* p)
{
    const int fb = p->A * p->P * (p->bits / 4), words = fb % 4 ? (fb + 6) / 4 : fb / 4;
    return 4 * (words | 1);
}

size_t grid_tc_smem(const epic_plan_s* p, int gc)
{
    return gt_raw_at(!p->jones.empty()) + (size_t)gc * (64 / p->P) * raw_stride(p) + 1024;  // + 1 KB to align the operands
}

}  // namespace

// Groups of frames per staged chunk (parameter grid_frames: 1, 2, 4 or 8 groups of 64 / pols frames, of which as
// many are staged as fit: values that the gather kernels take stay valid).
epic_status grid_tc_config(epic_plan_s* p, int gc)
{
    if (!p->tc.gt_tile0 || (gc != 1 && gc != 2 && gc != 4 && gc != 8)) return EPIC_ERR_UNSUPPORTED;
    const void* fn = (const void*)grid_tc_fn(p);
    cudaFuncAttributes fa{};
    cudaError_t e = cudaFuncGetAttributes(&fa, fn);
    if (e != cudaSuccess) return cuda_fail(p, e, "cudaFuncGetAttributes(k_dftgemm_grid_tc)");
    int fit = gc;
    while (fit > 1 && grid_tc_smem(p, fit) + fa.sharedSizeBytes > (size_t)p->smem_optin) fit >>= 1;
    if (grid_tc_smem(p, fit) + fa.sharedSizeBytes > (size_t)p->smem_optin) return EPIC_ERR_UNSUPPORTED;
    e = allow_max_smem(fn, p->smem_optin);
    if (e != cudaSuccess) return cuda_fail(p, e, "cudaFuncSetAttribute(k_dftgemm_grid_tc)");
    p->tc.grid_frames = gc;
    p->tc.gt_groups = fit;
    p->tc.grid_smem = (int)grid_tc_smem(p, fit);
    p->tc.grid_blocks = p->sm_count;
    return EPIC_OK;
}

// Tables of the tensor-core gridding kernel.  UNSUPPORTED (with nothing allocated) for plans it
// does not take: frames too large to stage, weights (or mixing matrices) outside the range in which
// FP16 hi + lo parts are as accurate as FP32.
epic_status grid_tc_setup(epic_plan_s* p)
{
    const int A = p->A, C = p->C, K = p->K, P = p->P;
    const bool cplx = p->gcf.kind != EPIC_GCF_GAUSSIAN;
    if (grid_tc_smem(p, 1) + 2048 > (size_t)p->smem_optin) return EPIC_ERR_UNSUPPORTED;
    // Mixed samples are split without scaling: at most 4 |J| of the largest sample, J's largest part, in FP16's
    // range, and the parts' absolute floor (2^-25) below the rounding of the tiles in every channel: with gains of
    // 1/64 it adds 1e-4 to the tiles' error squared (with 1e-5, images were off by 4.0e-4 of their norm; 2.6e-4
    // by the gather kernels).  A channel of zeros is exact.
    if (!p->jones.empty()) {
        float jmax = 0.f;
        for (int c = 0; c < C; ++c) {
            float m = 0.f;
            for (size_t i = (size_t)c * A * 8; i < (size_t)(c + 1) * A * 8; ++i) m = std::max(m, fabsf(p->jones[i]));
            if (m > 0.f && m < 0.015625f) return EPIC_ERR_UNSUPPORTED;
            jmax = std::max(jmax, m);
        }
        const float vmax = p->bits == 8 ? 128.f : 8.f;
        if (!(jmax >= 0.25f && jmax <= 128.f && 4.f * vmax * jmax <= 65504.f)) return EPIC_ERR_UNSUPPORTED;
    }
    double wmax = 0.0;
    for (double w : p->w_re) wmax = std::max(wmax, fabs(w));
    for (double w : p->w_im) wmax = std::max(wmax, fabs(w));
    // weights times 2^s and voltages times 2^-s: w_lo's last bit is then 2^-24-s, far below
    // FP32's rounding of the largest weights; |w| 2^s <= 2^14 keeps w_hi finite
    int ex = 0;
    frexp(wmax, &ex);  // wmax <= 2^ex
    const int s = std::min(10, 14 - ex);
    if (!std::isfinite(wmax) || ex < -8 || s < 0) return EPIC_ERR_UNSUPPORTED;
    const int EL = cplx ? 8 : 16;
    std::vector<int> tile0(C + 1, 0), unit0(1, 0), ent0(1, 0), el;
    std::vector<int2> ent;
    std::vector<long long> tcum(1, 0);
    ent.reserve(p->n_contrib * (cplx ? 2 : 1));
    struct En {
        int e, off;
        float wr, wi;
    };
    std::vector<std::vector<En>> lists;
    std::vector<int> at;  // position of an element in the tile's list
    for (int c = 0; c < C; ++c) {
        const Box b = p->box[c];
        const int half = b.nx / 2, pairs = p->tc.tbox_h[c].z * half, tiles = (pairs + 127) / 128;
        lists.assign(tiles, {});
        for (int e = 0; e < A; ++e) {  // in element order, so each list is
            const int fx = p->first_x[(size_t)c * A + e] - b.x0, fy = p->first_y[(size_t)c * A + e] - b.y0;
            for (int ty = 0; ty < K; ++ty)
                for (int tx = 0; tx < K; ++tx) {
                    const int x = fx + tx, pr = (fy + ty) * half + (x >> 1);
                    const size_t o = (((size_t)c * A + e) * K + ty) * K + tx;
                    lists[pr >> 7].push_back(En{e, (x & 1) * 4096 + (pr & 127) * 16, (float)p->w_re[o], (float)p->w_im[o]});
                }
        }
        for (const std::vector<En>& L : lists) {
            int n = 0;  // distinct elements
            for (size_t i = 0; i < L.size(); ++i) n += i == 0 || L[i].e != L[i - 1].e;
            const int steps = std::max(1, (n + EL - 1) / EL);
            const size_t u = unit0.back();
            el.resize((u + steps) * EL, 0);
            int k = -1;
            size_t i = 0;
            for (int st = 0; st < steps; ++st) {
                for (; i < L.size(); ++i) {
                    if (i == 0 || L[i].e != L[i - 1].e) {
                        if (k + 1 == (st + 1) * EL) break;
                        ++k;
                        el[u * EL + k] = L[i].e;
                    }
                    auto add = [&](int kk, float w) {
                        const float ws = (float)ldexp((double)w, s);
                        int bits;
                        std::memcpy(&bits, &ws, sizeof bits);
                        ent.push_back(make_int2(L[i].off + (kk >> 3) * 2048 + (kk & 7) * 2, bits));
                    };
                    const int kk = k - st * EL;
                    if (cplx) {
                        add(2 * kk, L[i].wr);
                        add(2 * kk + 1, L[i].wi);
                    } else {
                        add(kk, L[i].wr);
                    }
                }
                ent0.push_back((int)ent.size());
            }
            unit0.push_back((int)u + steps);
            // SM cycles of a group, as measured: the tile's stores, or its weight steps when they do not stay
            tcum.push_back(tcum.back() + (steps <= kGtRW ? 2700LL : 800LL * steps));
        }
        tile0[c + 1] = tile0[c] + tiles;
        if (ent.size() > (1u << 30) || el.size() > (1u << 30)) return EPIC_ERR_UNSUPPORTED;
    }
    size_t bytes = 0;
    cudaError_t e = put(&p->tc.gt_tile0, tile0, &bytes);
    if (e == cudaSuccess) e = put(&p->tc.gt_unit0, unit0, &bytes);
    if (e == cudaSuccess) e = put(&p->tc.gt_ent0, ent0, &bytes);
    if (e == cudaSuccess) e = put(&p->tc.gt_ent, ent, &bytes);
    if (e == cudaSuccess) e = put(&p->tc.gt_el, el, &bytes);
    if (e == cudaSuccess) e = put(&p->tc.gt_tcum, tcum, &bytes);
    p->tc.gt_scale = s;
    p->tc.gt_tiles_h = tile0;
    p->tc.gt_cost_h.resize(C + 1);
    for (int c = 0; c <= C; ++c) p->tc.gt_cost_h[c] = tcum[tile0[c]];
    p->dt.dft_bytes += bytes;
    if (e != cudaSuccess) return cuda_fail(p, e, "tensor-core gridding tables");
    return EPIC_OK;
}

// Whether the plan's launch configuration is this kernel's for its frames
bool grid_tc_configured(const epic_plan_s* p)
{
    return p->tc.gt_tile0 && (size_t)p->tc.grid_smem == grid_tc_smem(p, p->tc.gt_groups);
}

void grid_tc_launch(epic_plan_s* p, const uint8_t* volt, int t0, int nt, int c0, int n_ch, cudaStream_t s)
{
    GridTcArgs a{};
    a.volt = volt;
    a.t0 = t0;
    a.c0 = c0;
    a.n_ch = n_ch;
    a.nt = nt;
    a.C = p->C;
    a.A = p->A;
    a.box = p->dt.box;
    a.tbox = p->tc.tbox;
    a.tiles = (uint8_t*)p->scratch;
    a.tile_stride = p->tc.stride;
    a.dense = dftgemm_dense(p);
    a.status = p->tc.status;
    a.tile0 = p->tc.gt_tile0;
    a.unit0 = p->tc.gt_unit0;
    a.ent0 = p->tc.gt_ent0;
    a.ent = p->tc.gt_ent;
    a.el = p->tc.gt_el;
    a.tcum = p->tc.gt_tcum;
    const int fb = p->A * p->P * (p->bits / 4), FG = 64 / p->P;
    a.ngr = (nt + FG - 1) / FG;
    a.raw_stride = raw_stride(p);
    // a sample (all pols) of 4, 2 or 1 bytes is read from shared memory at its offset in the words, and
    // rows of whole words have no word to spare for an offset
    a.shift = (uintptr_t)volt % (p->P * p->bits / 4) != 0 || (fb % 4 == 0 && (uintptr_t)volt % 4 != 0) ? 1 : 0;
    a.edges = fb % 4 != 0 || (uintptr_t)volt % 4 != 0 ? 1 : 0;
    // chunks of equal numbers of groups, short enough for about 16 units a block
    const int tiles = p->tc.gt_tiles_h[c0 + n_ch] - p->tc.gt_tiles_h[c0], full = (a.ngr + p->tc.gt_groups - 1) / p->tc.gt_groups;
    const int want = std::max(full, std::min(a.ngr, (16 * p->sm_count + tiles - 1) / tiles));
    a.gc = (a.ngr + want - 1) / want;
    a.nch = (a.ngr + a.gc - 1) / a.gc;
    const int off = p->bits == 4 ? 1024 + 8 : 1024 + 128;
    const uint32_t sc = (uint32_t)(15 - p->tc.gt_scale) << 10;  // FP16 2^-s
    const __half hb = __float2half((float)-ldexp((double)off, -p->tc.gt_scale));
    uint16_t bb;
    std::memcpy(&bb, &hb, sizeof bb);
    a.jones = p->dt.jones;
    a.unscale = (float)ldexp(1.0, -p->tc.gt_scale);
    a.vscale = sc | (sc << 16);
    a.vbias = (uint32_t)bb | ((uint32_t)bb << 16);
    grid_tc_fn(p)<<<(unsigned)std::min<long long>(p->sm_count, (long long)tiles * a.nch), kGtThreads, p->tc.grid_smem, s>>>(a);
}

}  // namespace epic
