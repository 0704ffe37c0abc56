// Plain FP32 path of the EPIC hot loop (paper Sec. 2, Eq. 1-2).  Per chunk of time samples, two
// kernels with one HBM round trip of the occupied rows between them:
//   k_plain_rows     unpack the voltages (and mix polarisations, when the plan has a mixing
//                    kernel), gather-grid the occupied box of every (t, c) frame (Eq. 1 bracket)
//                    row by row into shared memory and FFT each row along x
//   k_plain_cols     the FFT along y on tiles of adjacent columns (rows outside the box are
//                    zero), the XX, YY, XY products, summed over the chunk's frames in registers
//                    and added to the images (Eq. 2)
//   k_plain_sum      adds the partial sums up where a chunk's frames were cut into slices
// The transforms are register-resident two-pass FFTs.  With full N x N grids going through HBM
// between four kernels (grid, rows, columns, products) the LWA-station block took 34.0 ms, six
// passes over 33.5 GB at 0.87 of the copy rate; the box rows are 48 of 128 there and go through
// once each way.  The tuner's second form (fft = 1) keeps the four kernels with radix-4/2 Stockham
// transforms in shared memory:
//   k_plain_grid, k_plain_fft_rows_smem, k_plain_fft_cols_smem, k_plain_sqacc
#include <algorithm>
#include <cmath>

#include "epic_internal.h"
#include "kcommon.cuh"
#include "tc_ptx.cuh"

namespace epic {

namespace {

constexpr int kThreads = 256;
constexpr int kColTile = 16;
constexpr size_t kGridBudget = 512ull << 20;  // bytes of the chunk grid buffer

// ---- register-resident two-pass FFT ------------------------------------------
// A length-N transform X[k] = sum_n x[n] w^(nk), w = exp(+2 pi i / N) (Eq. 1: + sign,
// unnormalised), is split with N = N1 N2, n = n1 + N1 n2 and k = k2 + N2 k1 into
//   Y[n1][k2] = w^(n1 k2) sum_n2 x[n1 + N1 n2] w_N2^(n2 k2)       (pass 1)
//   X[k2 + N2 k1] = sum_n1 Y[n1][k2] w_N1^(n1 k1)                 (pass 2)
// (the Cooley-Tukey "four-step" factorisation).  Each thread holds whole N2- or
// N1-point transforms in registers; Y goes once through shared memory between
// the passes.  N1 is N2 or 2 N2, so both are at most 32 for N <= 512.

// exp(+2 pi i m / 32), m < 16: the twiddles inside the register transforms.
__constant__ float2 c_w32[16] = {
    {1.0f, 0.0f},                    {0.980785251f, 0.195090324f}, {0.923879504f, 0.382683426f},
    {0.831469595f, 0.555570245f},    {0.707106769f, 0.707106769f}, {0.555570245f, 0.831469595f},
    {0.382683426f, 0.923879504f},    {0.195090324f, 0.980785251f}, {0.0f, 1.0f},
    {-0.195090324f, 0.980785251f},   {-0.382683426f, 0.923879504f}, {-0.555570245f, 0.831469595f},
    {-0.707106769f, 0.707106769f},   {-0.831469595f, 0.555570245f}, {-0.923879504f, 0.382683426f},
    {-0.980785251f, 0.195090324f}};

__host__ __device__ constexpr int ilog2(int n) { return n <= 1 ? 0 : 1 + ilog2(n >> 1); }

// k with its low `bits` bits reversed
__host__ __device__ constexpr int bit_reverse(int k, int bits)
{
    int r = 0;
    for (int i = 0; i < bits; ++i) r |= ((k >> i) & 1) << (bits - 1 - i);
    return r;
}

// d * exp(+2 pi i m / 32); m is a compile-time constant once the callers are unrolled
__device__ __forceinline__ float2 w32_mul(float2 d, int m)
{
    if (m == 0) return d;
    if (m == 8) return make_float2(-d.y, d.x);
    return cmul(d, c_w32[m]);
}

// In-place R-point transform (+ sign, unnormalised) of v by radix-2 decimation in
// frequency: afterwards v[bit_reverse(k, log2 R)] = sum_n v_in[n] exp(+2 pi i n k / R).
// A span-h stage maps (a, b) = (v[i], v[i + h]) to (a + b, (a - b) w_2h^j), j = i mod h.
template <int R>
__device__ __forceinline__ void dft_reg(float2 (&v)[R])
{
#pragma unroll
    for (int h = R / 2; h >= 1; h >>= 1) {
#pragma unroll
        for (int b = 0; b < R; b += 2 * h) {
#pragma unroll
            for (int j = 0; j < h; ++j) {
                const float2 x = v[b + j], y = v[b + j + h];
                v[b + j] = make_float2(x.x + y.x, x.y + y.y);
                v[b + j + h] = w32_mul(make_float2(x.x - y.x, x.y - y.y), j * (32 / (2 * h)));
            }
        }
    }
}

// tw[k2 N1 + n1] = w^(n1 k2) from the plan's table twg[m] = exp(+2 pi i m / N), m < N/2
template <int N1, int N2>
__device__ __forceinline__ void load_step_twiddles(float2* tw, const float2* __restrict__ twg)
{
    constexpr int N = N1 * N2;
    for (int i = threadIdx.x; i < N; i += blockDim.x) {
        const int m = (i / N1) * (i % N1);  // < N
        const float2 t = twg[m < N / 2 ? m : m - N / 2];
        tw[i] = m < N / 2 ? t : make_float2(-t.x, -t.y);
    }
}

// How k_plain_rows reads a frame's samples: decoded from the frame (which begins at an even byte where samples have
// 8 bits), staged FP32 pairs, or decoded by bytes.
enum RowForm { kRowDecode, kRowStaged, kRowBytes };

// Samples of element e (0 .. P-1 pols) of a frame.
template <int P, int FORM>
__device__ __forceinline__ void frame_sample(const float2* sv, const uint8_t* fr, int e, int bits, const float4* jm,
                                             float2 (&v)[P])
{
    if (FORM == kRowStaged) {
        if (P == 2) {
            const float4 q = *reinterpret_cast<const float4*>(sv + 2 * e);
            v[0] = make_float2(q.x, q.y);
            v[P - 1] = make_float2(q.z, q.w);
        } else {
            v[0] = sv[e];
        }
    } else if (P == 2) {
        const float4 q = load_pair<FORM == kRowDecode>(fr, e, bits, jm);
        v[0] = make_float2(q.x, q.y);
        v[P - 1] = make_float2(q.z, q.w);
    } else {
        v[0] = load_sample<FORM == kRowDecode>(fr, e, bits);
    }
}

constexpr int kRowThreads = 256;
constexpr int kRowFrames = 2;  // frames of a block: each list entry read from L1 serves both (one in short launches)

// bytes of k_plain_rows's shared memory beside the frames: twiddles, Y (whose rows the box columns share)
template <int N1, int N2>
__host__ __device__ constexpr size_t rows_fft_smem()
{
    return sizeof(float2) * ((size_t)N1 * N2 + (size_t)(kRowThreads / N2) * N2 * (N1 + 1));
}

// Gridded and row-transformed frames (LWA station: 5.1 ms a block, 2.9 ms of it the 12.6 GB of row
// stores, the rest the gather's dependent list and voltage reads; 5.6 ms with three blocks an SM instead of
// four, before a row's cells shared Y's memory): block = frames F blockIdx.x ... of
// channel blockIdx.y, slice blockIdx.z of the box rows.
// Rows go in batches of 256 / N2 (both frames, all pols, a few y): the batch's cells are gathered
// one per thread and step, both frames and pols at once, then N2 threads a row run the two FFT
// passes (thread j takes n1 = j, j + N2 in pass 1 and k2 = j in pass 2; Y is stored [k2][n1] with
// stride N1 + 1, which no pass-1 store or pass-2 load of a warp meets twice in one bank) and
// store rows[(t C + c) P + p][y - y0][N].
template <int N1, int N2, int P, int FORM, bool CPLX, int F>
__global__ void __launch_bounds__(kRowThreads) k_plain_rows(const uint8_t* __restrict__ volt, int t0, int nt, int C, int A,
                                                            int bits, const int4* __restrict__ box,
                                                            const int* __restrict__ cell_off,
                                                            const int* __restrict__ cell_ptr,
                                                            const int* __restrict__ ce, const float2* __restrict__ cw,
                                                            const float4* __restrict__ jones, int frame_in_smem,
                                                            int ny_max, const float2* __restrict__ twg,
                                                            float2* __restrict__ rows)
{
    constexpr int N = N1 * N2, RPC = kRowThreads / N2, S = N2 * (N1 + 1), T = N1 / N2;
    constexpr int L1 = ilog2(N1), L2 = ilog2(N2), YR = RPC / (F * P);
    static_assert(YR >= 1, "a batch holds a row of every frame and pol");
    extern __shared__ float2 sm[];
    tc::grid_launch_dependents();  // k_plain_cols
    const int tid = threadIdx.x, c = blockIdx.y, f0 = F * blockIdx.x;
    const int4 b = box[c];
    // box padding beyond the grid holds nothing; the rows end with this block's slice of the batches
    const int nx = min(b.z, N - b.x), nb = (min(b.w, N - b.y) + YR - 1) / YR;
    const int ny = min(min(b.w, N - b.y), nb * ((int)blockIdx.z + 1) / (int)gridDim.z * YR);
    float2* tw = sm;               // [N2][N1]
    float2* y = tw + N;            // [RPC][N2][N1 + 1]
    uint8_t* fr_s = reinterpret_cast<uint8_t*>(y + RPC * S);
    float2* sv = reinterpret_cast<float2*>(fr_s);  // [F][A][P]
    const int FB = A * P * (bits / 4);
    const float4* jm = jones ? jones + (size_t)c * A * 2 : nullptr;
    const uint8_t* fr[F];
#pragma unroll
    for (int f = 0; f < F; ++f) {
        fr[f] = volt + ((size_t)(t0 + min(f0 + f, nt - 1)) * C + c) * (size_t)FB;  // an odd last frame twice
        if (FORM == kRowStaged) {
            stage_frame(sv + (size_t)f * A * P, fr[f], A, P, bits, jm);
        } else if (frame_in_smem) {
            uint8_t* d = fr_s + (size_t)f * ((FB + 15) & ~15);
            if (((FB | (int)(uintptr_t)fr[f]) & 3) == 0)
                for (int i = tid; i < FB >> 2; i += kRowThreads)
                    reinterpret_cast<uint32_t*>(d)[i] = __ldg(reinterpret_cast<const uint32_t*>(fr[f]) + i);
            else
                for (int i = tid; i < FB; i += kRowThreads) d[i] = __ldg(fr[f] + i);
            fr[f] = d;
        }
    }
    load_step_twiddles<N1, N2>(tw, twg);
    const int* ptr = cell_ptr + cell_off[c];
    const int rl = tid / N2, j = tid % N2;             // this thread's row of a batch and its place in it
    const int rf = rl / (P * YR), rp = rl / YR % P, ry = rl % YR;
    for (int yb = nb * (int)blockIdx.z / (int)gridDim.z * YR; yb < ny; yb += YR) {
        __syncthreads();  // frames staged; the last batch's rows are read
        for (int i = tid; i < YR * nx; i += kRowThreads) {
            const int r = i / nx, x = i - r * nx;
            float2 acc[F][P];
#pragma unroll
            for (int f = 0; f < F; ++f)
#pragma unroll
                for (int p = 0; p < P; ++p) acc[f][p] = make_float2(0.f, 0.f);
            if (yb + r < ny) {
                const int cell = (yb + r) * b.z + x, q1 = __ldg(ptr + cell + 1);
                if constexpr (F == 1) {  // short launches: four entries' loads at once (lists of 81 entries: 227 -> 162 us)
                    auto entry = [&](int i) {
                        const float2 w = CPLX ? __ldg(cw + i) : make_float2(__ldg(&cw[i].x), 0.f);
                        float2 v[P];
                        frame_sample<P, FORM>(sv, fr[0], __ldg(ce + i), bits, jm, v);
#pragma unroll
                        for (int p = 0; p < P; ++p) acc[0][p] = cfma(w, v[p], acc[0][p]);
                    };
#pragma unroll 4
                    for (int q = __ldg(ptr + cell); q < q1; ++q) entry(q);
                } else {
                    for (int q = __ldg(ptr + cell); q < q1; ++q) {
                        const int e = __ldg(ce + q);
                        const float2 w = CPLX ? __ldg(cw + q) : make_float2(__ldg(&cw[q].x), 0.f);
#pragma unroll
                        for (int f = 0; f < F; ++f) {
                            float2 v[P];
                            frame_sample<P, FORM>(sv + (size_t)f * A * P, fr[f], e, bits, jm, v);
#pragma unroll
                            for (int p = 0; p < P; ++p) {
                                if (CPLX) acc[f][p] = cfma(w, v[p], acc[f][p]);
                                else acc[f][p] = make_float2(fmaf(w.x, v[p].x, acc[f][p].x), fmaf(w.x, v[p].y, acc[f][p].y));
                            }
                        }
                    }
                }
            }
#pragma unroll
            for (int f = 0; f < F; ++f)
#pragma unroll
                for (int p = 0; p < P; ++p) y[((f * P + p) * YR + r) * S + x] = acc[f][p];
        }
        __syncthreads();
        float2 u[T][N2];
        float2* yr = y + rl * S;  // the row's cells (nx <= N of them), then its Y
#pragma unroll
        for (int t = 0; t < T; ++t)
#pragma unroll
            for (int n2 = 0; n2 < N2; ++n2) {
                const int x = j + N2 * t + N1 * n2 - b.x;
                u[t][n2] = x >= 0 && x < nx ? yr[x] : make_float2(0.f, 0.f);
            }
        __syncwarp();  // a row's N2 threads are of one warp: its cells are read
#pragma unroll
        for (int t = 0; t < T; ++t) {
            dft_reg<N2>(u[t]);
            const int n1 = j + N2 * t;
#pragma unroll
            for (int k2 = 0; k2 < N2; ++k2) yr[k2 * (N1 + 1) + n1] = cmul(u[t][bit_reverse(k2, L2)], tw[k2 * N1 + n1]);
        }
        __syncthreads();
        float2 z[N1];
#pragma unroll
        for (int n1 = 0; n1 < N1; ++n1) z[n1] = yr[j * (N1 + 1) + n1];
        dft_reg<N1>(z);
        tc::grid_wait();  // the chunk before is read (later batches: at once)
        if (f0 + rf < nt && yb + ry < ny) {
            float2* o = rows + ((((size_t)(f0 + rf) * C + c) * P + rp) * ny_max + yb + ry) * N + j;
#pragma unroll
            for (int k1 = 0; k1 < N1; ++k1) o[N2 * k1] = z[bit_reverse(k1, L1)];
        }
    }
}

// One pixel's products added to its sums.
template <int P>
__device__ __forceinline__ void add_products(float2 X, float2 Y, float& xx, float& yy, float& rxy, float& ixy)
{
    xx = fmaf(X.x, X.x, fmaf(X.y, X.y, xx));
    if (P == 2) {
        yy = fmaf(Y.x, Y.x, fmaf(Y.y, Y.y, yy));
        rxy = fmaf(X.x, Y.x, fmaf(X.y, Y.y, rxy));
        ixy = fmaf(X.y, Y.x, fmaf(-X.x, Y.y, ixy));
    }
}

__device__ __forceinline__ void cp_async16(void* dst, const void* src)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src)
                 : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int K>
__device__ __forceinline__ void cp_async_wait()
{
    asm volatile("cp.async.wait_group %0;" ::"n"(K) : "memory");
}

// frames k_plain_cols sums in registers before it adds them to memory: the rounding error of long
// sums stays that of short ones
constexpr int kColRun = 64;

// frames of box columns k_plain_cols holds in shared memory (two in flight); none at N = 512, where
// one would take half an SM
constexpr int col_stages(int N) { return N <= 256 ? 3 : 0; }

// Column transforms and products: block = TX adjacent columns of channel blockIdx.y and slice
// blockIdx.z of the chunk's frames (with sub-integrations: of its intervals, or slice blockIdx.z % cuts of
// interval blockIdx.z / cuts); N2 threads a column,
// lanes on adjacent columns (every global access of a warp one contiguous run per row, Y
// [n1][k2][column] without bank conflicts).  The box rows of the next two frames are on their way
// into shared memory while a frame is transformed (loaded when needed, the HBM latency of each
// pol showed: 4.4 k cycles a tile and frame).  A thread ends up with the pixels ky = j + N2 k1 of
// its column and keeps their sums in registers; at N1 = 32 X's pixels wait in the thread's own
// slots of the exchange buffer while Y is transformed.  out: the images, or the slice's partial sums.
// CUT: that last form (a form of its own: the LWA station's columns took 2 % longer with the choice inside).
template <int N1, int N2, int TX, int P, bool CUT>
__global__ void __launch_bounds__(TX * N2) k_plain_cols(const float2* __restrict__ rows, int nt, int C, int ny_max,
                                                        const int4* __restrict__ box, const float2* __restrict__ twg,
                                                        float* __restrict__ out, float* __restrict__ partial,
                                                        int accumulate, int sub, int out_iv0, int cuts)
{
    constexpr int N = N1 * N2, T = N1 / N2, L1 = ilog2(N1), L2 = ilog2(N2), NP = P == 2 ? 4 : 1, ST = col_stages(N);
    constexpr size_t NN = (size_t)N * N;
    constexpr bool kKeep = N1 <= 16;  // X's pixels stay in registers
    extern __shared__ __align__(16) float2 sm[];
    float2* tw = sm;                          // [N2][N1]
    float2* y = sm + N;                       // [P][N1][N2][TX]
    float2* stage = y + (size_t)P * N * TX;   // [ST][P][ny_max][TX]
    const int xl = threadIdx.x % TX, j = threadIdx.x / TX, c = blockIdx.y, xb = blockIdx.x * TX;
    const int4 b = box[c];
    const int y0 = b.y, ny = min(b.w, N - b.y);
    load_step_twiddles<N1, N2>(tw, twg);
    const int unit = sub > 0 ? sub : 1, units = nt / unit, S = gridDim.z;
    const int z = CUT ? blockIdx.z % cuts : 0, i0 = CUT ? blockIdx.z / cuts * sub : 0;
    const int ta = CUT ? i0 + (int)((long long)sub * z / cuts) : (int)((long long)units * blockIdx.z / S) * unit;
    const int tb = CUT ? i0 + (int)((long long)sub * (z + 1) / cuts) : (int)((long long)units * (blockIdx.z + 1) / S) * unit;
    float xx[N1], yy[P == 2 ? N1 : 1], rxy[P == 2 ? N1 : 1], ixy[P == 2 ? N1 : 1];
    auto clear = [&]() {
#pragma unroll
        for (int i = 0; i < N1; ++i) {
            xx[i] = 0.f;
            if (P == 2) yy[i] = rxy[i] = ixy[i] = 0.f;
        }
    };
    auto store = [&](float* o, bool add) {
        o += (size_t)j * N + xb + xl;
#pragma unroll
        for (int k1 = 0; k1 < N1; ++k1) {
            float* q = o + (size_t)(N2 * k1) * N;
            q[0] = (add ? q[0] : 0.f) + xx[k1];
            if (P == 2) {
                q[NN] = (add ? q[NN] : 0.f) + yy[k1];
                q[2 * NN] = (add ? q[2 * NN] : 0.f) + rxy[k1];
                q[3 * NN] = (add ? q[3 * NN] : 0.f) + ixy[k1];
            }
        }
    };
    auto frame = [&](int t, int p) { return rows + (((size_t)t * C + c) * P + p) * (size_t)ny_max * N + xb; };
    auto fetch = [&](int t) {  // frame t's box columns -> its stage (a group is committed either way)
        if (t < tb) {
            float2* d = stage + (size_t)(t % (ST ? ST : 1)) * P * ny_max * TX;
            constexpr int Q = TX / 2;  // 16-byte chunks of a row
            for (int i = threadIdx.x; i < P * ny * Q; i += TX * N2) {
                const int row = i / Q, q = i % Q, p = P == 2 && row >= ny ? 1 : 0, r = row - p * ny;
                cp_async16(d + ((size_t)p * ny_max + r) * TX + 2 * q, frame(t, p) + (size_t)r * N + 2 * q);
            }
        }
        cp_async_commit();
    };
    auto image = [&](int t) {  // where frame t's sums go
        if (CUT) return partial + (((size_t)z * units + t / sub) * C + c) * NP * NN;  // this slice's sums of every interval
        return sub > 0 ? out + ((size_t)(out_iv0 + t / sub) * C + c) * NP * NN
                       : (partial ? partial + (size_t)blockIdx.z * C * NP * NN : out) + (size_t)c * NP * NN;
    };
    clear();
    bool add = accumulate != 0;
    tc::grid_launch_dependents();  // k_plain_rows of the next chunk
    tc::grid_wait();               // this chunk's rows are complete
    if (ST) {
        fetch(ta);
        fetch(ta + 1);
    }
    for (int t = ta; t < tb;) {
        // a run: up to kColRun frames of one image set
        const int te = min(min(t + kColRun, tb), sub > 0 ? t - t % sub + sub : tb);
        float* const target = image(t);
        const bool end = te == tb || (sub > 0 && te % sub == 0);
        for (; t < te; ++t) {
            if (ST) cp_async_wait<1>();
            __syncthreads();  // this frame's columns (and the twiddles) are in; the last frame's buffers are read
            if (ST) fetch(t + 2);
            else if (t + 1 < tb)  // the next one's into L2 meanwhile (512-pixel station: 1.63 -> 1.56 ms)
                for (int i = threadIdx.x; i < P * ny; i += TX * N2) {
                    const int p = P == 2 && i >= ny ? 1 : 0;
                    asm volatile("prefetch.global.L2 [%0];" ::"l"(frame(t + 1, p) + (size_t)(i - p * ny) * N));
                }
#pragma unroll
            for (int p = 0; p < P; ++p) {
                const float2* r = ST ? stage + ((size_t)(t % (ST ? ST : 1)) * P + p) * ny_max * TX + xl : frame(t, p) + xl;
                const int ld = ST ? TX : N;
                float2 u[T][N2];
#pragma unroll
                for (int i = 0; i < T; ++i)
#pragma unroll
                    for (int n2 = 0; n2 < N2; ++n2) {
                        const int row = j + N2 * i + N1 * n2 - y0;
                        u[i][n2] = row >= 0 && row < ny ? r[(size_t)row * ld] : make_float2(0.f, 0.f);
                    }
#pragma unroll
                for (int i = 0; i < T; ++i) {
                    dft_reg<N2>(u[i]);
                    const int n1 = j + N2 * i;
#pragma unroll
                    for (int k2 = 0; k2 < N2; ++k2)
                        y[((p * N1 + n1) * N2 + k2) * TX + xl] = cmul(u[i][bit_reverse(k2, L2)], tw[k2 * N1 + n1]);
                }
            }
            __syncthreads();
            float2* own = y + (size_t)j * TX + xl;  // this thread's k2 = j, stride N2 TX over n1
            float2 zx[N1];
#pragma unroll
            for (int n1 = 0; n1 < N1; ++n1) zx[n1] = own[n1 * N2 * TX];
            dft_reg<N1>(zx);
            if (P == 1) {
#pragma unroll
                for (int k1 = 0; k1 < N1; ++k1) {
                    const float2 X = zx[bit_reverse(k1, L1)];
                    add_products<1>(X, X, xx[k1], yy[0], rxy[0], ixy[0]);
                }
            } else {
                if (!kKeep) {
#pragma unroll
                    for (int k1 = 0; k1 < N1; ++k1) own[k1 * N2 * TX] = zx[bit_reverse(k1, L1)];
                }
                float2 zy[N1];
#pragma unroll
                for (int n1 = 0; n1 < N1; ++n1) zy[n1] = own[(N1 + n1) * N2 * TX];
                dft_reg<N1>(zy);
#pragma unroll
                for (int k1 = 0; k1 < N1; ++k1) {
                    const float2 X = kKeep ? zx[bit_reverse(k1, L1)] : own[k1 * N2 * TX];
                    constexpr int m = P == 2 ? 1 : 0;
                    add_products<P>(X, zy[bit_reverse(k1, L1)], xx[k1], yy[m * k1], rxy[m * k1], ixy[m * k1]);
                }
            }
        }
        store(target, add);
        clear();
        add = end ? accumulate != 0 : true;
    }
    if (ST) cp_async_wait<0>();
    if (sub == 0 && ta >= tb) store(image(ta), add);  // no frames: zeros
}

__device__ __forceinline__ float add(float a, float b) { return a + b; }
__device__ __forceinline__ float4 add(float4 a, float4 b) { return make_float4(a.x + b.x, a.y + b.y, a.z + b.z, a.w + b.w); }

// out (+)= the slices' partial sums, in slice order, a V at a time (float4 where `out` begins at 16 bytes,
// else float)
template <class V>
__global__ void __launch_bounds__(kThreads) k_plain_sum(const V* __restrict__ partial, size_t n, int S, V* __restrict__ out,
                                                        int accumulate)
{
    for (size_t i = (size_t)blockIdx.x * kThreads + threadIdx.x; i < n; i += (size_t)gridDim.x * kThreads) {
        V a = partial[i];
        for (int k = 1; k < S; ++k) a = add(a, partial[k * n + i]);
        out[i] = accumulate ? add(a, out[i]) : a;
    }
}

template <class V>
void sum_slices(const epic_plan_s* p, const float* partial, size_t n, int S, float* out, bool accumulate, cudaStream_t s)
{
    n /= sizeof(V) / sizeof(float);
    const unsigned blocks = (unsigned)std::min<size_t>((n + kThreads - 1) / kThreads, 8 * (size_t)p->sm_count);
    k_plain_sum<V><<<blocks, kThreads, 0, s>>>(reinterpret_cast<const V*>(partial), n, S, reinterpret_cast<V*>(out),
                                               accumulate ? 1 : 0);
}

// the register-FFT kernels of one N, number of pols and form of the frames and weights
struct RegFft {
    // of one frame a block, of kRowFrames
    void (*rows[2])(const uint8_t*, int, int, int, int, int, const int4*, const int*, const int*, const int*, const float2*,
                    const float4*, int, int, const float2*, float2*);
    // of one frame, read by bytes: 8-bit samples at an odd address in frames that are not staged at all
    void (*rows_bytes)(const uint8_t*, int, int, int, int, int, const int4*, const int*, const int*, const int*, const float2*,
                       const float4*, int, int, const float2*, float2*);
    void (*cols)(const float2*, int, int, int, const int4*, const float2*, float*, float*, int, int, int, int);
    void (*cut)(const float2*, int, int, int, const int4*, const float2*, float*, float*, int, int, int, int);
    int col_tile, col_threads;
    int rows_batch[2];            // box rows a block transforms at once
    size_t rows_fft;
    size_t cols_smem, cols_row;   // cols_row: per box row, the staged frames
};

template <int N1, int N2, int P>
RegFft reg_fft_p(bool staged, bool cplx)
{
    constexpr int N = N1 * N2;
    // 128 threads a block (fewer for the smallest grids): four to eight blocks an SM hide the barriers
    constexpr int TX = 128 / N2 < N ? 128 / N2 : N;
    RegFft f{};
#define EPIC_ROWS(form, F) (cplx ? k_plain_rows<N1, N2, P, form, true, F> : k_plain_rows<N1, N2, P, form, false, F>)
    f.rows[0] = staged ? EPIC_ROWS(kRowStaged, 1) : EPIC_ROWS(kRowDecode, 1);
    f.rows[1] = staged ? EPIC_ROWS(kRowStaged, kRowFrames) : EPIC_ROWS(kRowDecode, kRowFrames);
    f.rows_bytes = EPIC_ROWS(kRowBytes, 1);
#undef EPIC_ROWS
    f.cols = k_plain_cols<N1, N2, TX, P, false>;
    f.cut = k_plain_cols<N1, N2, TX, P, true>;
    f.col_tile = TX;
    f.col_threads = TX * N2;
    f.rows_batch[0] = kRowThreads / N2 / P;
    f.rows_batch[1] = kRowThreads / N2 / (kRowFrames * P);
    f.rows_fft = rows_fft_smem<N1, N2>();
    f.cols_smem = sizeof(float2) * ((size_t)N + (size_t)P * N * TX);
    f.cols_row = sizeof(float2) * (size_t)col_stages(N) * P * TX;
    return f;
}

template <int N1, int N2>
RegFft reg_fft(int P, bool staged, bool cplx)
{
    return P == 2 ? reg_fft_p<N1, N2, 2>(staged, cplx) : reg_fft_p<N1, N2, 1>(staged, cplx);
}

// Frames as staged FP32 samples (as many bytes as fit beside the FFT in a third of an SM), else as
// bytes in shared memory, else read through L1.
enum FrameForm { kFrameStaged, kFrameBytes, kFrameGlobal };

// N = 2^logN, 8 <= N <= 512
RegFft reg_fft_for(const epic_plan_s* p, bool staged)
{
    const bool cplx = p->gcf.kind != EPIC_GCF_GAUSSIAN;
    switch (p->logN) {
        case 3: return reg_fft<4, 2>(p->P, staged, cplx);
        case 4: return reg_fft<4, 4>(p->P, staged, cplx);
        case 5: return reg_fft<8, 4>(p->P, staged, cplx);
        case 6: return reg_fft<8, 8>(p->P, staged, cplx);
        case 7: return reg_fft<16, 8>(p->P, staged, cplx);
        case 8: return reg_fft<16, 16>(p->P, staged, cplx);
        default: return reg_fft<32, 16>(p->P, staged, cplx);
    }
}

size_t cols_smem_for(const epic_plan_s* p, const RegFft& f)
{
    return f.cols_smem + f.cols_row * std::min(p->box_max_y, p->N);
}

size_t frame_smem(const epic_plan_s* p, FrameForm form, int frames = kRowFrames)
{
    const size_t fb = (size_t)p->A * p->P * (p->bits / 4);
    if (form == kFrameStaged) return frames * sizeof(float2) * (size_t)p->A * p->P;
    return form == kFrameBytes ? frames * ((fb + 15) & ~(size_t)15) : 0;
}

FrameForm frame_form(const epic_plan_s* p)
{
    const size_t base = reg_fft_for(p, true).rows_fft, lim = (size_t)p->smem_optin;
    // in a third of an SM: three blocks hide the gather's latency (20 000 elements as bytes in one block an SM
    // 1.97 ms, through L1 1.45); mixed samples stay staged while they fit at all, or every tap would mix again
    if (base + frame_smem(p, kFrameStaged) <= (p->jones.empty() ? lim / 3 : lim)) return kFrameStaged;
    return base + frame_smem(p, kFrameBytes) <= lim / 3 ? kFrameBytes : kFrameGlobal;
}

// Slices of a chunk's frames for k_plain_cols: the number that loses least to the last wave -- of
// blocks over the resident ones and over the SMs, a part-filled wave running faster per block, half
// each -- and to the partial sums' traffic beside the rows'.  One for the LWA station's 1024 tiles
// (6.1 ms a block; 6.8 in three slices), nine for the 64 tiles of the one-channel 512 x 512 station
// (1.65 ms; 1.84 in four, 3.4 in two).
// With sub-integrations a slice is of whole intervals, or each interval is cut (`cuts` slices, whose partial
// sums k_plain_sum adds up): two 250-sample intervals of 8 channels of 64 x 64 pixels 188 us whole, 57 and
// 8 for the sums cut.
int col_slices(const epic_plan_s* p, const RegFft& f, int nt, int slots, int* cuts)
{
    const double B = (double)(p->N / f.col_tile) * p->C;
    const int iv = p->sub > 0 ? std::max(1, nt / p->sub) : 1;
    const double img = sizeof(float) * (double)p->C * p->nprod * p->N * p->N;
    const double rows = sizeof(float2) * (double)nt * p->C * p->P * p->box_max_y * p->N;
    int best = 1;
    double cost = 1e30;
    auto take = [&](int S, double sums) {  // sums: the partial sums' images
        const double w = B * S / slots, m = B * S / p->sm_count;
        const double k = 0.5 * std::ceil(w) / w + 0.5 * std::ceil(m) / m + 2.0 * sums * img / rows;
        if (k >= cost - 1e-9) return false;
        cost = k;
        best = S;
        return true;
    };
    *cuts = 1;
    for (int S = 1; S <= 16 && S <= std::max(1, p->sub > 0 ? std::min(nt / 4, iv) : nt / 4); ++S) take(S, S > 1 && p->sub == 0 ? S : 0);
    for (int q = 2; p->sub > 0 && q <= 16 && q <= p->sub / 4; ++q)
        if (take(iv * q, (double)iv * q)) *cuts = q;
    return best;
}

// Zeros of the N x N planes (P of them, NN apart) outside the occupied box b =
// (x0, y0, width, height): pairs of cells wholly outside take one 16-byte store.
__device__ __forceinline__ void zero_outside_box(float2* g, int N, int P, int4 b)
{
    const size_t NN = (size_t)N * N;
    const float4 z4 = make_float4(0.f, 0.f, 0.f, 0.f);
    for (int i = threadIdx.x; i < N * N / 2; i += blockDim.x) {
        const int cell = 2 * i, y = cell / N, x = cell - y * N;
        const bool row_in = y >= b.y && y < b.y + b.w;
        const bool in0 = row_in && x >= b.x && x < b.x + b.z;
        const bool in1 = row_in && x + 1 >= b.x && x + 1 < b.x + b.z;
        if (!in0 && !in1) {
            for (int p = 0; p < P; ++p) *reinterpret_cast<float4*>(g + p * NN + cell) = z4;
        } else if (in0 != in1) {
            const int zc = in0 ? cell + 1 : cell;
            for (int p = 0; p < P; ++p) g[p * NN + zc] = make_float2(0.f, 0.f);
        }
    }
}

__global__ void __launch_bounds__(kThreads) k_plain_grid(const uint8_t* __restrict__ volt, int t0, int C, int A,
                                                         int P, int N, int bits, const int4* __restrict__ box,
                                                         const int* __restrict__ cell_off,
                                                         const int* __restrict__ cell_ptr,
                                                         const int* __restrict__ ce, const float2* __restrict__ cw,
                                                         const float4* __restrict__ jones, float2* __restrict__ grid)
{
    extern __shared__ float2 sv[];  // [A][P] unpacked (and pol-mixed) voltages of this frame
    const int tl = blockIdx.x, c = blockIdx.y;
    const uint8_t* fr = volt + ((size_t)(t0 + tl) * C + c) * (size_t)A * P * (bits / 4);
    stage_frame(sv, fr, A, P, bits, jones ? jones + (size_t)c * A * 2 : nullptr);
    __syncthreads();
    const int4 b = box[c];
    const int* ptr = cell_ptr + cell_off[c];
    const size_t NN = (size_t)N * N;
    float2* g = grid + ((size_t)tl * C + c) * P * NN;
    // the occupied box (its padding clipped to the grid), one cell per thread and step
    for (int i = threadIdx.x; i < b.z * b.w; i += blockDim.x) {
        const int ry = i / b.z, rx = i - ry * b.z;
        if (b.y + ry >= N || b.x + rx >= N) continue;  // box padding beyond the grid (empty lists)
        const size_t cell = (size_t)(b.y + ry) * N + b.x + rx;
        float2 a0 = make_float2(0.f, 0.f), a1 = make_float2(0.f, 0.f);
        const int q1 = ptr[i + 1];
        for (int q = ptr[i]; q < q1; ++q) {
            const int e = ce[q];
            const float2 w = cw[q];
            a0 = cfma(w, sv[e * P], a0);
            if (P == 2) a1 = cfma(w, sv[e * P + 1], a1);
        }
        g[cell] = a0;
        if (P == 2) g[NN + cell] = a1;
    }
    zero_outside_box(g, N, P, b);
}

// Same as k_plain_grid for frames whose A*P voltages do not fit in shared memory
// (very large arrays): each contribution reads and unpacks its voltage byte
// through the read-only data cache.
__global__ void __launch_bounds__(kThreads) k_plain_grid_g(const uint8_t* __restrict__ volt, int t0, int C, int A,
                                                           int P, int N, int bits, const int4* __restrict__ box,
                                                           const int* __restrict__ cell_off,
                                                           const int* __restrict__ cell_ptr,
                                                           const int* __restrict__ ce, const float2* __restrict__ cw,
                                                           const float4* __restrict__ jones, float2* __restrict__ grid)
{
    const int tl = blockIdx.x, c = blockIdx.y;
    const uint8_t* fr = volt + ((size_t)(t0 + tl) * C + c) * (size_t)A * P * (bits / 4);
    const float4* jm = jones ? jones + (size_t)c * A * 2 : nullptr;
    const int4 b = box[c];
    const int* ptr = cell_ptr + cell_off[c];
    const size_t NN = (size_t)N * N;
    float2* g = grid + ((size_t)tl * C + c) * P * NN;
    for (int i = threadIdx.x; i < b.z * b.w; i += blockDim.x) {
        const int ry = i / b.z, rx = i - ry * b.z;
        if (b.y + ry >= N || b.x + rx >= N) continue;  // box padding beyond the grid (empty lists)
        const size_t cell = (size_t)(b.y + ry) * N + b.x + rx;
        float2 a0 = make_float2(0.f, 0.f), a1 = make_float2(0.f, 0.f);
        const int q1 = ptr[i + 1];
        for (int q = ptr[i]; q < q1; ++q) {
            const int e = ce[q];
            const float2 w = cw[q];
            if (jm) {
                const float4 v = load_pair(fr, e, bits, jm);
                a0 = cfma(w, make_float2(v.x, v.y), a0);
                a1 = cfma(w, make_float2(v.z, v.w), a1);
            } else {
                a0 = cfma(w, load_sample(fr, (size_t)e * P, bits), a0);
                if (P == 2) a1 = cfma(w, load_sample(fr, (size_t)e * P + 1, bits), a1);
            }
        }
        g[cell] = a0;
        if (P == 2) g[NN + cell] = a1;
    }
    zero_outside_box(g, N, P, b);
}

__global__ void __launch_bounds__(kThreads) k_plain_fft_rows_smem(float2* __restrict__ grid, size_t n_rows, int logN,
                                                                  int rows_per_cta, const float2* __restrict__ twg)
{
    extern __shared__ float2 sm[];
    const int N = 1 << logN;
    float2* tw = sm;                       // [N/2]
    float2* a = sm + N / 2;                // [rows][N]
    float2* b = a + (size_t)rows_per_cta * N;
    for (int i = threadIdx.x; i < N / 2; i += blockDim.x) tw[i] = twg[i];
    const size_t r0 = (size_t)blockIdx.x * rows_per_cta;
    const int nr = (int)min((size_t)rows_per_cta, n_rows - r0);
    const float2* src = grid + r0 * N;
    for (int i = threadIdx.x; i < nr * N; i += blockDim.x) a[i] = src[i];
    __syncthreads();
    float2* res = fft_stockham(a, b, logN, nr, 1, N, tw);
    float2* dst = grid + r0 * N;
    for (int i = threadIdx.x; i < nr * N; i += blockDim.x) dst[i] = res[i];
}

__global__ void __launch_bounds__(kThreads) k_plain_fft_cols_smem(float2* __restrict__ grid, int logN, int tile,
                                                                  const float2* __restrict__ twg)
{
    extern __shared__ float2 sm[];
    const int N = 1 << logN;
    const int ld = N + 1;                  // padded column stride in shared memory
    float2* tw = sm;
    float2* a = sm + N / 2;                // [tile][N + 1]
    float2* b = a + (size_t)tile * ld;
    for (int i = threadIdx.x; i < N / 2; i += blockDim.x) tw[i] = twg[i];
    const size_t frame = blockIdx.y;
    const int x0 = blockIdx.x * tile;
    float2* g = grid + frame * (size_t)N * N;
    for (int i = threadIdx.x; i < N * tile; i += blockDim.x) {
        const int row = i / tile, col = i - row * tile;
        a[col * ld + row] = g[(size_t)row * N + x0 + col];
    }
    __syncthreads();
    float2* res = fft_stockham(a, b, logN, tile, 1, ld, tw);
    for (int i = threadIdx.x; i < N * tile; i += blockDim.x) {
        const int row = i / tile, col = i - row * tile;
        g[(size_t)row * N + x0 + col] = res[col * ld + row];
    }
}

// Products summed over the chunk's frames (sub = 0), or over each interval of sub
// frames (sub-integrations, paper Sec. 4): interval k of the chunk goes to image
// set out_iv0 + k.
__global__ void __launch_bounds__(kThreads) k_plain_sqacc(const float2* __restrict__ grid, int nt, int C, int P, int N,
                                                          float* __restrict__ out, int accumulate, int sub, int out_iv0)
{
    const size_t NN = (size_t)N * N;
    const size_t pix = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int c = blockIdx.y;
    if (pix >= NN) return;
    const int nprod = P == 2 ? 4 : 1;
    const int span = sub > 0 ? sub : nt;
    for (int iv = 0; iv * span < nt; ++iv) {
    float xx = 0.f, yy = 0.f, rxy = 0.f, ixy = 0.f;
#pragma unroll 4
    for (int tl = iv * span; tl < (iv + 1) * span; ++tl) {
        const float2* g = grid + ((size_t)tl * C + c) * P * NN;
        const float2 X = g[pix];
        xx = fmaf(X.x, X.x, fmaf(X.y, X.y, xx));
        if (P == 2) {
            const float2 Y = g[NN + pix];
            yy = fmaf(Y.x, Y.x, fmaf(Y.y, Y.y, yy));
            rxy = fmaf(X.x, Y.x, fmaf(X.y, Y.y, rxy));
            ixy = fmaf(X.y, Y.x, fmaf(-X.x, Y.y, ixy));
        }
    }
    float* o = out + ((size_t)(out_iv0 + iv) * C + c) * nprod * NN + pix;
    if (accumulate) {
        o[0] += xx;
        if (P == 2) { o[NN] += yy; o[2 * NN] += rxy; o[3 * NN] += ixy; }
    } else {
        o[0] = xx;
        if (P == 2) { o[NN] = yy; o[2 * NN] = rxy; o[3 * NN] = ixy; }
    }
    }
}

int rows_per_cta_for(int N) { return std::max(1, 2048 / N); }

size_t rows_smem(int N) { return sizeof(float2) * ((size_t)N / 2 + 2ull * rows_per_cta_for(N) * N); }

int col_tile_for(int N) { return std::min(kColTile, N); }

size_t cols_smem(int N) { return sizeof(float2) * ((size_t)N / 2 + 2ull * col_tile_for(N) * (N + 1)); }

}  // namespace

// Time samples per chunk so that the chunk's rows (fft = 1: whole grids) take at most `budget`
// bytes (at least one sample), and the buffer for them and for the slices' partial sums.
epic_status plain_set_chunk(epic_plan_s* p, size_t budget)
{
    const int rows = p->plain_fft == 0 ? std::min(p->box_max_y, p->N) : p->N;
    const size_t per_t = (size_t)p->C * p->P * rows * p->N * sizeof(float2);
    // at most 65,535 (sample, channel, pol) columns: the second grid dimension of the column FFT
    const size_t max_t = 65535 / ((size_t)p->C * p->P);
    int tcn = (int)std::max<size_t>(1, std::min<size_t>(std::min<size_t>((size_t)p->max_time, max_t), budget / per_t));
    if (p->sub > 0) tcn = std::max(p->sub, tcn - tcn % p->sub);  // whole sub-integrations per chunk
    if ((size_t)tcn > max_t) {
        p->last_error = "plain path: sub_int x n_chan x n_pol exceeds 65,535";
        return EPIC_ERR_UNSUPPORTED;
    }
    size_t bytes = (per_t * tcn + 255) & ~(size_t)255;
    int slices = 1, cuts = 1;
    if (p->plain_fft == 0) {
        const RegFft f = reg_fft_for(p, frame_form(p) == kFrameStaged);
        int occ = 0;
        cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, (const void*)f.cols, f.col_threads, cols_smem_for(p, f));
        if (e != cudaSuccess) return cuda_fail(p, e, "cudaOccupancyMaxActiveBlocksPerMultiprocessor(k_plain_cols)");
        p->plain_slots = std::max(1, occ) * p->sm_count;
        slices = col_slices(p, f, tcn, p->plain_slots, &cuts);
        const int sums = p->sub == 0 ? (slices > 1 ? slices : 0) : cuts > 1 ? tcn / p->sub * cuts : 0;
        bytes += sizeof(float) * (size_t)sums * p->C * p->nprod * p->N * p->N;
    }
    const epic_status st = scratch_resize(p, bytes, false, "plain grid buffer");
    if (st != EPIC_OK) return st;
    p->chunk_budget = budget;
    p->plain_slices = slices;
    p->plain_cuts = cuts;
    p->time_chunk = tcn;
    return EPIC_OK;
}

// Form of the plain path: 0 two kernels with register two-pass transforms, 1 four kernels with
// shared-memory Stockham transforms
epic_status plain_set_fft(epic_plan_s* p, int v)
{
    if (v != 0 && v != 1) {
        p->last_error = "plain path: FFT form must be 0 or 1";
        return EPIC_ERR_INVALID_ARG;
    }
    if (v == p->plain_fft) return EPIC_OK;
    const int old = p->plain_fft;
    p->plain_fft = v;
    epic_status st = plain_set_chunk(p, p->chunk_budget);  // the chunk's buffer holds other rows
    if (st != EPIC_OK) {
        p->plain_fft = old;
        plain_set_chunk(p, p->chunk_budget);
    }
    return st;
}

epic_status plain_setup(epic_plan_s* p)
{
    p->plain_fft = 0;
    cudaError_t e = cudaSuccess;
    const size_t sg = sizeof(float2) * (size_t)p->A * p->P;
    if (sg > 48 * 1024 && (int)sg <= p->smem_optin) {  // larger frames use k_plain_grid_g
        e = allow_max_smem((const void*)k_plain_grid, p->smem_optin);
        if (e != cudaSuccess) return cuda_fail(p, e, "cudaFuncSetAttribute(k_plain_grid)");
    }
    e = allow_max_smem((const void*)k_plain_fft_rows_smem, p->smem_optin);
    if (e != cudaSuccess) return cuda_fail(p, e, "cudaFuncSetAttribute(k_plain_fft_rows_smem)");
    e = allow_max_smem((const void*)k_plain_fft_cols_smem, p->smem_optin);
    if (e != cudaSuccess) return cuda_fail(p, e, "cudaFuncSetAttribute(k_plain_fft_cols_smem)");
    const RegFft rf = reg_fft_for(p, frame_form(p) == kFrameStaged);
    if (rf.rows_fft > (size_t)p->smem_optin || cols_smem_for(p, rf) > (size_t)p->smem_optin) {
        p->last_error = "plain path: FFT shared memory exceeds the device limit";
        return EPIC_ERR_UNSUPPORTED;
    }
    for (int i = 0; i < 4 && e == cudaSuccess; ++i)  // short launches stage their frames
        e = allow_max_smem((const void*)(i < 2 ? rf : reg_fft_for(p, true)).rows[i & 1], p->smem_optin);
    if (e == cudaSuccess) e = allow_max_smem((const void*)rf.rows_bytes, p->smem_optin);
    if (e != cudaSuccess) return cuda_fail(p, e, "cudaFuncSetAttribute(k_plain_rows)");
    e = allow_max_smem((const void*)rf.cols, p->smem_optin);
    if (e == cudaSuccess) e = allow_max_smem((const void*)rf.cut, p->smem_optin);
    if (e != cudaSuccess) return cuda_fail(p, e, "cudaFuncSetAttribute(k_plain_cols)");
    return plain_set_chunk(p, kGridBudget);
}

// A launch that may start where blocks of the kernel before it on the stream have ended (early; that kernel
// allows it, and this one waits for its end before it touches what the other reads or writes): a chunk's two
// kernels of 0.2 ms each left the chip half empty at every end.
template <class F, class... X>
static void launch_early(bool early, F* fn, dim3 grid, int threads, size_t smem, cudaStream_t s, X... x)
{
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = grid;
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = early;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    cudaLaunchKernelEx(&cfg, fn, x...);  // errors: as after any launch, by cudaGetLastError
}

epic_status plain_run(epic_plan_s* p, const uint8_t* volt, int T, cudaStream_t s, float* out, bool accumulate)
{
    const int C = p->C, P = p->P, N = p->N, A = p->A;
    if (!p->scratch) return no_scratch(p);
    float2* grid = (float2*)p->scratch;
    const size_t sg = sizeof(float2) * (size_t)A * P;
    const int bits = p->bits;
    for (int t0 = 0; t0 < T; t0 += p->time_chunk) {
        const int nt = std::min(p->time_chunk, T - t0);
        const int acc = (accumulate || (t0 > 0 && p->sub == 0)) ? 1 : 0;
        if (p->plain_fft == 0) {
            FrameForm form = frame_form(p);
            RegFft rf = reg_fft_for(p, form == kFrameStaged);
            const int ny_max = std::min(p->box_max_y, N);
            ev_begin(p, "k_plain_rows", s);
            // slices of the rows where frames and channels alone leave fewer than eight blocks an SM (one channel
            // of a 512-pixel grid: 2.45 ms a block of 1024 samples with 128 blocks a chunk, 1.97 with slices)
            auto grid_of = [&](int frames) {
                const int batch = rf.rows_batch[frames > 1], fb = (nt + frames - 1) / frames;
                const int fill = (int)(8LL * p->sm_count / ((long long)fb * C));
                return dim3(fb, C, std::max(1, std::min((ny_max + batch - 1) / batch, fill)));
            };
            auto blocks = [](dim3 g) { return (long long)g.x * g.y * g.z; };
            // Short launches.  Frames are staged as FP32 samples wherever all blocks are resident with them (1861 elements,
            // 54 channels of 16 x 16 cells, one sample: 138 us, 337 as bytes).  Long lists: one frame a block while two
            // would leave SMs with fewer than four blocks, unless a thread then walks more of them: a walk takes 1.4 times as
            // long for two frames, but a batch of one has up to twice the rows.  Us of rows with two frames a block and
            // with one: 41 channels of 16 x 16 cells of 53 entries, 2 samples 66 and 45; 113 of 32 x 32 cells of 81
            // entries, one sample 227 and 113; 4 of 32 x 32 cells of 96 entries, one 77 and 130.  Short lists gain nothing
            // (44 channels of 16 x 16 cells of 2 entries, 24 samples: 21 us a call with two, 24 with one).
            auto fits = [&](int frames, dim3 g) {
                const size_t per_sm = (size_t)((blocks(g) + p->sm_count - 1) / p->sm_count);
                return form == kFrameStaged || rf.rows_fft + frame_smem(p, kFrameStaged, frames) <= (size_t)p->smem_optin / per_sm;
            };
            auto walks = [&](int i) { return (std::min(rf.rows_batch[i], ny_max) * p->box_max_x + kRowThreads - 1) / kRowThreads; };
            dim3 g = grid_of(kRowFrames);
            const bool longer = (double)A * p->K * p->K >= 8.0 * p->box_max_x * ny_max;  // eight entries a cell
            const int frames = longer && blocks(g) < 4LL * p->sm_count && 5 * walks(0) <= 7 * walks(1) && fits(1, grid_of(1))
                                   ? 1
                                   : kRowFrames;
            const bool odd = bits == 8 && ((uintptr_t)volt & 1) != 0 && form == kFrameGlobal;
            if (frames == 1 || odd) g = grid_of(1);
            if (form != kFrameStaged && !odd && fits(frames, g)) {
                form = kFrameStaged;
                rf = reg_fft_for(p, true);
            }
            launch_early(t0 > 0, odd ? rf.rows_bytes : rf.rows[frames > 1], g, kRowThreads,
                         rf.rows_fft + frame_smem(p, form, frames), s, volt, t0, nt, C, A, bits, p->dt.box, p->dt.cell_off,
                         p->dt.cell_ptr, p->dt.contrib_e, p->dt.contrib_w, p->dt.jones, form == kFrameBytes ? 1 : 0, ny_max, p->dt.twiddle, grid);
            ev_end(p, s);
            // slices of whole intervals, or of at least four frames; the same for every chunk of the call,
            // whose partial sums add up over the chunks
            const int iv = p->sub > 0 ? nt / p->sub : 0, cuts = p->plain_cuts;
            const int S = cuts > 1 ? iv * cuts
                                   : std::max(1, std::min(p->plain_slices, p->sub > 0 ? iv : std::min(p->time_chunk, T) / 4));
            float* partial = nullptr;
            if (cuts > 1 || (S > 1 && p->sub == 0))
                partial = reinterpret_cast<float*>(
                    (uint8_t*)p->scratch + ((sizeof(float2) * (size_t)p->time_chunk * C * P * ny_max * N + 255) & ~(size_t)255));
            ev_begin(p, "k_plain_cols", s);
            // Started early, few blocks would crowd onto the SMs that come free first (21 blocks of 100 frames: 158 us a call,
            // 62 in turn): they ask for as much shared memory as spreads them evenly (8 channels of 32 x 32 pixels, 243
            // samples in 16 slices: 35 us in turn, 49 early, 32 early and spread).
            const int per_sm = (int)(((long long)(N / rf.col_tile) * C * S + p->sm_count - 1) / p->sm_count);
            size_t smem = cols_smem_for(p, rf);
            if (per_sm < p->plain_slots / p->sm_count)  // an SM has 1 KB more than a block may take, and keeps 1 KB of each
                smem = std::max(smem, ((size_t)p->smem_optin + 1024) / per_sm - 1024);
            launch_early(true, cuts > 1 ? rf.cut : rf.cols, dim3(N / rf.col_tile, C, S), rf.col_threads, smem, s,
                         (const float2*)grid, nt, C, ny_max, p->dt.box, p->dt.twiddle, out, partial,
                         cuts > 1 ? 0 : partial ? t0 > 0 : acc, p->sub, p->sub > 0 ? t0 / p->sub : 0, cuts);
            ev_end(p, s);
            if (partial && (cuts > 1 || t0 + nt == T)) {
                const size_t set = (size_t)C * p->nprod * N * N, n = cuts > 1 ? iv * set : set;
                float* o = out + (cuts > 1 ? t0 / p->sub * set : 0);
                ev_begin(p, "k_plain_sum", s);
                if (((uintptr_t)o & 15) == 0) sum_slices<float4>(p, partial, n, cuts > 1 ? cuts : S, o, accumulate, s);
                else sum_slices<float>(p, partial, n, cuts > 1 ? cuts : S, o, accumulate, s);
                ev_end(p, s);
            }
        } else {
            ev_begin(p, "k_plain_grid", s);
            if ((int)sg <= p->smem_optin)
                k_plain_grid<<<dim3(nt, C), kThreads, sg, s>>>(volt, t0, C, A, P, N, bits, p->dt.box, p->dt.cell_off,
                                                               p->dt.cell_ptr, p->dt.contrib_e, p->dt.contrib_w, p->dt.jones, grid);
            else
                k_plain_grid_g<<<dim3(nt, C), kThreads, 0, s>>>(volt, t0, C, A, P, N, bits, p->dt.box, p->dt.cell_off,
                                                                p->dt.cell_ptr, p->dt.contrib_e, p->dt.contrib_w, p->dt.jones, grid);
            ev_end(p, s);
            const size_t n_rows = (size_t)nt * C * P * N;
            const int rpc = rows_per_cta_for(N);
            ev_begin(p, "k_plain_fft_rows_smem", s);
            k_plain_fft_rows_smem<<<(unsigned)((n_rows + rpc - 1) / rpc), kThreads, rows_smem(N), s>>>(
                grid, n_rows, p->logN, rpc, p->dt.twiddle);
            ev_end(p, s);
            ev_begin(p, "k_plain_fft_cols_smem", s);
            k_plain_fft_cols_smem<<<dim3(N / col_tile_for(N), (unsigned)((size_t)nt * C * P)), kThreads,
                                    cols_smem(N), s>>>(grid, p->logN, col_tile_for(N), p->dt.twiddle);
            ev_end(p, s);
            ev_begin(p, "k_plain_sqacc", s);
            k_plain_sqacc<<<dim3((unsigned)(((size_t)N * N + kThreads - 1) / kThreads), C), kThreads, 0, s>>>(
                grid, nt, C, P, N, out, acc, p->sub, p->sub > 0 ? t0 / p->sub : 0);
            ev_end(p, s);
        }
        cudaError_t e = cudaGetLastError();
        if (e != cudaSuccess) return cuda_fail(p, e, "plain path launch");
    }
    return EPIC_OK;
}

}  // namespace epic
