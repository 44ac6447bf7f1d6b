// CUDA-core (fp32 FMA) kernels of the TF_F32 path: the same LM-head pass and SwiGLU of Eq. 1
// as the tensor-core path, for fp32 inputs whose 1e-4 accuracy target rules out TF32 / bf16
// tensor-core arithmetic. Same partial format, same merge.
//
// Both contractions share one main loop: a CTA multiplies kTileW rows of W by RT rows of X (K
// contiguous in both). What bounds it is the fp32 FMA rate from about 16 rows on (W is read once
// per row group), and HBM below that, so
//  - each thread keeps 8 x TR outputs in registers (TR = 8 from 32 rows on): shared memory delivers
//    128 bytes per clock to an SM, so 128 FMAs per clock need at most one loaded byte per FMA, which
//    is what an 8 x 8 tile takes;
//  - an output is two sums, over even and odd k, so that one packed fma.rn.f32x2 takes two
//    neighbouring k of both operands as they lie in shared memory;
//  - stages of 32 k arrive by cp.async into a ring, rows padded to 36 floats so that the 16-byte
//    loads of eight neighbouring rows hit all banks once;
//  - the approximator's GEMMs, which have few output tiles, split K over the CTAs of a cluster:
//    each leaves its partial tile in shared memory and the cluster's CTAs add the tiles in K
//    order through distributed shared memory (no workspace, the same bits on every run).
// Measured on GB300 (V = 32768, d = 1024): LM head 33 us for 8 rows (4.0 TB/s) and 107 us for 57
// (45 TFLOP/s with padding, 63% of the FMA pipe; packed FMAs issue every other clock and 8 warps
// per SM are all that the accumulators leave room for, 12 with 8 x 4 outputs ran no faster), 276
// and 385 us with one column per thread; Eq. 1 (I = 3072, 57 rows) 72 us against 940.
#include <math.h>

#include "common.cuh"
#include "tc_ptx.cuh"

namespace tf {
namespace {

constexpr int kTileW = 128;         // rows of W per CTA tile: half a vocabulary block, 64 gate + 64 up, or 128 outputs
constexpr int kKC = 32;             // k per stage
constexpr int kLd = kKC + 4;        // padded row of a stage, in floats
constexpr int kZLd = kTileW + 4;    // row of the staged tile: 4 chunks of 33 floats, or 128 and a pad of 4
static_assert(kZLd == 4 * 33, "the chunk layout of the LM head fills a row");
constexpr int kMaxClusterK = 8;     // K-ranges of one approximator tile (the portable cluster size)

// A tile of RT rows of X: 16 thread columns of 8 W rows, RT / TR thread rows of TR X rows. Small
// tiles are bound by bytes in flight, large ones by registers.
template <int RT>
struct Tile {
    static constexpr int TR = RT <= 32 ? RT / 4 : 8;
    static constexpr int kThreads = 16 * (RT / TR);
    static constexpr int kStages = RT <= 16 ? 5 : 3;
    static constexpr int kStageFloats = (kTileW + RT) * kLd;
    static constexpr int kSmemBytes = kStages * kStageFloats * 4;
    static_assert(RT * kZLd <= kStages * kStageFloats, "the staged tile reuses the ring");
    // this thread's first W row (the others 16 apart) and first X row (the others RT / TR apart):
    // a warp holds 8 thread columns and 4 thread rows
    static __device__ __forceinline__ int vt() { return (threadIdx.x & 7) + 8 * ((threadIdx.x >> 5) & 1); }
    static __device__ __forceinline__ int rt() { return ((threadIdx.x >> 3) & 3) + 4 * (threadIdx.x >> 6); }
};

// 16 (VEC) or 4 bytes from global to shared memory, zeros where !ok (src then only has to be a
// valid address, nothing is read).
template <bool VEC>
__device__ __forceinline__ void copy_async(float* dst, const float* src, bool ok) {
    const int n = ok ? (VEC ? 16 : 4) : 0;
    if constexpr (VEC)
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(ptx::smem_u32(dst)), "l"(src), "r"(n) : "memory");
    else
        asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(ptx::smem_u32(dst)), "l"(src), "r"(n) : "memory");
}
__device__ __forceinline__ void copy_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void copy_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

__device__ __forceinline__ float sum2(unsigned long long v) { return f2_lo(v) + f2_hi(v); }

// rows [r0, r0 + n) of a [.., K] matrix (n <= 0: none)
struct RowsOf {
    const float* p;   // row r0
    int n;
};

// One stage of a tile: rows 0..63 of `lo` and 64..127 of `hi` into the stage's W part (for one
// matrix hi continues lo), or RT rows of X into its X part; k0 .. k0 + 31, zeros past kend.
template <bool VEC, int ROWS, int THREADS>
__device__ __forceinline__ void load_rows(float* dst, const RowsOf& m, int K, int k0, int kend) {
    constexpr int kPer = VEC ? 4 : 1;                 // floats per copy
    constexpr int kCols = kKC / kPer;                 // copies per row
    const int col = (threadIdx.x % kCols) * kPer, row0 = threadIdx.x / kCols;
    constexpr int kStep = THREADS / kCols;            // rows per pass of the CTA
    const bool kin = k0 + col < kend;
    const float* src = m.p + static_cast<size_t>(row0) * K + k0 + col;
#pragma unroll
    for (int r = row0; r < ROWS; r += kStep, src += static_cast<size_t>(kStep) * K) {
        const bool ok = kin && r < m.n;
        copy_async<VEC>(dst + r * kLd + col, ok ? src : m.p, ok);
    }
}

// acc[i][j] = W[vt + 16 i] . X[rt + RT / TR j] over k in [k0, k1): the pipelined main loop. The
// weights are no kernel's output: the first stages' W is requested before the dependency wait.
template <int RT, bool VEC>
__device__ __forceinline__ void mainloop(float* ring, const RowsOf& lo, const RowsOf& hi, const RowsOf& x, int K, int k0,
                                         int k1, unsigned long long (&acc)[8][Tile<RT>::TR]) {
    using T = Tile<RT>;
    constexpr int TR = T::TR, kStages = T::kStages;
    const int n = (k1 - k0 + kKC - 1) / kKC;
    auto load_w = [&](float* st, int t) {
        load_rows<VEC, 64, T::kThreads>(st, lo, K, k0 + t * kKC, k1);
        load_rows<VEC, 64, T::kThreads>(st + 64 * kLd, hi, K, k0 + t * kKC, k1);
    };
    auto load_x = [&](float* st, int t) { load_rows<VEC, RT, T::kThreads>(st + kTileW * kLd, x, K, k0 + t * kKC, k1); };
#pragma unroll 1
    for (int t = 0; t < kStages - 1 && t < n; ++t) load_w(ring + t * T::kStageFloats, t);
    pdl_wait();
#pragma unroll 1
    for (int t = 0; t < kStages - 1; ++t) {
        if (t < n) load_x(ring + t * T::kStageFloats, t);
        copy_commit();                                // (an empty group keeps the count)
    }
#pragma unroll
    for (int i = 0; i < 8; ++i)
#pragma unroll
        for (int j = 0; j < TR; ++j) acc[i][j] = 0ull;
    const float* ws = ring + T::vt() * kLd;
    const float* xs = ring + (kTileW + T::rt()) * kLd;
    int cur = 0, nxt = kStages - 1;                   // ring slots of stages t and t + kStages - 1
#pragma unroll 1
    for (int t = 0; t < n; ++t) {
        copy_wait<kStages - 2>();                     // stage t has landed (this thread's part)
        __syncthreads();                              // everyone's part, and stage t - 1 is free
        if (t + kStages - 1 < n) {
            load_w(ring + nxt * T::kStageFloats, t + kStages - 1);
            load_x(ring + nxt * T::kStageFloats, t + kStages - 1);
        }
        copy_commit();
        const float* wk = ws + cur * T::kStageFloats;
        const float* xk = xs + cur * T::kStageFloats;
#pragma unroll
        for (int k = 0; k < kKC; k += 4) {
            ulonglong2 xv[TR];
#pragma unroll
            for (int j = 0; j < TR; ++j) xv[j] = *reinterpret_cast<const ulonglong2*>(xk + (RT / TR) * j * kLd + k);
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                const ulonglong2 wv = *reinterpret_cast<const ulonglong2*>(wk + 16 * i * kLd + k);
#pragma unroll
                for (int j = 0; j < TR; ++j) acc[i][j] = f2_fma(wv.x, xv[j].x, acc[i][j]);
#pragma unroll
                for (int j = 0; j < TR; ++j) acc[i][j] = f2_fma(wv.y, xv[j].y, acc[i][j]);
            }
        }
        cur = cur + 1 == kStages ? 0 : cur + 1;
        nxt = nxt + 1 == kStages ? 0 : nxt + 1;
    }
    copy_wait<0>();
    __syncthreads();                                  // the ring may be reused
}

// ------------------------------------------------------------------------------------------
// LM head: one CTA per (row group of RT, half vocabulary block of 128). The logits of the tile go
// through shared memory to one thread per (row, 32-entry chunk), which keeps the chunk's three
// largest logits, the offsets of the first two (ties to the smaller id) and the sum of
// exp(z - max); the four threads of a row fold their chunks into the half's summary in id order.
// Row groups are the fastest grid dimension, so the groups of a half block share its W in L2.
// ------------------------------------------------------------------------------------------
template <int RT, bool VEC>
__global__ void __launch_bounds__(Tile<RT>::kThreads, 1)
    lmhead_simt_kernel(const float* __restrict__ W, const float* __restrict__ X, int n_rows, int d, int V,
                       float inv_temp, Partials partials, int* reset_status) {
    extern __shared__ __align__(16) float ring[];
    using T = Tile<RT>;
    pdl_trigger();
    const int r0 = blockIdx.x * RT, v0 = blockIdx.y * kTileW, t = threadIdx.x;
    const int rows = min(RT, n_rows - r0), cols = max(0, min(kTileW, V - v0));
    // (a half block wholly past V has no row of W: nothing is read from row 0 in its place)
    const float* wbase = W + (cols > 0 ? static_cast<size_t>(v0) * d : 0);
    const RowsOf lo{wbase, cols}, hi{cols > 64 ? wbase + static_cast<size_t>(64) * d : wbase, cols - 64};
    const RowsOf x{X + static_cast<size_t>(r0) * d, rows};
    unsigned long long acc[8][T::TR];
    mainloop<RT, VEC>(ring, lo, hi, x, d, 0, d, acc);
    if (reset_status && blockIdx.x == 0 && blockIdx.y == 0 && t == 0) *reset_status = 0;
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        const int v = T::vt() + 16 * i;
#pragma unroll
        for (int j = 0; j < T::TR; ++j)
            ring[(T::rt() + RT / T::TR * j) * kZLd + (v >> 5) * 33 + (v & 31)] = v < cols ? sum2(acc[i][j]) * inv_temp : -INFINITY;
    }
    __syncthreads();
#pragma unroll 1
    for (int q = t; q < 4 * RT; q += T::kThreads) {   // (whole warps)
        const int r = q >> 2, c = q & 3;              // row of the group, chunk of the half block
        const bool mine = r < rows;
        float a1 = -INFINITY, a2 = -INFINITY, a3 = -INFINITY, s = 0.0f;
        int i1 = 0, i2 = 0;
        if (mine) {
            const float* z = ring + r * kZLd + c * 33;
            float v[kChunk];
#pragma unroll
            for (int i = 0; i < kChunk; ++i) v[i] = z[i];
#pragma unroll
            for (int i = 0; i < kChunk; ++i) {
                // strict comparisons: among equal values the smaller id ranks first
                const bool g1 = v[i] > a1, g2 = v[i] > a2;
                a3 = g2 ? a2 : fmaxf(a3, v[i]);
                i2 = g1 ? i1 : (g2 ? i : i2);
                a2 = g1 ? a1 : (g2 ? v[i] : a2);
                i1 = g1 ? i : i1;
                a1 = g1 ? v[i] : a1;
            }
            if (a1 > -INFINITY) {
#pragma unroll
                for (int i = 0; i < kChunk; ++i) s += expf(v[i] - a1);
            }
            const int tile = blockIdx.y >> 1, chunk = (blockIdx.y & 1) * (kChunks / 2) + c;
            partials.chunks[partials.chunk_at(tile, chunk, r0 + r)] = make_float4(a1, a2, a3, __int_as_float(i1 | (i2 << 8)));
        }
        // the half's summary: chunk pairs, then pairs of pairs; the lower chunk keeps its entry on a tie
        float m = a1, bv = a1;
        int bid = a1 > -INFINITY ? v0 + c * kChunk + i1 : -1;
#pragma unroll
        for (int o = 1; o < 4; o <<= 1) {
            const float m2 = __shfl_down_sync(0xffffffffu, m, o), s2 = __shfl_down_sync(0xffffffffu, s, o);
            const float bv2 = __shfl_down_sync(0xffffffffu, bv, o);
            const int bid2 = __shfl_down_sync(0xffffffffu, bid, o);
            const float mn = fmaxf(m, m2);
            if (mn > -INFINITY) s = s * expf(m - mn) + s2 * expf(m2 - mn);
            m = mn;
            if (bv2 > bv) {
                bv = bv2;
                bid = bid2;
            }
        }
        if (mine && c == 0)
            partials.halves[partials.half_at(blockIdx.y >> 1, blockIdx.y & 1, r0 + r)] = make_float4(m, s, bv, __int_as_float(bid));
    }
}

// ------------------------------------------------------------------------------------------
// C[n_rows, N] = X[n_rows, K] W[N, K]^T, one cluster per (N tile, row group), its CTAs on
// consecutive K-ranges.
// GATEUP (N tile of 64): out = SiLU(X Wg^T) * (X Wu^T); DOWN (N tile of 128): out = hidden of the
// stage-2 row's depth + X Wd^T.
// ------------------------------------------------------------------------------------------
template <bool GATEUP, int RT, bool VEC>
__global__ void __launch_bounds__(Tile<RT>::kThreads, 1)
    swiglu_simt_kernel(const float* __restrict__ X, const float* __restrict__ W0, const float* __restrict__ W1, int n_rows,
                       int K, int N, int n_rg, float* __restrict__ out, const float* __restrict__ hidden, int R, int M,
                       int gamma) {
    extern __shared__ __align__(16) float ring[];
    using T = Tile<RT>;
    constexpr int kOut = GATEUP ? kTileW / 2 : kTileW;    // output columns of a tile
    pdl_trigger();
    const int ks = static_cast<int>(ptx::cluster_nctarank()), kr = static_cast<int>(ptx::cluster_ctarank());
    const int unit = blockIdx.x / ks, rg = unit % n_rg, nt = unit / n_rg;
    const int r0 = rg * RT, c0 = nt * kOut;
    const int rows = min(RT, n_rows - r0), cols = min(kOut, N - c0);
    RowsOf lo{W0 + static_cast<size_t>(c0) * K, cols}, hi;
    if (GATEUP)
        hi = RowsOf{W1 + static_cast<size_t>(c0) * K, cols};
    else
        hi = RowsOf{cols > 64 ? lo.p + static_cast<size_t>(64) * K : lo.p, cols - 64};
    const RowsOf x{X + static_cast<size_t>(r0) * K, rows};
    // K-ranges in whole stages
    const int nst = (K + kKC - 1) / kKC;
    const int k0 = static_cast<int>(static_cast<long long>(nst) * kr / ks) * kKC;
    const int k1 = min(K, static_cast<int>(static_cast<long long>(nst) * (kr + 1) / ks) * kKC);
    unsigned long long acc[8][T::TR];
    mainloop<RT, VEC>(ring, lo, hi, x, K, k0, k1, acc);
#pragma unroll
    for (int i = 0; i < 8; ++i)
#pragma unroll
        for (int j = 0; j < T::TR; ++j) ring[(T::rt() + RT / T::TR * j) * kZLd + T::vt() + 16 * i] = sum2(acc[i][j]);
    ptx::cluster_sync();                              // every partial tile of the cluster is in place
    // this CTA's share of the tile: four columns of one row per step, summed in K order
    const bool vec_out = N % 4 == 0;
    for (int idx = kr * T::kThreads + static_cast<int>(threadIdx.x); idx < RT * kOut / 4; idx += ks * T::kThreads) {
        const int r = idx / (kOut / 4), c = (idx - r * (kOut / 4)) * 4;
        if (r >= rows || c >= cols) continue;
        const uint32_t at = ptx::smem_u32(ring + r * kZLd + c);
        float g[4] = {}, u[4] = {};
        for (int s = 0; s < ks; ++s) {
            const float4 a = ptx::ld_cluster_f4(ptx::mapa_shared(at, s));
            g[0] += a.x; g[1] += a.y; g[2] += a.z; g[3] += a.w;
            if (GATEUP) {
                const float4 b = ptx::ld_cluster_f4(ptx::mapa_shared(at + 64 * 4, s));
                u[0] += b.x; u[1] += b.y; u[2] += b.z; u[3] += b.w;
            }
        }
        float v[4];
        if (GATEUP) {
#pragma unroll
            for (int e = 0; e < 4; ++e) v[e] = g[e] / (1.0f + expf(-g[e])) * u[e];
        } else {
            const int row = r0 + r, sq = row / R, rr = row - sq * R;
            const float* h = hidden + static_cast<size_t>(sq * gamma + stage2_hidden_index(rr, M)) * N + c0 + c;
#pragma unroll
            for (int e = 0; e < 4; ++e) v[e] = c + e < cols ? h[e] + g[e] : 0.0f;
        }
        float* dst = out + static_cast<size_t>(r0 + r) * N + c0 + c;
        if (vec_out) {
            *reinterpret_cast<float4*>(dst) = make_float4(v[0], v[1], v[2], v[3]);
        } else {
            for (int e = 0; e < 4; ++e)
                if (c + e < cols) dst[e] = v[e];
        }
    }
    ptx::cluster_sync();                              // no CTA leaves while its tile may still be read
}

template <int RT, bool VEC>
cudaError_t run_lmhead(const Ctx& ctx, const float* W, const float* X, int n_rows, int d, int V, float inv_temp,
                       const Partials& partials, bool reset_status) {
    auto kern = lmhead_simt_kernel<RT, VEC>;
    const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, Tile<RT>::kSmemBytes);
    if (e != cudaSuccess) return e;
    const dim3 grid((n_rows + RT - 1) / RT, 2 * ((V + kBlockV - 1) / kBlockV));
    return launch_pdl(kern, grid, dim3(Tile<RT>::kThreads), Tile<RT>::kSmemBytes, ctx.stream, W, X, n_rows, d, V, inv_temp, partials,
                      reset_status ? ctx.status : static_cast<int*>(nullptr));
}

template <bool GATEUP, int RT, bool VEC>
cudaError_t run_swiglu(const Ctx& ctx, const float* X, const float* W0, const float* W1, int n_rows, int K, int N,
                       float* out, const float* hidden, int R, int M, int gamma, int ks) {
    auto kern = swiglu_simt_kernel<GATEUP, RT, VEC>;
    const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, Tile<RT>::kSmemBytes);
    if (e != cudaSuccess) return e;
    constexpr int kOut = GATEUP ? kTileW / 2 : kTileW;
    const int n_rg = (n_rows + RT - 1) / RT;
    const long long ctas = static_cast<long long>((N + kOut - 1) / kOut) * n_rg * ks;
    if (ctas > 0x7fffffffll) return cudaErrorInvalidConfiguration;
    return launch_pdl_cluster(kern, dim3(static_cast<unsigned>(ctas)), dim3(Tile<RT>::kThreads), Tile<RT>::kSmemBytes, ctx.stream,
                              ks, X, W0, W1, n_rows, K, N, n_rg, out, hidden, R, M, gamma);
}

// Row group of a contraction with n_rows rows: the smallest that holds them all; beyond 64 rows
// groups of 64, or of 32 where those pad less (the thread tile is the same, W is read twice as
// often from L2). Rows that do not start at multiples of 16 bytes (!vec) arrive by copies of four bytes, 80
// per thread and stage with the 64 threads of a group of 32: groups of 16 up to 32 rows, of 64 from there
// on (V = 9001, d = 2050: 17 rows 541 -> 117 us, 65 rows 680 -> 252, 200 rows 1240 -> 300).
int row_group(int n_rows, bool vec) {
    if (n_rows <= 16) return n_rows <= 8 ? 8 : 16;
    if (!vec) return n_rows <= 32 ? 16 : 64;
    return (n_rows + 31) / 32 % 2 == 0 ? 64 : 32;
}

template <bool GATEUP>
cudaError_t swiglu_gemm(const Ctx& ctx, const float* X, const float* W0, const float* W1, int n_rows, int K, int N,
                        float* out, const float* hidden, int R, int M, int gamma) {
    constexpr int kOut = GATEUP ? kTileW / 2 : kTileW;
    // K-ranges per tile: enough CTAs for three on every SM, at least two stages each. Where even
    // eight ranges per tile leave SMs idle, smaller row groups make more tiles.
    const long long tiles = (N + kOut - 1) / kOut;
    const bool vec = K % 4 == 0;
    int rt = row_group(n_rows, vec);
    while (rt > 16 && tiles * ((n_rows + rt - 1) / rt) * kMaxClusterK < 2ll * ctx.num_sms) rt /= vec ? 2 : 4;
    const long long base = tiles * ((n_rows + rt - 1) / rt);
    int ks = 1;
    while (ks < kMaxClusterK && base * ks * 2 <= 3ll * ctx.num_sms && K >= 2 * kKC * ks * 2) ks *= 2;
    auto run = vec ? (rt == 8    ? run_swiglu<GATEUP, 8, true>
                      : rt == 16 ? run_swiglu<GATEUP, 16, true>
                      : rt == 32 ? run_swiglu<GATEUP, 32, true>
                                 : run_swiglu<GATEUP, 64, true>)
                   : (rt == 8    ? run_swiglu<GATEUP, 8, false>
                      : rt == 16 ? run_swiglu<GATEUP, 16, false>
                                 : run_swiglu<GATEUP, 64, false>);
    return run(ctx, X, W0, W1, n_rows, K, N, out, hidden, R, M, gamma, ks);
}

}  // namespace

cudaError_t launch_lmhead_simt(const Ctx& ctx, int dtype, const void* lm_head, const void* x, int n_rows, int d,
                               int V, float inv_temp, Partials partials, bool reset_status) {
    if (dtype != TF_F32) return cudaErrorNotSupported;
    if (n_rows <= 0) return cudaSuccess;
    const float* W = static_cast<const float*>(lm_head);
    const float* X = static_cast<const float*>(x);
    const int rt = row_group(n_rows, d % 4 == 0);
    auto run = d % 4 == 0 ? (rt == 8    ? run_lmhead<8, true>
                             : rt == 16 ? run_lmhead<16, true>
                             : rt == 32 ? run_lmhead<32, true>
                                        : run_lmhead<64, true>)
                          : (rt == 8    ? run_lmhead<8, false>
                             : rt == 16 ? run_lmhead<16, false>
                                        : run_lmhead<64, false>);
    const cudaError_t e = run(ctx, W, X, n_rows, d, V, inv_temp, partials, reset_status);
    return e != cudaSuccess ? e : cudaGetLastError();
}

cudaError_t launch_swiglu_simt(const Ctx& ctx, const void* X, int k_in, const void* w_gate, const void* w_up,
                               const void* w_down, const void* hidden, int n_rows, int d, int I, int R, int M,
                               int gamma, void* A, void* h_prime) {
    if (n_rows <= 0) return cudaSuccess;
    cudaError_t e = swiglu_gemm<true>(ctx, static_cast<const float*>(X), static_cast<const float*>(w_gate),
                                      static_cast<const float*>(w_up), n_rows, k_in, I, static_cast<float*>(A),
                                      nullptr, R, M, gamma);
    if (e == cudaSuccess) e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    e = swiglu_gemm<false>(ctx, static_cast<const float*>(A), static_cast<const float*>(w_down), nullptr, n_rows, I, d,
                           static_cast<float*>(h_prime), static_cast<const float*>(hidden), R, M, gamma);
    return e != cudaSuccess ? e : cudaGetLastError();
}

// The "w/ Linear" approximator: the residual GEMM above with x (K = 2d) in place of A.
cudaError_t launch_linear_simt(const Ctx& ctx, const void* X, const void* w_lin, const void* hidden, int n_rows, int d,
                               int R, int M, int gamma, void* h_prime) {
    if (n_rows <= 0) return cudaSuccess;
    const cudaError_t e = swiglu_gemm<false>(ctx, static_cast<const float*>(X), static_cast<const float*>(w_lin), nullptr,
                                             n_rows, 2 * d, d, static_cast<float*>(h_prime),
                                             static_cast<const float*>(hidden), R, M, gamma);
    return e != cudaSuccess ? e : cudaGetLastError();
}

}  // namespace tf
