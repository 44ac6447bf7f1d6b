// Tensor-core (tcgen05 + TMA) GEMM kernels of the bf16 path.
//
//   D[r, n] = sum_k X[r, k] * W[n, k]          X: activations [rows, K], W: weights [N, K]
//
// X rows sit in the 128 TMEM lanes (M = 128 per tile), weight rows in the MMA N dimension, so
// every epilogue thread owns one activation row and walks its logits / outputs serially.
// Fused epilogues:
//   LMHEAD  the LM-head pass of Algorithm 1 (stage 1 and stage 2): for each (row, block of 256
//           vocabulary entries) it keeps per half block the max, the sum of exp(z - max) and the
//           best (z, id), and per 32-wide chunk the three largest z with the ids of the first
//           two. Logits never leave the SM.
//   GATEUP  SwiGLU of Eq. 1, first half: A = SiLU(X W_gate^T) * (X W_up^T), bf16 out.
//   DOWN    SwiGLU of Eq. 1, second half plus the residual: h' = h + A W_down^T, bf16 out; the
//           same epilogue serves the linear approximator of the ablations, h' = h + x W_lin^T.
//   CGATEUP, CDOWN  the same two results where K is split over the CTAs of a cluster.
//   PARTIAL fp32 sums of a K-range, for the reduction kernels, where no cluster can take the split.
//
// Warp roles (576 threads, one CTA per SM, persistent over work units):
//   warp 0      TMA producer: one elected lane streams X and W tiles into a ring of stages.
//   warp 1      TMEM allocator and MMA issuer (one lane issues tcgen05.mma and commits).
//   warps 2..17 epilogue, two groups of eight; group g drains accumulator slot g (TMEM columns
//               [256 g, 256 g + 256)); warp w may only touch TMEM lanes 32 (w % 4) .. + 31, and
//               the two warps of a group on the same lanes split the columns in halves.
// A work unit is (N tile, group of MT M-tiles). With MT = 2 both slots hold one unit (M-tile j
// in slot j); with MT = 1 consecutive units alternate slots so the epilogue of one overlaps the
// MMAs of the next. With clusters of CL = 2 CTAs (most LM heads over more than 128 rows, the down
// projection of many rows) the two CTAs are a tcgen05 CTA pair: units are dealt to clusters, CTA r of a cluster stages M-tile r of
// the unit's pair of M-tiles and weight rows [128 r, 128 r + 128) of the unit's 256-row weight
// tile, and the even CTA issues one cta_group::2 MMA (M = 256, N = 256) per K slice that reads
// both CTAs' shared memory and writes each CTA's 128 rows into its own TMEM. W is read once, each
// CTA stages 32 KB per stage instead of 48 KB, and each keeps one TMEM slot per unit, so its
// epilogue overlaps the next unit's MMAs. Every wait is bounded: after a time limit the kernel
// raises TF_DEV_TIMEOUT, drains its in-flight copies and MMAs, frees TMEM and returns.
#include <cuda.h>
#include <math.h>

#include "common.cuh"
#include "tc_ptx.cuh"

namespace tf {
namespace {

constexpr int kBK = 64;       // K elements per stage: one 128-byte swizzle row of bf16
constexpr int kBM = 128;      // activation rows per M-tile (TMEM lanes)
constexpr int kEpiWarps = 16;  // two groups (one per TMEM slot) of eight warps
constexpr int kThreads = 64 + 32 * kEpiWarps;
constexpr uint64_t kWaitLimitNs = 2000000000ull;

// EPI_CGATEUP / EPI_CDOWN: the GATEUP / DOWN results from split-K over the CTAs of a cluster, the
// partial sums exchanged through an area of the workspace that stays in L2.
enum { EPI_LMHEAD = 0, EPI_GATEUP = 1, EPI_DOWN = 2, EPI_PARTIAL = 3, EPI_CGATEUP = 4, EPI_CDOWN = 5 };

struct EpiParams {
    Partials partials;           // LMHEAD: per (row, vocabulary block) summaries
    int V;
    float inv_temp;
    __nv_bfloat16* out;          // GATEUP: A [n_rows, ld_out]; DOWN: h' [n_rows, ld_out]
    int ld_out;
    const __nv_bfloat16* hidden; // DOWN: residual rows, [b * gamma, ld_out]
    int R, M, gamma;
    float* partial;              // PARTIAL: fp32 sums [k_splits][n_cols / 4][n_rows][4] (float4-major),
    int n_cols;                  //          accumulator nb of N tile nt at columns nb * n_total + nt * BN
    int n_total;                 // N of the whole GEMM (n_ntiles * BN)
    int reset_status;            // LMHEAD: zero *status first (the first kernel of a stage-1 call)
    unsigned long long wait_ns;  // limit of every wait for progress (0: kWaitLimitNs); the waits
                                 // that drain in-flight copies and MMAs always take kWaitLimitNs
    // GATEUP / DOWN of fixed width, single CTAs or pairs: units n_full.. (the last, partial round) run as
    // tail_split K-chunks each (0: none). A chunk writes its fp32 partial sums to `partial`, laid
    // out [tail unit][chunk][M-tile][col / 4][128 rows][4]; the chunk that finishes last (counted
    // in sem[tail unit * MT + M-tile], zero between calls) adds them in chunk order and applies
    // the epilogue.
    int n_full, tail_split;
    int* sem;
    // kernels with a width chosen at launch: columns per N tile (a multiple of 8) and ring stages
    int bn, stages;
    // LMHEAD with single CTAs: 2 copies of 33 to 64 rows, 4 of up to 32, one per half (quarter) of the TMEM
    // lanes, so that all epilogue warps share the chunks of a block (each of them has rows: they wait for
    // one another); otherwise 1
    int copies;
};

// Work unit u -> (N tile, M-tile group, K split); consecutive units share the N tile and K split
// (the same weight tile) and differ in the M-tile group, so batched rows reuse it from L2.
struct Unit {
    int nt, mg, kx;
};
__device__ __forceinline__ Unit decode_unit(int u, int n_mgroups, int k_splits) {
    Unit w;
    w.mg = u % n_mgroups;
    const int rest = u / n_mgroups;
    w.kx = rest % k_splits;
    w.nt = rest / k_splits;
    return w;
}

// PAIR: a CTA of a cta_group::2 pair, which stages half of the weight tile (BN / 2 rows).
// VAR: tiles of up to BN columns and up to STAGES stages, as many as fit the ring.
template <int MT, int NB, int BN, int STAGES, bool PAIR = false, bool VAR = false>
struct TileCfg {
    static constexpr int kABytes = kBM * kBK * 2;
    static constexpr int kBBytes = BN * kBK * 2;                    // the whole weight tile of a stage
    static constexpr int kBBytesCta = PAIR ? kBBytes / 2 : kBBytes;  // the part this CTA stages
    static constexpr int kStageBytes = MT * kABytes + NB * kBBytesCta;
    static constexpr int kRingBytes = VAR ? 208 * 1024 : STAGES * kStageBytes;
    static constexpr int kBarrierBytes = 256;
    static constexpr int kSmemBytes = kRingBytes + kBarrierBytes + 1024;
    static_assert(NB * BN <= 256, "one accumulator slot is 256 TMEM columns");
    static_assert(BN % 64 == 0 && BN >= 64 && BN <= 256, "N tile (two epilogue warps split it in 32-column steps)");
    static_assert(kStageBytes % 1024 == 0, "stages must stay 1024-byte aligned for 128B swizzle");
};

constexpr int kShortRows = 64;     // rows of a last M-tile that is loaded through a shorter box
constexpr int kVarMaxStages = 8;   // ring stages of the kernels whose tile width is chosen at launch

__device__ __forceinline__ float silu_f(float g) { return g / (1.0f + __expf(-g)); }

__device__ __forceinline__ uint32_t pack_bf16x2(float lo, float hi) {
    __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
    return *reinterpret_cast<uint32_t*>(&v);
}

// Summary of one 32-column chunk of one row: the three largest logits, the chunk-local offsets of the
// first two (the smaller first among equals) and the sum of exp(z - max). The same instructions for
// every lane whatever the data (a per-lane sorted insertion would diverge across the warp's 32 rows).
// What bounds it is the instructions issued: with d of 512 to 2048 the epilogue, not the contraction,
// sets the pace of the LM head. The three values come from a network of min/max (a merge of two sorted
// triples: a third largest is one of two thirds and two cross minima), the offsets from four selects
// per merge, and the exponentials from one pass over the values once the maximum is known, in packed
// pairs. A warp issues 508 instructions per chunk of its 32 rows (loads, tests and stores included),
// where a tree whose every node rescaled its sum of exponentials took 1040 (V = 151936, 256 rows: d = 512 66 -> 47 us, d = 1024 78 -> 64, d = 2048 122 ->
// 115, d = 4096 222 -> 217 on GB300).
struct Top3 {
    float a1, a2, a3;  // a1 >= a2 >= a3
    int i1, i2;        // offsets of a1, a2
};
// p covers smaller offsets than q, so on equal values p's entry ranks first.
__device__ __forceinline__ void top3_first_two(const Top3& p, const Top3& q, int winner_second, Top3& n) {
    const float t = fminf(p.a1, q.a1);
    n.a1 = fmaxf(p.a1, q.a1);
    n.a2 = fmaxf(fmaxf(p.a2, q.a2), t);
    // the winner's second against the loser's first (whichever of the two tests does not apply is false)
    const bool second = p.a2 >= q.a1 || q.a2 > p.a1;
    n.i2 = second ? winner_second : (p.a1 >= q.a1 ? q.i1 : p.i1);
}
template <int OFF, int N>
__device__ __forceinline__ Top3 top3(const float (&z)[32]) {
    static_assert(N >= 4, "");
    Top3 n;
    if constexpr (N == 4) {
        Top3 p, q;   // pairs: a3 and i2 unused
        const bool g0 = z[OFF] >= z[OFF + 1], g1 = z[OFF + 2] >= z[OFF + 3];
        p.a1 = fmaxf(z[OFF], z[OFF + 1]);
        p.a2 = fminf(z[OFF], z[OFF + 1]);
        p.i1 = g0 ? OFF : OFF + 1;
        q.a1 = fmaxf(z[OFF + 2], z[OFF + 3]);
        q.a2 = fminf(z[OFF + 2], z[OFF + 3]);
        q.i1 = g1 ? OFF + 2 : OFF + 3;
        n.i1 = p.a1 >= q.a1 ? p.i1 : q.i1;
        top3_first_two(p, q, n.i1 ^ 1, n);
        n.a3 = fmaxf(fminf(p.a2, q.a1), fminf(p.a1, q.a2));
    } else {
        const Top3 p = top3<OFF, N / 2>(z), q = top3<OFF + N / 2, N / 2>(z);
        const bool pw = p.a1 >= q.a1;
        n.i1 = pw ? p.i1 : q.i1;
        top3_first_two(p, q, pw ? p.i2 : q.i2, n);
        n.a3 = fmaxf(fmaxf(fmaxf(p.a3, q.a3), fminf(p.a2, q.a1)), fminf(p.a1, q.a2));
    }
    return n;
}
__device__ __forceinline__ float ex2(float x) {
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
// sum of exp(z - m) over a chunk whose two largest values are m = t.a1 and t.a2
__device__ __forceinline__ float sum_exp(const float (&z)[32], const Top3& t) {
    constexpr float kLog2e = 1.4426950408889634f;
    const unsigned long long m2 = f2_pack(t.a1, t.a1), l2 = f2_pack(kLog2e, kLog2e);
    unsigned long long s[4];
#pragma unroll
    for (int i = 0; i < 16; ++i) {
        const unsigned long long x = f2_mul(f2_sub(f2_pack(z[2 * i], z[2 * i + 1]), m2), l2);
        const unsigned long long e = f2_pack(ex2(f2_lo(x)), ex2(f2_hi(x)));
        s[i & 3] = i < 4 ? e : f2_add(s[i & 3], e);
    }
    const unsigned long long u = f2_add(f2_add(s[0], s[1]), f2_add(s[2], s[3]));
    const float sum = f2_lo(u) + f2_hi(u);
    if (t.a1 == INFINITY) return t.a2 == INFINITY ? NAN : 1.0f;   // (inf - inf above)
    return t.a1 > -INFINITY ? sum : 0.0f;                         // no entry in the chunk
}

// VAR: the tile is ep.bn <= BN columns wide and the ring has ep.stages <= STAGES stages.
template <int EPI, int MT, int NB, int BN, int STAGES, int CL, bool VAR>
__global__ void __launch_bounds__(kThreads, 1)
tc_gemm_kernel(const __grid_constant__ CUtensorMap tmap_x, const __grid_constant__ CUtensorMap tmap_xl,
               const __grid_constant__ CUtensorMap tmap_w0, const __grid_constant__ CUtensorMap tmap_w1, int n_rows, int K, int n_ntiles,
               int n_mgroups, int k_splits, int w_stream_once, EpiParams ep, int* status) {
    // Two kinds of cluster: kPair, a CTA pair on two M-tiles sharing each weight tile through
    // cta_group::2 MMAs; kSplitK, up to CL CTAs on the K-ranges of one output tile (one tile per
    // cluster), whose accumulators are summed through an exchange area in L2.
    constexpr bool kSplitK = EPI == EPI_CGATEUP || EPI == EPI_CDOWN;
    constexpr bool kPair = CL > 1 && !kSplitK;
    using C = TileCfg<MT, NB, BN, STAGES, kPair, VAR>;
    static_assert(CL == 1 || kSplitK || (CL == 2 && MT == 1 && NB == 1), "a CTA pair: one M-tile each, one weight matrix");
    static_assert(!kSplitK || (CL == 4 && kMaxKSplits == 4 && (VAR || (MT == 2 && BN == 128))), "cluster split-K");
    constexpr bool kCopies = EPI == EPI_LMHEAD && CL == 1;
    // copies: half summaries of the copies' chunks, [group][half][parity of the unit][copy][row]
    __shared__ float4 copy_sums[kCopies ? 2 * 2 * 2 * kBM : 1];
    constexpr bool kShare = kSplitK && VAR && MT == 1;   // both epilogue groups work on one accumulator
    static_assert(!VAR || (!kPair && EPI != EPI_LMHEAD), "variable width: single CTAs and K-splitting clusters");
    pdl_trigger();
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = reinterpret_cast<uint8_t*>(
        (reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~static_cast<uintptr_t>(1023));
    const int bn = VAR ? ep.bn : BN, stages = VAR ? ep.stages : STAGES;
    const int stage_bytes = VAR ? MT * C::kABytes + NB * bn * kBK * 2 : C::kStageBytes;
    uint64_t* full = reinterpret_cast<uint64_t*>(smem + C::kRingBytes);
    uint64_t* empty = full + STAGES;
    uint64_t* tfull = empty + STAGES;
    uint64_t* tempty = tfull + 2;
    uint64_t* drain = tempty + 2;
    uint64_t* meet = drain + 1;   // [4]: where epilogue warps wait for one another
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(meet + 4);
    volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
    volatile int* last_chunk = abort_flag + 1;   // [2]: this group's chunk was its unit's last

    const int warp = threadIdx.x >> 5;
    const int lane = threadIdx.x & 31;
    // Units are dealt to clusters. Pair: CTA `crank` of a cluster takes M-tile group member crank
    // of every unit. Split-K: a unit is an output tile and CTA crank takes K-range crank. With
    // CL = 1 a cluster is one CTA.
    const int n_units = kSplitK ? n_ntiles * n_mgroups : n_ntiles * n_mgroups * k_splits;
    const int crank = CL > 1 ? static_cast<int>(ptx::cluster_ctarank()) : 0;
    const int m_cl = kPair ? CL : 1, m_rank = kPair ? crank : 0;   // M-tiles of a cluster, this CTA's
    const bool leader = !kPair || crank == 0;                     // the pair's MMA issuer
    const int cid = CL > 1 ? static_cast<int>(ptx::cluster_id_x()) : static_cast<int>(blockIdx.x);
    const int ncl = CL > 1 ? static_cast<int>(ptx::cluster_count_x()) : static_cast<int>(gridDim.x);
    const int nk = K / kBK / k_splits;      // K-steps per unit (K % (64 * k_splits) == 0)
    const uint64_t wait_ns = ep.wait_ns ? ep.wait_ns : kWaitLimitNs;
    auto unit_of = [&](int u) {
        if constexpr (kSplitK) return Unit{u / n_mgroups, u % n_mgroups, crank};
        return decode_unit(u, n_mgroups, k_splits);
    };
    // Work items: the units, except that with a tail split each unit of the last round becomes
    // tail_split items over consecutive K-chunks of its range ([kb0, kb1) in K-steps).
    constexpr bool kTail = !VAR && (EPI == EPI_GATEUP || EPI == EPI_DOWN);
    constexpr int kUnitTiles = kPair ? 2 : MT;   // M-tiles of a unit
    const int n_split = kTail ? ep.tail_split : 0;
    const int n_items = n_split ? ep.n_full + (n_units - ep.n_full) * n_split : n_units;
    struct Item {
        Unit w;
        int kb0, kb1, tail, chunk;   // tail unit and chunk index (-1: a whole unit)
    };
    auto item_of = [&](int i) {
        Item it;
        const int ns = n_split > 0 ? n_split : 1;   // (a constant 1 in kernels without a tail split)
        if (n_split == 0 || i < ep.n_full) {
            it.w = unit_of(i);
            it.kb0 = it.w.kx * nk;
            it.kb1 = it.kb0 + nk;
            it.tail = it.chunk = -1;
        } else {
            const int r = i - ep.n_full;
            it.tail = r / ns;
            it.chunk = r - it.tail * ns;
            it.w = unit_of(ep.n_full + it.tail);
            it.kb0 = it.w.kx * nk + nk * it.chunk / ns;
            it.kb1 = it.w.kx * nk + nk * (it.chunk + 1) / ns;
        }
        return it;
    };
    // shared::cluster address of this CTA's barrier `bar` as seen at the same offset in the pair's
    // even CTA (pair mode: the barriers the issuer waits on) or in the odd one
    auto in_leader = [&](uint64_t* bar) {
        return kPair && crank != 0 ? ptx::mapa_shared(ptx::smem_u32(bar), 0) : ptx::smem_u32(bar);
    };
    auto in_peer = [&](uint64_t* bar) { return ptx::mapa_shared(ptx::smem_u32(bar), 1); };

    if (threadIdx.x == 0) {
        for (int s = 0; s < STAGES; ++s) {
            ptx::mbar_init(&full[s], 1);
            ptx::mbar_init(&empty[s], 1);
        }
        for (int g = 0; g < 2; ++g) {
            ptx::mbar_init(&tfull[g], 1);
            // pair: one arrival per epilogue warp of both CTAs (used in the even CTA only)
            ptx::mbar_init(&tempty[g], kPair ? 2 * (kEpiWarps / 2) : 32 * kEpiWarps / 2);
        }
        ptx::mbar_init(drain, 1);
        // one arrival per warp: the warps of a group (tail split), of a group and column half (copies)
        for (int i = 0; i < 4; ++i) ptx::mbar_init(&meet[i], EPI == EPI_LMHEAD ? kEpiWarps / 4 : kEpiWarps / 2);
        *abort_flag = 0;
        ptx::fence_barrier_init();
    }
    if constexpr (kPair) {
        // both CTAs of the pair are running and their barriers exist before the collective
        // allocation and before either CTA signals the other's barriers
        ptx::cluster_sync();
        if (warp == 1) {
            ptx::tmem_alloc_pair(tmem_slot, 512);
            ptx::tmem_relinquish_pair();
        }
        ptx::tc_fence_before();
        __syncthreads();
        ptx::tc_fence_after();
    } else {
        if (warp == 1) {
            ptx::tmem_alloc(tmem_slot, 512);
            ptx::tmem_relinquish();
        }
        ptx::tc_fence_before();
        __syncthreads();
        if constexpr (CL > 1) ptx::cluster_sync();   // the peers' barriers exist before any remote access
        ptx::tc_fence_after();
    }
    const uint32_t tmem_base = *tmem_slot;
    if (!(warp == 0 && lane == 0)) pdl_wait();   // the producer waits after its weight prefetch
    // a call's status word starts at zero; cleared here, after every earlier kernel has finished,
    // instead of by a separate memset that would end the overlap with the previous kernel
    if (EPI == EPI_LMHEAD && ep.reset_status && blockIdx.x == 0 && threadIdx.x == 64 && status) *status = 0;

    if (warp == 0) {
        // ------------------------------------------------------------------ TMA producer
        if (lane == 0) {
            const bool short_box = EPI == EPI_LMHEAD ? kCopies && ep.copies > 1 : !kPair;
            const int rem = n_rows % kBM, x_last = (rem + 7) / 8 * 8;
            const int m_all = (n_rows + kBM - 1) / kBM, m_short = short_box && rem > 0 && rem <= kShortRows ? m_all - 1 : -1;
            const CUtensorMap* only = m_short == 0 ? &tmap_xl : &tmap_x;
            ptx::prefetch_tmap(only);
            ptx::prefetch_tmap(&tmap_w0);
            if (NB == 2) ptx::prefetch_tmap(&tmap_w1);
            const uint64_t pol_x = ptx::policy_evict_last();
            const uint64_t pol_w = w_stream_once ? ptx::policy_evict_first() : ptx::policy_evict_last();
            // Pair: both CTAs' copies of a stage complete on the even CTA's full barrier, which
            // the even CTA alone arms with the bytes of both halves.
            // X rows: M-tiles through tmap_x; a last one of at most kShortRows rows through tmap_xl, whose box
            // ends with the rows (in whole 8-row swizzle groups: a box mostly outside the tensor is slow
            // to fill); an M-tile past the rows not at all. Pairs, and the LM head but for copies of the rows,
            // always take whole boxes: their MMAs cover the padding, and zeros there cost less than what the
            // stage held before (V = 151936, d = 4096: 320 rows on pairs 383 against 440 us under the board's
            // power cap, 270 on single CTAs 315 against 325; V = 9001, 16 rows 27 against 30).
            const int copies = kCopies ? ep.copies : 1;
            auto load_x = [&](uint8_t* sp, uint64_t* bar, int j, int kb, int mt) {
                uint8_t* dst = sp + j * C::kABytes;
                if constexpr (kPair) {
                    ptx::tma_load_2d_pair(dst, &tmap_x, in_leader(bar), kb * kBK, mt * kBM, pol_x);
                } else if (MT == 1 && !kCopies) {        // one M-tile in all
                    ptx::tma_load_2d(dst, only, bar, kb * kBK, 0, pol_x);
                } else if (mt != m_short) {
                    if (mt < m_all) ptx::tma_load_2d(dst, &tmap_x, bar, kb * kBK, mt * kBM, pol_x);
                } else {
                    for (int c = 0; c < copies; ++c)
                        ptx::tma_load_2d(dst + (kCopies ? c * (C::kABytes / copies) : 0), &tmap_xl, bar, kb * kBK, mt * kBM, pol_x);
                }
            };
            // Bytes that land on a stage's full barrier. Pair: both CTAs' copies of a stage complete on the
            // even CTA's barrier, which the even CTA alone arms.
            auto stage_tx = [&](const Unit& w) {
                if constexpr (kPair) return static_cast<uint32_t>(2 * C::kStageBytes);
                uint32_t n = NB * bn * kBK * 2;
                for (int j = 0; j < MT; ++j) {
                    const int mt = w.mg * MT + j;
                    n += mt == m_short ? copies * x_last * kBK * 2 : mt < m_all ? C::kABytes : 0;
                }
                return n;
            };
            // Weight tiles of one stage; in a pair each CTA stages its half of the rows (tmap_w0's box is then
            // BN / 2 rows high).
            auto load_w = [&](uint8_t* sp, uint64_t* bar, int kb, int nt) {
                if constexpr (kPair) {
                    ptx::tma_load_2d_pair(sp + MT * C::kABytes, &tmap_w0, in_leader(bar), kb * kBK,
                                          nt * BN + crank * (BN / 2), pol_w);
                } else {
                    ptx::tma_load_2d(sp + MT * C::kABytes, &tmap_w0, bar, kb * kBK, nt * bn, pol_w);
                    if (NB == 2)
                        ptx::tma_load_2d(sp + MT * C::kABytes + bn * kBK * 2, &tmap_w1, bar, kb * kBK, nt * bn, pol_w);
                }
            };
            // The weights are no kernel's output: the first unit's first weight tiles are
            // requested before waiting for the previous kernel (which may be writing X).
            int pre = 0;
            if (cid < n_items) {
                const Item f = item_of(cid);
                const uint32_t tx = stage_tx(f.w);
                pre = f.kb1 - f.kb0 < stages ? f.kb1 - f.kb0 : stages;
                for (int i = 0; i < pre; ++i) {
                    if (leader) ptx::mbar_arrive_expect_tx(&full[i], tx);
                    load_w(smem + i * stage_bytes, &full[i], f.kb0 + i, f.w.nt);
                }
            }
            pdl_wait();
            int stage = 0;
            uint32_t phase = 0;
            uint32_t issued_mask = 0;                 // stages that ever received a load
            uint32_t last_parity[STAGES > 0 ? STAGES : 1];
            bool ok = true;
            int it = 0;                               // k-steps issued so far by this CTA
            for (int u = cid; u < n_items && ok; u += ncl) {
                const Item itm = item_of(u);
                const int nt = itm.w.nt, mt0 = (itm.w.mg * m_cl + m_rank) * MT;
                const uint32_t tx = stage_tx(itm.w);
                for (int kb = itm.kb0; kb < itm.kb1; ++kb, ++it) {
                    if (!ptx::mbar_wait(&empty[stage], phase ^ 1u, abort_flag, wait_ns)) {
                        ok = false;
                        break;
                    }
                    uint8_t* sp = smem + stage * stage_bytes;
                    const bool w_done = it < pre;     // weight tiles already requested above
                    if (!w_done && leader) ptx::mbar_arrive_expect_tx(&full[stage], tx);
#pragma unroll
                    for (int j = 0; j < MT; ++j) load_x(sp, &full[stage], j, kb, mt0 + j);
                    if (!w_done) load_w(sp, &full[stage], kb, nt);
                    issued_mask |= 1u << stage;
                    last_parity[stage] = phase;
                    if (++stage == stages) {
                        stage = 0;
                        phase ^= 1u;
                    }
                }
            }
            if (!ok) {
                *abort_flag = 1;
                set_status(status, TF_DEV_TIMEOUT);
            }
            // No copy may still be writing this CTA's shared memory when it exits: wait for the
            // last load of every stage (already complete unless another role gave up early). The
            // odd CTA of a pair has no barrier of its own to wait on: its copies complete on the
            // even CTA's barriers, which the even CTA's producer waits for here before both CTAs
            // meet at the final cluster barrier; after giving up it waits a fixed 100 us, far
            // longer than any copy takes once issued.
            if (leader) {
                for (int s = 0; s < STAGES; ++s)
                    if (issued_mask & (1u << s)) ptx::mbar_wait(&full[s], last_parity[s], nullptr, kWaitLimitNs);
            } else if (!ok) {
                const uint64_t t0 = ptx::globaltimer_ns();
                while (ptx::globaltimer_ns() - t0 < 100000ull) {
                }
            }
        }
    } else if (warp == 1) {
        // ------------------------------------------------------------------ MMA issuer
        if (lane == 0 && leader) {
            // the NB weight tiles of a stage are adjacent in shared memory with the same swizzle, so
            // one MMA of N = NB * BN covers them: A is read from shared memory once per k-step
            const uint32_t idesc = ptx::idesc_bf16_f32(kPair ? 2 * kBM : kBM, NB * bn);
            int stage = 0;
            uint32_t phase = 0;
            uint32_t use[2] = {0u, 0u};
            bool ok = true;
            int kl = 0;
            for (int u = cid; u < n_items && ok; u += ncl, ++kl) {
                const int g0 = (MT == 2) ? 0 : (kl & 1);
                const Item itm = item_of(u);
                const int nk_u = itm.kb1 - itm.kb0;
                // M-tiles past the rows are left out
                const int mts = MT == 1 ? 1 : min(MT, (n_rows + kBM - 1) / kBM - itm.w.mg * MT);
                for (int j = 0; j < MT && ok; ++j)
                    ok = kPair ? ptx::mbar_wait_cluster(&tempty[g0 + j], (use[g0 + j] & 1u) ^ 1u, abort_flag, wait_ns)
                               : ptx::mbar_wait(&tempty[g0 + j], (use[g0 + j] & 1u) ^ 1u, abort_flag, wait_ns);
                if (!ok) break;
                ptx::tc_fence_after();
                for (int kb = 0; kb < nk_u; ++kb) {   // position inside the item's K range
                    const bool landed = kPair ? ptx::mbar_wait_cluster(&full[stage], phase, abort_flag, wait_ns)
                                              : ptx::mbar_wait(&full[stage], phase, abort_flag, wait_ns);
                    if (!landed) {
                        ok = false;
                        break;
                    }
                    ptx::tc_fence_after();
                    const uint32_t a0 = ptx::smem_u32(smem + stage * stage_bytes);
                    const uint32_t b0 = a0 + MT * C::kABytes;
#pragma unroll
                    for (int kk = 0; kk < kBK / 16; ++kk) {
                        const uint64_t bd = ptx::sw128_kmajor_desc(b0 + kk * 32);
#pragma unroll
                        for (int j = 0; j < MT; ++j) {
                            const uint64_t ad = ptx::sw128_kmajor_desc(a0 + j * C::kABytes + kk * 32);
                            const uint32_t acc = (kb | kk) != 0 ? 1u : 0u;
                            if constexpr (kPair)
                                ptx::mma_bf16_pair(tmem_base + 256u * (g0 + j), ad, bd, idesc, acc);
                            else if (MT == 1 || j == 0 || j < mts)
                                ptx::mma_bf16(tmem_base + 256u * (g0 + j), ad, bd, idesc, acc);
                        }
                    }
                    // frees the stage (in both CTAs of a pair) once these MMAs finish
                    if constexpr (kPair) {
                        ptx::mma_commit_pair(ptx::smem_u32(&empty[stage]));
                        ptx::mma_commit_pair(in_peer(&empty[stage]));
                    } else {
                        ptx::mma_commit(&empty[stage]);
                    }
                    if (++stage == stages) {
                        stage = 0;
                        phase ^= 1u;
                    }
                }
                if (!ok) break;
                for (int j = 0; j < MT; ++j) {
                    if constexpr (kPair) {
                        ptx::mma_commit_pair(ptx::smem_u32(&tfull[g0 + j]));
                        ptx::mma_commit_pair(in_peer(&tfull[g0 + j]));
                    } else {
                        ptx::mma_commit(&tfull[g0 + j]);
                    }
                    ++use[g0 + j];
                }
            }
            if (!ok) {
                *abort_flag = 1;
                set_status(status, TF_DEV_TIMEOUT);
            }
            // every MMA issued so far must finish before TMEM is released
            if constexpr (kPair)
                ptx::mma_commit_pair(ptx::smem_u32(drain));
            else
                ptx::mma_commit(drain);
            ptx::mbar_wait(drain, 0, nullptr, kWaitLimitNs);
        }
    } else {
        // ------------------------------------------------------------------ epilogue
        const int e = warp - 2;
        const int g = e / (kEpiWarps / 2);          // accumulator slot of this group
        const int q = warp & 3;                     // TMEM lane quarter of this warp
        const int half = (e % (kEpiWarps / 2)) / 4; // which half of the columns this warp takes
        uint32_t use = 0, met = 0;
        int kl = 0;
        // A wait of this warp, with one outcome for its 32 lanes: a lane that gave up alone would be missing
        // from the warp-collective loads that follow.
        auto wait_warp = [&](uint64_t* bar, uint32_t parity) {
            if (__all_sync(0xffffffffu, ptx::mbar_wait(bar, parity, abort_flag, wait_ns))) return true;
            *abort_flag = 1;
            set_status(status, TF_DEV_TIMEOUT);
            return false;
        };
        // Meeting i of the epilogue warps that share it, after which each sees what the others wrote. Each warp
        // decides by itself whether its accumulator came in time, so one that has given up never
        // arrives here: the others give up in turn, where a hardware barrier would keep them for ever.
        auto meet_warps = [&](int i) {
            __syncwarp();
            if (lane == 0) ptx::mbar_arrive(&meet[i]);
            return wait_warp(&meet[i], met++ & 1u);
        };
        // hands the accumulator slot back to the MMA issuer; in a pair one arrival per warp on
        // the even CTA's barrier, after the warp's TMEM loads have completed
        auto release_slot = [&](int slot) {
            ptx::tc_fence_before();
            if constexpr (kPair) {
                __syncwarp();
                if (lane == 0) ptx::mbar_arrive_cluster(in_leader(&tempty[slot]));
            } else {
                ptx::mbar_arrive(&tempty[slot]);
            }
        };
        for (int u = cid; u < n_items; u += ncl, ++kl) {
            if (MT == 1 && !kShare && (kl & 1) != g) continue;
            if (!wait_warp(&tfull[kShare ? 0 : g], use & 1u)) break;
            ++use;
            ptx::tc_fence_after();
            const Item itm = item_of(u);
            const Unit w = itm.w;
            const int nt = w.nt;
            [[maybe_unused]] const int row = ((w.mg * m_cl + m_rank) * MT + (MT == 2 ? g : 0)) * kBM + q * 32 + lane;
            [[maybe_unused]] const uint32_t tb = tmem_base + 256u * g + (static_cast<uint32_t>(q * 32) << 16);

            if (kTail && itm.chunk >= 0) {
                // ---- a K-chunk of a tail unit: its partial sums to `partial`; the group whose
                // chunk completes the unit's count adds all chunks in chunk order
                const int j = kPair ? crank : MT == 2 ? g : 0; // M-tile of the unit in this slot
                const int r = q * 32 + lane;                   // row within the M-tile
                constexpr int kUnitF4 = kBM * NB * BN / 4;     // float4s of one (chunk, M-tile)
                float4* part = reinterpret_cast<float4*>(ep.partial);
                auto at = [&](int ch, int col) {               // float4 of columns col..col+3, row r
                    return (static_cast<size_t>((itm.tail * n_split + ch) * kUnitTiles + j) * kUnitF4) +
                           static_cast<size_t>(col >> 2) * kBM + r;
                };
#pragma unroll 1
                for (int nb = 0; nb < NB; ++nb) {
#pragma unroll 1
                    for (int c = half * (BN / 2); c < (half + 1) * (BN / 2); c += 32) {
                        uint32_t ra[32];
                        ptx::tmem_ld_32cols(tb + nb * BN + c, ra);
#pragma unroll
                        for (int f = 0; f < 8; ++f)
                            part[at(itm.chunk, nb * BN + c + 4 * f)] =
                                make_float4(__uint_as_float(ra[4 * f]), __uint_as_float(ra[4 * f + 1]),
                                            __uint_as_float(ra[4 * f + 2]), __uint_as_float(ra[4 * f + 3]));
                    }
                }
                release_slot(g);
                __threadfence();                                // this thread's partial sums, device-wide
                if (!meet_warps(g)) break;
                if (e % (kEpiWarps / 2) == 0 && lane == 0) {
                    __threadfence();
                    const int done = atomicAdd(ep.sem + itm.tail * kUnitTiles + j, 1);
                    last_chunk[g] = done == n_split - 1 ? 1 : 0;
                }
                if (!meet_warps(g)) break;
                if (last_chunk[g]) {
                    __threadfence();                            // every chunk's partial sums
                    // 8 output columns at a time: this warp's half of the tile
#pragma unroll 1
                    for (int c = half * (BN / 2); c < (half + 1) * (BN / 2); c += 8) {
                        float a0[8], a1[8];
#pragma unroll
                        for (int t = 0; t < 8; ++t) a0[t] = a1[t] = 0.0f;
                        // the chunks' loads in groups of kBatch, all in flight before the first add (one
                        // chunk at a time, this sum alone took some 35 us: 1928 rows, d = I = 5120, Eq. 1
                        // 403 -> 378 us)
                        constexpr int kBatch = 4 / NB;
#pragma unroll 1
                        for (int ch0 = 0; ch0 < n_split; ch0 += kBatch) {
                            float4 p[kBatch][2 * NB];
#pragma unroll
                            for (int t = 0; t < kBatch; ++t)
#pragma unroll
                                for (int f = 0; f < 2 * NB; ++f)
                                    p[t][f] = ch0 + t < n_split ? part[at(ch0 + t, (f >> 1) * BN + c + 4 * (f & 1))]
                                                                : make_float4(0.0f, 0.0f, 0.0f, 0.0f);
#pragma unroll
                            for (int t = 0; t < kBatch; ++t) {
                                if (ch0 + t >= n_split) break;
                                a0[0] += p[t][0].x; a0[1] += p[t][0].y; a0[2] += p[t][0].z; a0[3] += p[t][0].w;
                                a0[4] += p[t][1].x; a0[5] += p[t][1].y; a0[6] += p[t][1].z; a0[7] += p[t][1].w;
                                if constexpr (NB == 2) {
                                    a1[0] += p[t][2].x; a1[1] += p[t][2].y; a1[2] += p[t][2].z; a1[3] += p[t][2].w;
                                    a1[4] += p[t][3].x; a1[5] += p[t][3].y; a1[6] += p[t][3].z; a1[7] += p[t][3].w;
                                }
                            }
                        }
                        if (row < n_rows) {
                            uint32_t o[4];
                            if constexpr (EPI == EPI_GATEUP) {
#pragma unroll
                                for (int t = 0; t < 4; ++t)
                                    o[t] = pack_bf16x2(silu_f(a0[2 * t]) * a1[2 * t], silu_f(a0[2 * t + 1]) * a1[2 * t + 1]);
                            } else {
                                const int sq = row / ep.R, rr = row - sq * ep.R;
                                const int hid_row = sq * ep.gamma + stage2_hidden_index(rr, ep.M);
                                const uint4 hv = *reinterpret_cast<const uint4*>(
                                    ep.hidden + static_cast<size_t>(hid_row) * ep.ld_out + nt * BN + c);
                                const uint32_t hw[4] = {hv.x, hv.y, hv.z, hv.w};
#pragma unroll
                                for (int t = 0; t < 4; ++t) {
                                    const __nv_bfloat162 h2 = *reinterpret_cast<const __nv_bfloat162*>(&hw[t]);
                                    o[t] = pack_bf16x2(__bfloat162float(h2.x) + a0[2 * t], __bfloat162float(h2.y) + a0[2 * t + 1]);
                                }
                            }
                            *reinterpret_cast<uint4*>(ep.out + static_cast<size_t>(row) * ep.ld_out + nt * BN + c) =
                                make_uint4(o[0], o[1], o[2], o[3]);
                        }
                    }
                    // the count starts from zero for the next call (nothing reads it before: every chunk has
                    // been counted)
                    if (e % (kEpiWarps / 2) == 0 && lane == 0) ep.sem[itm.tail * kUnitTiles + j] = 0;
                }
            } else if constexpr (kSplitK) {
                // the accumulators are summed across the cluster below, once every CTA has them
            } else if constexpr (EPI == EPI_LMHEAD) {
                static_assert(BN == kBlockV, "one LM-head N tile is one vocabulary block");
                // this warp's chunks: a half of the block, or with copies of the rows its copy's part
                constexpr int kHalf = kChunks / 2;
                const Partials& P = ep.partials;
                const int copies = kCopies ? ep.copies : 1;
                const int per = kHalf / copies;          // chunks of this warp
                const int copy = q * copies / 4;         // (4 / copies row quarters per copy)
                const int crow = kCopies ? row - copy * (kBM / copies) : row;
                // warps whose 32 rows are all padding skip the accumulators entirely (with copies there
                // are none)
                const bool on = crow - lane < n_rows;
                float hm = -INFINITY, hsum = 0.0f;       // max of the chunks so far, sum of exp(z - hm)
                int hid = -1;
                if (on) {
                    // one chunk at a time (a second one in flight would not fit the registers; the other
                    // warps of the scheduler cover the TMEM load)
#pragma unroll 1
                    for (int j = 0; j < per; ++j) {
                        const int ci = half * kHalf + copy * per + j, v0 = nt * BN + ci * kChunk;
                        uint32_t ra[32];
                        ptx::tmem_ld_32cols(tb + ci * kChunk, ra);
                        float z[32];
#pragma unroll
                        for (int i = 0; i < 32; ++i) z[i] = __uint_as_float(ra[i]);
                        if (ep.inv_temp != 1.0f) {
#pragma unroll
                            for (int i = 0; i < 32; ++i) z[i] *= ep.inv_temp;
                        }
                        if (v0 + kChunk > ep.V) {
#pragma unroll
                            for (int i = 0; i < 32; ++i) z[i] = v0 + i < ep.V ? z[i] : -INFINITY;
                        }
                        const Top3 t = top3<0, 32>(z);
                        const float cs = sum_exp(z, t);
                        // chunks arrive in id order, so strict > keeps the smaller id
                        if (t.a1 > hm) hid = v0 + t.i1;
                        const float m = fmaxf(hm, t.a1);
                        if (t.a1 > -INFINITY) hsum = hsum * __expf(hm - m) + cs * __expf(t.a1 - m);
                        hm = m;
                        if (crow < n_rows)
                            P.chunks[P.chunk_at(nt, ci, crow)] = make_float4(t.a1, t.a2, t.a3, __int_as_float(t.i1 | (t.i2 << 8)));
                        __syncwarp();   // converged for the warp-collective TMEM loads
                    }
                }
                release_slot(g);
                if (on) {
                    if (!kCopies || copies == 1) {
                        if (crow < n_rows) P.halves[P.half_at(nt, half, crow)] = make_float4(hm, hsum, hm, __int_as_float(hid));
                    } else {
                        // the half's copies meet in shared memory; the first one folds them in chunk order.
                        // (A buffer is written again two units later, after a meeting that its readers have come to.)
                        float4* sums = copy_sums + ((g * 2 + half) * 2 + (use & 1u)) * kBM;
                        sums[copy * (kBM / copies) + crow] = make_float4(hm, hsum, 0.0f, __int_as_float(hid));
                        if (!meet_warps(g * 2 + half)) break;
                        if (copy == 0 && crow < n_rows) {
                            for (int c = 1; c < copies; ++c) {
                                const float4 o = sums[c * (kBM / copies) + crow];
                                if (o.x > hm) hid = __float_as_int(o.w);
                                const float m = fmaxf(hm, o.x);
                                if (m > -INFINITY) hsum = hsum * __expf(hm - m) + o.y * __expf(o.x - m);
                                hm = m;
                            }
                            P.halves[P.half_at(nt, half, crow)] = make_float4(hm, hsum, hm, __int_as_float(hid));
                        }
                    }
                }
            } else if constexpr (VAR) {
                // Columns in steps of 8, alternating between the two warps of a row quarter; a last
                // tile may run past the matrix (its weight rows there are zero, its columns dropped).
                const int n_tot = EPI == EPI_PARTIAL ? ep.n_total : ep.ld_out;
                const int cols = n_tot - nt * bn < bn ? n_tot - nt * bn : bn;
                int hid_row = 0;
                if (EPI == EPI_DOWN && row < n_rows) {
                    const int sq = row / ep.R, rr = row - sq * ep.R;
                    hid_row = sq * ep.gamma + stage2_hidden_index(rr, ep.M);
                }
#pragma unroll 1
                for (int c = 8 * half; c < cols; c += 16) {
                    uint32_t ra[NB][8];
#pragma unroll
                    for (int nb = 0; nb < NB; ++nb) ptx::tmem_ld_8cols(tb + nb * bn + c, ra[nb]);
                    const size_t col = static_cast<size_t>(nt) * bn + c;
                    if (row >= n_rows) {
                    } else if constexpr (EPI == EPI_PARTIAL) {
                        float4* split = reinterpret_cast<float4*>(ep.partial + static_cast<size_t>(w.kx) * ep.n_cols * n_rows);
#pragma unroll
                        for (int nb = 0; nb < NB; ++nb) {
                            float4* dst = split + (nb * static_cast<size_t>(ep.n_total) + col) / 4 * n_rows + row;
#pragma unroll
                            for (int j = 0; j < 2; ++j)
                                dst[static_cast<size_t>(j) * n_rows] =
                                    make_float4(__uint_as_float(ra[nb][4 * j]), __uint_as_float(ra[nb][4 * j + 1]),
                                                __uint_as_float(ra[nb][4 * j + 2]), __uint_as_float(ra[nb][4 * j + 3]));
                        }
                    } else {
                        uint32_t o[4];
                        if constexpr (EPI == EPI_GATEUP) {
#pragma unroll
                            for (int t = 0; t < 4; ++t)
                                o[t] = pack_bf16x2(silu_f(__uint_as_float(ra[0][2 * t])) * __uint_as_float(ra[NB - 1][2 * t]),
                                                   silu_f(__uint_as_float(ra[0][2 * t + 1])) * __uint_as_float(ra[NB - 1][2 * t + 1]));
                        } else {
                            const uint4 hv = *reinterpret_cast<const uint4*>(ep.hidden + static_cast<size_t>(hid_row) * ep.ld_out + col);
                            const uint32_t hw[4] = {hv.x, hv.y, hv.z, hv.w};
#pragma unroll
                            for (int t = 0; t < 4; ++t) {
                                const __nv_bfloat162 h2 = *reinterpret_cast<const __nv_bfloat162*>(&hw[t]);
                                o[t] = pack_bf16x2(__bfloat162float(h2.x) + __uint_as_float(ra[0][2 * t]),
                                                   __bfloat162float(h2.y) + __uint_as_float(ra[0][2 * t + 1]));
                            }
                        }
                        *reinterpret_cast<uint4*>(ep.out + static_cast<size_t>(row) * ep.ld_out + col) = make_uint4(o[0], o[1], o[2], o[3]);
                    }
                    __syncwarp();   // converged again for the next TMEM load
                }
                release_slot(g);
            } else if constexpr (EPI == EPI_PARTIAL) {
                // float4-major: each store instruction writes the warp's 32 rows of 4 columns, 512
                // contiguous bytes
                float4* split = reinterpret_cast<float4*>(ep.partial + static_cast<size_t>(w.kx) * ep.n_cols * n_rows);
#pragma unroll 1
                for (int nb = 0; nb < NB; ++nb) {
#pragma unroll 1
                    for (int c = half * (BN / 2); c < (half + 1) * (BN / 2); c += 32) {
                        uint32_t ra[32];
                        ptx::tmem_ld_32cols(tb + nb * BN + c, ra);
                        if (row < n_rows) {
                            const int col = nb * ep.n_total + nt * BN + c;
                            float4* dst = split + static_cast<size_t>(col >> 2) * n_rows + row;
#pragma unroll
                            for (int j = 0; j < 8; ++j)
                                dst[static_cast<size_t>(j) * n_rows] = make_float4(__uint_as_float(ra[4 * j]), __uint_as_float(ra[4 * j + 1]),
                                                     __uint_as_float(ra[4 * j + 2]), __uint_as_float(ra[4 * j + 3]));
                        }
                    }
                }
                release_slot(g);
            } else if constexpr (EPI == EPI_GATEUP) {
#pragma unroll 1
                for (int c = half * (BN / 2); c < (half + 1) * (BN / 2); c += 32) {
                    uint32_t rg[32], ru[32];
                    ptx::tmem_ld_32cols(tb + c, rg);
                    ptx::tmem_ld_32cols(tb + BN + c, ru);
                    uint32_t packed[16];
#pragma unroll
                    for (int j = 0; j < 16; ++j) {
                        const float a0 = silu_f(__uint_as_float(rg[2 * j])) * __uint_as_float(ru[2 * j]);
                        const float a1 = silu_f(__uint_as_float(rg[2 * j + 1])) * __uint_as_float(ru[2 * j + 1]);
                        packed[j] = pack_bf16x2(a0, a1);
                    }
                    if (row < n_rows) {
                        uint4* dst = reinterpret_cast<uint4*>(ep.out + static_cast<size_t>(row) * ep.ld_out + nt * BN + c);
#pragma unroll
                        for (int j = 0; j < 4; ++j)
                            dst[j] = make_uint4(packed[4 * j], packed[4 * j + 1], packed[4 * j + 2], packed[4 * j + 3]);
                    }
                }
                release_slot(g);
            } else {  // EPI_DOWN
                int hid_row = 0;
                if (row < n_rows) {
                    const int sq = row / ep.R, rr = row - sq * ep.R;
                    hid_row = sq * ep.gamma + stage2_hidden_index(rr, ep.M);
                }
#pragma unroll 1
                for (int c = half * (BN / 2); c < (half + 1) * (BN / 2); c += 32) {
                    uint32_t ra[32];
                    ptx::tmem_ld_32cols(tb + c, ra);
                    if (row < n_rows) {
                        const uint4* res = reinterpret_cast<const uint4*>(
                            ep.hidden + static_cast<size_t>(hid_row) * ep.ld_out + nt * BN + c);
                        uint4* dst = reinterpret_cast<uint4*>(ep.out + static_cast<size_t>(row) * ep.ld_out + nt * BN + c);
#pragma unroll
                        for (int j = 0; j < 4; ++j) {
                            const uint4 hv = res[j];
                            const uint32_t hw[4] = {hv.x, hv.y, hv.z, hv.w};
                            uint32_t o[4];
#pragma unroll
                            for (int t = 0; t < 4; ++t) {
                                const __nv_bfloat162 h2 = *reinterpret_cast<const __nv_bfloat162*>(&hw[t]);
                                const float x0 = __bfloat162float(h2.x) + __uint_as_float(ra[8 * j + 2 * t]);
                                const float x1 = __bfloat162float(h2.y) + __uint_as_float(ra[8 * j + 2 * t + 1]);
                                o[t] = pack_bf16x2(x0, x1);
                            }
                            dst[j] = make_uint4(o[0], o[1], o[2], o[3]);
                        }
                    }
                }
                release_slot(g);
            }
        }
    }

    if constexpr (kSplitK && !VAR) {
        // ------------------------------------------------------------------ split-K sum, 128 columns
        // The tile's output columns are owned in CL blocks of BN / CL: CTA o adds the CL partial
        // sums of block o in K-range order (the order of the split-K reduction kernels) and
        // applies the epilogue. Every CTA writes the blocks it does not own to the exchange area
        // in global memory (it stays in L2; through L2 this takes half the time of remote
        // shared-memory stores), laid out [cluster][owner][sender slot][16-byte unit][row] so that
        // the 32 lanes (rows) of a warp store and load 512 contiguous bytes; one cluster barrier
        // (release/acquire at cluster scope) then makes them visible to their owners.
        constexpr int kOwn = BN / CL;                    // output columns per owner
        constexpr int kRowF4 = NB * kOwn / 4;            // 16-byte units per row of a block
        constexpr int kSlotF4 = MT * kBM * kRowF4;       // 16-byte units of one block
        static_assert(kOwn == 32, "one TMEM load per block and accumulator");
        const bool has_unit = cid < n_units;
        const int e = warp - 2;
        const int g = e / (kEpiWarps / 2), q = warp & 3, half = (e % (kEpiWarps / 2)) / 4;
        const int r = g * kBM + q * 32 + lane;           // tile row: TMEM slot g, lane q * 32 + lane
        const uint32_t tb = tmem_base + 256u * g + (static_cast<uint32_t>(q * 32) << 16);
        float4* xchg = reinterpret_cast<float4*>(ep.partial);
        // (the epilogue warps waited for this CTA's accumulators in the loop above)
        if (warp >= 2 && has_unit) {
            // the warp's half of the columns holds the blocks of owners 2 half and 2 half + 1
            for (int o = 2 * half; o < 2 * half + 2; ++o) {
                if (o == crank) continue;
                const int slot = crank < o ? crank : crank - 1;
                float4* dst = xchg + (static_cast<size_t>(cid * CL + o) * (CL - 1) + slot) * kSlotF4 + r;
#pragma unroll
                for (int nb = 0; nb < NB; ++nb) {
                    uint32_t ra[32];
                    ptx::tmem_ld_32cols(tb + nb * BN + o * kOwn, ra);
#pragma unroll
                    for (int f = 0; f < 8; ++f)
                        dst[(nb * 8 + f) * (MT * kBM)] = make_float4(__uint_as_float(ra[4 * f]), __uint_as_float(ra[4 * f + 1]),
                                                                   __uint_as_float(ra[4 * f + 2]), __uint_as_float(ra[4 * f + 3]));
                }
            }
        }
        __syncwarp();
        ptx::tc_fence_before();
        ptx::cluster_sync();   // every block is in the exchange area
        ptx::tc_fence_after();
        if (warp >= 2 && has_unit) {
            // this warp: 16 of the own block's columns, c0 .. c0 + 15 of the tile
            const Unit w = unit_of(cid);
            const int c0 = crank * kOwn + half * 16;
            const int row = w.mg * MT * kBM + r;
            float acc[NB][16];
#pragma unroll
            for (int kx = 0; kx < CL; ++kx) {
#pragma unroll
                for (int nb = 0; nb < NB; ++nb) {
                    float v[16];
                    if (kx == crank) {
                        uint32_t ra[16];
                        ptx::tmem_ld_16cols(tb + nb * BN + c0, ra);
#pragma unroll
                        for (int j = 0; j < 16; ++j) v[j] = __uint_as_float(ra[j]);
                    } else {
                        const int slot = kx < crank ? kx : kx - 1;
                        const float4* src = xchg + (static_cast<size_t>(cid * CL + crank) * (CL - 1) + slot) * kSlotF4 + r;
#pragma unroll
                        for (int f = 0; f < 4; ++f) {
                            const float4 t = src[(nb * 8 + half * 4 + f) * (MT * kBM)];
                            v[4 * f] = t.x;
                            v[4 * f + 1] = t.y;
                            v[4 * f + 2] = t.z;
                            v[4 * f + 3] = t.w;
                        }
                    }
#pragma unroll
                    for (int j = 0; j < 16; ++j) acc[nb][j] = kx == 0 ? v[j] : acc[nb][j] + v[j];
                }
            }
            if (row < n_rows) {
                const size_t col = static_cast<size_t>(w.nt) * BN + c0;
                uint32_t packed[8];
                if constexpr (EPI == EPI_CGATEUP) {
#pragma unroll
                    for (int j = 0; j < 8; ++j)
                        packed[j] = pack_bf16x2(silu_f(acc[0][2 * j]) * acc[NB - 1][2 * j],
                                                silu_f(acc[0][2 * j + 1]) * acc[NB - 1][2 * j + 1]);
                } else {
                    const int sq = row / ep.R, rr = row - sq * ep.R;
                    const int hid_row = sq * ep.gamma + stage2_hidden_index(rr, ep.M);
                    const uint4* res = reinterpret_cast<const uint4*>(ep.hidden + static_cast<size_t>(hid_row) * ep.ld_out + col);
#pragma unroll
                    for (int j = 0; j < 2; ++j) {
                        const uint4 hv = res[j];
                        const uint32_t hw[4] = {hv.x, hv.y, hv.z, hv.w};
#pragma unroll
                        for (int t = 0; t < 4; ++t) {
                            const __nv_bfloat162 h2 = *reinterpret_cast<const __nv_bfloat162*>(&hw[t]);
                            packed[4 * j + t] = pack_bf16x2(__bfloat162float(h2.x) + acc[0][8 * j + 2 * t],
                                                            __bfloat162float(h2.y) + acc[0][8 * j + 2 * t + 1]);
                        }
                    }
                }
                uint4* dst = reinterpret_cast<uint4*>(ep.out + static_cast<size_t>(row) * ep.ld_out + col);
                dst[0] = make_uint4(packed[0], packed[1], packed[2], packed[3]);
                dst[1] = make_uint4(packed[4], packed[5], packed[6], packed[7]);
            }
        }
    }

    if constexpr (kSplitK && VAR) {
        // ------------------------------------------------------------------ split-K sum, any width
        // The same with up to CL K-ranges, one or two M-tiles and columns owned in steps of 8; the
        // exchange area is laid out [cluster][sender][16-byte unit][row].
        const bool has_unit = cid < n_units;
        const int e = warp - 2;
        const int g = e / (kEpiWarps / 2), q = warp & 3, half = (e % (kEpiWarps / 2)) / 4;
        // a warp's M-tile and its share of the column steps: two warps per row quarter and M-tile
        // with two M-tiles, four with one
        constexpr int kColWarps = kShare ? 4 : 2;
        const int mt = kShare ? 0 : g, cw = kShare ? 2 * g + half : half;
        const int r = mt * kBM + q * 32 + lane;          // tile row: TMEM slot mt, lane q * 32 + lane
        const uint32_t tb = tmem_base + 256u * mt + (static_cast<uint32_t>(q * 32) << 16);
        const int ks = k_splits, n8 = bn / 8;
        const int o0 = n8 * crank / ks, o1 = n8 * (crank + 1) / ks;    // this CTA's column steps
        float4* xchg = reinterpret_cast<float4*>(ep.partial);
        auto at = [&](int sender, int nb, int c8, int f) {              // float4 f of step c8
            return (static_cast<size_t>(cid * ks + sender) * (NB * n8 * 2) + (nb * n8 + c8) * 2 + f) * (MT * kBM) + r;
        };
        // (the epilogue warps waited for this CTA's accumulators in the loop above; warps whose rows are
        // all padding have nothing to exchange)
        const bool rows_on = warp >= 2 && has_unit && unit_of(cid).mg * MT * kBM + r - lane < n_rows;
        if (rows_on) {
            // four column steps per TMEM wait: the steps of the other owners, in order
            const int others = n8 - (o1 - o0);
#pragma unroll 1
            for (int i = cw; i < others; i += 4 * kColWarps) {
                int c8[4];
#pragma unroll
                for (int t = 0; t < 4; ++t) {
                    const int j = i + t * kColWarps;
                    c8[t] = j < others ? (j < o0 ? j : j + o1 - o0) : -1;
                }
#pragma unroll
                for (int nb = 0; nb < NB; ++nb) {
                    uint32_t ra[32];
                    ptx::tmem_ld_8cols_nowait<0>(tb + nb * bn + 8 * c8[0], ra);
                    ptx::tmem_ld_8cols_nowait<8>(tb + nb * bn + 8 * (c8[1] < 0 ? c8[0] : c8[1]), ra);
                    ptx::tmem_ld_8cols_nowait<16>(tb + nb * bn + 8 * (c8[2] < 0 ? c8[0] : c8[2]), ra);
                    ptx::tmem_ld_8cols_nowait<24>(tb + nb * bn + 8 * (c8[3] < 0 ? c8[0] : c8[3]), ra);
                    ptx::tmem_wait_ld_regs(ra);
#pragma unroll
                    for (int t = 0; t < 4; ++t)
                        if (c8[t] >= 0) {
                            float4* dst = xchg + at(crank, nb, c8[t], 0);
#pragma unroll
                            for (int f = 0; f < 2; ++f)
                                dst[f * (MT * kBM)] = make_float4(__uint_as_float(ra[8 * t + 4 * f]), __uint_as_float(ra[8 * t + 4 * f + 1]),
                                                                  __uint_as_float(ra[8 * t + 4 * f + 2]), __uint_as_float(ra[8 * t + 4 * f + 3]));
                        }
                }
            }
        }
        __syncwarp();
        ptx::tc_fence_before();
        ptx::cluster_sync();   // every column step is in the exchange area
        ptx::tc_fence_after();
        if (rows_on) {
            const Unit w = unit_of(cid);
            const int row = w.mg * MT * kBM + r;
            int hid_row = 0;
            if (EPI == EPI_CDOWN && row < n_rows) {
                const int sq = row / ep.R, rr = row - sq * ep.R;
                hid_row = sq * ep.gamma + stage2_hidden_index(rr, ep.M);
            }
            // the first step of this warp at or after o0
#pragma unroll 1
            for (int c8 = o0 + (cw + kColWarps - o0 % kColWarps) % kColWarps; c8 < o1; c8 += kColWarps) {
                const int col = w.nt * bn + 8 * c8;
                float4 in[CL][NB][2];
#pragma unroll
                for (int kx = 0; kx < CL; ++kx)
#pragma unroll
                    for (int nb = 0; nb < NB; ++nb)
#pragma unroll
                        for (int f = 0; f < 2; ++f)
                            in[kx][nb][f] = kx < ks && kx != crank ? xchg[at(kx, nb, c8, f)] : make_float4(0.0f, 0.0f, 0.0f, 0.0f);
                float acc[NB][8];
#pragma unroll
                for (int nb = 0; nb < NB; ++nb) {
                    uint32_t ra[8];
                    ptx::tmem_ld_8cols(tb + nb * bn + 8 * c8, ra);
#pragma unroll
                    for (int kx = 0; kx < CL; ++kx) {
                        if (kx >= ks) break;
                        const float4 p0 = in[kx][nb][0], p1 = in[kx][nb][1];
                        const float v[8] = {p0.x, p0.y, p0.z, p0.w, p1.x, p1.y, p1.z, p1.w};
#pragma unroll
                        for (int j = 0; j < 8; ++j) {
                            const float t = kx == crank ? __uint_as_float(ra[j]) : v[j];
                            acc[nb][j] = kx == 0 ? t : acc[nb][j] + t;
                        }
                    }
                }
                if (row < n_rows && col < ep.ld_out) {
                    uint32_t o[4];
                    if constexpr (EPI == EPI_CGATEUP) {
#pragma unroll
                        for (int t = 0; t < 4; ++t)
                            o[t] = pack_bf16x2(silu_f(acc[0][2 * t]) * acc[NB - 1][2 * t],
                                               silu_f(acc[0][2 * t + 1]) * acc[NB - 1][2 * t + 1]);
                    } else {
                        const uint4 hv = *reinterpret_cast<const uint4*>(ep.hidden + static_cast<size_t>(hid_row) * ep.ld_out + col);
                        const uint32_t hw[4] = {hv.x, hv.y, hv.z, hv.w};
#pragma unroll
                        for (int t = 0; t < 4; ++t) {
                            const __nv_bfloat162 h2 = *reinterpret_cast<const __nv_bfloat162*>(&hw[t]);
                            o[t] = pack_bf16x2(__bfloat162float(h2.x) + acc[0][2 * t], __bfloat162float(h2.y) + acc[0][2 * t + 1]);
                        }
                    }
                    *reinterpret_cast<uint4*>(ep.out + static_cast<size_t>(row) * ep.ld_out + col) = make_uint4(o[0], o[1], o[2], o[3]);
                }
                __syncwarp();   // converged again for the next TMEM load
            }
        }
    }

    // the producer and MMA lanes rejoin their warps first: the CTA-wide barrier below must wait
    // for every thread, not only for each warp's first arrivals
    __syncwarp();
    ptx::tc_fence_before();
    __syncthreads();
    // no CTA of the cluster may still write into this CTA's shared memory or barriers
    if constexpr (CL > 1) ptx::cluster_sync();
    if (warp == 1) {
        __syncwarp();
        ptx::tc_fence_after();
        if constexpr (kPair)
            ptx::tmem_dealloc_pair(tmem_base, 512);
        else
            ptx::tmem_dealloc(tmem_base, 512);
    }
}

// ------------------------------------------------------------------------------ host side

typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

EncodeTiledFn encode_fn() {
    static EncodeTiledFn fn = [] {
        void* p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) !=
                cudaSuccess ||
            q != cudaDriverEntryPointSuccess)
            p = nullptr;
        return reinterpret_cast<EncodeTiledFn>(p);
    }();
    return fn;
}

// Row-major bf16 matrix [outer, inner] read in boxes of box_inner x box_outer with 128B swizzle.
cudaError_t make_tmap(CUtensorMap* map, const void* base, uint64_t inner, uint64_t outer, uint32_t box_inner,
                      uint32_t box_outer) {
    EncodeTiledFn fn = encode_fn();
    if (!fn) return cudaErrorNotSupported;
    const cuuint64_t dims[2] = {inner, outer};
    const cuuint64_t strides[1] = {inner * 2};
    const cuuint32_t box[2] = {box_inner, box_outer};
    const cuuint32_t es[2] = {1, 1};
    CUresult r = fn(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(base), dims, strides, box, es,
                    CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                    CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    return r == CUDA_SUCCESS ? cudaSuccess : cudaErrorInvalidValue;
}

// The maps of a kernel's X operand [n_rows, K]: whole M-tiles, and the rows of the last one.
struct XMaps {
    CUtensorMap whole, last;
};
cudaError_t make_xmaps(XMaps* m, const void* x, int K, int n_rows) {
    const int rem = n_rows % kBM;
    cudaError_t e = make_tmap(&m->whole, x, K, n_rows, kBK, kBM);
    if (e == cudaSuccess) e = make_tmap(&m->last, x, K, n_rows, kBK, rem ? (rem + 7) / 8 * 8 : kBM);
    return e;
}

// Clusters of cl CTAs that can be resident at once for this kernel (at most num_sms / cl).
template <typename K>
int resident_clusters(K kern, int smem, int cl, int num_sms) {
    int cap = num_sms / cl;
    if (cl == 1) return cap;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(cl * cap);
    cfg.blockDim = dim3(kThreads);
    cfg.dynamicSmemBytes = smem;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = cl;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    int n = 0;
    if (cudaOccupancyMaxActiveClusters(&n, kern, &cfg) != cudaSuccess || n < 1) {
        (void)cudaGetLastError();
        return cap;
    }
    return n < cap ? n : cap;
}

// Tail split: when the units overflow the SMs by a last round that would leave most of them idle, each
// unit of that round runs as up to kMaxTailSplit K-chunks on the idle SMs, summed by the chunk that
// finishes last (fp32 partial sums in the workspace). K-chunks per unit, or 0: no tail split. slots: the
// units that run at once, one per SM or pair of SMs.
int tail_chunks(const Ctx& ctx, int n_units, int slots, int m_tiles, int cols, int K, size_t partial_bytes) {
    const int tail = n_units % slots;
    int split = tail > 0 ? slots / tail : 0;
    split = split < kMaxTailSplit ? split : kMaxTailSplit;
    split = split < K / kBK ? split : K / kBK;
    const size_t need = static_cast<size_t>(tail) * split * m_tiles * kBM * cols * sizeof(float);
    const bool fits = ctx.status && tail * m_tiles <= kTailSems && need <= partial_bytes;
    return n_units > slots && split >= 2 && fits ? split : 0;
}

template <int EPI, int MT, int NB, int BN, int STAGES, int CL = 1>
cudaError_t run_gemm(const Ctx& ctx, const XMaps& tx, const CUtensorMap& tw0, const CUtensorMap& tw1,
                     int n_rows, int K, int n_ntiles, int n_mgroups, const EpiParams& ep_in, int k_splits = 1,
                     size_t partial_bytes = 0) {
    constexpr bool kSplitK = EPI == EPI_CGATEUP || EPI == EPI_CDOWN;
    using C = TileCfg<MT, NB, BN, STAGES, CL == 2 && !kSplitK>;
    auto kern = tc_gemm_kernel<EPI, MT, NB, BN, STAGES, CL, false>;
    EpiParams ep = ep_in;
    ep.wait_ns = wait_limit_ns();
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, C::kSmemBytes);
    if (e != cudaSuccess) return e;
    const int n_units = n_ntiles * n_mgroups * k_splits;
    const int stream_once = n_mgroups == 1 ? 1 : 0;
    if constexpr (kSplitK) {   // one output tile per cluster, its K-ranges on the cluster's CTAs
        e = launch_pdl_cluster(kern, dim3(CL * n_ntiles * n_mgroups), dim3(kThreads), C::kSmemBytes, ctx.stream, CL,
                               tx.whole, tx.last, tw0, tw1, n_rows, K, n_ntiles, n_mgroups, CL, stream_once, ep, ctx.status);
        return e != cudaSuccess ? e : cudaGetLastError();
    }
    int n_items = n_units;
    if constexpr (EPI == EPI_GATEUP || EPI == EPI_DOWN) {
        constexpr int kTiles = CL == 1 ? MT : 2;
        const int slots = CL == 2 ? ctx.num_sms / 2 : ctx.num_sms;
        const int split = k_splits == 1 && ep.partial
                              ? tail_chunks(ctx, n_units, slots, kTiles, NB * BN, K, partial_bytes) : 0;
        if (split) {
            const int tail = n_units % slots;
            ep.n_full = n_units - tail;
            ep.tail_split = split;
            ep.sem = ctx.status + 1;
            n_items = ep.n_full + tail * split;
        }
    }
    if constexpr (CL == 1) {
        const int grid = n_items < ctx.num_sms ? n_items : ctx.num_sms;
        e = launch_pdl(kern, dim3(grid), dim3(kThreads), C::kSmemBytes, ctx.stream, tx.whole, tx.last, tw0, tw1, n_rows, K,
                       n_ntiles, n_mgroups, k_splits, stream_once, ep, ctx.status);
    } else {
        static const int max_cl = resident_clusters(kern, C::kSmemBytes, CL, ctx.num_sms);
        const int n_cl = n_items < max_cl ? n_items : max_cl;
        e = launch_pdl_cluster(kern, dim3(CL * n_cl), dim3(kThreads), C::kSmemBytes, ctx.stream, CL, tx.whole, tx.last, tw0, tw1,
                               n_rows, K, n_ntiles, n_mgroups, k_splits, stream_once, ep, ctx.status);
    }
    return e != cudaSuccess ? e : cudaGetLastError();
}

}  // namespace

cudaError_t launch_lmhead_tc(const Ctx& ctx, const void* lm_head, const void* x, int n_rows, int d, int V,
                             float inv_temp, Partials partials, bool reset_status) {
    if (n_rows <= 0) return cudaSuccess;
    const int n_tiles = (V + kBlockV - 1) / kBlockV;
    const int m_tiles = (n_rows + kBM - 1) / kBM;
    // More than one M-tile: CTA pairs (clusters of two), one M-tile each, share every weight tile
    // through cta_group::2 MMAs (each stages half of its rows), so W_lm is read once while each
    // CTA keeps one TMEM slot per unit and overlaps its epilogue with the next unit's MMAs; 32 KB
    // per CTA and stage leaves room for seven stages. Three and five M-tiles run on single CTAs, which
    // read each weight tile once per M-tile from L2 but leave out the missing half of the last pair
    // (V = 151936, d = 4096: 320 rows 390 -> 345 us, 322 with whole boxes of X, 600 rows 575 -> 552; d = 1024:
    // 115 -> 92, 174 -> 150;
    // seven M-tiles gain nothing), and so do small d, where the epilogue sets the pace and single CTAs
    // hand over their accumulators sooner (d = 512: 250 rows 46 -> 41 us, 1020 rows 147 -> 139; d = 1024:
    // 64 -> 71, so pairs from there on).
    const bool single = m_tiles == 1 || m_tiles == 3 || m_tiles == 5 || d <= 512;
    const int cl = single ? 1 : 2;
    XMaps tx;
    CUtensorMap tw;
    // Few rows would leave all epilogue work to the warps of one TMEM lane quarter, which share one
    // scheduler (the TMA producer's): copies of the rows in the other quarters spread it over all sixteen
    // warps (V = 151936, 16 rows: d = 512 37 -> 28 us, d = 1024 64 -> 49, d = 2048 116 -> 101, d = 3072 174 ->
    // 144 on GB300). None from d = 4096 on, where the stream of W sets the pace and more copies per stage delay
    // it (V = 45000 79 against 85 us with copies), nor where a CTA's only block waits for its loads, with
    // half of the SMs idle (V = 9001: d = 2048 16.5 against 20.6, but d = 512 9.6 against 9.1).
    const bool copied = d < 4096 && (2 * n_tiles > ctx.num_sms || d <= 512);
    const int copies = !copied ? 1 : n_rows <= 32 ? 4 : n_rows <= 64 ? 2 : 1;
    cudaError_t e = make_xmaps(&tx, x, d, n_rows);
    if (e == cudaSuccess) e = make_tmap(&tw, lm_head, d, V, kBK, kBlockV / cl);
    if (e != cudaSuccess) return e;
    EpiParams ep{};
    ep.partials = partials;
    ep.V = V;
    ep.inv_temp = inv_temp;
    ep.reset_status = reset_status ? 1 : 0;
    ep.copies = copies;
    if (single) return run_gemm<EPI_LMHEAD, 1, 1, kBlockV, 4>(ctx, tx, tw, tw, n_rows, d, n_tiles, m_tiles, ep);
    return run_gemm<EPI_LMHEAD, 1, 1, kBlockV, 7, 2>(ctx, tx, tw, tw, n_rows, d, n_tiles, (m_tiles + 1) / 2, ep);
}

// Split-K factor for a GEMM with `base_units` (N tiles x M-tile groups) and nk K-steps: enough
// units to cover the SMs, at most kMaxKSplits, and a divisor of nk.
int choose_k_splits(int base_units, int nk, int num_sms) {
    int ks = base_units >= num_sms ? 1 : num_sms / base_units;
    if (ks > kMaxKSplits) ks = kMaxKSplits;
    while (ks > 1 && nk % ks != 0) --ks;
    return ks < 1 ? 1 : ks;
}

// Units from which CTA pairs take over from single CTAs of chosen width in the down projection (GB300,
// 152 SMs): d = 4096, 723 rows, 48 pairs: Eq. 1 111 against 114 us; d = 2560, 241 rows, 40 pairs: 84.5
// against 85.8; d = 2048, 32 pairs: 37.0 against 35.3.
constexpr int kMinPairs = 40;
constexpr int kMinClusterCtas = 96;

// A GEMM of single CTAs whose tile width is chosen for the SM count: [n_rows, K] x [N, K]^T (NB
// matrices side by side), in k_splits K-ranges. A round of units costs about what an SM loads per
// K-step (its weight tile, and X, mostly from L2, at half weight), so the width in [32, 128] that
// makes the cheapest whole rounds is taken: 12288 columns of one M-tile run as 140 tiles of 88 on 152
// SMs instead of 96 of 128 (121 rows, gate/up and down: 114 -> 102 us), 1024 columns in 4 K-ranges as
// 128 units of 32 instead of 32 of 128. The width does not change any output's sum.
template <int EPI, int MT, int NB>
cudaError_t run_gemm_var(const Ctx& ctx, const XMaps& tx, const void* w0, const void* w1, int N, int n_rows, int K,
                         int n_mgroups, int k_splits, const EpiParams& ep_in) {
    using C = TileCfg<MT, NB, 128, kVarMaxStages, false, true>;
    auto kern = tc_gemm_kernel<EPI, MT, NB, 128, kVarMaxStages, 1, true>;
    int bn = 128;
    double best = 0.0;
    // N of an MMA with M = 128 is a multiple of 16; boxes of whole 8-row swizzle groups
    constexpr int kStep = NB == 1 ? 16 : 8;
    for (int w = 128; w >= 32; w -= kStep) {
        const long long units = static_cast<long long>((N + w - 1) / w) * n_mgroups * k_splits;
        const long long rounds = (units + ctx.num_sms - 1) / ctx.num_sms;
        const double cost = static_cast<double>(rounds) * (MT * 8.0 + NB * w / 8.0 + 2.0);
        if (w == 128 || cost < best) {
            best = cost;
            bn = w;
        }
    }
    CUtensorMap t0, t1;
    cudaError_t e = make_tmap(&t0, w0, K, N, kBK, bn);
    if (e == cudaSuccess) e = make_tmap(&t1, NB == 2 ? w1 : w0, K, N, kBK, bn);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, C::kSmemBytes);
    if (e != cudaSuccess) return e;
    EpiParams ep = ep_in;
    ep.wait_ns = wait_limit_ns();
    ep.bn = bn;
    const int stages = C::kRingBytes / (MT * C::kABytes + NB * bn * kBK * 2);
    ep.stages = stages < kVarMaxStages ? stages : kVarMaxStages;
    const int n_ntiles = (N + bn - 1) / bn;
    const long long n_units = static_cast<long long>(n_ntiles) * n_mgroups * k_splits;
    const int grid = static_cast<int>(n_units < ctx.num_sms ? n_units : ctx.num_sms);
    e = launch_pdl(kern, dim3(grid), dim3(kThreads), C::kSmemBytes, ctx.stream, tx.whole, tx.last, t0, t1, n_rows, K, n_ntiles, n_mgroups,
                   k_splits, n_mgroups == 1 ? 1 : 0, ep, ctx.status);
    return e != cudaSuccess ? e : cudaGetLastError();
}

// Clusters of three left unused of those that fit an empty GPU: with as many as fit, one often finds no place
// beside clusters of the next or the previous kernel, and runs a round of its own (46 clusters, Eq. 1 of 241 rows,
// d = 1920, I = 5120 57 to 66 us; with two to spare 49, with reduction kernels 50). Clusters of two and four
// always found one (d = I = 4608, 36 of four: 64 us, 73 with two to spare).
constexpr int kSpareTriples = 2;

// The same where K is split: k_splits CTAs form a cluster on one output tile and exchange their partial
// sums, so no reduction kernel follows. All clusters must be resident at once (one tile each), which
// bounds their number; the tile width follows from it. *done stays false, and nothing runs, where there
// are too many tiles for that.
template <int EPI, int MT, int NB>
cudaError_t run_gemm_cluster(const Ctx& ctx, const XMaps& tx, const void* w0, const void* w1, int N, int n_rows, int K,
                             int n_mgroups, int k_splits, const EpiParams& ep_in, size_t partial_bytes, bool* done) {
    using C = TileCfg<MT, NB, 128, kVarMaxStages, false, true>;
    auto kern = tc_gemm_kernel<EPI, MT, NB, 128, kVarMaxStages, kMaxKSplits, true>;
    constexpr int kStep = NB == 1 ? 16 : 8;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, C::kSmemBytes);
    if (e != cudaSuccess) return e;
    static const struct Fit {
        int n[kMaxKSplits + 1];
    } fit = [&] {
        Fit f{};
        for (int c = 2; c <= kMaxKSplits; ++c) f.n[c] = resident_clusters(kern, C::kSmemBytes, c, ctx.num_sms);
        return f;
    }();
    const int max_cl = fit.n[k_splits] - (k_splits == 3 ? kSpareTriples : 0);
    int bn = 32;
    while (bn < 128 && static_cast<long long>((N + bn - 1) / bn) * n_mgroups > max_cl) bn += kStep;
    const int n_ntiles = (N + bn - 1) / bn;
    const long long n_cl = static_cast<long long>(n_ntiles) * n_mgroups;
    const size_t need = static_cast<size_t>(n_cl) * k_splits * NB * bn * MT * kBM * sizeof(float);
    if (n_cl > max_cl || !ep_in.partial || need > partial_bytes) return cudaSuccess;
    CUtensorMap t0, t1;
    if constexpr (MT == 2) {
        // Four ranges of two M-tiles in whole tiles of 128 columns that fill the SMs: the kernel with
        // that width fixed, whose exchange keeps more loads in flight (d = I = 4096, 241 rows: Eq. 1
        // 59.6 against 63.0 us; d = 2048 would leave half of the SMs idle, 36.8 against 33.2).
        if (n_mgroups == 1 && k_splits == 4 && N % 128 == 0 && N / 128 * 4 >= kMinClusterCtas && N / 128 <= max_cl) {
            e = make_tmap(&t0, w0, K, N, kBK, 128);
            if (e == cudaSuccess) e = make_tmap(&t1, NB == 2 ? w1 : w0, K, N, kBK, 128);
            if (e != cudaSuccess) return e;
            *done = true;
            return run_gemm<EPI, MT, NB, 128, NB == 2 ? 3 : 4, 4>(ctx, tx, t0, t1, n_rows, K, N / 128, 1, ep_in, 4);
        }
    }
    e = make_tmap(&t0, w0, K, N, kBK, bn);
    if (e == cudaSuccess) e = make_tmap(&t1, NB == 2 ? w1 : w0, K, N, kBK, bn);
    if (e != cudaSuccess) return e;
    EpiParams ep = ep_in;
    ep.wait_ns = wait_limit_ns();
    ep.bn = bn;
    const int stages = C::kRingBytes / (MT * C::kABytes + NB * bn * kBK * 2);
    ep.stages = stages < kVarMaxStages ? stages : kVarMaxStages;
    *done = true;
    e = launch_pdl_cluster(kern, dim3(static_cast<unsigned>(k_splits * n_cl)), dim3(kThreads), C::kSmemBytes, ctx.stream,
                           k_splits, tx.whole, tx.last, t0, t1, n_rows, K, n_ntiles, n_mgroups, k_splits, n_mgroups == 1 ? 1 : 0, ep,
                           ctx.status);
    return e != cudaSuccess ? e : cudaGetLastError();
}

// h' = h + In W^T with In [n_rows, K] (tmap_in, boxes of kBK x kBM) and W [d, K]: the SwiGLU down
// projection (K = I, In = A) and the linear approximator (K = 2d, In = x). The residual row of
// stage-2 row r is the hidden state of its depth; the epilogue adds it in fp32 and rounds once to
// bf16.
static cudaError_t run_residual_gemm(const Ctx& ctx, const XMaps& ta, const void* W, int K, const void* hidden,
                              int n_rows, int d, int R, int M, int gamma, void* h_prime, float* partial,
                              size_t partial_bytes) {
    constexpr int BN = 128;
    const int m_tiles = (n_rows + kBM - 1) / kBM;
    const int n_mg = m_tiles == 1 ? 1 : (m_tiles + 1) / 2;
    const int bn_d = d % BN == 0 ? BN : 64;
    const int ks2 = choose_k_splits((d / bn_d) * n_mg, K / kBK, ctx.num_sms);
    CUtensorMap td;
    cudaError_t e = make_tmap(&td, W, K, d, kBK, bn_d);
    if (e != cudaSuccess) return e;
    EpiParams ed{};
    ed.out = static_cast<__nv_bfloat16*>(h_prime);
    ed.ld_out = d;
    ed.hidden = static_cast<const __nv_bfloat16*>(hidden);
    ed.R = R;
    ed.M = M;
    ed.gamma = gamma;
    ed.partial = partial;
    ed.n_cols = d;
    ed.n_total = d;
    // K split: clusters that exchange their partial sums. Two or more M-tiles
    // otherwise: CTA pairs on 256-column tiles, which stage a third less per SM and overlap their
    // epilogue with the next unit (1928 rows, K = 8192, d = 4096: 131 -> 108 us with the gather; gate/up
    // gains nothing from pairs: single CTAs already run N = 256 MMAs there), where their units fill
    // the SMs.
    bool done = false;
    if (ks2 > 1)
        e = m_tiles == 1 ? run_gemm_cluster<EPI_CDOWN, 1, 1>(ctx, ta, W, nullptr, d, n_rows, K, 1, ks2, ed, partial_bytes, &done)
                         : run_gemm_cluster<EPI_CDOWN, 2, 1>(ctx, ta, W, nullptr, d, n_rows, K, n_mg, ks2, ed, partial_bytes, &done);
    if (done || e != cudaSuccess) return e;
    // With a tail split pairs take over only where they chunk the same outputs, and widths are not
    // chosen, so that which outputs are summed in chunks, and so their bits, does not depend on the kernel
    // that runs: near ties of a tree follow the last bit of h'. Pairs for other tails would save 0.5 % of a
    // step (32 sequences, 3872 rows, d = 4096: 4132 against 4155 us), widths chosen all the same most where
    // they replace tiles of 64 (720 rows, d = 3776, I = 11072: 671 against 730 us).
    const int units = d / bn_d * n_mg;
    const int tail = ks2 == 1 && tail_chunks(ctx, units, ctx.num_sms, m_tiles == 1 ? 1 : 2, bn_d, K, partial_bytes)
                         ? units % ctx.num_sms : 0;
    const bool pair = m_tiles > 1 && d % 256 == 0 && d / 256 * n_mg * ks2 >= kMinPairs && tail % (2 * n_mg) == 0;
    if (ks2 == 1) {
        if (tail && !pair) {
            if (bn_d == BN)
                return m_tiles == 1 ? run_gemm<EPI_DOWN, 1, 1, BN, 6>(ctx, ta, td, td, n_rows, K, d / BN, 1, ed, 1, partial_bytes)
                                    : run_gemm<EPI_DOWN, 2, 1, BN, 4>(ctx, ta, td, td, n_rows, K, d / BN, n_mg, ed, 1, partial_bytes);
            return m_tiles == 1 ? run_gemm<EPI_DOWN, 1, 1, 64, 8>(ctx, ta, td, td, n_rows, K, d / 64, 1, ed, 1, partial_bytes)
                                : run_gemm<EPI_DOWN, 2, 1, 64, 5>(ctx, ta, td, td, n_rows, K, d / 64, n_mg, ed, 1, partial_bytes);
        }
        if (pair) return run_gemm<EPI_DOWN, 1, 1, 256, 7, 2>(ctx, ta, td, td, n_rows, K, d / 256, n_mg, ed, 1, partial_bytes);
        return m_tiles == 1 ? run_gemm_var<EPI_DOWN, 1, 1>(ctx, ta, W, nullptr, d, n_rows, K, 1, 1, ed)
                            : run_gemm_var<EPI_DOWN, 2, 1>(ctx, ta, W, nullptr, d, n_rows, K, n_mg, 1, ed);
    }
    if (pair)
        e = run_gemm<EPI_PARTIAL, 1, 1, 256, 7, 2>(ctx, ta, td, td, n_rows, K, d / 256, n_mg, ed, ks2);
    else
        e = m_tiles == 1 ? run_gemm_var<EPI_PARTIAL, 1, 1>(ctx, ta, W, nullptr, d, n_rows, K, 1, ks2, ed)
                         : run_gemm_var<EPI_PARTIAL, 2, 1>(ctx, ta, W, nullptr, d, n_rows, K, n_mg, ks2, ed);
    if (e != cudaSuccess) return e;
    return launch_down_reduce(ctx, partial, ks2, n_rows, d, static_cast<const __nv_bfloat16*>(hidden), R, M, gamma,
                              static_cast<__nv_bfloat16*>(h_prime));
}

cudaError_t launch_swiglu_tc(const Ctx& ctx, const void* X, int k_in, const void* w_gate, const void* w_up,
                             const void* w_down, const void* hidden, int n_rows, int d, int I, int R, int M,
                             int gamma, void* A, void* h_prime, float* partial, size_t partial_bytes) {
    if (n_rows <= 0) return cudaSuccess;
    constexpr int BN = 128;
    const int m_tiles = (n_rows + kBM - 1) / kBM;
    const int n_mg = m_tiles == 1 ? 1 : (m_tiles + 1) / 2;
    const int bn_gu = I % BN == 0 ? BN : 64;
    XMaps tx, ta;
    CUtensorMap tg, tu;
    cudaError_t e = make_xmaps(&tx, X, k_in, n_rows);
    if (e == cudaSuccess) e = make_tmap(&tg, w_gate, k_in, I, kBK, bn_gu);
    if (e == cudaSuccess) e = make_tmap(&tu, w_up, k_in, I, kBK, bn_gu);
    if (e == cudaSuccess) e = make_xmaps(&ta, A, I, n_rows);
    if (e != cudaSuccess) return e;

    // ---- gate/up: A = SiLU(X Wg^T) * (X Wu^T)
    const int ks1 = choose_k_splits((I / bn_gu) * n_mg, k_in / kBK, ctx.num_sms);
    EpiParams ep{};
    ep.out = static_cast<__nv_bfloat16*>(A);
    ep.ld_out = I;
    ep.partial = partial;
    ep.n_cols = 2 * I;
    ep.n_total = I;
    bool done = false;
    if (ks1 > 1)
        e = m_tiles == 1 ? run_gemm_cluster<EPI_CGATEUP, 1, 2>(ctx, tx, w_gate, w_up, I, n_rows, k_in, 1, ks1, ep, partial_bytes, &done)
                         : run_gemm_cluster<EPI_CGATEUP, 2, 2>(ctx, tx, w_gate, w_up, I, n_rows, k_in, n_mg, ks1, ep, partial_bytes, &done);
    const int units = I / bn_gu * n_mg;
    if (done || e != cudaSuccess) {
    } else if (ks1 == 1 && tail_chunks(ctx, units, ctx.num_sms, m_tiles == 1 ? 1 : 2, 2 * bn_gu, k_in, partial_bytes)) {
        // a tail split: fixed widths, as in the down projection
        if (bn_gu == BN)
            e = m_tiles == 1 ? run_gemm<EPI_GATEUP, 1, 2, BN, 4>(ctx, tx, tg, tu, n_rows, k_in, I / BN, 1, ep, 1, partial_bytes)
                             : run_gemm<EPI_GATEUP, 2, 2, BN, 3>(ctx, tx, tg, tu, n_rows, k_in, I / BN, n_mg, ep, 1, partial_bytes);
        else
            e = m_tiles == 1 ? run_gemm<EPI_GATEUP, 1, 2, 64, 6>(ctx, tx, tg, tu, n_rows, k_in, I / 64, 1, ep, 1, partial_bytes)
                             : run_gemm<EPI_GATEUP, 2, 2, 64, 4>(ctx, tx, tg, tu, n_rows, k_in, I / 64, n_mg, ep, 1, partial_bytes);
    } else if (m_tiles > 1 && bn_gu == BN && ks1 == 1 && I / BN * n_mg > ctx.num_sms) {
        e = run_gemm<EPI_GATEUP, 2, 2, BN, 3>(ctx, tx, tg, tu, n_rows, k_in, I / BN, n_mg, ep);
    } else if (ks1 == 1) {
        e = m_tiles == 1 ? run_gemm_var<EPI_GATEUP, 1, 2>(ctx, tx, w_gate, w_up, I, n_rows, k_in, 1, 1, ep)
                         : run_gemm_var<EPI_GATEUP, 2, 2>(ctx, tx, w_gate, w_up, I, n_rows, k_in, n_mg, 1, ep);
    } else {
        e = m_tiles == 1 ? run_gemm_var<EPI_PARTIAL, 1, 2>(ctx, tx, w_gate, w_up, I, n_rows, k_in, 1, ks1, ep)
                         : run_gemm_var<EPI_PARTIAL, 2, 2>(ctx, tx, w_gate, w_up, I, n_rows, k_in, n_mg, ks1, ep);
        if (e == cudaSuccess) e = launch_swiglu_reduce(ctx, partial, ks1, n_rows, I, static_cast<__nv_bfloat16*>(A));
    }
    if (e != cudaSuccess) return e;

    // ---- down + residual: h' = h + A Wd^T
    return run_residual_gemm(ctx, ta, w_down, I, hidden, n_rows, d, R, M, gamma, h_prime, partial, partial_bytes);
}

cudaError_t launch_linear_tc(const Ctx& ctx, const void* X, const void* w_lin, const void* hidden, int n_rows, int d,
                             int R, int M, int gamma, void* h_prime, float* partial, size_t partial_bytes) {
    if (n_rows <= 0) return cudaSuccess;
    XMaps tx;
    const cudaError_t e = make_xmaps(&tx, X, 2 * d, n_rows);
    if (e != cudaSuccess) return e;
    return run_residual_gemm(ctx, tx, w_lin, 2 * d, hidden, n_rows, d, R, M, gamma, h_prime, partial, partial_bytes);
}

}  // namespace tf
