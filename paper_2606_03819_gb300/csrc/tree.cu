// Stage-2 input rows (Eq. 1), Part 2 of Algorithm 1 (OPT-Tree best-first selection) and the
// verifier's tree-attention mask.
#include <math.h>

#include "common.cuh"

namespace tf {
namespace {

// ------------------------------------------------------------------------------------------
// Inputs of stage-2 row `row` (R rows per sequence).
//  TreeFlash (Eq. 1): row 0 refines depth 1 with the root token; row 1 + (i-2) M + m refines
//  depth i with candidate m of depth i-1.
//  Two previous tokens (the ablations' two-token variant): row 0 refines depth 1 with (x_t,
//  x_{t-1}) = root_tok[2 sq], root_tok[2 sq + 1]; rows 1..M depth 2 with (candidate m of depth 1,
//  x_t); row 1 + M + (i-3) M^2 + m1 M + m2 depth i >= 3 with (candidate m1 of depth i-1,
//  candidate m2 of depth i-2).
// ------------------------------------------------------------------------------------------
__device__ __forceinline__ int stage2_row_hidden(int row, int R, int gamma, int M, bool two_prev) {
    const int sq = row / R, r = row - sq * R;
    if (!two_prev) return sq * gamma + stage2_hidden_index(r, M);
    const int depth = r == 0 ? 1 : r <= M ? 2 : 3 + (r - 1 - M) / (M * M);
    return sq * gamma + depth - 1;
}
// The previous token (p[0]) and, with two_prev, the one before it (p[1]).
__device__ __forceinline__ void stage2_row_tokens(int row, int R, int gamma, int M, int K1, bool two_prev,
                                                  const int32_t* root_tok, const int32_t* top_ids, int* p) {
    const int sq = row / R, r = row - sq * R;
    const int32_t* top = top_ids + static_cast<size_t>(sq) * gamma * K1;   // [gamma][K1] of this sequence
    if (!two_prev) {
        p[0] = r == 0 ? root_tok[sq] : top[((r - 1) / M) * K1 + (r - 1) % M];
        return;
    }
    const int32_t* root = root_tok + 2 * static_cast<size_t>(sq);
    if (r == 0) {
        p[0] = root[0];
        p[1] = root[1];
    } else if (r <= M) {
        p[0] = top[r - 1];
        p[1] = root[0];
    } else {
        const int q = r - 1 - M, i = 3 + q / (M * M), w = q - (i - 3) * M * M;
        p[0] = top[(i - 2) * K1 + w / M];
        p[1] = top[(i - 3) * K1 + w % M];
    }
}

// ------------------------------------------------------------------------------------------
// x = [RMSNorm(h_{t+i}) * norm_h ; RMSNorm(Embd(prev)) * norm_e] for every stage-2 row
// (Eq. 1, h~ first), and with NE = 2 a third part RMSNorm(Embd(token before prev)) * norm_e.
// One CTA per row; the embedding rows are gathered by token id here, so the candidate
// embeddings are never materialised on their own. hres (NE = 2): the row's hidden state.
// ------------------------------------------------------------------------------------------
template <typename T, int NE>
__global__ void __launch_bounds__(256) gather_norm_kernel(const T* __restrict__ hidden, const T* __restrict__ embed,
                                                          const T* __restrict__ norm_h, const T* __restrict__ norm_e,
                                                          const int32_t* __restrict__ root_tok,
                                                          const int32_t* __restrict__ top_ids, int gamma, int M,
                                                          int K1, int R, int d, int V, float eps, T* __restrict__ X,
                                                          T* __restrict__ hres, int* status) {
    pdl_trigger();
    pdl_wait();
    // the approximator GEMMs' tail-split counters (after the status word) start each call at zero
    if (blockIdx.x == 0 && status)
        for (int i = threadIdx.x; i < kTailSems; i += blockDim.x) status[1 + i] = 0;
    __shared__ float red[1 + NE][8];
    const int row = blockIdx.x;
    const int hid = stage2_row_hidden(row, R, gamma, M, NE == 2);
    int tok[2] = {0, 0};
    stage2_row_tokens(row, R, gamma, M, K1, NE == 2, root_tok, top_ids, tok);
    const T* seg[1 + NE];
    seg[0] = hidden + static_cast<size_t>(hid) * d;
#pragma unroll
    for (int j = 0; j < NE; ++j) {
        if (tok[j] < 0 || tok[j] >= V) {
            if (threadIdx.x == 0) set_status(status, TF_DEV_BAD_TOKEN);
            tok[j] = 0;
        }
        seg[1 + j] = embed + static_cast<size_t>(tok[j]) * d;
    }
    float sumsq[1 + NE];
#pragma unroll
    for (int j = 0; j <= NE; ++j) sumsq[j] = 0.0f;
    for (int k = threadIdx.x; k < d; k += blockDim.x) {
#pragma unroll
        for (int j = 0; j <= NE; ++j) {
            const float a = to_f32(seg[j][k]);
            sumsq[j] = fmaf(a, a, sumsq[j]);
        }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1)
#pragma unroll
        for (int j = 0; j <= NE; ++j) sumsq[j] += __shfl_xor_sync(0xffffffffu, sumsq[j], o);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (lane == 0)
#pragma unroll
        for (int j = 0; j <= NE; ++j) red[j][warp] = sumsq[j];
    __syncthreads();
    if (threadIdx.x <= NE) {
        float a = 0.0f;
        for (int w = 0; w < (int)(blockDim.x >> 5); ++w) a += red[threadIdx.x][w];
        red[threadIdx.x][0] = rsqrtf(a / d + eps);
    }
    __syncthreads();
    T* xr = X + static_cast<size_t>(row) * (1 + NE) * d;
    for (int k = threadIdx.x; k < d; k += blockDim.x) {
        const float hk = to_f32(seg[0][k]);
        xr[k] = from_f32<T>(hk * red[0][0] * to_f32(norm_h[k]));
#pragma unroll
        for (int j = 1; j <= NE; ++j) xr[j * d + k] = from_f32<T>(to_f32(seg[j][k]) * red[j][0] * to_f32(norm_e[k]));
        if (NE == 2) hres[static_cast<size_t>(row) * d + k] = seg[0][k];
    }
}

// ------------------------------------------------------------------------------------------
// OPT-Tree selection (Algorithm 1 Part 2) by a queue, one warp per sequence. It holds one entry per
// open child list: (path score, depth, parent node) packed into one 64-bit key, plus the list
// row, the rank in the list, the parent's score and the token. Popping rank k of a list
// replaces the entry by rank k+1 of the same list (its next sibling), and an expandable popped
// node adds rank 0 of its own child list. Every list is sorted (value desc, id asc), so this
// pops exactly what pushing whole distributions would, with at most B + 1 live entries.
//
// Queue order: larger score, then smaller depth, then smaller parent index. Two live entries
// never share (depth, parent): each node opens at most one child list. So the key
//   float_key(score) << 32 | (127 - depth) << 24 | (0xFFFFFF - parent)
// is unique and its integer maximum is the next pop. Each lane keeps the best key of its own
// slots (j = lane mod 32) and rescans only when one of them changed; a pop is two warp max
// reductions and a ballot.
// ------------------------------------------------------------------------------------------
struct TreeArgs {
    int gamma, M, K1, K2, B, V, mode, R;
    int two_prev;      // child lists by the ablations' two-token rule; root_tok holds 2 tokens per sequence
    const int32_t* root_tok;
    const int32_t* top_ids;
    const float* top_logp;
    const int32_t* child_ids;
    const float* child_logp;
    int32_t* node_tok;
    int32_t* node_parent;
    int32_t* node_depth;
    float* node_score;
    int32_t* dev_status;
    // optional, with B + 1 <= kFusedMaskMaxNodes: the builder also writes the verification mask and
    // position ids (tf_tree_mask's outputs) from the tree it holds in shared memory
    const int32_t* root_pos;
    uint8_t* mask;
    int32_t* pos_ids;
    // optional: the workspace status word, final once the builder runs (every earlier kernel of
    // the step has finished). Each dev_status[s] then becomes seq_bits | w | w << 16 with w that
    // word, so that a caller that reads dev_status alone also learns w by itself.
    const int32_t* ws_status;
};

// The status word of sequence s: its own bits, and with a.ws_status the folded workspace word.
__device__ __forceinline__ int32_t sequence_status(const TreeArgs& a, int flags) {
    if (!a.ws_status) return flags;
    const int32_t w = *a.ws_status;
    return flags | w | (w << 16);
}

// Index m of `tok` among the M <= 64 stage-1 candidates of depth `dep` (the M-ary rule of
// Algorithm 1 Part 2: the node is expandable iff its token is one of them), or -1; two warp
// ballots, so every lane of the warp must call it (active = false gives -1).
__device__ __forceinline__ int mary_index(const int* topm, int dep, int M, int tok, int lane, bool active) {
    const int* t = topm + (dep - 1) * M;
    const bool h0 = active && lane < M && t[lane] == tok;
    const bool h1 = active && lane + 32 < M && t[lane + 32] == tok;
    const unsigned b0 = __ballot_sync(0xffffffffu, h0), b1 = __ballot_sync(0xffffffffu, h1);
    return b0 ? __ffs(b0) - 1 : (b1 ? 32 + __ffs(b1) - 1 : -1);
}

// Child list of a popped node under the two-previous-token rule: the node (depth dep, candidate
// m of its depth, or m < 0 outside the M-ary tree) gets the row conditioned on its own token and
// its parent's, 1 + m for dep = 1 and 1 + M + (dep - 2) M^2 + m M + mp for dep >= 2, mp the
// parent's candidate index at depth dep - 1 (the parent was expanded, so it has one). o_tok holds
// the tokens of the nodes placed so far, written by lane 0, which alone reads the parent's token.
// Every lane must call it (ballots); returns -1 for a leaf.
__device__ __forceinline__ int child_row_2prev(const int* topm, const int* o_tok, int M, int dep, int m, int par,
                                               int lane) {
    const bool deep = m >= 0 && dep >= 2;
    int ptok = 0;
    if (lane == 0 && deep) ptok = o_tok[par];
    ptok = __shfl_sync(0xffffffffu, ptok, 0);
    const int mp = mary_index(topm, deep ? dep - 1 : 1, M, ptok, lane, deep);
    if (m < 0) return -1;
    if (dep == 1) return 1 + m;
    return mp >= 0 ? 1 + M + (dep - 2) * M * M + m * M + mp : -1;
}

__device__ __forceinline__ unsigned long long queue_key(float score, int depth, int parent) {
    return (static_cast<unsigned long long>(float_key(score)) << 32) |
           (static_cast<unsigned long long>(127 - depth) << 24) | static_cast<unsigned long long>(0xFFFFFF - parent);
}


// Shared-memory bytes of the general builder: queue, node arrays, stage-1 top-M, mask bits.
__host__ __device__ inline size_t tree_mask_words(int n) { return static_cast<size_t>(n) * ((n + 31) / 32); }
__host__ __device__ inline size_t tree_smem_fixed(int B, int gamma, int M, bool with_mask) {
    return static_cast<size_t>(B + 2) * (8 + 4 * 4) + static_cast<size_t>(B + 1) * 4 * 4 +
           static_cast<size_t>(gamma) * M * 4 + 16 + (with_mask ? tree_mask_words(B + 1) * 4 + 16 : 0);
}
constexpr size_t kTreeSmemLimit = 200 * 1024;

// The child lists of one sequence, in global memory.
struct ListView {
    const int32_t* ids;     // [rows][stride]
    const float* lps;
    int stride;
    __device__ __forceinline__ int tok(int row, int rank) const { return ids[static_cast<size_t>(row) * stride + rank]; }
    __device__ __forceinline__ float lp(int row, int rank) const { return lps[static_cast<size_t>(row) * stride + rank]; }
};
__device__ __forceinline__ ListView sequence_lists(const TreeArgs& a, int s) {
    if (a.mode == TF_MODE_AR)
        return ListView{a.child_ids + static_cast<size_t>(s) * a.R * a.K2, a.child_logp + static_cast<size_t>(s) * a.R * a.K2, a.K2};
    return ListView{a.top_ids + static_cast<size_t>(s) * a.gamma * a.K1, a.top_logp + static_cast<size_t>(s) * a.gamma * a.K1, a.K1};
}

// Shared memory of the general builder: the queue, the output nodes and the stage-1 top-M.
struct TreeSmem {
    unsigned long long* qkey;
    float* qps;
    int *qrow, *qrank, *qtok;
    int *o_tok, *o_par, *o_dep;
    float* o_score;
    int* topm;        // [gamma, M]
    uint32_t* anc;    // with the fused mask: ancestor-or-self bits of B + 1 rows
};
__device__ __forceinline__ TreeSmem tree_smem(uint8_t* base, const TreeArgs& a) {
    TreeSmem t;
    const int cap = a.B + 2, n_out = a.B + 1;
    t.qkey = reinterpret_cast<unsigned long long*>(base);
    t.qps = reinterpret_cast<float*>(t.qkey + cap);
    t.qrow = reinterpret_cast<int*>(t.qps + cap);
    t.qrank = t.qrow + cap;
    t.qtok = t.qrank + cap;
    t.o_tok = t.qtok + cap;
    t.o_par = t.o_tok + n_out;
    t.o_dep = t.o_par + n_out;
    t.o_score = reinterpret_cast<float*>(t.o_dep + n_out);
    t.topm = reinterpret_cast<int*>(t.o_score + n_out);
    t.anc = reinterpret_cast<uint32_t*>(t.topm + a.gamma * a.M);
    return t;
}

// Nodes from shared memory to the outputs.
__device__ __forceinline__ void write_nodes(const TreeArgs& a, int s, const TreeSmem& t) {
    const int n_out = a.B + 1;
    for (int i = threadIdx.x; i < n_out; i += static_cast<int>(blockDim.x)) {
        const size_t o = static_cast<size_t>(s) * n_out + i;
        a.node_tok[o] = t.o_tok[i];
        a.node_parent[o] = t.o_par[i];
        a.node_depth[o] = t.o_dep[i];
        a.node_score[o] = t.o_score[i];
    }
}

// Rows r0 .. r1-1 of one sequence's tree-attention mask and their position ids. mask[i][j] = 1
// iff node j is node i or one of its ancestors; pos = root_pos + depth. Each node walks its own
// parent chain (at most kMaxGamma links) and sets the bits of its row, so no thread waits for
// another level. A node is present iff every link of its chain goes to a smaller index exactly
// one level up and the chain ends at the root (node 0, depth 0); absent nodes (missing from an
// underfull tree, or behind a broken link) get an empty row and column and pos -1.
// par, dep: the tree's n parents and depths (shared memory); bits: a bit per entry of the rows, without
// padding between rows, so that any four entries are one shift of two words (with padded rows every
// warp went through a path for words that run into the next row as well: 65 nodes 1.8 -> 1.4 us); mask_s [n][n] and pos_s [n]: this sequence's outputs.
__device__ __forceinline__ void mask_rows(int n, const int* par, const int* dep, int root_pos, int r0, int r1,
                                          uint32_t* bits, uint8_t* mask_s, int32_t* pos_s) {
    const int total = (r1 - r0) * n;
    for (int w = threadIdx.x; w < (total + 31) / 32; w += blockDim.x) bits[w] = 0u;
    __syncthreads();
    for (int i = r0 + static_cast<int>(threadIdx.x); i < r1; i += blockDim.x) {
        const int row = (i - r0) * n;
        bool ok = true;
        int j = i, dj = dep[i], links = 0;
        for (; ok && j != 0; ++links) {
            const int p = par[j];
            const bool link = p >= 0 && p < j;
            const int dp = link ? dep[p] : -1;
            ok = links < kMaxGamma && dj >= 1 && dj <= kMaxGamma && link && dp == dj - 1;
            atomicOr(&bits[(row + j) >> 5], 1u << ((row + j) & 31));   // (no result: the walk does not wait)
            j = p;
            dj = dp;
        }
        ok = ok && dep[0] == 0;
        if (ok) {
            atomicOr(&bits[row >> 5], 1u << (row & 31));   // the root
        } else {
            for (j = i; links > 0; --links) {              // absent: empty row
                atomicAnd(&bits[(row + j) >> 5], ~(1u << ((row + j) & 31)));
                j = par[j];
            }
        }
        pos_s[i] = ok ? root_pos + dep[i] : -1;
    }
    __syncthreads();
    // The rows are contiguous bytes: aligned words of four entries, single bytes before the first and
    // after the last.
    uint8_t* out = mask_s + static_cast<size_t>(r0) * n;
    const int head = min(total, static_cast<int>(-reinterpret_cast<intptr_t>(out) & 3));
    const int words = (total - head) / 4;
    for (int w = threadIdx.x; w < words; w += blockDim.x) {
        const int at = head + 4 * w, sh = at & 31;
        const uint32_t x = __funnelshift_r(bits[at >> 5], sh > 28 ? bits[(at >> 5) + 1] : 0u, sh);
        *reinterpret_cast<uint32_t*>(out + at) = (x & 1u) | ((x & 2u) << 7) | ((x & 4u) << 14) | ((x & 8u) << 21);
    }
    for (int k = threadIdx.x; k < total - 4 * words; k += blockDim.x) {
        const int at = k < head ? k : 4 * words + k;
        out[at] = static_cast<uint8_t>((bits[at >> 5] >> (at & 31)) & 1u);
    }
}

// The fused mask of a builder CTA, once its tree is complete in shared memory.
__device__ __forceinline__ void fused_mask(const TreeArgs& a, int s, const TreeSmem& t) {
    if (!a.mask) return;
    const int n = a.B + 1;
    mask_rows(n, t.o_par, t.o_dep, a.root_pos[s], 0, n, t.anc, a.mask + static_cast<size_t>(s) * n * n,
              a.pos_ids + static_cast<size_t>(s) * n);
}

// General builder (any lists): the queue in shared memory, popped by the CTA's first warp. Every
// thread of the CTA calls it; on return the nodes are in shared memory and the status is written.
__device__ void build_tree_queue(const TreeArgs& a, int s, const TreeSmem& t, const ListView& lv) {
    unsigned long long* qkey = t.qkey;
    float* qps = t.qps;
    int* qrow = t.qrow;
    int* qrank = t.qrank;
    int* qtok = t.qtok;
    int* o_tok = t.o_tok;
    int* o_par = t.o_par;
    int* o_dep = t.o_dep;
    float* o_score = t.o_score;
    int* topm = t.topm;
    const int n_out = a.B + 1;
    const int tid = threadIdx.x;
    const bool ar = a.mode == TF_MODE_AR;

    if (tid < 32) {
        const int lane = tid;
        constexpr unsigned kFull = 0xffffffffu;
        int flags = 0;
        const int root = a.root_tok[a.two_prev ? 2 * s : s];
        if (root < 0 || root >= a.V) flags |= TF_DEV_BAD_TOKEN;
        const int list_len = a.K2;
        if (lane == 0) {
            o_tok[0] = root;
            o_par[0] = -1;
            o_dep[0] = 0;
            o_score[0] = 0.0f;
            qkey[0] = queue_key(lv.lp(0, 0), 1, 0);
            qps[0] = 0.0f;
            qrow[0] = 0;
            qrank[0] = 0;
            qtok[0] = lv.tok(0, 0);
        }
        int n_e = 1;
        int count = 1;
        __syncwarp();
        unsigned long long lbest = 0ull;
        int lidx = -1;
        auto rescan = [&]() {
            lbest = 0ull;
            lidx = -1;
            for (int j = lane; j < n_e; j += 32) {
                const unsigned long long k = qkey[j];
                if (k > lbest) {
                    lbest = k;
                    lidx = j;
                }
            }
        };
        rescan();
        while (count < n_out && n_e > 0) {
            const uint32_t hi = static_cast<uint32_t>(lbest >> 32), lo = static_cast<uint32_t>(lbest);
            const uint32_t mhi = __reduce_max_sync(kFull, hi);
            const uint32_t mlo = __reduce_max_sync(kFull, hi == mhi ? lo : 0u);
            const unsigned win = __ballot_sync(kFull, lbest != 0ull && hi == mhi && lo == mlo);
            if (win == 0u) break;
            const int best = __shfl_sync(kFull, lidx, __ffs(win) - 1);
            const float sc = key_float(mhi);
            const int dep = 127 - static_cast<int>(mlo >> 24);
            const int par = 0xFFFFFF - static_cast<int>(mlo & 0xFFFFFFu);
            const int row = qrow[best], rank = qrank[best], tok = qtok[best];
            const float psc = qps[best];
            __syncwarp();
            const int node = count++;
            if (tok < 0 || tok >= a.V) flags |= TF_DEV_BAD_TOKEN;
            if (!isfinite(sc)) flags |= TF_DEV_NONFINITE;
            // expandable? (depth cap; M-ary rule)
            int crow = -1;
            if (dep < a.gamma) {
                if (a.mode == TF_MODE_MARGINAL) {
                    crow = dep;
                } else {
                    const int m = mary_index(topm, dep, a.M, tok, lane, true);
                    if (m >= 0) crow = ar ? 1 + (dep - 1) * a.M + m : dep;
                    if (ar && a.two_prev) crow = child_row_2prev(topm, o_tok, a.M, dep, m, par, lane);
                }
            }
            const bool sibling = rank + 1 < list_len;
            const int last = n_e - 1;
            if (lane == 0) {
                o_tok[node] = tok;
                o_par[node] = par;
                o_dep[node] = dep;
                o_score[node] = sc;
                if (sibling) {                   // next sibling of the popped entry
                    qrank[best] = rank + 1;
                    qtok[best] = lv.tok(row, rank + 1);
                    qkey[best] = queue_key(psc + lv.lp(row, rank + 1), dep, par);
                } else if (best != last) {       // list exhausted: move the last entry here
                    qkey[best] = qkey[last];
                    qps[best] = qps[last];
                    qrow[best] = qrow[last];
                    qrank[best] = qrank[last];
                    qtok[best] = qtok[last];
                }
            }
            if (!sibling) --n_e;
            int fresh = -1;
            if (crow >= 0) {
                fresh = n_e;
                if (lane == 0) {
                    qkey[n_e] = queue_key(sc + lv.lp(crow, 0), dep + 1, node);
                    qps[n_e] = sc;
                    qrow[n_e] = crow;
                    qrank[n_e] = 0;
                    qtok[n_e] = lv.tok(crow, 0);
                }
                ++n_e;
            }
            __syncwarp();
            if (lane == (best & 31) || (!sibling && lane == (last & 31)) || (fresh >= 0 && lane == (fresh & 31)))
                rescan();
        }
        if (count < n_out) flags |= TF_DEV_UNDERFULL;
        for (int i = count + lane; i < n_out; i += 32) {
            o_tok[i] = -1;
            o_par[i] = -1;
            o_dep[i] = -1;
            o_score[i] = -INFINITY;
        }
        if (lane == 0) a.dev_status[s] = sequence_status(a, flags);
    }
    __syncthreads();
}

// ------------------------------------------------------------------------------------------
// Builder with a sorted queue, for B <= 64 with every reachable list entry staged. The same pops, tie
// rules and results as build_tree_queue. After t pops only the B - t best live entries can still be popped (each
// needs every better entry popped first), and at most t + 1 entries are live (a pop replaces its
// entry by the next sibling and adds at most the node's first child), so at most
// min(t + 1, B - t) <= 32 entries matter: lane i of one warp holds the i-th best. A pop takes
// lane 0's entry, tests its token against the stage-1 candidates of its depth with a ballot
// (the M-ary rule), and places its two successors (next sibling, first child) with two ballots
// over the remaining keys; every lane then takes its new entry from itself or a neighbour by
// shuffle. There is no warp-wide max and no divergent branch. The queue carries keys and list
// entries only (a sibling's parent score is the placed parent's o_score); a pop costs about
// 250 ns on GB300, a chain of about a hundred dependent single-warp instructions.
// ------------------------------------------------------------------------------------------
constexpr int kFastThreads = 512;
constexpr int kSortedQueueMax = 64;
// Shared-memory bytes of build_tree_fast_kernel: nodes, candidates, mask bits and the staged
// lists (token and log-probability of every entry).
__host__ __device__ inline size_t fast_tree_smem(int B, int gamma, int M, int rows, int sw, bool with_mask) {
    const size_t n = static_cast<size_t>(B) + 1;
    size_t bytes = n * 20 + static_cast<size_t>(gamma) * M * 4;
    bytes = (bytes + 15) & ~static_cast<size_t>(15);
    if (with_mask) bytes += (tree_mask_words(static_cast<int>(n)) * 4 + 15) & ~static_cast<size_t>(15);
    return bytes + static_cast<size_t>(rows) * sw * 8 + 16;
}

__device__ __forceinline__ bool key_gt(uint32_t ahi, uint32_t alo, uint32_t bhi, uint32_t blo) {
    return ahi > bhi || (ahi == bhi && alo > blo);
}

template <bool TWO>   // the two-previous-token rule
__global__ void __launch_bounds__(kFastThreads) build_tree_fast_kernel(TreeArgs a, int sw) {
    pdl_trigger();
    pdl_wait();
    extern __shared__ __align__(16) uint8_t smem_raw[];
    constexpr unsigned kFull = 0xffffffffu;
    const int n_out = a.B + 1, s = blockIdx.x, tid = threadIdx.x;
    const int T = blockDim.x;
    const bool ar = a.mode == TF_MODE_AR, mary = a.mode != TF_MODE_MARGINAL;
    const int rows_l = ar ? a.R : a.gamma;
    const int stride = ar ? a.K2 : a.K1;
    // every array is carved by a byte offset into smem_raw, so that all accesses stay
    // shared-memory accesses
    int* o_tok = reinterpret_cast<int*>(smem_raw);
    int* o_par = o_tok + n_out;
    int* o_dep = o_par + n_out;
    float* o_score = reinterpret_cast<float*>(o_dep + n_out);
    int* o_m = reinterpret_cast<int*>(o_score + n_out);   // candidate index (two-token rule)
    int* topm = o_m + n_out;
    size_t off = (static_cast<size_t>(reinterpret_cast<uint8_t*>(topm + a.gamma * a.M) - smem_raw) + 15) & ~static_cast<size_t>(15);
    uint32_t* anc = reinterpret_cast<uint32_t*>(smem_raw + off);
    if (a.mask) off += (tree_mask_words(n_out) * 4 + 15) & ~static_cast<size_t>(15);
    const int n = rows_l * sw;
    int* l_tok = reinterpret_cast<int*>(smem_raw + off);
    float* l_lp = reinterpret_cast<float*>(l_tok + n);

    // ---- the lists and the stage-1 candidates
    const int32_t* g_ids = ar ? a.child_ids + static_cast<size_t>(s) * a.R * a.K2
                              : a.top_ids + static_cast<size_t>(s) * a.gamma * a.K1;
    const float* g_lp = ar ? a.child_logp + static_cast<size_t>(s) * a.R * a.K2
                           : a.top_logp + static_cast<size_t>(s) * a.gamma * a.K1;
    const bool vec = sw == stride && (sw & 3) == 0 &&
                     ((reinterpret_cast<uintptr_t>(g_ids) | reinterpret_cast<uintptr_t>(g_lp)) & 15) == 0;
    if (vec) {
        const int n4 = n >> 2;
        const int4* gi = reinterpret_cast<const int4*>(g_ids);
        const float4* gl = reinterpret_cast<const float4*>(g_lp);
        for (int base = tid; base < n4; base += 8 * T) {
            int4 vi[8];
            float4 vl[8];
#pragma unroll
            for (int u = 0; u < 8; ++u)
                if (base + u * T < n4) {
                    vi[u] = gi[base + u * T];
                    vl[u] = gl[base + u * T];
                }
#pragma unroll
            for (int u = 0; u < 8; ++u)
                if (base + u * T < n4) {
                    reinterpret_cast<int4*>(l_tok)[base + u * T] = vi[u];
                    reinterpret_cast<float4*>(l_lp)[base + u * T] = vl[u];
                }
        }
    } else {
        for (int i = tid; i < n; i += T) {
            const int r = i / sw;
            const size_t g = static_cast<size_t>(r) * stride + (i - r * sw);
            l_tok[i] = g_ids[g];
            l_lp[i] = g_lp[g];
        }
    }
    for (int i = tid; i < a.gamma * a.M; i += T)
        topm[i] = a.top_ids[(static_cast<size_t>(s) * a.gamma + i / a.M) * a.K1 + i % a.M];
    __syncthreads();
    // ---- the pops (one warp): lane i holds the i-th best live entry, as its key (score, depth,
    // parent) and its list entry (row << 10 | rank); key 0 marks an empty lane. The parent's
    // score, which a sibling's score needs, is read from the placed nodes (o_score[parent]).
    if (tid < 32) {
        const int lane = tid;
        const int list_len = a.K2 < sw ? a.K2 : sw;   // staged ranks; a pop never reaches rank sw
        int flags = 0;
        const int root = a.root_tok[TWO ? 2 * s : s];
        if (root < 0 || root >= a.V) flags |= TF_DEV_BAD_TOKEN;
        uint32_t khi = 0u, klo = 0u;
        int rr = 0;
        if (lane == 0) {
            const unsigned long long k0 = queue_key(l_lp[0], 1, 0);
            khi = static_cast<uint32_t>(k0 >> 32);
            klo = static_cast<uint32_t>(k0);
            o_tok[0] = root;
            o_par[0] = -1;
            o_dep[0] = 0;
            o_score[0] = 0.0f;
        }
        int count = 1;    // nodes placed
        while (count < n_out) {
            __syncwarp();                              // lane 0's node writes, for o_score below
            // the head: lane 0's entry
            const uint32_t hhi = __shfl_sync(kFull, khi, 0);
            if (hhi == 0u) break;                      // queue empty
            const uint32_t hlo = __shfl_sync(kFull, klo, 0);
            const int hrr = __shfl_sync(kFull, rr, 0);
            // the rest shifted by one: lane i sees entries i + 1 (next) and i - 1 (prev)
            uint32_t nhi = __shfl_down_sync(kFull, khi, 1), nlo = __shfl_down_sync(kFull, klo, 1);
            const int nrr = __shfl_down_sync(kFull, rr, 1);
            if (lane == 31) nhi = nlo = 0u;
            const uint32_t phi = __shfl_up_sync(kFull, khi, 1), plo = __shfl_up_sync(kFull, klo, 1);
            const int prr = __shfl_up_sync(kFull, rr, 1);
            // the popped node
            const int row = hrr >> 10, rank = hrr & 1023, idx = row * sw + rank;
            const int dep = 127 - static_cast<int>(hlo >> 24);
            const int par = 0xFFFFFF - static_cast<int>(hlo & 0xFFFFFFu);
            const float sc = key_float(hhi);
            const int node = count++;
            const int tok = l_tok[idx];
            const float hpsc = o_score[par];           // the parent's score
            // its children: none at the depth cap; DDTree: the next depth's marginal row;
            // otherwise only for a stage-1 candidate m of its depth (Algorithm 1 Part 2), found by
            // ballots over the depth's candidates (the first equal one counts): stage-2 row
            // 1 + (dep - 1) M + m, or the next marginal row
            const int* cand = topm + (dep < a.gamma && mary ? (dep - 1) * a.M : 0);
            const int c0 = lane < a.M ? cand[lane] : -1;
            const unsigned b0 = __ballot_sync(kFull, lane < a.M && c0 == tok);
            int m = b0 ? __ffs(b0) - 1 : -1;
            if (a.M > 32) {                            // (the same for every lane)
                const int c1 = lane + 32 < a.M ? cand[lane + 32] : -1;
                const unsigned b1 = __ballot_sync(kFull, lane + 32 < a.M && c1 == tok);
                m = b0 ? m : b1 ? 32 + __ffs(b1) - 1 : -1;
            }
            int crow = dep >= a.gamma ? -1 : !mary ? dep : m < 0 ? -1 : ar ? 1 + (dep - 1) * a.M + m : dep;
            // two-token rule: the row of (this node's candidate, its parent's); the parent was expanded,
            // so it has one
            if (TWO && crow >= 0 && dep >= 2) crow = 1 + a.M + (dep - 2) * a.M * a.M + m * a.M + o_m[par];
            const bool sib_ok = rank + 1 < list_len;
            const float slp = l_lp[sib_ok ? idx + 1 : idx];
            const bool ch_ok = crow >= 0 && node + 1 < n_out;   // nothing is popped after the last node
            const float clp = l_lp[ch_ok ? crow * sw : 0];
            if (lane == 0) {
                if (tok < 0 || tok >= a.V) flags |= TF_DEV_BAD_TOKEN;
                if (!isfinite(sc)) flags |= TF_DEV_NONFINITE;
                o_tok[node] = tok;
                o_par[node] = par;
                o_dep[node] = dep;
                o_score[node] = sc;
                if (TWO) o_m[node] = m;
            }
            // its successors, A before B in queue order (0 = none): the next sibling shares the
            // head's depth and parent (the low word of its key), the child is one level deeper
            // with this node as parent
            const uint32_t shi = sib_ok ? float_key(hpsc + slp) : 0u, slo = sib_ok ? hlo : 0u;
            const uint32_t chi = ch_ok ? float_key(sc + clp) : 0u;
            const uint32_t clo = ch_ok ? (static_cast<uint32_t>(126 - dep) << 24) | static_cast<uint32_t>(0xFFFFFF - node) : 0u;
            const bool s_first = key_gt(shi, slo, chi, clo);
            const uint32_t ahi = s_first ? shi : chi, alo = s_first ? slo : clo;
            const uint32_t bhi = s_first ? chi : shi, blo = s_first ? clo : slo;
            const int arr = s_first ? hrr + 1 : crow << 10, brr = s_first ? crow << 10 : hrr + 1;
            // their places among the remaining entries (sorted, so the larger keys are a prefix)
            const int pA = __popc(__ballot_sync(kFull, key_gt(nhi, nlo, ahi, alo)));
            const int pB = __popc(__ballot_sync(kFull, key_gt(nhi, nlo, bhi, blo)));
            // new entry i: rest[i] before A, A, rest[i - 1] up to B, B, rest[i - 2] after it
            const int j = lane;
            const bool takeA = j == pA, takeB = j == pB + 1;
            const bool fromN = j < pA, fromO = j > pA && j <= pB;
            khi = takeA ? ahi : takeB ? bhi : fromN ? nhi : fromO ? khi : phi;
            klo = takeA ? alo : takeB ? blo : fromN ? nlo : fromO ? klo : plo;
            rr = takeA ? arr : takeB ? brr : fromN ? nrr : fromO ? rr : prr;
        }
        flags = static_cast<int>(__reduce_or_sync(kFull, static_cast<unsigned>(flags)));
        if (count < n_out) flags |= TF_DEV_UNDERFULL;
        for (int i = count + lane; i < n_out; i += 32) {
            o_tok[i] = -1;
            o_par[i] = -1;
            o_dep[i] = -1;
            o_score[i] = -INFINITY;
        }
        if (lane == 0) a.dev_status[s] = sequence_status(a, flags);
    }
    __syncthreads();
    for (int i = tid; i < n_out; i += T) {
        const size_t o = static_cast<size_t>(s) * n_out + i;
        a.node_tok[o] = o_tok[i];
        a.node_parent[o] = o_par[i];
        a.node_depth[o] = o_dep[i];
        a.node_score[o] = o_score[i];
    }
    if (a.mask)
        mask_rows(n_out, o_par, o_dep, a.root_pos[s], 0, n_out, anc, a.mask + static_cast<size_t>(s) * n_out * n_out,
                  a.pos_ids + static_cast<size_t>(s) * n_out);
}

// ------------------------------------------------------------------------------------------
// Builder by levels, for large budgets and for few depths. A pop sequence is a chain: with the queue in shared
// memory 512 pops took 343 us on GB300, about 0.65 us each on one warp (33 us this way). But the B popped nodes are simply
// the B first of all nodes in the order (score, smaller depth, earlier parent, earlier list entry),
// as long as no node outscores its parent or its list predecessor (log-probabilities <= 0, lists
// sorted): then the first B nodes contain every ancestor and predecessor of each of them. So the
// CTA grows all of them level by level, a warp per (parent, 32 list entries), and keeps only nodes
// that can still be among the first B: theta, a lower bound of the B-th best score so far, rises
// after each pass. The survivors (a few more than B) are sorted once.
// What bounds it is instructions on a few warps and block barriers: per pass about 1.4 us, of which a
// third waits for the lists in L2. So up to kLvExact nodes the B-th best and the order come from
// counting, several threads per node (one phase instead of the five of a histogram: 1.3 -> 0.7 us,
// the order 2.2 -> 1.5 us), more nodes are ordered by buckets and counting within a bucket (513 nodes
// 6 -> 3.5 us; a bitonic sort has 55 phases), and the root token and position, which may lie in host
// memory, are read at the start (B = 512 with the mask 44.9 -> 37.5 us, B = 1023 76 -> 63).
//  - Two nodes of equal score and depth under different parents are ordered by their parents' places
//    in the order, known once shallower levels are: the few such ties are resolved after the sort.
//  - A score of -inf ends its list (as padding of short lists does). A list entry above its predecessor or
//    its parent, NaN, fewer finite nodes than B where lists ended early, more than kLvTies ties near
//    the tree, or more nodes at theta than there is room for send the sequence to the queue
//    (build_tree_queue) instead: the same results, at the queue's speed on top of the levels done by then.
// ------------------------------------------------------------------------------------------
constexpr int kLvThreads = 512;
constexpr int kLvWarps = kLvThreads / 32;
constexpr int kLvCap = 4096;       // nodes held at once
constexpr int kLvBins = 2 * kLvThreads;
constexpr int kLvSort = 2048;      // nodes that can be sorted
constexpr int kLvExact = 128;      // up to this many nodes: order statistics by counting
constexpr int kLvTies = 32;        // ties resolved in place, and the longest run of equal nodes
// The lowest score that theta's histogram covers: entries far below (lists padded with a type's lowest
// value) would leave one bin for all others.
constexpr float kLvFloor = -1024.0f;

// Nodes to expand: the node (kNoNode: dropped), the next 32-entry chunk of its child list, the list.
struct ActList {
    int* row;
    uint16_t* node;
    uint8_t* chunk;
};
struct LevelSmem {
    unsigned long long* key;   // [kLvSort]
    float* score;          // [kLvCap]; node 0 is the root
    int* tok;
    int* hist;             // [kLvBins]
    uint16_t *par, *rank;
    uint16_t* place;       // new index in a compaction; 1 + place in the order at the end
    uint8_t* dep;
    int8_t* m;             // candidate index of an expandable node (two-token rule)
    ActList act[3];        // [kLvCap] each: this pass, the lists that go on, the next level
    int* topm;             // [gamma * M]
};
constexpr uint16_t kNoNode = 0xffff;
constexpr size_t kLvFixedBytes = kLvCap * (4 + 4 + 2 + 2 + 2 + 1 + 1 + 3 * 7) + kLvSort * 8 + kLvBins * 4;
__host__ __device__ inline size_t level_smem_bytes(int B, int gamma, int M, bool with_mask) {
    const size_t mine = kLvFixedBytes + static_cast<size_t>(gamma) * M * 4;
    const size_t queue = tree_smem_fixed(B, gamma, M, with_mask);
    return mine > queue ? mine : queue;
}
__device__ __forceinline__ LevelSmem level_smem(uint8_t* p) {
    LevelSmem t;
    auto take = [&](size_t bytes) {
        uint8_t* q = p;
        p += bytes;
        return q;
    };
    t.key = reinterpret_cast<unsigned long long*>(take(kLvSort * 8));
    t.score = reinterpret_cast<float*>(take(kLvCap * 4));
    t.tok = reinterpret_cast<int*>(take(kLvCap * 4));
    t.hist = reinterpret_cast<int*>(take(kLvBins * 4));
    for (ActList& l : t.act) l.row = reinterpret_cast<int*>(take(kLvCap * 4));
    t.par = reinterpret_cast<uint16_t*>(take(kLvCap * 2));
    t.rank = reinterpret_cast<uint16_t*>(take(kLvCap * 2));
    t.place = reinterpret_cast<uint16_t*>(take(kLvCap * 2));
    for (ActList& l : t.act) l.node = reinterpret_cast<uint16_t*>(take(kLvCap * 2));
    for (ActList& l : t.act) l.chunk = take(kLvCap);
    t.dep = take(kLvCap);
    t.m = reinterpret_cast<int8_t*>(take(kLvCap));
    t.topm = reinterpret_cast<int*>(p);
    return t;
}

// Sort key of node idx: larger score, smaller depth, smaller list rank, then index (unique).
__device__ __forceinline__ unsigned long long level_key(float score, int dep, int rank, int idx) {
    return (static_cast<unsigned long long>(float_key(score)) << 32) | (static_cast<unsigned>(127 - dep) << 24) |
           (static_cast<unsigned>(0xfff - rank) << 12) | static_cast<unsigned>(idx);
}
static_assert(kLvCap <= 1 << 12 && kMaxK <= 1 << 12 && kMaxGamma <= 127, "fields of level_key");

// What builders by levels have done on this device: trees left to the queue, compactions of their nodes.
__device__ unsigned long long g_builder_counts[2];

__global__ void __launch_bounds__(kLvThreads) build_tree_level_kernel(TreeArgs a) {
    pdl_trigger();
    pdl_wait();
    extern __shared__ __align__(16) uint8_t smem_raw[];
    __shared__ float theta_s, wmin[kLvWarps];
    // n_cont_s, n_next_s: lists that go on after a pass, nodes that the next level expands; a pass
    // (level) uses one of three counters and zeroes the next one, whose last readers are a pass
    // (level) behind
    __shared__ int wsum[kLvWarps], count_s, bad_s, ended_s, n_cont_s[3], n_next_s[3], n_ties_s, ties[kLvTies], flags_s;
    constexpr unsigned kFull = 0xffffffffu;
    const LevelSmem t = level_smem(smem_raw);
    const int s = blockIdx.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const bool ar = a.mode == TF_MODE_AR, mary = a.mode != TF_MODE_MARGINAL;
    const ListView lists = sequence_lists(a, s);
    const int n_chunks = (a.K2 + 31) / 32;
    // read here (they may lie in host memory), used at the end
    const int root = a.root_tok[a.two_prev ? 2 * s : s];
    const int root_pos = a.mask ? a.root_pos[s] : 0;
    if (mary)
        for (int i = tid; i < a.gamma * a.M; i += kLvThreads)
            t.topm[i] = a.top_ids[(static_cast<size_t>(s) * a.gamma + i / a.M) * a.K1 + i % a.M];
    if (tid == 0) {
        t.score[0] = 0.0f;
        t.par[0] = t.rank[0] = 0;
        t.dep[0] = 0;
        t.m[0] = -1;
        t.act[0].node[0] = 0;
        t.act[0].chunk[0] = 0;
        t.act[0].row[0] = 0;
        n_cont_s[0] = n_next_s[1] = 0;
        count_s = 1;
        bad_s = ended_s = 0;
        flags_s = 0;
        theta_s = -INFINITY;
    }
    __syncthreads();

    // Threads per item when up to kLvExact items are ranked by counting
    auto sharers = [](int n) { return n <= 64 ? 8 : 4; };
    // Raises theta to the B-th best score, with more than kLvExact nodes to the lower edge of the
    // histogram bin that holds it (a little below it: the bins' arithmetic is rounded). Nothing happens
    // while there are fewer than B (with more than kLvExact nodes: fewer than B from kLvFloor up).
    auto raise_theta = [&](int count) {
        if (count - 1 < a.B) return;
        if (count <= kLvExact) {
            // the root counts as a node here: it scores no less than any other, so that the B-th best
            // of the others is the (B + 1)-th of all
            const int per = sharers(count), i = tid / per, part = tid % per, whole = count / 4;
            const float x = t.score[i < count ? i : 0];
            int gt = 0, ge = 0;
            auto tally = [&](float y) {
                gt += y > x ? 1 : 0;
                ge += y >= x ? 1 : 0;
            };
            for (int q = part; q < whole; q += per) {
                const float4 y = reinterpret_cast<const float4*>(t.score)[q];
                tally(y.x);
                tally(y.y);
                tally(y.z);
                tally(y.w);
            }
            if (part < count - 4 * whole) tally(t.score[4 * whole + part]);
            for (int o = 1; o < per; o <<= 1) {
                gt += __shfl_xor_sync(kFull, gt, o);
                ge += __shfl_xor_sync(kFull, ge, o);
            }
            // (all writers hold the same value)
            if (i < count && part == 0 && gt <= a.B && ge > a.B && x > theta_s) theta_s = x;
            __syncthreads();
            return;
        }
        float lo = theta_s;
        if (lo < kLvFloor) {
            float mn = 0.0f;
            for (int i = 1 + tid; i < count; i += kLvThreads) {
                const float x = t.score[i];
                if (x >= kLvFloor) mn = fminf(mn, x);
            }
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) mn = fminf(mn, __shfl_xor_sync(kFull, mn, o));
            if (lane == 0) wmin[warp] = mn;
            __syncthreads();
            lo = wmin[0];
            for (int w = 1; w < kLvWarps; ++w) lo = fminf(lo, wmin[w]);
        }
        if (!(lo < 0.0f)) return;                        // (uniform: every thread holds the same lo)
        t.hist[2 * tid] = t.hist[2 * tid + 1] = 0;
        __syncthreads();
        const float scale = static_cast<float>(kLvBins) / -lo;
        for (int i = 1 + tid; i < count; i += kLvThreads) {
            const float x = t.score[i] - lo;
            if (x >= 0.0f) atomicAdd(&t.hist[min(kLvBins - 1, static_cast<int>(x * scale))], 1);
        }
        __syncthreads();
        const int h0 = t.hist[2 * tid], h1 = t.hist[2 * tid + 1];
        int incl = h0 + h1;                              // bins 2 tid and above, within the warp
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int v = __shfl_down_sync(kFull, incl, o);
            if (lane + o < 32) incl += v;
        }
        if (lane == 0) wsum[warp] = incl;
        __syncthreads();
        for (int w = warp + 1; w < kLvWarps; ++w) incl += wsum[w];
        const int excl = incl - h0 - h1;
        if (incl >= a.B && excl < a.B) {
            const int bin = 2 * tid + (excl + h1 >= a.B ? 1 : 0);
            const float edge = lo + (-lo) * (static_cast<float>(bin) / kLvBins) + lo * 4e-6f;
            if (edge > theta_s) theta_s = edge;
        }
        __syncthreads();
    };

    // Drops the nodes below theta, keeping the others' order; the nodes still to expand move along: in `act`
    // a dropped one leaves a gap, of `next` those kept go to `spare` (n_spare of them, zero before).
    // Returns the new count.
    auto compact = [&](int count, const ActList& act, int n_act, const ActList& next, int n_next, const ActList& spare,
                       int& n_spare) {
        constexpr int kPer = kLvCap / kLvThreads;
        const float theta = theta_s;
        float sc[kPer];
        int tk[kPer];
        uint16_t pr[kPer], rk[kPer];
        uint8_t dp[kPer];
        int8_t mm[kPer];
        bool keep[kPer];
        int mine = 0;
#pragma unroll
        for (int j = 0; j < kPer; ++j) {
            const int i = tid * kPer + j;
            keep[j] = i < count && (i == 0 || t.score[i] >= theta);
            mine += keep[j] ? 1 : 0;
            if (keep[j]) {
                sc[j] = t.score[i];
                tk[j] = t.tok[i];
                pr[j] = t.par[i];
                rk[j] = t.rank[i];
                dp[j] = t.dep[i];
                mm[j] = t.m[i];
            }
        }
        int incl = mine;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int v = __shfl_up_sync(kFull, incl, o);
            if (lane >= o) incl += v;
        }
        if (lane == 31) wsum[warp] = incl;
        __syncthreads();
        int base = incl - mine, total = 0;
        for (int w = 0; w < kLvWarps; ++w) {
            if (w < warp) base += wsum[w];
            total += wsum[w];
        }
#pragma unroll
        for (int j = 0; j < kPer; ++j) {
            const int i = tid * kPer + j;
            t.place[i] = static_cast<uint16_t>(keep[j] ? base : kNoNode);
            base += keep[j] ? 1 : 0;
        }
        __syncthreads();
        for (int i = tid; i < n_act; i += kLvThreads)
            act.node[i] = act.node[i] == kNoNode ? kNoNode : t.place[act.node[i]];
        for (int i = tid; i < n_next; i += kLvThreads) {
            const uint16_t to = t.place[next.node[i]];
            if (to == kNoNode) continue;
            const int q = atomicAdd(&n_spare, 1);
            spare.node[q] = to;
            spare.chunk[q] = 0;
            spare.row[q] = next.row[i];
        }
        uint16_t to[kPer], np[kPer];
#pragma unroll
        for (int j = 0; j < kPer; ++j)
            if (keep[j]) {
                to[j] = t.place[tid * kPer + j];
                np[j] = t.place[pr[j]];                  // a kept node's parent scores no less: kept
            }
        __syncthreads();
#pragma unroll
        for (int j = 0; j < kPer; ++j)
            if (keep[j]) {
                t.score[to[j]] = sc[j];
                t.tok[to[j]] = tk[j];
                t.par[to[j]] = np[j];
                t.rank[to[j]] = rk[j];
                t.dep[to[j]] = dp[j];
                t.m[to[j]] = mm[j];
            }
        if (tid == 0) count_s = total;
        __syncthreads();
        return total;
    };

    int li = 0, lc = 1, ln = 2;                          // act lists: this pass, going on, next level
    int n_act = 1, count = 1, seen = 1, pass = 0;        // seen: the count at the last raise_theta
    for (int d = 1; d <= a.gamma && n_act > 0; ++d) {
        // the nodes of depth d: children of the n_act expandable nodes of depth d - 1
        int& n_next = n_next_s[d % 3];
        if (tid == 0) n_next_s[(d + 1) % 3] = 0;
        const int* cand = t.topm + (d - 1) * a.M;
        const bool deeper = d < a.gamma;
        // list chunks taken of each parent per pass: small budgets rarely want a second one, so no more
        // than the warps take in one go (B = 96 22.8 -> 21.9 us, B = 65 of 16 levels 49.0 -> 46.7)
        int g = (a.B <= 128 ? kLvWarps : 2 * kLvWarps) / n_act;
        g = g < 1 ? 1 : g > n_chunks ? n_chunks : g;
        while (n_act > 0) {
            if (kLvCap - count < 32 * kLvWarps) {
                __syncthreads();                         // (n_next is final for the passes so far)
                raise_theta(count);
                int& n_spare = n_next_s[(d + 1) % 3];    // (zero, and zero again below)
                count = seen = compact(count, t.act[li], n_act, t.act[ln], n_next, t.act[lc], n_spare);
                if (tid == 0) {
                    n_next = n_spare;
                    n_spare = 0;
                    atomicAdd(&g_builder_counts[1], 1ull);
                }
                const int old = ln;
                ln = lc;
                lc = old;
                __syncthreads();
            }
            const ActList act = t.act[li], cont = t.act[lc], next = t.act[ln];
            int nb = (kLvCap - count) / (32 * g);        // parents of this pass: all their entries fit
            nb = nb < n_act ? nb : n_act;
            if (nb < 1) {                                // too many nodes at theta
                if (tid == 0) bad_s = 1;
                __syncthreads();
                break;
            }
            int& n_cont = n_cont_s[pass % 3];
            if (tid == 0) n_cont_s[(pass + 1) % 3] = 0;
            ++pass;
            const float theta = theta_s;
            for (int item = warp; item < nb * g; item += kLvWarps) {
                const int pi = item / g, c = act.chunk[pi] + (item - pi * g);
                const int p = act.node[pi], row = act.row[pi];
                if (p == kNoNode || c >= n_chunks) continue;
                const float ps = t.score[p];
                if (ps < theta) continue;
                const int rank = c * 32 + lane;
                const bool in = rank < a.K2;
                const float lp = in ? lists.lp(row, rank) : 0.0f;
                const int tok = in ? lists.tok(row, rank) : 0;
                const float before = lane == 0 && c > 0 ? lists.lp(row, rank - 1) : 0.0f;
                const float sc = ps + lp;
                float prev = __shfl_up_sync(kFull, sc, 1);
                if (lane == 0) prev = ps + before;       // the parent itself above a list's first entry
                if (in && !(sc <= prev)) bad_s = 1;      // (also for NaN)
                const bool finite = sc > -INFINITY;
                if (in && !finite) ended_s = 1;          // the list ends before its length
                const bool take = in && finite && sc >= theta;
                const unsigned bal = __ballot_sync(kFull, take);
                if (bal == 0u) continue;
                int base = 0;
                if (lane == 0) {
                    base = atomicAdd(&count_s, __popc(bal));
                    // every entry so far counts: the list goes on in the next pass
                    if (item - pi * g == g - 1 && bal == kFull && c + 1 < n_chunks) {
                        const int q = atomicAdd(&n_cont, 1);
                        cont.node[q] = static_cast<uint16_t>(p);
                        cont.chunk[q] = static_cast<uint8_t>(c + 1);
                        cont.row[q] = row;
                    }
                }
                base = __shfl_sync(kFull, base, 0);
                if (!take) continue;
                const int i = base + __popc(bal & ((1u << lane) - 1u));
                // expandable? (M-ary rule: the first equal candidate of its depth) and its child list
                int m = -1, crow = -1;
                if (deeper) {
                    if (!mary) {
                        crow = d;
                    } else {
                        for (int j = a.M - 1; j >= 0; --j) m = cand[j] == tok ? j : m;
                        if (m >= 0)
                            crow = !ar              ? d
                                   : !a.two_prev    ? 1 + (d - 1) * a.M + m
                                   : d == 1         ? 1 + m
                                                    : 1 + a.M + (d - 2) * a.M * a.M + m * a.M + t.m[p];
                    }
                }
                t.score[i] = sc;
                t.tok[i] = tok;
                t.par[i] = static_cast<uint16_t>(p);
                t.rank[i] = static_cast<uint16_t>(rank);
                t.dep[i] = static_cast<uint8_t>(d);
                t.m[i] = static_cast<int8_t>(m);
                if (crow >= 0) {
                    const int q = atomicAdd(&n_next, 1); // (one entry per node held: it fits)
                    next.node[q] = static_cast<uint16_t>(i);
                    next.chunk[q] = 0;
                    next.row[q] = crow;
                }
            }
            __syncthreads();
            count = count_s;
            const int more = n_cont, rest = n_act - nb;
            const bool bad = bad_s != 0;
            __syncthreads();                             // everyone has read them before the next pass writes
            if (bad) break;
            if (rest > 0) {                              // parents left out of this pass
                for (int i = tid; i < rest; i += kLvThreads) {
                    cont.node[more + i] = act.node[nb + i];
                    cont.chunk[more + i] = act.chunk[nb + i];
                    cont.row[more + i] = act.row[nb + i];
                }
                __syncthreads();
            }
            n_act = more + rest;
            const int old = li;
            li = lc;
            lc = old;
            if (count - seen >= (a.B >> 1) || n_act > 0) {
                raise_theta(count);
                seen = count;
            }
        }
        if (n_act > 0) break;                            // (left by one of the breaks above)
        n_act = n_next;
        const int old = li;
        li = ln;
        ln = old;
        if (n_act > 2 * kLvWarps) {                      // many: only those that theta leaves
            const ActList all = t.act[li], few = t.act[lc];
            int& n_few = n_cont_s[pass % 3];
            if (tid == 0) n_cont_s[(pass + 1) % 3] = 0;
            ++pass;
            const float theta = theta_s;
            for (int i = tid; i < n_act; i += kLvThreads) {
                const uint16_t p = all.node[i];
                if (t.score[p] < theta) continue;
                const int q = atomicAdd(&n_few, 1);
                few.node[q] = p;
                few.chunk[q] = 0;
                few.row[q] = all.row[i];
            }
            __syncthreads();
            n_act = n_few;
            __syncthreads();
            const int o = li;
            li = lc;
            lc = o;
        }
    }
    __syncthreads();

    // ---- the order of the survivors. (Entries of -inf come after all others; the tree holds some only
    // where there are too few others, and then the queue places them.)
    int n = 0;
    if (tid == 0 && ended_s && count - 1 < a.B) bad_s = 1;
    __syncthreads();
    if (!bad_s) {
        if (tid == 0) n_ties_s = 0;
        if (count <= kLvExact) {
            // few: each node's place by counting the larger keys, those below theta included
            n = count - 1;
            const int per = sharers(n), i = tid / per, part = tid % per;
            if (tid < n) t.key[tid] = level_key(t.score[tid + 1], t.dep[tid + 1], t.rank[tid + 1], tid + 1);
            __syncthreads();
            const unsigned long long x = i < n ? t.key[i] : 0ull;
            int r = 0;
#pragma unroll 4
            for (int j = part; j < n; j += per) r += t.key[j] > x ? 1 : 0;
            for (int o = 1; o < per; o <<= 1) r += __shfl_xor_sync(kFull, r, o);
            __syncthreads();
            if (i < n && part == 0) t.key[r] = x;
            __syncthreads();
        } else {
            // Those at theta or above by buckets of equal width (bucket 0 holds the best), then by
            // counting within the bucket.
            raise_theta(count);
            __syncthreads();
            const float theta = theta_s;
            // (fewer than B nodes leave theta unknown: any scale serves)
            const float scale = theta < 0.0f ? static_cast<float>(kLvBins) / fmaxf(theta, -64.0f) : 0.0f;
            auto bucket = [&](float x) { return min(kLvBins - 1, static_cast<int>(x * scale)); };
            t.hist[2 * tid] = t.hist[2 * tid + 1] = 0;
            __syncthreads();
            for (int i = 1 + tid; i < count; i += kLvThreads)
                if (t.score[i] >= theta) atomicAdd(&t.hist[bucket(t.score[i])], 1);
            __syncthreads();
            const int h0 = t.hist[2 * tid], h1 = t.hist[2 * tid + 1];
            int incl = h0 + h1;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int v = __shfl_up_sync(kFull, incl, o);
                if (lane >= o) incl += v;
            }
            if (lane == 31) wsum[warp] = incl;
            __syncthreads();
            int base = incl - h0 - h1;
            for (int w = 0; w < kLvWarps; ++w) {
                n += wsum[w];
                base += w < warp ? wsum[w] : 0;
            }
            t.hist[2 * tid] = base;                      // the next free place of each bucket
            t.hist[2 * tid + 1] = base + h0;
            __syncthreads();
            if (n <= kLvSort) {
                for (int i = 1 + tid; i < count; i += kLvThreads)
                    if (t.score[i] >= theta)
                        t.key[atomicAdd(&t.hist[bucket(t.score[i])], 1)] = level_key(t.score[i], t.dep[i], t.rank[i], i);
                __syncthreads();                         // bucket b's keys: from hist[b - 1] up to hist[b]
                unsigned long long x[kLvSort / kLvThreads];
                int r[kLvSort / kLvThreads];
#pragma unroll
                for (int k = 0; k < kLvSort / kLvThreads; ++k) {
                    const int i = tid + k * kLvThreads;
                    if (i < n) {
                        x[k] = t.key[i];
                        const int bk = bucket(t.score[x[k] & 0xfff]), end = t.hist[bk];
                        r[k] = bk > 0 ? t.hist[bk - 1] : 0;
#pragma unroll 1
                        for (int j = r[k]; j < end; ++j) r[k] += t.key[j] > x[k] ? 1 : 0;
                    }
                }
                __syncthreads();
#pragma unroll
                for (int k = 0; k < kLvSort / kLvThreads; ++k)
                    if (tid + k * kLvThreads < n) t.key[r[k]] = x[k];
                __syncthreads();
            }
        }
        if (n > kLvSort) {
            if (tid == 0) bad_s = 1;
        } else {
            for (int i = tid; i < n; i += kLvThreads) {
                const unsigned long long x = t.key[i];
                const int xi = static_cast<int>(x & 0xfff);
                t.place[xi] = static_cast<uint16_t>(i + 1);
                // (runs of equal nodes that begin behind the last place are not part of the tree)
                if (i + 1 < n && (i < a.B || (x >> 24) == (t.key[a.B - 1] >> 24))) {
                    const unsigned long long y = t.key[i + 1];
                    if ((x >> 24) == (y >> 24) && t.par[xi] != t.par[y & 0xfff]) {
                        const int q = atomicAdd(&n_ties_s, 1);
                        if (q < kLvTies) ties[q] = i;
                    }
                }
            }
            __syncthreads();
            if (tid == 0 && n_ties_s > 0) {
                // equal score and depth, different parents: shallower levels first, each run of
                // equal nodes by its parents' places, then by list rank
                const int nt = n_ties_s;
                bool ok = nt <= kLvTies;
                for (int dd = 1; ok && dd <= a.gamma; ++dd)
                    for (int q = 0; ok && q < nt; ++q) {
                        const unsigned long long x = t.key[ties[q]] >> 24;
                        if (127 - static_cast<int>(x & 0xff) != dd) continue;
                        int l = ties[q], r = ties[q] + 1;
                        while (l > 0 && (t.key[l - 1] >> 24) == x) --l;
                        while (r + 1 < n && (t.key[r + 1] >> 24) == x) ++r;
                        ok = r - l < kLvTies;
                        for (int i = l + 1; ok && i <= r; ++i) {
                            const unsigned long long v = t.key[i];
                            const int vp = t.place[t.par[v & 0xfff]], vr = t.rank[v & 0xfff];
                            int j = i - 1;
                            for (; j >= l; --j) {
                                const int u = static_cast<int>(t.key[j] & 0xfff);
                                const int up = t.place[t.par[u]];
                                if (up < vp || (up == vp && t.rank[u] < vr)) break;
                                t.key[j + 1] = t.key[j];
                            }
                            t.key[j + 1] = v;
                        }
                        for (int i = l; i <= r; ++i) t.place[t.key[i] & 0xfff] = static_cast<uint16_t>(i + 1);
                    }
                if (!ok) bad_s = 1;
            }
        }
    }
    __syncthreads();
    const int n_out = a.B + 1;
    if (bad_s) {
        __syncthreads();
        if (tid == 0) atomicAdd(&g_builder_counts[0], 1ull);
        const TreeSmem q = tree_smem(smem_raw, a);
        for (int i = tid; i < a.gamma * a.M; i += kLvThreads)
            q.topm[i] = a.top_ids[(static_cast<size_t>(s) * a.gamma + i / a.M) * a.K1 + i % a.M];
        __syncthreads();
        build_tree_queue(a, s, q, sequence_lists(a, s));
        write_nodes(a, s, q);
        fused_mask(a, s, q);
        return;
    }
    const size_t o0 = static_cast<size_t>(s) * n_out;
    for (int i = tid; i < n_out; i += kLvThreads) {
        int tok = -1, par = -1, dep = -1;
        float sc = -INFINITY;
        if (i == 0) {
            tok = root;
            dep = 0;
            sc = 0.0f;
            if (root < 0 || root >= a.V) atomicOr(&flags_s, TF_DEV_BAD_TOKEN);
        } else if (i <= n) {
            const int x = static_cast<int>(t.key[i - 1] & 0xfff), p = t.par[x];
            tok = t.tok[x];
            par = p == 0 ? 0 : t.place[p];
            dep = t.dep[x];
            sc = t.score[x];
            if (tok < 0 || tok >= a.V) atomicOr(&flags_s, TF_DEV_BAD_TOKEN);
        } else {
            atomicOr(&flags_s, TF_DEV_UNDERFULL);
        }
        a.node_tok[o0 + i] = tok;
        a.node_parent[o0 + i] = par;
        a.node_depth[o0 + i] = dep;
        a.node_score[o0 + i] = sc;
        if (a.mask) {                                    // (hist: at most kFusedMaskMaxNodes entries of each)
            t.hist[i] = par;
            t.hist[kFusedMaskMaxNodes + i] = dep;
        }
    }
    __syncthreads();
    if (tid == 0) a.dev_status[s] = sequence_status(a, flags_s);
    if (a.mask)
        mask_rows(n_out, t.hist, t.hist + kFusedMaskMaxNodes, root_pos, 0, n_out, reinterpret_cast<uint32_t*>(t.key),
                  a.mask + static_cast<size_t>(s) * n_out * n_out, a.pos_ids + o0);
}

// ------------------------------------------------------------------------------------------
// The tree-attention mask and position ids (mask_rows) of a drafted tree in global memory: one
// CTA per sequence and block of kMaskRows rows. Blocks of 16 rows and four-byte stores: 513 nodes take
// about 4 us on GB300 instead of 23 with blocks of 128 and single bytes (8 or 32 rows: the same
// within 2 us).
// ------------------------------------------------------------------------------------------
constexpr int kMaskRows = 16;
__global__ void __launch_bounds__(256) tree_mask_kernel(int n, const int32_t* __restrict__ node_parent,
                                                        const int32_t* __restrict__ node_depth,
                                                        const int32_t* __restrict__ root_pos,
                                                        uint8_t* __restrict__ mask, int32_t* __restrict__ pos_ids) {
    pdl_trigger();
    pdl_wait();
    extern __shared__ uint32_t sm[];
    const int s = blockIdx.x;
    const int r0 = blockIdx.y * kMaskRows, r1 = min(n, r0 + kMaskRows);   // this CTA's rows
    int* par = reinterpret_cast<int*>(sm);
    int* dep = par + n;
    uint32_t* anc = reinterpret_cast<uint32_t*>(dep + n);   // ancestor-or-self bits of kMaskRows rows
    const int32_t* P = node_parent + static_cast<size_t>(s) * n;
    const int32_t* D = node_depth + static_cast<size_t>(s) * n;
    for (int i = threadIdx.x; i < n; i += blockDim.x) {
        par[i] = P[i];
        dep[i] = D[i];
    }
    __syncthreads();
    mask_rows(n, par, dep, root_pos[s], r0, r1, anc, mask + static_cast<size_t>(s) * n * n,
              pos_ids + static_cast<size_t>(s) * n);
}

// ------------------------------------------------------------------------------------------
// Verification walk (Sec. 3: a drafted token is accepted iff it equals the verifier's token at
// its parent's position; Sec. 4: the step gains the accepted tokens plus the verifier's residual
// token). One warp per sequence: from the root, each step finds the child of the current node
// whose token equals the verifier's token there (a ballot over all nodes; the smallest index if
// an invalid tree repeats a token) and moves to it. At most gamma steps (the depth cap), so a
// corrupt parent array cannot loop.
// ------------------------------------------------------------------------------------------
__global__ void __launch_bounds__(32) accept_walk_kernel(int n, int gamma, const int32_t* __restrict__ node_tok,
                                                         const int32_t* __restrict__ node_parent,
                                                         const int32_t* __restrict__ verifier_tok,
                                                         int32_t* __restrict__ accept_len,
                                                         int32_t* __restrict__ accept_path,
                                                         int32_t* __restrict__ next_tok) {
    pdl_trigger();
    pdl_wait();
    constexpr unsigned kFull = 0xffffffffu;
    const int s = blockIdx.x, lane = threadIdx.x;
    const int32_t* tok = node_tok + static_cast<size_t>(s) * n;
    const int32_t* par = node_parent + static_cast<size_t>(s) * n;
    const int32_t* ver = verifier_tok + static_cast<size_t>(s) * n;
    int32_t* path = accept_path + static_cast<size_t>(s) * (gamma + 1);
    int cur = 0, len = 0;
    if (lane == 0) path[0] = 0;
    for (int step = 0; step < gamma; ++step) {
        const int want = ver[cur];
        int found = -1;
        for (int c0 = 1; c0 < n && found < 0; c0 += 32) {
            const int c = c0 + lane;
            const bool m = c < n && par[c] == cur && tok[c] == want;
            const unsigned bal = __ballot_sync(kFull, m);
            if (bal) found = c0 + __ffs(bal) - 1;
        }
        if (found < 0) break;
        cur = found;
        ++len;
        if (lane == 0) path[len] = cur;
    }
    for (int i = len + 1 + lane; i <= gamma; i += 32) path[i] = -1;
    if (lane == 0) {
        accept_len[s] = len;
        next_tok[s] = ver[cur];
    }
}

}  // namespace

// Error-free sum (Knuth's TwoSum): s + c tracks a running sum to about twice fp32 precision.
__device__ __forceinline__ void two_sum_acc(float& s, float& c, float x) {
    const float t = s + x;
    const float z = t - s;
    c += (s - (t - z)) + (x - z);
    s = t;
}

// bf16 nearest-even rounding of the real value r + t, where r is an fp32 value and |t| is below
// two fp32 ulps of r. Only an r within a few ulps of a bf16 midpoint can round differently from
// r alone; for those the side of the midpoint is decided from (r - midpoint) + t, where
// r - midpoint is exact (both share r's binade).
__device__ __forceinline__ __nv_bfloat16 bf16_round_sum(float r, float t) {
    const uint32_t u = __float_as_uint(r);
    const uint32_t low = u & 0xffffu;
    if ((u & 0x7f800000u) == 0x7f800000u || low < 0x8000u - 4u || low > 0x8000u + 4u) return __float2bfloat16_rn(r);
    const uint32_t trunc = u & 0xffff0000u;
    const float mid = __uint_as_float(trunc | 0x8000u);
    const float dm = (r - mid) + t;
    const float away = (u & 0x80000000u) ? -dm : dm;   // > 0: beyond the midpoint in magnitude
    uint32_t bits = trunc;
    if (away > 0.0f || (away == 0.0f && (trunc & 0x10000u))) bits += 0x10000u;
    return __ushort_as_bfloat16(static_cast<unsigned short>(bits >> 16));
}

// the two bf16 values of a 32-bit word
__device__ __forceinline__ unsigned long long f2_bf16x2(uint32_t w) {
    return f2_pack(__uint_as_float(w << 16), __uint_as_float(w & 0xffff0000u));
}

// ------------------------------------------------------------------------------------------
// The stage-2 input rows for bf16 with d <= 8192: one item per normalised vector, not per row. The
// M rows (two tokens: M^2) of a depth share their hidden state, so its part of x is computed once
// per depth and stored to all of them (at most kHRows per item); every embedding is an item of its
// own. Only the norm weights are read before the dependency wait: the hidden states may be the output
// of the kernel just before.
// An item is a CTA of eight warps. (Items of one or two warps save the block barrier but hold so
// much in registers that too few warps are in flight: 1928 rows of d = 5120 took 38 us with one CTA
// per row, 73 with a warp per item.)
// x is the correctly rounded bf16 value of the definition (an element off by one bf16 ulp would
// perturb every gate/up output and flip many later roundings), computed in fp32 only (GB300's fp64
// is too slow even for the few scalar steps of a row):
//  - mean(h^2): every square of a bf16 value is exact in fp32; the sums, and their warp and block
//    reductions, are compensated (TwoSum pairs);
//  - 1 / sqrt(mean + eps) as hi + lo: hi = rsqrtf, then one Newton step in double-float
//    arithmetic (the squares and products formed exactly with FMAs), about 2^-46 relative;
//  - h * w is exact in fp32 (two 8-bit significands); (h w) * hi is rounded once and its
//    rounding error recovered with an FMA, so (h w) / sqrt(mean + eps) is known as r + t to
//    about 2^-45 relative, which decides the bf16 rounding (bf16_round_sum).
// ------------------------------------------------------------------------------------------
constexpr int kHRows = 8;       // rows that one hidden-state item stores to (16: up to 3% slower, one row each: 2%)
struct GatherArgs {
    const uint4 *hidden, *embed, *norm_h, *norm_e;
    const int32_t *root_tok, *top_ids;
    int gamma, M, K1, R, d, V, two_prev;
    float eps;
    uint4 *X, *hres;
    int* status;
    int h_chunks;     // items per hidden state
    int n_h;          // hidden-state items, the first ones
};

template <int NV>      // 16-byte units per thread: ceil(d / 2048)
__global__ void __launch_bounds__(256) gather_norm_bf16_kernel(GatherArgs a) {
    pdl_trigger();
    __shared__ float red[8][2];
    const int t = threadIdx.x, warp = t >> 5, lane = t & 31;
    const int item = blockIdx.x;
    const bool is_h = item < a.n_h;
    const int dv = a.d / 8, NS = a.two_prev ? 3 : 2;
    // the norm weights are no kernel's output: requested before the dependency wait
    const uint4* wt = is_h ? a.norm_h : a.norm_e;
    uint4 wv[NV];
#pragma unroll
    for (int j = 0; j < NV; ++j) {
        const int c = t + j * 256;
        wv[j] = c < dv ? wt[c] : make_uint4(0u, 0u, 0u, 0u);
    }
    pdl_wait();
    // the rows that the item stores to: r0 .. r0 + n - 1 (an embedding: one row, part `part`)
    int r0 = 0, n = 1, part = 0;
    const uint4* src = a.hidden;
    if (is_h) {
        const int q = item / a.h_chunks, c = item - q * a.h_chunks, sq = q / a.gamma, i = q - sq * a.gamma;
        const int per = i == 0 ? 1 : a.two_prev && i > 1 ? a.M * a.M : a.M;          // rows of depth i + 1
        const int at = i == 0 ? 0 : !a.two_prev ? 1 + (i - 1) * a.M : i == 1 ? 1 : 1 + a.M + (i - 2) * a.M * a.M;
        r0 = sq * a.R + at + c * kHRows;
        n = min(kHRows, per - c * kHRows);    // (at most 0: nothing to store)
        src += static_cast<size_t>(sq * a.gamma + i) * dv;
    } else {
        const int q = item - a.n_h;
        r0 = a.two_prev ? q >> 1 : q;
        part = a.two_prev ? 1 + (q & 1) : 1;
        int tok[2] = {0, 0};
        stage2_row_tokens(r0, a.R, a.gamma, a.M, a.K1, a.two_prev != 0, a.root_tok, a.top_ids, tok);
        int token = tok[part - 1];
        if (token < 0 || token >= a.V) {
            if (t == 0) set_status(a.status, TF_DEV_BAD_TOKEN);
            token = 0;
        }
        src = a.embed + static_cast<size_t>(token) * dv;
    }
    uint4 v[NV];
#pragma unroll
    for (int j = 0; j < NV; ++j) {
        const int c = t + j * 256;
        v[j] = n > 0 && c < dv ? src[c] : make_uint4(0u, 0u, 0u, 0u);
    }
    // sums of squares, two packed running sums
    unsigned long long s2 = 0ull, c2 = 0ull;
#pragma unroll
    for (int j = 0; j < NV; ++j) {
        const uint32_t w[4] = {v[j].x, v[j].y, v[j].z, v[j].w};
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const unsigned long long h = f2_bf16x2(w[k]), x = f2_mul(h, h);
            const unsigned long long u = f2_add(s2, x), z = f2_sub(u, s2);
            c2 = f2_add(c2, f2_add(f2_sub(s2, f2_sub(u, z)), f2_sub(x, z)));
            s2 = u;
        }
    }
    float S = f2_lo(s2), C = f2_lo(c2);
    two_sum_acc(S, C, f2_hi(s2));
    C += f2_hi(c2);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const float so = __shfl_down_sync(0xffffffffu, S, o), co = __shfl_down_sync(0xffffffffu, C, o);
        two_sum_acc(S, C, so);
        C += co;
    }
    if (lane == 0) {
        red[warp][0] = S;
        red[warp][1] = C;
    }
    __syncthreads();
    S = C = 0.0f;
#pragma unroll
    for (int w = 0; w < 8; ++w) {
        two_sum_acc(S, C, red[w][0]);
        C += red[w][1];
    }
    // m = (S + C) / d + eps as a double-float (mh, ml); d is scaled exactly when it is a power of
    // two, otherwise the quotient's rounding error is recovered by an FMA
    float hi, lo;
    {
        const float fd = static_cast<float>(a.d);
        const float q = S / fd;
        const float qerr = fmaf(-q, fd, S) / fd + C / fd;
        float mh = q + a.eps;
        float ml = (q - (mh - (mh - q))) + (a.eps - (mh - q)) + qerr;   // TwoSum(q, eps) plus the rest
        const float u = mh + ml;
        ml = ml - (u - mh);
        mh = u;
        // y = 1 / sqrt(m): y0 = rsqrtf(mh), then one Newton step in double-float arithmetic,
        // y = y0 + y0 (1 - m y0^2) / 2, with y0^2 and m y0^2 formed by exact FMA products
        const float y0 = rsqrtf(mh);
        const float p = y0 * y0, pl = fmaf(y0, y0, -p);          // y0^2 = p + pl exactly
        const float w = mh * p, wl = fmaf(mh, p, -w);              // mh p = w + wl exactly
        const float r = ((1.0f - w) - wl) - (mh * pl + ml * p);    // 1 - m y0^2, ~2^-23
        hi = y0;
        lo = 0.5f * y0 * r;
    }
    // the approximator GEMMs' tail-split counters (after the status word) start each call at zero
    if (item == 0 && a.status)
        for (int i = t; i < kTailSems; i += 256) a.status[1 + i] = 0;
    uint4* out = a.X + static_cast<size_t>(r0) * NS * dv + static_cast<size_t>(part) * dv;
    uint4* res = a.two_prev && is_h ? a.hres + static_cast<size_t>(r0) * dv : nullptr;
    const unsigned long long hi2 = f2_pack(hi, hi), lo2 = f2_pack(lo, lo);
#pragma unroll
    for (int j = 0; j < NV; ++j) {
        const int c = t + j * 256;
        if (c >= dv) break;
        const uint32_t xb[4] = {v[j].x, v[j].y, v[j].z, v[j].w}, wb[4] = {wv[j].x, wv[j].y, wv[j].z, wv[j].w};
        uint32_t o[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const unsigned long long pv = f2_mul(f2_bf16x2(xb[k]), f2_bf16x2(wb[k]));
            const unsigned long long rv = f2_mul(pv, hi2);
            const float r0v = f2_lo(rv), r1v = f2_hi(rv);
            const unsigned long long tv = f2_fma(pv, lo2, f2_fma(pv, hi2, f2_pack(-r0v, -r1v)));
            const __nv_bfloat16 b0 = bf16_round_sum(r0v, f2_lo(tv)), b1 = bf16_round_sum(r1v, f2_hi(tv));
            o[k] = static_cast<uint32_t>(__bfloat16_as_ushort(b1)) << 16 | __bfloat16_as_ushort(b0);
        }
        const uint4 ov = make_uint4(o[0], o[1], o[2], o[3]);
        for (int r = 0; r < n; ++r) out[static_cast<size_t>(r) * NS * dv + c] = ov;
        if (res)
            for (int r = 0; r < n; ++r) res[static_cast<size_t>(r) * dv + c] = v[j];
    }
}

cudaError_t launch_gather_norm(const Ctx& ctx, int dtype, const void* hidden, const void* embed, const void* norm_h,
                               const void* norm_e, const int32_t* root_tok, const int32_t* top_ids, int b, int gamma,
                               int M, int K1, int R, int two_prev, int d, int V, float eps, void* X, void* hres) {
    const int rows = b * R;
    if (rows <= 0) return cudaSuccess;
    if (two_prev && !hres) return cudaErrorInvalidValue;
    cudaError_t e;
    if (dtype == TF_BF16 && d % 8 == 0 && d <= 8192) {
        GatherArgs a{};
        a.hidden = static_cast<const uint4*>(hidden);
        a.embed = static_cast<const uint4*>(embed);
        a.norm_h = static_cast<const uint4*>(norm_h);
        a.norm_e = static_cast<const uint4*>(norm_e);
        a.root_tok = root_tok;
        a.top_ids = top_ids;
        a.gamma = gamma;
        a.M = M;
        a.K1 = K1;
        a.R = R;
        a.d = d;
        a.V = V;
        a.two_prev = two_prev;
        a.eps = eps;
        a.X = static_cast<uint4*>(X);
        a.hres = static_cast<uint4*>(hres);
        a.status = ctx.status;
        a.h_chunks = ((two_prev && gamma > 2 ? M * M : M) + kHRows - 1) / kHRows;
        const long long n_h = static_cast<long long>(b) * gamma * a.h_chunks;
        const long long n_items = n_h + static_cast<long long>(rows) * (two_prev ? 2 : 1);
        if (n_items > 0x7fffffffll) return cudaErrorInvalidConfiguration;
        a.n_h = static_cast<int>(n_h);
        auto kern = d <= 2048   ? gather_norm_bf16_kernel<1>
                    : d <= 4096 ? gather_norm_bf16_kernel<2>
                    : d <= 6144 ? gather_norm_bf16_kernel<3>
                                : gather_norm_bf16_kernel<4>;
        e = launch_pdl(kern, dim3(static_cast<unsigned>(n_items)), dim3(256), 0, ctx.stream, a);
    } else if (dtype == TF_BF16) {
        using B16 = __nv_bfloat16;
        auto kern = two_prev ? gather_norm_kernel<B16, 2> : gather_norm_kernel<B16, 1>;
        e = launch_pdl(kern, dim3(rows), dim3(256), 0, ctx.stream, static_cast<const B16*>(hidden),
                       static_cast<const B16*>(embed), static_cast<const B16*>(norm_h), static_cast<const B16*>(norm_e),
                       root_tok, top_ids, gamma, M, K1, R, d, V, eps, static_cast<B16*>(X), static_cast<B16*>(hres),
                       ctx.status);
    } else {
        auto kern = two_prev ? gather_norm_kernel<float, 2> : gather_norm_kernel<float, 1>;
        e = launch_pdl(kern, dim3(rows), dim3(256), 0, ctx.stream, static_cast<const float*>(hidden),
                       static_cast<const float*>(embed), static_cast<const float*>(norm_h),
                       static_cast<const float*>(norm_e), root_tok, top_ids, gamma, M, K1, R, d, V, eps,
                       static_cast<float*>(X), static_cast<float*>(hres), ctx.status);
    }
    return e != cudaSuccess ? e : cudaGetLastError();
}

cudaError_t launch_build_tree(const Ctx& ctx, int b, int gamma, int M, int K1, int K2, int B, int V, int mode, int R,
                              int two_prev, const int32_t* root_tok, const int32_t* top_ids, const float* top_logp,
                              const int32_t* child_ids, const float* child_logp, int32_t* node_tok,
                              int32_t* node_parent, int32_t* node_depth, float* node_score, int32_t* dev_status,
                              const int32_t* root_pos, uint8_t* mask, int32_t* pos_ids, const int32_t* ws_status) {
    if (mask && B + 1 > kFusedMaskMaxNodes) return cudaErrorInvalidValue;
    TreeArgs a{gamma, M, K1, K2, B, V, mode, R, mode == TF_MODE_AR && two_prev ? 1 : 0, root_tok, top_ids, top_logp,
               child_ids, child_logp, node_tok, node_parent, node_depth, node_score, dev_status, root_pos, mask,
               pos_ids, ws_status};
    const int rows_l = mode == TF_MODE_AR ? R : gamma;
    const int stride = mode == TF_MODE_AR ? K2 : K1;
    const int sw = stride < B + 1 ? stride : B + 1;   // list entries that a tree can reach
    // The sorted-queue builder for small budgets with every reachable entry in shared memory. Its cost is the
    // pops, about 3.2 us + 0.26 B, whatever the lists and the number of sequences. The builder by levels
    // costs what the deepest of the trees does, 1.7 to 3 us per level, which no size tells: gamma at
    // worst. So up to 64 nodes it takes over where all gamma levels cost no more than the pops. Measured on
    // GB300 (with the mask; queue against levels for trees of two to five kinds, one and eight sequences): gamma =
    // 1, B = 16 6.9, 6.5; gamma = 2, B = 32 11.0, 8.5 to 9.1; gamma = 3, B = 48 15.2, 12.4 to 14.3, B = 32
    // 11.1, 10.9 to 11.7; gamma = 4, B = 64 19.5, 15.7 to 19.6, B = 48 15.4, 13.9 to 17.9; gamma = 16, B = 64
    // 20.2, 15.9 (4 levels) to 40.5 (16). Two-token rule: gamma = 4, B = 64 21, 13.8 to 16.2; gamma = 12 23, 16 to 35.
    // Beyond 64 nodes the queue lies in shared memory (0.6 us per pop).
    const size_t fsm = fast_tree_smem(B, gamma, M, rows_l, sw, mask != nullptr);
    if (B <= kSortedQueueMax && B < 16 * gamma && fsm <= kTreeSmemLimit) {
        auto kern = a.two_prev ? build_tree_fast_kernel<true> : build_tree_fast_kernel<false>;
        cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(fsm));
        if (e != cudaSuccess) return e;
        e = launch_pdl(kern, dim3(b), dim3(kFastThreads), fsm, ctx.stream, a, sw);
        return e != cudaSuccess ? e : cudaGetLastError();
    }
    const size_t lsm = level_smem_bytes(B, gamma, M, mask != nullptr);
    cudaError_t e = cudaFuncSetAttribute(build_tree_level_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         static_cast<int>(lsm));
    if (e != cudaSuccess) return e;
    e = launch_pdl(build_tree_level_kernel, dim3(b), dim3(kLvThreads), lsm, ctx.stream, a);
    return e != cudaSuccess ? e : cudaGetLastError();
}

cudaError_t builder_counts(unsigned long long out[2]) {
    const cudaError_t e = cudaDeviceSynchronize();
    return e != cudaSuccess ? e : cudaMemcpyFromSymbol(out, g_builder_counts, sizeof(g_builder_counts));
}

cudaError_t launch_tree_mask(const Ctx& ctx, int b, int B, const int32_t* node_parent, const int32_t* node_depth,
                             const int32_t* root_pos, uint8_t* mask, int32_t* pos_ids) {
    const int n = B + 1;
    const int W = (n + 31) / 32;
    const size_t smem = static_cast<size_t>(2 * n + kMaskRows * W) * 4;
    cudaError_t e = cudaFuncSetAttribute(tree_mask_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         static_cast<int>(smem));
    if (e != cudaSuccess) return e;
    e = launch_pdl(tree_mask_kernel, dim3(b, (n + kMaskRows - 1) / kMaskRows), dim3(256), smem, ctx.stream, n,
                   node_parent, node_depth, root_pos, mask, pos_ids);
    return e != cudaSuccess ? e : cudaGetLastError();
}

cudaError_t launch_accept_walk(const Ctx& ctx, int b, int B, int gamma, const int32_t* node_tok,
                               const int32_t* node_parent, const int32_t* verifier_tok, int32_t* accept_len,
                               int32_t* accept_path, int32_t* next_tok) {
    const cudaError_t e = launch_pdl(accept_walk_kernel, dim3(b), dim3(32), 0, ctx.stream, B + 1, gamma, node_tok,
                                     node_parent, verifier_tok, accept_len, accept_path, next_tok);
    return e != cudaSuccess ? e : cudaGetLastError();
}

}  // namespace tf
