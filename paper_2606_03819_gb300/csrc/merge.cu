// Merge of the LM-head partials into log-softmax top-k (Algorithm 1 "TopM" of stage 1 and the
// log-softmax + top-k of every stage-2 row).
//
// One CTA per row. The CTA
//   1. combines the row's half-block (max, sum of exp) pairs into its log-sum-exp;
//   2. keeps the halves whose best entry can be among the k best: a histogram of the halves' best
//      values over 256 equal-width buckets gives the bucket of the k-th, and the halves in it or
//      above are kept (k and a few: every other half's best, hence all of its entries, is below k
//      other values). Their chunks' two largest entries in those buckets are the candidates;
//   3. certifies: a kept chunk whose third-largest value reaches the k-th candidate may hide
//      further members of the top k. Those chunks' 32 logits are recomputed exactly from lm_head
//      and x (in rounds of at most 64 chunks), replace the chunk's two candidates, and the
//      selection is redone;
//   4. writes the k winners sorted, as (id, logit - LSE): the candidates' ranks, by counting.
// What bounds it is the chain of loads and block barriers, eight in the usual case (an exact k-th
// half and an exact k-th candidate by two further selections took 21): on GB300, k = 32, 3872 rows
// 143 -> 90 us, 512 rows 21 -> 12.5; k = 64, 1928 rows 81 -> 60, 241 rows 13.7 -> 10.8. The selections
// remain for rows with equal or non-finite values, crowded buckets, fewer halves than k, more
// halves than registers hold, or more candidates than are worth counting.
// The result is the exact top-k of the full vocabulary whatever the input; a recompute needs
// three members of the top k in one 32-column chunk (about one row in 500 on random data).
#include <math.h>

#include "common.cuh"

namespace tf {
namespace {

constexpr int kRegHalves = 8;     // half summaries a thread can hold in registers (V <= 262144)
constexpr int kKeepSlack = 64;    // room for halves beyond the k-th in its bucket
constexpr int kThreads = 256;   // 512 or more: two CTAs no longer fit an SM, so 241 rows take two waves
// Candidates that are ranked by counting: one per thread. Two per thread cost more than a selection (V =
// 151936, d = 1024, 1000 rows, k = 256: 87 against 76 us).
constexpr int kRankCands = kThreads;

__device__ __forceinline__ void lse_combine(float& m, float& s, float m2, float s2) {
    if (m2 > m) {
        s = s * __expf(m - m2) + s2;
        m = m2;
    } else if (m2 > -INFINITY) {
        s += s2 * __expf(m2 - m);
    }
}

// k-th largest of keys[0..n) (n >= k >= 1), by 8-bit digits from the most significant byte. Once
// the chosen digit's bin holds a single key, that key is the answer and is looked up directly
// (float keys of one row share their top bytes, so this usually ends the search after two or
// three digits instead of eight).
__device__ unsigned long long block_kth_largest(const unsigned long long* keys, int n, int k, int* hist,
                                                int* sel, unsigned long long* found) {
    unsigned long long prefix = 0;
    int rem = k;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    for (int shift = 56; shift >= 0; shift -= 8) {
        for (int i = tid; i < 256; i += kThreads) hist[i] = 0;
        __syncthreads();
        const unsigned long long hi_mask = shift == 56 ? 0ull : (~0ull << (shift + 8));
        // shared-memory atomics: lanes of a warp on one bin are combined by the hardware (a
        // warp match to aggregate them first costs far more on GB300)
        for (int i = tid; i < n; i += kThreads) {
            const unsigned long long key = keys[i];
            if ((key & hi_mask) == prefix) atomicAdd(&hist[static_cast<int>((key >> shift) & 255)], 1);
        }
        __syncthreads();
        if (warp == 0) {
            int local[8];
            int sum = 0;
#pragma unroll
            for (int b = 0; b < 8; ++b) {
                local[b] = hist[lane * 8 + b];
                sum += local[b];
            }
            // inclusive suffix sum over lanes (higher lanes hold higher digits)
            int incl = sum;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int v = __shfl_down_sync(0xffffffffu, incl, o);
                if (lane + o < 32) incl += v;
            }
            const int excl = incl - sum;
            if (excl < rem && rem <= incl) {
                int c = excl;
                for (int b = 7; b >= 0; --b) {
                    if (c + local[b] >= rem) {
                        sel[0] = lane * 8 + b;
                        sel[1] = rem - c;
                        sel[2] = local[b];
                        break;
                    }
                    c += local[b];
                }
            }
        }
        __syncthreads();
        prefix |= static_cast<unsigned long long>(sel[0]) << shift;
        rem = sel[1];
        if (sel[2] == 1 && shift > 0) {
            // the k-th key is the only key with this prefix
            const unsigned long long mask = ~0ull << shift;
            for (int i = tid; i < n; i += kThreads)
                if ((keys[i] & mask) == prefix) *found = keys[i];
            __syncthreads();
            const unsigned long long r = *found;
            __syncthreads();   // every thread has read *found and sel before either is reused
            return r;
        }
        __syncthreads();       // every thread has read sel before the next digit rewrites it
    }
    return prefix;
}

// Shared state of block_kth_largest_fast.
constexpr int kBuckets = 256;
constexpr int kCollectCap = 256;
struct alignas(16) SelectSmem {
    int hist[kBuckets];
    unsigned long long coll[kCollectCap];
    float wmax[kThreads / 32], wmin[kThreads / 32];
    int wcnt[kThreads / 32];
    float vmin, scale;
    int total, bucket, rem, count, n_coll;
    unsigned long long found;
};

// The k-th largest non-zero key of keys[0..n) (zero keys are empty slots and rank below all),
// or 0 when fewer than k keys are non-zero. One histogram pass over 256 equal-width buckets of
// the key values (a monotone map, so the k-th largest key lies in the bucket where the count from
// the top reaches k), then an exact rank among the few keys of that bucket. Falls back to the
// byte-wise radix select when the values are all equal, not finite, or crowd one bucket.
__device__ unsigned long long block_kth_largest_fast(const unsigned long long* keys, int n, int k, SelectSmem& B,
                                                     int* hist, int* sel, unsigned long long* found) {
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    float vmax = -INFINITY, vmin = INFINITY;
    int cnt = 0;
    for (int i = tid; i < n; i += kThreads) {
        const unsigned long long key = keys[i];
        if (key != 0ull) {
            const float v = key_value(key);
            vmax = fmaxf(vmax, v);
            vmin = fminf(vmin, v);
            ++cnt;
        }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        vmax = fmaxf(vmax, __shfl_xor_sync(0xffffffffu, vmax, o));
        vmin = fminf(vmin, __shfl_xor_sync(0xffffffffu, vmin, o));
        cnt += __shfl_xor_sync(0xffffffffu, cnt, o);
    }
    if (lane == 0) {
        B.wmax[warp] = vmax;
        B.wmin[warp] = vmin;
        B.wcnt[warp] = cnt;
    }
    for (int i = tid; i < kBuckets; i += kThreads) B.hist[i] = 0;
    __syncthreads();
    if (warp == 0) {
        float mx = lane < kThreads / 32 ? B.wmax[lane] : -INFINITY;
        float mn = lane < kThreads / 32 ? B.wmin[lane] : INFINITY;
        int c = lane < kThreads / 32 ? B.wcnt[lane] : 0;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
            mn = fminf(mn, __shfl_xor_sync(0xffffffffu, mn, o));
            c += __shfl_xor_sync(0xffffffffu, c, o);
        }
        if (lane == 0) {
            B.total = c;
            B.vmin = mn;
            const float range = mx - mn;
            B.scale = (range > 0.0f && isfinite(range)) ? static_cast<float>(kBuckets) / range : 0.0f;
            B.n_coll = 0;
        }
    }
    __syncthreads();
    const int total = B.total;
    const float scale = B.scale, vlo = B.vmin;
    if (total < k) {
        __syncthreads();
        return 0ull;
    }
    if (scale == 0.0f) {
        __syncthreads();
        return block_kth_largest(keys, n, k, hist, sel, found);
    }
    auto bucket_of = [&](unsigned long long key) {
        const int b = static_cast<int>((key_value(key) - vlo) * scale);
        return b < 0 ? 0 : (b >= kBuckets ? kBuckets - 1 : b);
    };
    for (int i = tid; i < n; i += kThreads) {
        const unsigned long long key = keys[i];
        if (key != 0ull) atomicAdd(&B.hist[bucket_of(key)], 1);
    }
    __syncthreads();
    if (warp == 0) {
        // lane l holds buckets 8l .. 8l+7; inclusive suffix sums over lanes (high buckets first)
        int local[8];
        int sum = 0;
#pragma unroll
        for (int b = 0; b < 8; ++b) {
            local[b] = B.hist[lane * 8 + b];
            sum += local[b];
        }
        int incl = sum;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int v = __shfl_down_sync(0xffffffffu, incl, o);
            if (lane + o < 32) incl += v;
        }
        const int excl = incl - sum;
        if (excl < k && k <= incl) {
            int c = excl;
            for (int b = 7; b >= 0; --b) {
                if (c + local[b] >= k) {
                    B.bucket = lane * 8 + b;
                    B.rem = k - c;
                    B.count = local[b];
                    break;
                }
                c += local[b];
            }
        }
    }
    __syncthreads();
    const int bk = B.bucket, rem = B.rem, cb = B.count;
    if (cb > kCollectCap) {
        __syncthreads();
        return block_kth_largest(keys, n, k, hist, sel, found);
    }
    for (int i = tid; i < n; i += kThreads) {
        const unsigned long long key = keys[i];
        if (key != 0ull && bucket_of(key) == bk) B.coll[atomicAdd(&B.n_coll, 1)] = key;
    }
    __syncthreads();
    // keys are distinct: exactly one has rem - 1 larger keys in the bucket
    for (int i = tid; i < cb; i += kThreads) {
        const unsigned long long key = B.coll[i];
        int rank = 0;
        for (int j = 0; j < cb; ++j) rank += B.coll[j] > key ? 1 : 0;
        if (rank == rem - 1) B.found = key;
    }
    __syncthreads();
    const unsigned long long r = B.found;
    __syncthreads();   // every thread has read the shared results before they are reused
    return r;
}

// <w_c, x> for four weight rows of d elements (row c at w + c * d), by one warp: lanes take 8-element
// slices, four slices of all rows in flight; every sum in the order of its slices. acc[c] on every lane.
__device__ __forceinline__ void dot_rows4(const __nv_bfloat16* const (&w)[4], const __nv_bfloat16* x, int d, int lane,
                                          float (&acc)[4]) {
#pragma unroll
    for (int c = 0; c < 4; ++c) acc[c] = 0.0f;
    if ((d & 255) == 0 && ((reinterpret_cast<uintptr_t>(w[0]) | reinterpret_cast<uintptr_t>(x)) & 15) == 0) {
        const uint4* x4 = reinterpret_cast<const uint4*>(x);
        const int n = d / 256;                       // 16-byte slices per lane
        for (int base = 0; base < n; base += 4) {
            uint4 xb[4], wb[4][4];
#pragma unroll
            for (int i = 0; i < 4; ++i)
                if (base + i < n) {
                    xb[i] = x4[(base + i) * 32 + lane];
#pragma unroll
                    for (int c = 0; c < 4; ++c) wb[c][i] = reinterpret_cast<const uint4*>(w[c])[(base + i) * 32 + lane];
                }
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                if (base + i >= n) break;
                const __nv_bfloat16* xv = reinterpret_cast<const __nv_bfloat16*>(&xb[i]);
#pragma unroll
                for (int c = 0; c < 4; ++c) {
                    const __nv_bfloat16* b = reinterpret_cast<const __nv_bfloat16*>(&wb[c][i]);
#pragma unroll
                    for (int j = 0; j < 8; ++j) acc[c] = fmaf(__bfloat162float(b[j]), __bfloat162float(xv[j]), acc[c]);
                }
            }
        }
    } else {
        for (int k = lane; k < d; k += 32) {
            const float xk = __bfloat162float(x[k]);
#pragma unroll
            for (int c = 0; c < 4; ++c) acc[c] = fmaf(__bfloat162float(w[c][k]), xk, acc[c]);
        }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1)
#pragma unroll
        for (int c = 0; c < 4; ++c) acc[c] += __shfl_xor_sync(0xffffffffu, acc[c], o);
}
__device__ __forceinline__ void dot_rows4(const float* const (&w)[4], const float* x, int d, int lane, float (&acc)[4]) {
#pragma unroll
    for (int c = 0; c < 4; ++c) acc[c] = 0.0f;
#pragma unroll 4
    for (int k = lane; k < d; k += 32) {
        const float xk = x[k];
#pragma unroll
        for (int c = 0; c < 4; ++c) acc[c] = fmaf(w[c][k], xk, acc[c]);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1)
#pragma unroll
        for (int c = 0; c < 4; ++c) acc[c] += __shfl_xor_sync(0xffffffffu, acc[c], o);
}

// Shared-memory layout of one merge CTA (dynamic part), for a top-k of k and room for kc >= k halves.
struct MergeSmem {
    unsigned long long* hkey;   // [n_halves] best key of every half block (0 = empty); once the halves are chosen,
    float* zbuf;                // in its place, [kMergeExpandChunks * kChunk] recomputed logits
    unsigned long long* cand;   // [2 * 4kc + kMergeExpandChunks * kChunk]
    unsigned long long* cand2;  // the same size: the compacted set of the next round
    unsigned long long* sel;    // [k] the winners
    float* c3;                  // [4kc] third value of each kept chunk (bound on the rest)
    int* cbase;                 // [4kc] first vocabulary id of each kept chunk
    int* chalf;                 // [kc] the halves kept
    uint8_t* expanded;          // [4kc] chunk recomputed
};
constexpr size_t kZbufBytes = static_cast<size_t>(kMergeExpandChunks) * kChunk * sizeof(float);
__host__ __device__ inline size_t merge_key_bytes(int n_tiles) { return static_cast<size_t>(2) * n_tiles * 8; }
// The static part is 4.7 KB: with the most that the dims check lets through, a CTA stays within the 227 KB
// of a block.
constexpr size_t kMergeStaticBytes = 5 * 1024;
static_assert(kMaxMergeSmem + kMergeStaticBytes <= 227 * 1024, "shared memory of a merge CTA");
__host__ __device__ inline size_t merge_layout(int n_tiles, int k, int kc, uint8_t* base, MergeSmem* m) {
    const size_t detail = static_cast<size_t>(kc) * (kChunks / 2);  // chunks of the halves kept
    size_t off = 0;
    auto take = [&](size_t bytes) {
        uint8_t* p = base ? base + off : nullptr;
        off += (bytes + 15) / 16 * 16;
        return p;
    };
    uint8_t* hk = take(merge_key_bytes(n_tiles) > kZbufBytes ? merge_key_bytes(n_tiles) : kZbufBytes);
    uint8_t* cd = take((2 * detail + static_cast<size_t>(kMergeExpandChunks) * kChunk) * 8);
    uint8_t* cd2 = take((2 * detail + static_cast<size_t>(kMergeExpandChunks) * kChunk) * 8);
    uint8_t* se = take(static_cast<size_t>(k) * 8);
    uint8_t* c3 = take(detail * 4);
    uint8_t* cb = take(detail * 4);
    uint8_t* ch = take(static_cast<size_t>(kc) * 4);
    uint8_t* ex = take(detail);
    if (m) {
        m->hkey = reinterpret_cast<unsigned long long*>(hk);
        m->zbuf = reinterpret_cast<float*>(hk);
        m->cand = reinterpret_cast<unsigned long long*>(cd);
        m->cand2 = reinterpret_cast<unsigned long long*>(cd2);
        m->sel = reinterpret_cast<unsigned long long*>(se);
        m->c3 = reinterpret_cast<float*>(c3);
        m->cbase = reinterpret_cast<int*>(cb);
        m->chalf = reinterpret_cast<int*>(ch);
        m->expanded = ex;
    }
    return off;
}

template <typename T>
__global__ void __launch_bounds__(kThreads, 2) lmhead_merge_kernel(Partials partials, int n_rows, int n_tiles, int V,
                                                                int d, int k, int kc, float inv_temp,
                                                                const T* __restrict__ lm_head,
                                                                const T* __restrict__ x, int32_t* __restrict__ out_ids,
                                                                float* __restrict__ out_logp, int* status) {
    pdl_trigger();
    pdl_wait();
    extern __shared__ __align__(16) uint8_t dsm[];
    MergeSmem S;
    merge_layout(n_tiles, k, kc, dsm, &S);
    const int n_detail = kc * (kChunks / 2);
    __shared__ int hist[256];
    __shared__ SelectSmem SB;
    __shared__ float red_m[kThreads / 32], red_s[kThreads / 32];
    __shared__ uint32_t wkmax[kThreads / 32], wkmin[kThreads / 32];
    __shared__ int wcnt[kThreads / 32];
    __shared__ int sel_info[3], n_flag, flag_list[kMergeExpandChunks], n_cand, n_next, n_sel, n_valid, n_chalf;
    __shared__ unsigned long long found;
    __shared__ float lse_s;

    const int row = blockIdx.x;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int nh = 2 * n_tiles;
    if (tid == 0) {
        n_cand = 0;
        n_valid = 0;
        n_chalf = 0;
    }

    for (int i = tid; i < n_detail; i += kThreads) S.expanded[i] = 0;
    const float4* half_of = partials.halves + row;   // half i at half_of[i * n_rows]
    const size_t half_stride = static_cast<size_t>(partials.n_rows);
    int nch = 0;                 // halves kept
    bool kept = false;
    // The usual case (up to kRegHalves halves per thread, finite values): the summaries stay in
    // registers, one histogram of the halves' best values gives the bucket of the k-th, and every
    // half in that bucket or above is kept (a few more than k: unless they exceed the room for them,
    // the exact rank inside the bucket is not needed).
    if (nh <= kRegHalves * kThreads) {
        float4 v[kRegHalves];
#pragma unroll
        for (int j = 0; j < kRegHalves; ++j) {
            const int i = tid + j * kThreads;
            v[j] = i < nh ? half_of[static_cast<size_t>(i) * half_stride] : make_float4(0.0f, 0.0f, 0.0f, __int_as_float(-1));
        }
        uint32_t kmax = 0u, kmin = 0xffffffffu;
        int cnt = 0;
#pragma unroll
        for (int j = 0; j < kRegHalves; ++j)
            if (__float_as_int(v[j].w) >= 0) {
                const uint32_t key = float_key(v[j].z);
                kmax = max(kmax, key);
                kmin = min(kmin, key);
                ++cnt;
            }
        kmax = __reduce_max_sync(0xffffffffu, kmax);
        kmin = __reduce_min_sync(0xffffffffu, kmin);
        cnt = __reduce_add_sync(0xffffffffu, cnt);
        if (lane == 0) {
            wkmax[warp] = kmax;
            wkmin[warp] = kmin;
            wcnt[warp] = cnt;
        }
        SB.hist[tid] = 0;
        __syncthreads();
        cnt = 0;
#pragma unroll
        for (int w = 0; w < kThreads / 32; ++w) {
            kmax = max(kmax, wkmax[w]);
            kmin = min(kmin, wkmin[w]);
            cnt += wcnt[w];
        }
        const float M = key_float(kmax), lo = key_float(kmin), range = M - lo;
        if (cnt >= k && range > 0.0f && isfinite(range) && isfinite(M)) {     // (uniform)
            const float scale = static_cast<float>(kBuckets) / range;
            auto bucket_of = [&](float x) {
                const int b = static_cast<int>((x - lo) * scale);
                return b < 0 ? 0 : b >= kBuckets ? kBuckets - 1 : b;
            };
            float s = 0.0f;
#pragma unroll
            for (int j = 0; j < kRegHalves; ++j)
                if (__float_as_int(v[j].w) >= 0) {
                    atomicAdd(&SB.hist[bucket_of(v[j].z)], 1);
                    s += v[j].y * __expf(v[j].x - M);
                }
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
            if (lane == 0) red_s[warp] = s;
            __syncthreads();
            if (warp == 0) {
                // lane l holds buckets 8l .. 8l + 7; inclusive suffix sums over lanes
                const int4 h0 = reinterpret_cast<const int4*>(SB.hist)[2 * lane], h1 = reinterpret_cast<const int4*>(SB.hist)[2 * lane + 1];
                const int local[8] = {h0.x, h0.y, h0.z, h0.w, h1.x, h1.y, h1.z, h1.w};
                int incl = 0;
#pragma unroll
                for (int b = 0; b < 8; ++b) incl += local[b];
                const int sum = incl;
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const int u = __shfl_down_sync(0xffffffffu, incl, o);
                    if (lane + o < 32) incl += u;
                }
                const int excl = incl - sum;
                if (excl < k && k <= incl) {
                    int c = excl, bk = 7;
#pragma unroll
                    for (int b = 7; b >= 0; --b)
                        if (c < k) {
                            c += local[b];
                            bk = b;
                        }
                    SB.bucket = lane * 8 + bk;
                    SB.count = c;                        // halves in that bucket or above
                }
            } else if (tid == 32) {
                float t = 0.0f;
                for (int w = 0; w < kThreads / 32; ++w) t += red_s[w];
                const float lse = M + logf(t);
                lse_s = lse;
                if (!isfinite(lse)) set_status(status, TF_DEV_NONFINITE);
            }
            __syncthreads();
            const int bk = SB.bucket;
            nch = SB.count;
            kept = nch <= kc;                            // (uniform)
            if (kept) {
#pragma unroll
                for (int j = 0; j < kRegHalves; ++j)
                    if (__float_as_int(v[j].w) >= 0 && bucket_of(v[j].z) >= bk) S.chalf[atomicAdd(&n_chalf, 1)] = tid + j * kThreads;
                __syncthreads();
                // their chunks: the two largest entries in those buckets become candidates
                for (int i = tid; i < nch * (kChunks / 2); i += kThreads) {
                    const int h = S.chalf[i >> 2];
                    const int tile = h >> 1, chunk = (h & 1) * (kChunks / 2) + (i & 3);
                    const float4 q = partials.chunks[partials.chunk_at(tile, chunk, row)];
                    const int v0 = tile * kBlockV + chunk * kChunk;
                    const int ids = __float_as_int(q.w);
                    S.cbase[i] = v0;
                    S.c3[i] = q.z;
                    if (q.x > -INFINITY && bucket_of(q.x) >= bk) S.cand[atomicAdd(&n_cand, 1)] = cand_key(q.x, v0 + (ids & 255));
                    if (q.y > -INFINITY && bucket_of(q.y) >= bk) S.cand[atomicAdd(&n_cand, 1)] = cand_key(q.y, v0 + ((ids >> 8) & 255));
                }
                __syncthreads();
            }
        }
        if (!kept) __syncthreads();                      // the shared words above are reused below
    }

    if (!kept) {
        // 1. half-block summaries (strided by n_rows, eight loads in flight per thread): the row's
        //    log-sum-exp and one key per half
        float m = -INFINITY, s = 0.0f;
        int my_valid = 0;
        {
            for (int base = tid; base < nh; base += 8 * kThreads) {
                float4 v[8];
#pragma unroll
                for (int j = 0; j < 8; ++j) {
                    const int i = base + j * kThreads;
                    if (i < nh) v[j] = half_of[static_cast<size_t>(i) * half_stride];
                }
#pragma unroll
                for (int j = 0; j < 8; ++j) {
                    const int i = base + j * kThreads;
                    if (i >= nh) break;
                    const int id = __float_as_int(v[j].w);
                    unsigned long long key = 0ull;
                    if (id >= 0) {
                        lse_combine(m, s, v[j].x, v[j].y);
                        key = cand_key(v[j].z, id);
                        ++my_valid;
                    }
                    S.hkey[i] = key;
                }
            }
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            const float m2 = __shfl_xor_sync(0xffffffffu, m, o);
            const float s2 = __shfl_xor_sync(0xffffffffu, s, o);
            lse_combine(m, s, m2, s2);
        }
        if (lane == 0) {
            red_m[warp] = m;
            red_s[warp] = s;
        }
        __syncthreads();
        atomicAdd(&n_valid, my_valid);
        __syncthreads();
        if (warp == 0) {
            float M = lane < kThreads / 32 ? red_m[lane] : -INFINITY;
            float Ssum = lane < kThreads / 32 ? red_s[lane] : 0.0f;
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
                const float m2 = __shfl_xor_sync(0xffffffffu, M, o);
                const float s2 = __shfl_xor_sync(0xffffffffu, Ssum, o);
                lse_combine(M, Ssum, m2, s2);
            }
            if (lane == 0) {
                const float lse = M + logf(Ssum);
                lse_s = lse;
                if (!isfinite(lse)) set_status(status, TF_DEV_NONFINITE);
            }
        }

        // 2. theta0 and the halves at or above it (at most k: the keys are distinct)
        const unsigned long long theta0 =
            n_valid >= k ? block_kth_largest_fast(S.hkey, nh, k, SB, hist, sel_info, &found) : 0ull;
        for (int i = tid; i < nh; i += kThreads) {
            const unsigned long long key = S.hkey[i];
            if (key != 0ull && key >= theta0) {
                const int slot = atomicAdd(&n_chalf, 1);
                if (slot < k) S.chalf[slot] = i;
            }
        }
        __syncthreads();
        nch = min(n_chalf, k);
        // their chunks: the two largest entries at or above theta0 become candidates
        for (int i = tid; i < nch * (kChunks / 2); i += kThreads) {
            const int h = S.chalf[i >> 2];
            const int tile = h >> 1, chunk = (h & 1) * (kChunks / 2) + (i & 3);
            const float4 q = partials.chunks[partials.chunk_at(tile, chunk, row)];
            const int v0 = tile * kBlockV + chunk * kChunk;
            const int ids = __float_as_int(q.w);
            S.cbase[i] = v0;
            S.c3[i] = q.z;
            if (q.x > -INFINITY) {
                const unsigned long long key = cand_key(q.x, v0 + (ids & 255));
                if (key >= theta0) S.cand[atomicAdd(&n_cand, 1)] = key;
            }
            if (q.y > -INFINITY) {
                const unsigned long long key = cand_key(q.y, v0 + ((ids >> 8) & 255));
                if (key >= theta0) S.cand[atomicAdd(&n_cand, 1)] = key;
            }
        }
        __syncthreads();
    }

    // 3. select; a kept chunk whose third value reaches the k-th candidate may hide members of
    //    the top k, so its 32 logits are recomputed exactly and the selection is redone. Chunks
    //    are recomputed in rounds of at most kMergeExpandChunks; after each round the keys at or
    //    above the k-th candidate survive (the candidates are logits of the row, so every member
    //    of the true top k is at or above it), and all logits of the round's chunks join them, which bounds
    //    the set by k + kMergeExpandChunks * kChunk whatever the input. (All: a recomputed logit is summed in
    //    another order, so one that was at the k-th candidate may come out a little below it. Without it the
    //    set could fall below k and be filled up with far smaller ones.) Few candidates (the usual case)
    //    are ranked by counting, which sorts the winners as well.
    unsigned long long theta = 0;
    unsigned long long* cand = S.cand;
    unsigned long long* spare = S.cand2;
    for (;;) {
        const int nc = n_cand;
        const bool few = nc >= k && nc <= kRankCands;
        unsigned long long mine = 0ull;
        int rank = 0;
        if (few) {
            if (tid < nc) {
                mine = cand[tid];
#pragma unroll 8
                for (int i = 0; i < nc; ++i) rank += cand[i] > mine ? 1 : 0;
                if (rank == k - 1) found = mine;
            }
        } else {
            theta = nc >= k ? block_kth_largest_fast(cand, nc, k, SB, hist, sel_info, &found) : 0ull;
        }
        if (tid == 0) n_flag = 0;
        __syncthreads();
        if (few) theta = found;
        const float tval = key_value(theta);
        for (int i = tid; i < nch * (kChunks / 2); i += kThreads) {
            if (S.expanded[i] || !(S.c3[i] > -INFINITY)) continue;
            if (nc < k || S.c3[i] >= tval) {
                const int slot = atomicAdd(&n_flag, 1);
                if (slot < kMergeExpandChunks) flag_list[slot] = i;
            }
        }
        __syncthreads();
        const int nf = min(n_flag, kMergeExpandChunks);   // the rest wait for the next round
        if (nf == 0) {
            if (!few) break;
            if (mine != 0ull && rank < k) {
                out_ids[static_cast<size_t>(row) * k + rank] = key_id(mine);
                out_logp[static_cast<size_t>(row) * k + rank] = key_value(mine) - lse_s;
            }
            return;
        }
        if (tid == 0) {
            set_status(status, TF_DEV_RECOMPUTED);
            n_next = 0;
        }
        // exact logits of this round's chunks, four columns per warp
        for (int q = 4 * warp; q < nf * kChunk; q += 4 * (kThreads / 32)) {
            const int v = S.cbase[flag_list[q / kChunk]] + q % kChunk;
            const T* w[4];
#pragma unroll
            for (int c = 0; c < 4; ++c) w[c] = lm_head + static_cast<size_t>(min(v + c, V - 1)) * d;
            float acc[4];
            dot_rows4(w, x + static_cast<size_t>(row) * d, d, lane, acc);
            if (lane < 4) {
                const float z = lane == 0 ? acc[0] : lane == 1 ? acc[1] : lane == 2 ? acc[2] : acc[3];
                S.zbuf[q + lane] = v + lane < V ? z * inv_temp : -INFINITY;
            }
        }
        __syncthreads();
        // the next set: surviving keys not from this round's chunks, then their exact logits
        for (int j = tid; j < nc; j += kThreads) {
            const unsigned long long key = cand[j];
            if (key == 0ull || key < theta) continue;
            const int id = key_id(key);
            bool mine = false;
            for (int f = 0; f < nf; ++f) {
                const int v0 = S.cbase[flag_list[f]];
                mine = mine || (id >= v0 && id < v0 + kChunk);
            }
            if (!mine) spare[atomicAdd(&n_next, 1)] = key;
        }
        for (int q = tid; q < nf * kChunk; q += kThreads) {
            const int f = q / kChunk, cc = q - f * kChunk;
            const int v = S.cbase[flag_list[f]] + cc;
            if (v < V) {
                const unsigned long long key = cand_key(S.zbuf[q], v);
                if (key >= theta || S.zbuf[q] > -INFINITY) spare[atomicAdd(&n_next, 1)] = key;
            }
        }
        for (int f = tid; f < nf; f += kThreads) S.expanded[flag_list[f]] = 1;
        __syncthreads();
        if (tid == 0) n_cand = n_next;
        unsigned long long* t = cand;
        cand = spare;
        spare = t;
        __syncthreads();
    }

    // 4. the k winners, sorted
    if (tid == 0) n_sel = 0;
    __syncthreads();
    const int nc = n_cand;
    for (int i = tid; i < nc; i += kThreads) {
        const unsigned long long key = cand[i];
        if (key != 0ull && key >= theta) {
            const int slot = atomicAdd(&n_sel, 1);
            if (slot < k) S.sel[slot] = key;
        }
    }
    __syncthreads();
    const int ns = min(n_sel, k);
    const float lse = lse_s;
    for (int i = tid; i < ns; i += kThreads) {
        const unsigned long long key = S.sel[i];
        int rank = 0;
        for (int j = 0; j < ns; ++j) rank += S.sel[j] > key ? 1 : 0;
        out_ids[static_cast<size_t>(row) * k + rank] = key_id(key);
        out_logp[static_cast<size_t>(row) * k + rank] = key_value(key) - lse;
    }
    for (int i = ns + tid; i < k; i += kThreads) {
        out_ids[static_cast<size_t>(row) * k + i] = -1;
        out_logp[static_cast<size_t>(row) * k + i] = -INFINITY;
    }
    if (tid == 0 && ns < k) set_status(status, TF_DEV_UNDERFULL);
}

}  // namespace

// What the dims check counts per merge CTA: the keys alone in their place, and a row of x in fp32, which
// bounds d. (Where the recomputed logits need more room than the keys, the rest is far below the limit.)
size_t merge_smem_bytes(int n_tiles, int d, int k) {
    const size_t keys = merge_key_bytes(n_tiles), more = keys < kZbufBytes ? kZbufBytes - keys : 0;
    return merge_layout(n_tiles, k, k, nullptr, nullptr) - more + (static_cast<size_t>(d) * 4 + 15) / 16 * 16;
}

cudaError_t launch_lmhead_merge(const Ctx& ctx, int dtype, Partials partials, int n_rows, int V, int d, int k,
                                float inv_temp, const void* lm_head, const void* x, int32_t* out_ids,
                                float* out_logp) {
    if (n_rows <= 0) return cudaSuccess;
    const int n_tiles = (V + kBlockV - 1) / kBlockV;
    // Room for up to kKeepSlack halves more than k, as far as it leaves as many CTAs on an SM (228 KB, 1 KB of
    // it per CTA for the system) as k alone (V = 151936, d = 1024, 241 rows: k = 320 32 -> 23 us, k = 384 41 ->
    // 32).
    auto resident = [&](int c) {
        const size_t smem = merge_layout(n_tiles, k, c, nullptr, nullptr);
        return smem > kMaxMergeSmem ? 0 : (228 * 1024) / (smem + kMergeStaticBytes + 1024);
    };
    int kc = k + kKeepSlack;
    while (kc > k && resident(kc) < resident(k)) kc -= 8;
    if (kc < k) kc = k;
    const size_t smem = merge_layout(n_tiles, k, kc, nullptr, nullptr);
    if (dtype == TF_BF16) {
        auto kern = lmhead_merge_kernel<__nv_bfloat16>;
        cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(smem));
        if (e != cudaSuccess) return e;
        e = launch_pdl(kern, dim3(n_rows), dim3(kThreads), smem, ctx.stream, partials, n_rows, n_tiles, V, d, k, kc,
                       inv_temp, static_cast<const __nv_bfloat16*>(lm_head), static_cast<const __nv_bfloat16*>(x),
                       out_ids, out_logp, ctx.status);
        if (e != cudaSuccess) return e;
    } else {
        auto kern = lmhead_merge_kernel<float>;
        cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(smem));
        if (e != cudaSuccess) return e;
        e = launch_pdl(kern, dim3(n_rows), dim3(kThreads), smem, ctx.stream, partials, n_rows, n_tiles, V, d, k, kc,
                       inv_temp, static_cast<const float*>(lm_head), static_cast<const float*>(x), out_ids, out_logp,
                       ctx.status);
        if (e != cudaSuccess) return e;
    }
    return cudaGetLastError();
}

}  // namespace tf
