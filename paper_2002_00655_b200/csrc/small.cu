// Calls of few key occurrences (kSmallOcc at most): the cumulative push without a sort.
//
// A push of a few thousand rows is a microsecond or two of memory traffic; sorted, it is a fork to another stream, a
// cooperative sort with a grid barrier per pass, a reduction and a fix-up launch: 27 us for 13 rows, of which the host
// spends 20.  Here ONE launch does it.  Every block reads all keys of the call and keeps those of its hash bucket (one to
// four dozen, in the order of the call: lane masks of the warps' shares, no sort), finds the first occurrence and the
// number of occurrences of each in a table in shared memory, and a warp per distinct key adds its occurrences' rows in
// the order of the call, in fp64, and rounds once, as the sorted reduction does.  Keys with more than kShortRun
// occurrences are shared by four to sixteen of the block's warps (a range of the list each, partial sums added in range order).
// Hot keys, which are a large part of the call, are shared by all blocks: 8,192 occurrences of one key took its block 118 us
// at 128 values and 242 at 400, where a sort and the tiled reduction take 39 and 52.  Every block finds the same ones by itself
// in a sample of kSample keys at jittered positions (hot_hits of one key make it hot: a key that is a quarter of the call is
// missed once in some hundred calls, which costs time only; at four in a hundred the largest key of 6,000 Zipf(0.9) ones,
// 300 occurrences, is shared as well: a pull, push and relocation of them take 39 us instead of 26).  The call is cut into
// pieces, a block sums a hot key's occurrences of one piece and parks the sum; the last block to finish a key adds its pieces
// in order.
// What grows with the call is the reading of all keys by every block: kSmallOcc is where the sort takes over.
// (A first form compared every occurrence with all others, 128 keys per instruction: 1,200 to 1,800 warp instructions
// per occurrence, 11 us at 2,048 and 27 us at 3,328 occurrences of AdaGrad.)
//
// Training steps take the same launch after their gradient kernel, which leaves the key of every occurrence slot in
// a buffer (num_keys: no key; all ones: an index out of range, the whole call is a no-op).
#include <string.h>

#include "ps_internal.cuh"

namespace psb {

namespace {

constexpr int kThreads = 512;
constexpr int kWarps = kThreads / 32;
constexpr uint32_t kShortRun = 8;               // occurrences of one key that a warp adds alone
__device__ __forceinline__ uint32_t long_warps(uint32_t occurrences) { return occurrences <= 16 ? 4 : occurrences <= 32 ? 8 : 16; }   // ... that add a longer one
constexpr int kTableBits = 10, kTable = 1 << kTableBits;
constexpr uint32_t kSample = 64;
__host__ __device__ constexpr uint32_t hot_hits(int kCh) { return kCh == 1 ? 7 : 10; }   // (a warp has half as many rows of several column blocks in flight)
constexpr uint32_t kHotCall = 2049;             // smaller calls are not sampled: 2,048 occurrences of one key take 33 us, sorted 31
constexpr uint32_t kHotPiece = 256;             // occurrences per piece, at least
static_assert(kSmallOcc <= 32 * kThreads, "a lane per round of the bucket's selection");

// which of the blocks takes a key: a multiplicative hash, so that neighbouring keys (the frequent ones) are spread
__device__ __forceinline__ uint32_t bucket_of(uint32_t key, uint32_t n_buckets) {
    return (((key * 0x9e3779b1u) >> 16) * n_buckets) >> 16;
}

struct acc4 {
    double x, y, z, w;
};

enum { kPlain = 0, kScaled = 1, kAdaGrad = 2 };

struct SmallArgs {
    const uint64_t* keys64;         // caller's keys (range-checked here), or null:
    const uint32_t* keys32;         // keys a gradient kernel left
    uint32_t n, K;
    const float4* upd;              // kPlain: a row per occurrence; kScaled: two source rows per example; kAdaGrad: a gradient per occurrence
    const float* scales;
    uint32_t slots;                 // kScaled: occurrences per example
    float lr, eps;                  // kAdaGrad
    float4* store;
    const uint2* table;
    uint64_t S;
    uint32_t L4, F4;                // float4 of a store row; of an update row (kAdaGrad: half a row)
    const double* loss_partial;
    uint32_t loss_blocks;
    double* loss_accum;
    DevStatus* st;
    uint32_t pieces, piece_len;     // of the call, for hot keys; piece_len a multiple of kWarps
    double* parked;                 // [stretch][hot key][piece][stretch_vals]
    uint32_t stretch_vals;
    unsigned int* tickets;          // [stretch][hot key], zero between calls
};

// position s of the sample: one in each of kSample equal parts of the call, so that no period of the batch escapes it
__device__ __forceinline__ uint32_t sample_pos(uint32_t s, uint32_t n) {
    const uint32_t jitter = (s * 0x9e3779b1u) >> 16;
    return (uint32_t)(((uint64_t)(s * 0x10000u + jitter) * n) >> 22);
}
static_assert(kSample * 8 == kThreads && kSample == 1u << 6, "sample_pos divides by 2^16 times this");

__device__ __forceinline__ uint32_t key_at(const SmallArgs& A, uint32_t i) {     // kSentinelPad: out of range
    if (A.keys64) {
        const uint64_t k = A.keys64[i];
        return k < A.K ? (uint32_t)k : kSentinelPad;
    }
    return A.keys32[i];
}


// Hot keys: a piece of the call at a time, a sixteenth of it per warp, kFly rows of a warp in flight.  (A function of its own, so
// that the registers of calls without hot keys stay as they are.)
template <int kMode, int kCh>
__device__ __noinline__ void hot_keys(const SmallArgs A, const uint32_t* s_hot, uint32_t n_hot, acc4 (*s_part)[32], uint32_t* s_ticket) {
    constexpr int kHalves = kMode == kAdaGrad ? 2 : 1, kFly = kCh == 4 ? 2 : 4;
    const unsigned full = 0xffffffffu;
    const uint32_t tid = threadIdx.x, lane = tid & 31, w = tid >> 5, n = A.n, f0 = blockIdx.y * (32 * kCh) + lane;
    for (uint32_t task = blockIdx.x; task < n_hot * A.pieces; task += gridDim.x - 1) {
        const uint32_t h = task / A.pieces, p = task - h * A.pieces, k = s_hot[h], slot = blockIdx.y * kMaxHot + h;
        float4* target = A.store + phys_row(A.table[k], A.S) * A.L4;
        float4 G[kCh];                          // kAdaGrad: the accumulators before the call
        acc4 a[kHalves][kCh];
#pragma unroll
        for (int c = 0; c < kCh; ++c) {
            G[c] = kMode == kAdaGrad && f0 + 32 * c < A.F4 ? target[A.F4 + f0 + 32 * c] : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
            for (int half = 0; half < kHalves; ++half) a[half][c] = acc4{0.0, 0.0, 0.0, 0.0};
        }
        const uint32_t from = tmin(p * A.piece_len + w * (A.piece_len / kWarps), n), to = tmin(from + A.piece_len / kWarps, n);
        for (uint32_t b = from; b < to; b += 32) {
            for (unsigned todo = __ballot_sync(full, b + lane < to && key_at(A, b + lane) == k); todo;) {
                float4 u[kFly][kCh];
                float sc[kFly];
                bool have[kFly];
#pragma unroll
                for (int q = 0; q < kFly; ++q) {
                    have[q] = todo != 0;
                    const uint32_t o = b + (todo ? __ffs(todo) - 1 : 0);
                    todo &= todo - 1;           // 0 stays 0
                    uint64_t row = o;
                    sc[q] = 1.f;
                    if (kMode == kScaled) {
                        sc[q] = A.scales[o];
                        const uint32_t e = o / A.slots;
                        row = 2u * e + (o != e * A.slots ? 1u : 0u);
                    }
#pragma unroll
                    for (int c = 0; c < kCh; ++c)
                        u[q][c] = have[q] && f0 + 32 * c < A.F4 ? A.upd[row * A.F4 + f0 + 32 * c] : make_float4(0.f, 0.f, 0.f, 0.f);
                }
#pragma unroll
                for (int q = 0; q < kFly; ++q) {
                    if (!have[q]) break;
#pragma unroll
                    for (int c = 0; c < kCh; ++c) {
                        float4 v = u[q][c];
                        if (kMode == kAdaGrad) {
                            const float4 sq = make_float4(v.x * v.x, v.y * v.y, v.z * v.z, v.w * v.w);
                            adagrad_steps4(u[q][c], make_float4(G[c].x + sq.x, G[c].y + sq.y, G[c].z + sq.z, G[c].w + sq.w), A.lr, A.eps, v);
                            acc4& g = a[kHalves - 1][c];
                            g.x += (double)sq.x; g.y += (double)sq.y; g.z += (double)sq.z; g.w += (double)sq.w;
                        }
                        const double d = (double)sc[q];
                        a[0][c].x += d * (double)v.x; a[0][c].y += d * (double)v.y;
                        a[0][c].z += d * (double)v.z; a[0][c].w += d * (double)v.w;
                    }
                }
            }
        }
        // the warps' sums in warp order, parked
        double* const mine = A.parked + (uint64_t)slot * A.pieces * A.stretch_vals;
        const uint32_t per_half = tmin<uint32_t>(32 * kCh, A.F4);                // float4 from one half's sums to the other's
#pragma unroll
        for (int half = 0; half < kHalves; ++half)
#pragma unroll
            for (int c = 0; c < kCh; ++c) {
                s_part[w][lane] = a[half][c];
                __syncthreads();
                if (w == 0 && f0 + 32 * c < A.F4) {
                    acc4 tot = s_part[0][lane];
                    for (int i = 1; i < kWarps; ++i) {
                        tot.x += s_part[i][lane].x; tot.y += s_part[i][lane].y;
                        tot.z += s_part[i][lane].z; tot.w += s_part[i][lane].w;
                    }
                    double2* to2 = reinterpret_cast<double2*>(mine + (uint64_t)p * A.stretch_vals) + 2 * (half * per_half + 32 * c + lane);
                    to2[0] = make_double2(tot.x, tot.y);
                    to2[1] = make_double2(tot.z, tot.w);
                }
                __syncthreads();
            }
        if (w == 0) __threadfence();
        __syncthreads();
        if (tid == 0) {
            *s_ticket = atomicAdd(A.tickets + slot, 1u);
            if (*s_ticket == A.pieces - 1) A.tickets[slot] = 0u;                // (nobody draws it again in this call)
        }
        __syncthreads();
        if (*s_ticket != A.pieces - 1) continue;
        __threadfence();
        if (w < kHalves * kCh) {                // a warp per half and column block adds the pieces
            const uint32_t half = w / kCh, c = w % kCh, f = f0 + 32 * c;
            if (f < A.F4) {
                const double2* at2 = reinterpret_cast<const double2*>(mine) + 2 * (half * per_half + 32 * c + lane);
                acc4 tot = {0.0, 0.0, 0.0, 0.0};
#pragma unroll 8
                for (uint32_t i = 0; i < A.pieces; ++i) {
                    const double2 x = __ldcg(at2 + (uint64_t)i * (A.stretch_vals / 2)), y = __ldcg(at2 + (uint64_t)i * (A.stretch_vals / 2) + 1);
                    tot.x += x.x; tot.y += x.y; tot.z += y.x; tot.w += y.y;
                }
                float4 r = target[half * A.F4 + f];
                r.x = (float)((double)r.x + tot.x); r.y = (float)((double)r.y + tot.y);
                r.z = (float)((double)r.z + tot.z); r.w = (float)((double)r.w + tot.w);
                target[half * A.F4 + f] = r;
            }
        }
    }
}

// kCh: float4 per lane; blockIdx.y counts stretches of 32 kCh float4 of the row.  kHot: hot keys are looked for (compiled apart:
// that costs calls without any half a microsecond)
template <int kMode, int kCh, bool kHot>
__global__ void __launch_bounds__(kThreads, kCh == 1 ? 2 : 1) small_push_kernel(const SmallArgs A) {
    extern __shared__ __align__(16) uint32_t s_dyn[];
    uint32_t* const s_key = s_dyn;                          // the bucket: keys of its occurrences, in the order of the call
    uint16_t* const s_pos = reinterpret_cast<uint16_t*>(s_dyn + A.n);      // ... and their numbers
    __shared__ uint32_t t_key[kTable], t_first[kTable], t_count[kTable];
    __shared__ uint16_t s_firsts[kTable];
    __shared__ uint32_t s_cnt[kWarps], s_n_firsts, s_over;
    __shared__ acc4 s_part[kWarps * (kMode == kAdaGrad ? 2 : 1)][32];
    __shared__ uint32_t s_n_longs;                          // keys with many occurrences: the last of s_firsts, backwards
    __shared__ __align__(16) uint32_t s_sample[kHot ? kSample : 4];
    __shared__ uint32_t s_hot[kMaxHot], s_hot_mask[kWarps], s_ticket;
    constexpr int kHalves = kMode == kAdaGrad ? 2 : 1;      // AdaGrad: sums for the parameters and for their accumulators
    // update rows a warp has in flight (AdaGrad in 64 registers: two; four spill 300 bytes per thread, a step of 256 ComplEx triples of
    // 12 dimensions 24.5 us, with two 23.3, with one 23.6)
    constexpr int kFly = kCh == 1 ? (kMode == kAdaGrad ? 2 : 4) : (kCh == 2 && kMode != kAdaGrad ? 4 : 2) / (kCh == 4 ? 2 : 1);
    const unsigned full = 0xffffffffu;
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    const uint32_t n = A.n, K = A.K, n_buckets = gridDim.x - 1, bucket = blockIdx.x;
    auto key_at = [&](uint32_t i) -> uint32_t {             // kSentinelPad: out of range
        if (A.keys64) {
            const uint64_t k = A.keys64[i];
            return k < K ? (uint32_t)k : kSentinelPad;
        }
        return A.keys32[i];
    };
    pdl_trigger();
    for (int i = tid; i < kTable; i += kThreads) {
        t_key[i] = t_first[i] = kSentinelPad;
        t_count[i] = 0;
    }
    if (tid == 0) s_n_firsts = s_n_longs = s_over = 0;
    pdl_wait();
    uint32_t sample = K;
    if constexpr (kHot) {
        if (tid < (int)kSample) sample = key_at(sample_pos(tid, n));
    }
    // ---- the occurrences whose keys fall into this block's bucket; warp w looks at its 16th of the call ----
    const uint32_t rounds = (n + kThreads - 1) / kThreads;  // at most 32: lane r keeps the bucket's lanes of round r
    const uint32_t w0 = w * rounds * 32;
    uint32_t mask_of = 0, cnt_w = 0;
    int bad = 0;
#pragma unroll 8
    for (uint32_t r = 0; r < rounds; ++r) {
        const uint32_t i = w0 + r * 32 + lane;
        const uint32_t k = i < n ? key_at(i) : K;
        bad |= k == kSentinelPad;
        const unsigned m = __ballot_sync(full, k < K && bucket_of(k, n_buckets) == bucket);
        if (lane == (int)r) mask_of = m;
        cnt_w += __popc(m);
    }
    if (lane == 0) s_cnt[w] = cnt_w;
    if constexpr (kHot) {
        if (tid < (int)kSample) s_sample[tid] = sample;
    }
    if (__syncthreads_or(bad)) {                // the same decision in every block: nothing has been written yet
        if (A.keys64 && bucket == 0 && blockIdx.y == 0 && tid == 0) latch_error(A.st, 0u, PS_ERR_KEY_RANGE);
        return;
    }
    if (bucket == n_buckets) {                  // the last block adds the loss partials: strided per thread, then a tree
        if (blockIdx.y != 0 || !A.loss_accum) return;
        double* ws = reinterpret_cast<double*>(s_part);
        double t = 0;
        for (uint32_t b = tid; b < A.loss_blocks; b += kThreads) t += A.loss_partial[b];
        t = warp_sum_d(t);
        if (lane == 0) ws[w] = t;
        __syncthreads();
        if (tid == 0) {
            double tot = 0;
            for (int i = 0; i < kWarps; ++i) tot += ws[i];
            *A.loss_accum += tot;
        }
        return;
    }
    if constexpr (kHot) {                       // eight threads compare a key of the sample with all of it
        const uint32_t sampled = s_sample[tid / 8];
        uint32_t hits = 0;
#pragma unroll
        for (uint32_t i = 0; i < kSample / 32; ++i) {
            const uint4 x = reinterpret_cast<const uint4*>(s_sample)[8 * i + tid % 8];
            hits += (x.x == sampled) + (x.y == sampled) + (x.z == sampled) + (x.w == sampled);
        }
        hits += __shfl_xor_sync(full, hits, 1);
        hits += __shfl_xor_sync(full, hits, 2);
        hits += __shfl_xor_sync(full, hits, 4);
        bool is_hot = hits >= hot_hits(kCh) && sampled < K && tid % 8 == 0;
        if (__builtin_expect(__syncthreads_or(is_hot), 0)) {
            if (is_hot)                         // (its first place in the sample)
                for (int i = 0; i < tid / 8; ++i) is_hot = is_hot && s_sample[i] != sampled;
            const unsigned mine = __ballot_sync(full, is_hot);
            if (lane == 0) s_hot_mask[w] = mine;
            __syncthreads();
            uint32_t rank = __popc(mine & ((1u << lane) - 1u)), n_hot = 0;
            for (int i = 0; i < kWarps; ++i) {
                if (i < w) rank += __popc(s_hot_mask[i]);
                n_hot += __popc(s_hot_mask[i]);
            }
            n_hot = tmin(n_hot, kMaxHot);       // the same list, in the order of the sample, in every block
            if (is_hot && rank < kMaxHot) s_hot[rank] = sampled;
            __syncthreads();
            // they leave the block's list
            cnt_w = 0;
            for (unsigned some = __ballot_sync(full, mask_of != 0); some; some &= some - 1) {
                const int r = __ffs(some) - 1;
                const unsigned mk = __shfl_sync(full, mask_of, r);
                bool keep = (mk >> lane) & 1u;
                if (keep) {
                    const uint32_t k = key_at(w0 + r * 32 + lane);
                    for (uint32_t h = 0; h < n_hot; ++h) keep = keep && k != s_hot[h];
                }
                const unsigned kept = __ballot_sync(full, keep);
                if (lane == r) mask_of = kept;
                cnt_w += __popc(kept);
            }
            if (lane == 0) s_cnt[w] = cnt_w;
            hot_keys<kMode, kCh>(A, s_hot, n_hot, s_part, &s_ticket);
            __syncthreads();
        }
    }
    uint32_t at = 0, m = 0;                     // where the warp's part of the list begins; the length of the list
#pragma unroll
    for (int i = 0; i < kWarps; ++i) {
        if (i < w) at += s_cnt[i];
        m += s_cnt[i];
    }
    if (m == 0) return;
    if (cnt_w) {
        for (unsigned some = __ballot_sync(full, mask_of != 0); some; some &= some - 1) {
            const int r = __ffs(some) - 1;
            const unsigned mk = __shfl_sync(full, mask_of, r);
            if ((mk >> lane) & 1u) {
                const uint32_t i = w0 + r * 32 + lane, to = at + __popc(mk & ((1u << lane) - 1u));
                s_key[to] = key_at(i);
                s_pos[to] = (uint16_t)i;
            }
            at += __popc(mk);
        }
    }
    __syncthreads();
    // ---- first occurrence and number of occurrences of every key of the bucket ----
    auto probe = [&](uint32_t k) -> uint32_t { return (k * 0x85ebca6bu) >> (32 - kTableBits); };
    for (uint32_t i = tid; i < m; i += kThreads) {
        const uint32_t k = s_key[i];
        uint32_t s = probe(k), tries = 0;
        for (; tries < kTable; ++tries, s = (s + 1) & (kTable - 1)) {
            const uint32_t was = atomicCAS(&t_key[s], kSentinelPad, k);
            if (was == kSentinelPad || was == k) break;
        }
        if (tries == kTable) {
            s_over = 1;
        } else {
            atomicMin(&t_first[s], i);
            atomicAdd(&t_count[s], 1u);
        }
    }
    __syncthreads();
    const bool over = s_over != 0;              // more keys than the table has room for: a warp compares for itself, below
    for (uint32_t i = tid; i < m && !over; i += kThreads) {
        const uint32_t k = s_key[i];
        uint32_t s = probe(k);
        while (t_key[s] != k) s = (s + 1) & (kTable - 1);
        if (t_first[s] != i) continue;
        if (t_count[s] <= kShortRun) {
            s_firsts[atomicAdd(&s_n_firsts, 1u)] = (uint16_t)s;
            continue;
        }
        const uint32_t at = atomicAdd(&s_n_longs, 1u);
        s_firsts[kTable - 1 - at] = (uint16_t)s;
    }
    __syncthreads();
    // ---- sums ----
    const uint32_t f0 = blockIdx.y * (32 * kCh) + lane;
    // one occurrence's update row: where it is, and what it is multiplied by
    auto source = [&](uint32_t o, float& sc) -> const float4* {
        sc = 1.f;
        if (kMode == kScaled) {
            sc = A.scales[o];
            const uint32_t e = o / A.slots;
            return A.upd + (uint64_t)(2u * e + (o != e * A.slots ? 1u : 0u)) * A.F4;
        }
        return A.upd + (uint64_t)o * A.F4;
    };
    auto add = [&](acc4& a, const float4& u, double d) {
        if (kMode == kScaled) {
            a.x += d * (double)u.x; a.y += d * (double)u.y; a.z += d * (double)u.z; a.w += d * (double)u.w;
        } else {
            a.x += (double)u.x; a.y += (double)u.y; a.z += (double)u.z; a.w += (double)u.w;
        }
    };
    auto ada = [&](const float4& g, const float4& G, float4& step, float4& q) {
        q = make_float4(g.x * g.x, g.y * g.y, g.z * g.z, g.w * g.w);
        adagrad_steps4(g, make_float4(G.x + q.x, G.y + q.y, G.z + q.z, G.w + q.w), A.lr, A.eps, step);
    };
    auto finish = [&](float4 r, const acc4& a) {
        r.x = (float)((double)r.x + a.x); r.y = (float)((double)r.y + a.y);
        r.z = (float)((double)r.z + a.z); r.w = (float)((double)r.w + a.w);
        return r;
    };
    auto load_row = [&](const float4* target, float4 (*row)[kCh]) {
#pragma unroll
        for (int c = 0; c < kCh; ++c)
#pragma unroll
            for (int h = 0; h < kHalves; ++h)
                row[h][c] = f0 + 32 * c < A.F4 ? target[h * A.F4 + f0 + 32 * c] : make_float4(0.f, 0.f, 0.f, 0.f);
    };
    // the occurrences of key k among list entries [lo, hi), in order, kFly rows in flight; G: the accumulators before the call
    auto sum_range = [&](uint32_t k, uint32_t lo, uint32_t hi, acc4 (*a)[kCh], const float4* G) {
#pragma unroll
        for (int h = 0; h < kHalves; ++h)
#pragma unroll
            for (int c = 0; c < kCh; ++c) a[h][c] = acc4{0.0, 0.0, 0.0, 0.0};
        for (uint32_t b = lo; b < hi; b += 32) {
            const uint32_t e = b + lane;
            const bool hit = e < hi && s_key[e] == k;
            const uint32_t mine = hit ? s_pos[e] : 0u;
            unsigned todo = __ballot_sync(full, hit);
            while (todo) {
                float4 u[kFly][kCh];
                float sc[kFly];
                int got = 0;
#pragma unroll
                for (int q = 0; q < kFly; ++q) {
                    const int src = todo ? __ffs(todo) - 1 : 0;
                    if (todo) got = q + 1;
                    todo &= todo - 1;                       // 0 stays 0
                    const uint32_t o = __shfl_sync(full, mine, src);
                    if (q < got) {
                        const float4* p = source(o, sc[q]);
#pragma unroll
                        for (int c = 0; c < kCh; ++c)
                            u[q][c] = f0 + 32 * c < A.F4 ? p[f0 + 32 * c] : make_float4(0.f, 0.f, 0.f, 0.f);
                    }
                }
#pragma unroll
                for (int q = 0; q < kFly; ++q) {
                    if (q >= got) break;
                    const double d = (double)sc[q];
#pragma unroll
                    for (int c = 0; c < kCh; ++c) {
                        if (kMode == kAdaGrad) {
                            float4 step, sq;
                            ada(u[q][c], G[c], step, sq);
                            add(a[0][c], step, d);
                            add(a[kHalves - 1][c], sq, d);
                        } else {
                            add(a[0][c], u[q][c], d);
                        }
                    }
                }
            }
        }
    };
    // a key whose occurrences one warp adds alone: entry i of the list is the first of `count`
    auto one_key = [&](uint32_t i, uint32_t count) {
        const uint32_t k = s_key[i];
        float4* target = A.store + phys_row(A.table[k], A.S) * A.L4;
        float4 row[kHalves][kCh];
        if (count > 1) {
            acc4 a[kHalves][kCh];
            load_row(target, row);
            sum_range(k, i & ~31u, m, a, row[kHalves - 1]);
#pragma unroll
            for (int c = 0; c < kCh; ++c)
#pragma unroll
                for (int h = 0; h < kHalves; ++h)
                    if (f0 + 32 * c < A.F4) target[h * A.F4 + f0 + 32 * c] = finish(row[h][c], a[h][c]);
            return;
        }
        // one occurrence (most keys): the exact sum is rounded once in fp32
        float sc;
        const float4* p = source(s_pos[i], sc);
        float4 own[kCh];
#pragma unroll
        for (int c = 0; c < kCh; ++c) own[c] = f0 + 32 * c < A.F4 ? p[f0 + 32 * c] : make_float4(0.f, 0.f, 0.f, 0.f);
        load_row(target, row);
#pragma unroll
        for (int c = 0; c < kCh; ++c) {
            const uint32_t f = f0 + 32 * c;
            if (f >= A.F4) continue;
            float4 r = row[0][c];
            const float4 u = own[c];
            if (kMode == kAdaGrad) {
                float4 step, q, G = row[kHalves - 1][c];
                ada(u, G, step, q);
                r.x += step.x; r.y += step.y; r.z += step.z; r.w += step.w;
                G.x += q.x; G.y += q.y; G.z += q.z; G.w += q.w;
                target[A.F4 + f] = G;
            } else if (kMode == kScaled) {
                r.x = fmaf(sc, u.x, r.x); r.y = fmaf(sc, u.y, r.y); r.z = fmaf(sc, u.z, r.z); r.w = fmaf(sc, u.w, r.w);
            } else {
                r.x += u.x; r.y += u.y; r.z += u.z; r.w += u.w;
            }
            target[f] = r;
        }
    };
    if (over) {
        for (uint32_t i = w; i < m; i += kWarps) {
            const uint32_t k = s_key[i];
            uint32_t before = 0, count = 0;
            for (uint32_t e = lane; e < m; e += 32) {
                before += s_key[e] == k && e < i;
                count += s_key[e] == k;
            }
            if (!__any_sync(full, before != 0)) one_key(i, __reduce_add_sync(full, count));
        }
        return;
    }
    const uint32_t n_firsts = s_n_firsts, n_longs = s_n_longs;
    for (uint32_t j = w; j < n_firsts; j += kWarps) {
        const uint32_t s = s_firsts[j];
        one_key(t_first[s], t_count[s]);
    }
    // ---- keys with many occurrences: a range of the list per warp, partial sums added in range order; up to four keys at a time ----
    // (One after the other, all warps on each and a meeting of the block per half and column block, they took 3 to 6 us a key: the
    // last 9 of 15 us in a push of 6,000 Zipf(0.9) keys, where every fifth block has one.  That push with its pull and relocation
    // 26.6 -> 25.3 us, 8,000 of 256 values 40.2 -> 34.3, 4,000 cells of rank 64 20.8 -> 17.5, 600 ComplEx triples of 100 dimensions
    // 38.6 -> 33.1.  Four warps for every such key: 256 triples 23.2 -> 26.6, the longer ones then take eight trips.  Their rows
    // asked for ahead: no gain.)
    for (uint32_t at = 0; at < n_longs;) {      // the same decisions in every warp
        uint32_t used = 0, key_slot = kTable, first_warp = 0, warps = 0;
        for (; at < n_longs; ++at) {            // (how many warps depends on the key's count alone; what each adds also on the bucket's list: the same in every such call)
            const uint32_t s = s_firsts[kTable - 1 - at], r = long_warps(t_count[s]);
            if (used + r > (uint32_t)kWarps) break;
            if ((uint32_t)w >= used && (uint32_t)w < used + r) {
                key_slot = s;
                first_warp = used;
                warps = r;
            }
            used += r;
        }
        float4* target = nullptr;
        float4 row[kHalves][kCh];
        acc4 a[kHalves][kCh];
        if (warps) {
            const uint32_t k = t_key[key_slot];
            target = A.store + phys_row(A.table[k], A.S) * A.L4;
            load_row(target, row);
            const uint32_t per = (m + warps - 1) / warps, lo = tmin<uint32_t>((w - first_warp) * per, m);
            sum_range(k, lo, tmin<uint32_t>(lo + per, m), a, row[kHalves - 1]);
        }
#pragma unroll
        for (int c = 0; c < kCh; ++c) {
            if (warps) {
#pragma unroll
                for (int h = 0; h < kHalves; ++h) s_part[w * kHalves + h][lane] = a[h][c];
            }
            __syncthreads();                    // (every warp has read the row by now)
            const uint32_t half = w - first_warp;
            if (half < (uint32_t)kHalves && warps && f0 + 32 * c < A.F4) {      // a warp per half
                acc4 tot = s_part[first_warp * kHalves + half][lane];
                for (uint32_t i = 1; i < warps; ++i) {
                    const acc4 x = s_part[(first_warp + i) * kHalves + half][lane];
                    tot.x += x.x; tot.y += x.y; tot.z += x.z; tot.w += x.w;
                }
                float4* to = target + half * A.F4 + f0 + 32 * c;
                *to = finish(kHalves == 2 && half ? row[kHalves - 1][c] : row[0][c], tot);
            }
            __syncthreads();
        }
    }
}

template <int kMode, int kCh, bool kHot>
void launch_kernel(ps_store* ps, const SmallArgs& a, uint32_t strips, cudaStream_t s) {
    // About a dozen occurrences per block of 16 warps, two blocks per SM at most (more would only read the keys again).  Up to 48 where
    // the blocks of all stretches of columns would not be resident at once, as a second round of blocks reads the keys anew: 120
    // ComplEx triples of 1,000 dimensions 47 -> 35 us, 240 of 500 58 -> 38; pull and push of 4,000 rows of 1,024 values 28 -> 23.  Larger
    // plain calls and small skip-gram steps have hot keys that want more blocks (100 centers of 300 values 34 -> 36.6): they keep
    // the dozen.  Time with 48 over time with a dozen, pulls and pushes of 500 to 8,192 rows of 132 to 4,096 values (378 sizes): up to 4,096
    // rows 0.57 to 1.04 with uniform and Zipf(0.6) keys, 0.77 to 1.12 (median 0.89) with Zipf(1); above 0.71 to 1.07 and 0.84 to 1.11
    // (median 1.00); one stretch of 388 to 512 values above 2,560 rows 0.73 to 1.03, and 1.02 to 1.09 with Zipf(1); ComplEx steps
    // 0.69 to 1.07.
    const uint32_t wide = div_up_u32(strips, kCh), places = (uint32_t)ps->sm_count * (kCh == 1 ? 2 : 1) / wide;
    const uint32_t dozens = div_up_u32(a.n, 12), limit = (uint32_t)ps->sm_count * 2 - 1;
    const bool fewer = kMode == kAdaGrad || (kMode == kPlain && a.n <= (kCh == 4 && wide == 1 ? 2560u : 4096u));
    const uint32_t fit = fewer ? tmax<uint32_t>(places > 1 ? places - 1 : 1u, div_up_u32(a.n, 48)) : limit;
    const uint32_t buckets = tmax<uint32_t>(1u, tmin<uint32_t>(dozens, tmin<uint32_t>(fit, limit)));
    const size_t smem = ((size_t)a.n * 6 + 15) & ~(size_t)15;
    static std::atomic<unsigned long long> smem_set{0};
    opt_in_smem((const void*)small_push_kernel<kMode, kCh, kHot>, (size_t)kSmallOcc * 6, &smem_set);
    const char* name = kMode == kAdaGrad ? "small_push_kernel<adagrad>" : kMode == kScaled ? "small_push_kernel<scaled>" : "small_push_kernel";
    PS_LAUNCH_PDL(ps, name, (small_push_kernel<kMode, kCh, kHot>), dim3(buckets + 1, div_up_u32(strips, kCh)), dim3(kThreads), smem, s, a);
}
template <int kMode, int kCh>
void launch_as(ps_store* ps, const SmallArgs& a, uint32_t strips, cudaStream_t s) {
    SmallArgs b = a;
    const uint32_t stretches = div_up_u32(strips, kCh);
    b.stretch_vals = tmin<uint32_t>(32 * kCh, a.F4) * 4 * (kMode == kAdaGrad ? 2 : 1);
    const uint64_t room = (uint64_t)ps->tile_cap * 2 * ps->cfg.row_len / ((uint64_t)stretches * kMaxHot * b.stretch_vals);
    b.pieces = a.n < kHotCall || stretches > kHotStretches ? 0u : (uint32_t)tmin<uint64_t>(div_up_u32(a.n, kHotPiece), room);
    if (b.pieces < 2) return launch_kernel<kMode, kCh, false>(ps, a, strips, s);
    b.piece_len = div_up_u32(a.n, b.pieces * kWarps) * kWarps;
    launch_kernel<kMode, kCh, true>(ps, b, strips, s);
}
template <int kMode>
void launch(ps_store* ps, const SmallArgs& a, cudaStream_t s) {
    const uint32_t strips = div_up_u32(a.F4, 32);
    // Few rows: a warp per 32 float4, for latency.  Once that is more than about two waves of warps the
    // selection of the bucket, done anew for every stretch of columns, should serve more of the row.
    const bool narrow = strips == 1 || (uint64_t)a.n * strips <= (uint64_t)ps->sm_count * kWarps * 4;
    if (narrow) launch_as<kMode, 1>(ps, a, strips, s);
    else if (kMode == kAdaGrad || strips == 2) launch_as<kMode, 2>(ps, a, strips, s);
    else launch_as<kMode, kMode == kAdaGrad ? 2 : 4>(ps, a, strips, s);
}

SmallArgs common(ps_store* ps, uint32_t n, double* d_loss_accum, uint32_t loss_blocks) {
    SmallArgs a;
    memset(&a, 0, sizeof a);
    a.keys32 = small_keys(ps);
    a.n = n;
    a.K = (uint32_t)ps->cfg.num_keys;
    a.upd = (const float4*)ps->upd;
    a.store = (float4*)ps->store;
    a.table = ps->table;
    a.S = ps->cfg.slots_per_part;
    a.L4 = a.F4 = ps->cfg.row_len / 4;
    a.loss_partial = ps->loss_partial;
    a.loss_blocks = loss_blocks;
    a.loss_accum = loss_blocks ? d_loss_accum : nullptr;
    a.st = ps->status;
    a.parked = ps->carry;           // (the sorted reductions' partial sums: on the caller's stream, as all of this is)
    a.tickets = ps->hot_tickets;
    return a;
}

}  // namespace

// (the list of rows staged by the sorted matrix-factorization step: on the caller's stream, as all of this is)
uint32_t* small_keys(ps_store* ps) { return (uint32_t*)ps->apply_rows; }

void run_small_push_keys(ps_store* ps, const uint64_t* d_keys, uint32_t n, const float* d_upd, cudaStream_t s) {
    SmallArgs a = common(ps, n, nullptr, 0);
    a.keys64 = d_keys;
    a.upd = (const float4*)d_upd;
    launch<kPlain>(ps, a, s);
}

void run_small_reduce(ps_store* ps, uint32_t n, double* d_loss_accum, uint32_t loss_blocks, cudaStream_t s,
                      const float* d_scales, uint32_t slots) {
    SmallArgs a = common(ps, n, d_loss_accum, loss_blocks);
    a.scales = d_scales;
    a.slots = slots;
    if (d_scales) launch<kScaled>(ps, a, s);
    else launch<kPlain>(ps, a, s);
}

void run_small_adagrad(ps_store* ps, uint32_t n, float lr, float eps, double* d_loss_accum, uint32_t loss_blocks,
                       cudaStream_t s, const double* loss_terms) {
    SmallArgs a = common(ps, n, d_loss_accum, loss_blocks);
    if (loss_terms) a.loss_partial = loss_terms;
    a.F4 /= 2;
    a.lr = lr;
    a.eps = eps;
    launch<kAdaGrad>(ps, a, s);
}

}  // namespace psb
