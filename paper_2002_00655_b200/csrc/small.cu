// Calls of few key occurrences (kSmallOcc at most): the cumulative push without a sort.
//
// A push of a few thousand rows is a microsecond or two of memory traffic; sorted, it is a fork to another stream, a
// cooperative sort with a grid barrier per pass, a reduction and a fix-up launch: 27 us for 13 rows, of which the host
// spends 20.  Here ONE launch does it.  Every block reads all keys of the call and keeps those of its hash bucket (a
// dozen or two, in the order of the call: lane masks of the warps' shares, no sort), finds the first occurrence and the
// number of occurrences of each in a table in shared memory, and a warp per distinct key adds its occurrences' rows in
// the order of the call, in fp64, and rounds once, as the sorted reduction does.  A key with more than kShortRun
// occurrences is shared by the block's warps (a range of the list each, partial sums added in range order).
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
constexpr int kTableBits = 10, kTable = 1 << kTableBits;
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
};

// kCh: float4 per lane; blockIdx.y counts stretches of 32 kCh float4 of the row
template <int kMode, int kCh>
__global__ void __launch_bounds__(kThreads, kCh == 1 ? 2 : 1) small_push_kernel(const SmallArgs A) {
    extern __shared__ __align__(16) uint32_t s_dyn[];
    uint32_t* const s_key = s_dyn;                          // the bucket: keys of its occurrences, in the order of the call
    uint16_t* const s_pos = reinterpret_cast<uint16_t*>(s_dyn + A.n);      // ... and their numbers
    __shared__ uint32_t t_key[kTable], t_first[kTable], t_count[kTable];
    __shared__ uint16_t s_firsts[kTable];
    __shared__ uint32_t s_cnt[kWarps], s_n_firsts, s_over;
    __shared__ acc4 s_part[kWarps][32];
    constexpr int kHalves = kMode == kAdaGrad ? 2 : 1;      // AdaGrad: sums for the parameters and for their accumulators
    constexpr int kFly = kCh == 1 ? 4 : (kCh == 2 && kMode != kAdaGrad ? 4 : 2) / (kCh == 4 ? 2 : 1);      // update rows a warp has in flight
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
    if (tid == 0) s_n_firsts = s_over = 0;
    pdl_wait();
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
        if (t_first[s] == i) s_firsts[atomicAdd(&s_n_firsts, 1u)] = (uint16_t)s;
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
    const uint32_t n_firsts = s_n_firsts;
    bool any_long = false;
    for (uint32_t j = 0; j < n_firsts; ++j) {
        const uint32_t s = s_firsts[j], count = t_count[s];
        if (count > kShortRun) any_long = true;
        else if (j % kWarps == (uint32_t)w) one_key(t_first[s], count);
    }
    if (!any_long) return;                      // the same decision in every warp
    // ---- keys with many occurrences: the whole block on one at a time, a range of the list per warp ----
    const uint32_t per = (m + kWarps - 1) / kWarps, lo = tmin<uint32_t>(w * per, m), hi = tmin<uint32_t>(lo + per, m);
    for (uint32_t j = 0; j < n_firsts; ++j) {
        const uint32_t s = s_firsts[j];
        if (t_count[s] <= kShortRun) continue;
        const uint32_t k = t_key[s];
        float4* target = A.store + phys_row(A.table[k], A.S) * A.L4;
        float4 row[kHalves][kCh];
        acc4 a[kHalves][kCh];
        load_row(target, row);
        sum_range(k, lo, hi, a, row[kHalves - 1]);
#pragma unroll
        for (int h = 0; h < kHalves; ++h)
#pragma unroll
            for (int c = 0; c < kCh; ++c) {
                s_part[w][lane] = a[h][c];
                __syncthreads();                // (every warp has read the row by now)
                if (w == 0 && f0 + 32 * c < A.F4) {
                    acc4 tot = s_part[0][lane];
#pragma unroll
                    for (int i = 1; i < kWarps; ++i) {
                        tot.x += s_part[i][lane].x; tot.y += s_part[i][lane].y;
                        tot.z += s_part[i][lane].z; tot.w += s_part[i][lane].w;
                    }
                    target[h * A.F4 + f0 + 32 * c] = finish(row[h][c], tot);
                }
                __syncthreads();
            }
    }
}

template <int kMode, int kCh>
void launch_as(ps_store* ps, const SmallArgs& a, uint32_t strips, cudaStream_t s) {
    // about a dozen occurrences per block of 16 warps, two blocks per SM at most (more would only read the keys again)
    const uint32_t buckets = tmax<uint32_t>(1u, tmin<uint32_t>(div_up_u32(a.n, 12), (uint32_t)ps->sm_count * 2 - 1));
    const size_t smem = ((size_t)a.n * 6 + 15) & ~(size_t)15;
    static std::atomic<unsigned long long> smem_set{0};
    opt_in_smem((const void*)small_push_kernel<kMode, kCh>, (size_t)kSmallOcc * 6, &smem_set);
    const char* name = kMode == kAdaGrad ? "small_push_kernel<adagrad>" : kMode == kScaled ? "small_push_kernel<scaled>" : "small_push_kernel";
    PS_LAUNCH_PDL(ps, name, (small_push_kernel<kMode, kCh>), dim3(buckets + 1, div_up_u32(strips, kCh)), dim3(kThreads), smem, s, a);
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
