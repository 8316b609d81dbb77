// Calls of few key occurrences (kSmallOcc at most): the cumulative push without a sort.
//
// A push of a few thousand rows is a microsecond or two of memory traffic; sorted, it is a fork to another stream, a
// cooperative sort with a grid barrier per pass, a reduction and a fix-up launch, 27 us of which the host spends 20
// (push of 13 rows).  Here ONE launch does it: every block reads all keys of the call into shared memory (16 KB at
// most), a warp takes one occurrence, compares its key with all the others (32 x 4 keys per instruction) and is done if
// an earlier occurrence has the same key; otherwise the occurrence is the first of its key and the warp adds the rows of
// all of them, in the order of the call, in fp64, and rounds once, as the sorted reduction does.  The comparison costs n^2 / 128
// warp instructions in all, a microsecond at 4,096 keys, and twice the keys would cost four times that: the limit.
// A key with more than kShortRun occurrences is shared by the block's warps (a range of the keys each, partial sums
// added in range order), so one hot key costs n / 16 rows of latency and not n.
//
// Training steps take the same launch after their gradient kernel, which leaves the key of every occurrence slot in
// a buffer (num_keys: no key; all ones: an index out of range, the whole call is a no-op).
#include <string.h>

#include "ps_internal.cuh"

namespace psb {

namespace {

constexpr int kThreads = 512;
constexpr int kWarps = kThreads / 32;
constexpr uint32_t kShortRun = 64;              // occurrences of one key that a warp adds alone
constexpr uint32_t kRange = kSmallOcc / kWarps; // keys per warp in the shared walk

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
__global__ void __launch_bounds__(kThreads) small_push_kernel(const SmallArgs A) {
    __shared__ __align__(16) uint32_t s_key[kSmallOcc];
    __shared__ uint16_t s_list[kWarps][kRange];
    __shared__ uint32_t s_long[kWarps];         // the warp's occurrence starts a long run
    __shared__ acc4 s_part[kWarps][32];
    constexpr int kHalves = kMode == kAdaGrad ? 2 : 1;      // AdaGrad: sums for the parameters and for their accumulators
    const unsigned full = 0xffffffffu;
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    const uint32_t n = A.n, K = A.K;
    const uint32_t n_pad = (n + 127) & ~127u;
    int bad = 0;
    for (uint32_t i = tid; i < n_pad; i += kThreads) {
        uint32_t k = K;
        if (i < n) {
            if (A.keys64) {
                const uint64_t k64 = A.keys64[i];
                bad |= k64 >= K;
                k = (uint32_t)k64;
            } else {
                k = A.keys32[i];
                bad |= k == kSentinelPad;
            }
        }
        s_key[i] = k;
    }
    if (__syncthreads_or(bad)) {                // the same decision in every block: nothing has been written yet
        if (A.keys64 && blockIdx.x == 0 && blockIdx.y == 0 && tid == 0) latch_error(A.st, 0u, PS_ERR_KEY_RANGE);
        return;
    }
    if (blockIdx.x == gridDim.x - 1) {          // the last block adds the loss partials: strided per thread, then a tree
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
    const uint32_t f0 = blockIdx.y * (32 * kCh) + lane;
    const uint32_t t = blockIdx.x * kWarps + w;
    const uint32_t my = t < n ? s_key[t] : K;
    const bool usable = my < K;
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
    // Asked for before the keys are compared, used after: the target row and this occurrence's own update.
    float4 row[kHalves][kCh], own[kCh];
    float own_sc = 1.f;
    float4* target = A.store;
    if (usable) {
        target = A.store + phys_row(A.table[my], A.S) * A.L4;
        const float4* u = source(t, own_sc);
#pragma unroll
        for (int c = 0; c < kCh; ++c) {
            const uint32_t f = f0 + 32 * c;
            own[c] = f < A.F4 ? u[f] : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
            for (int h = 0; h < kHalves; ++h)
                row[h][c] = f < A.F4 ? target[h * A.F4 + f] : make_float4(0.f, 0.f, 0.f, 0.f);
        }
    }
    bool earlier = false;
    uint32_t same = 0;
    const uint4* k4 = reinterpret_cast<const uint4*>(s_key);
#pragma unroll 4
    for (uint32_t b = 0; b < n_pad; b += 128) {
        const uint4 q = k4[b / 4 + lane];
        const uint32_t i = b + 4 * lane;
        same += (q.x == my) + (q.y == my) + (q.z == my) + (q.w == my);
        earlier |= (q.x == my && i < t) || (q.y == my && i + 1 < t) || (q.z == my && i + 2 < t) || (q.w == my && i + 3 < t);
    }
    same = __reduce_add_sync(full, same);
    const bool first = usable && !__any_sync(full, earlier);
    const bool is_long = first && same > kShortRun;
    if (lane == 0) s_long[w] = is_long;
    // positions of a key's occurrences among keys [lo, hi), ascending, into the warp's list; how many
    auto find = [&](uint32_t key, uint32_t lo, uint32_t hi) -> uint32_t {
        const unsigned lt = (1u << lane) - 1u;
        uint32_t cnt = 0;
        for (uint32_t b = lo; b < hi; b += 128) {
            const uint32_t i = b + 4 * lane;
            const uint4 q = i < hi ? k4[i / 4] : make_uint4(kSentinelPad, kSentinelPad, kSentinelPad, kSentinelPad);
            const bool m0 = q.x == key, m1 = q.y == key, m2 = q.z == key, m3 = q.w == key;
            const unsigned b0 = __ballot_sync(full, m0), b1 = __ballot_sync(full, m1), b2 = __ballot_sync(full, m2),
                           b3 = __ballot_sync(full, m3);
            uint32_t at = cnt + __popc(b0 & lt) + __popc(b1 & lt) + __popc(b2 & lt) + __popc(b3 & lt);
            if (m0) s_list[w][at++] = (uint16_t)i;
            if (m1) s_list[w][at++] = (uint16_t)(i + 1);
            if (m2) s_list[w][at++] = (uint16_t)(i + 2);
            if (m3) s_list[w][at++] = (uint16_t)(i + 3);
            cnt += __popc(b0) + __popc(b1) + __popc(b2) + __popc(b3);
        }
        __syncwarp();
        return cnt;
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
        step = make_float4(adagrad_step(g.x, G.x + q.x, A.lr, A.eps), adagrad_step(g.y, G.y + q.y, A.lr, A.eps),
                           adagrad_step(g.z, G.z + q.z, A.lr, A.eps), adagrad_step(g.w, G.w + q.w, A.lr, A.eps));
    };
    auto finish = [&](float4 r, const acc4& a) {
        r.x = (float)((double)r.x + a.x); r.y = (float)((double)r.y + a.y);
        r.z = (float)((double)r.z + a.z); r.w = (float)((double)r.w + a.w);
        return r;
    };
    // the warp's list summed into a[][], several occurrences' rows in flight; G: the accumulators before the call
    auto sum_list = [&](uint32_t cnt, acc4 (*a)[kCh], const float4* G, int n_ch, uint32_t fa) {
        constexpr int kFly = kCh == 4 ? 2 : 4;
        for (uint32_t j = 0; j < cnt; j += kFly) {
            float4 u[kFly][kCh];
            float sc[kFly];
#pragma unroll
            for (int k = 0; k < kFly; ++k) {
                const float4* p = source(s_list[w][j + k < cnt ? j + k : j], sc[k]);
#pragma unroll
                for (int c = 0; c < kCh; ++c)
                    u[k][c] = (c < n_ch && fa + 32 * c < A.F4) ? p[fa + 32 * c] : make_float4(0.f, 0.f, 0.f, 0.f);
            }
#pragma unroll
            for (int k = 0; k < kFly; ++k) {
                if (j + k >= cnt) break;
                const double d = (double)sc[k];
#pragma unroll
                for (int c = 0; c < kCh; ++c) {
                    if (c >= n_ch) break;
                    if (kMode == kAdaGrad) {
                        float4 step, q;
                        ada(u[k][c], G[c], step, q);
                        add(a[0][c], step, d);
                        add(a[kHalves - 1][c], q, d);
                    } else {
                        add(a[0][c], u[k][c], d);
                    }
                }
            }
        }
    };
    if (first && same == 1) {                   // most keys: the exact sum is rounded once in fp32
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
                r.x = fmaf(own_sc, u.x, r.x); r.y = fmaf(own_sc, u.y, r.y);
                r.z = fmaf(own_sc, u.z, r.z); r.w = fmaf(own_sc, u.w, r.w);
            } else {
                r.x += u.x; r.y += u.y; r.z += u.z; r.w += u.w;
            }
            target[f] = r;
        }
    } else if (first && !is_long) {
        const uint32_t cnt = find(my, t & ~127u, n_pad);
        acc4 a[kHalves][kCh];
#pragma unroll
        for (int h = 0; h < kHalves; ++h)
#pragma unroll
            for (int c = 0; c < kCh; ++c) a[h][c] = acc4{0.0, 0.0, 0.0, 0.0};
        sum_list(cnt, a, row[kHalves - 1], kCh, f0);
#pragma unroll
        for (int c = 0; c < kCh; ++c) {
            const uint32_t f = f0 + 32 * c;
            if (f >= A.F4) continue;
#pragma unroll
            for (int h = 0; h < kHalves; ++h) target[h * A.F4 + f] = finish(row[h][c], a[h][c]);
        }
    }
    __syncthreads();
    for (int j = 0; j < kWarps; ++j) {          // long runs: the whole block on one key at a time
        if (!s_long[j]) continue;               // the same decision in every warp
        const uint32_t key = s_key[blockIdx.x * kWarps + j];
        float4* dst = A.store + phys_row(A.table[key], A.S) * A.L4;
        const uint32_t lo = tmin<uint32_t>(w * kRange, n_pad), hi = tmin<uint32_t>(lo + kRange, n_pad);
        const uint32_t cnt = find(key, lo, hi);
        for (int c = 0; c < kCh; ++c) {
            const uint32_t f = f0 + 32 * c;
            float4 r[kHalves];
#pragma unroll
            for (int h = 0; h < kHalves; ++h) r[h] = f < A.F4 ? dst[h * A.F4 + f] : make_float4(0.f, 0.f, 0.f, 0.f);
            acc4 a[kHalves][kCh];
#pragma unroll
            for (int h = 0; h < kHalves; ++h) a[h][0] = acc4{0.0, 0.0, 0.0, 0.0};
            sum_list(cnt, a, r + kHalves - 1, 1, f);
#pragma unroll
            for (int h = 0; h < kHalves; ++h) {
                s_part[w][lane] = a[h][0];
                __syncthreads();                // (every warp has read the row by now)
                if (w == 0 && f < A.F4) {
                    acc4 tot = s_part[0][lane];
#pragma unroll
                    for (int i = 1; i < kWarps; ++i) {
                        tot.x += s_part[i][lane].x; tot.y += s_part[i][lane].y;
                        tot.z += s_part[i][lane].z; tot.w += s_part[i][lane].w;
                    }
                    dst[h * A.F4 + f] = finish(r[h], tot);
                }
                __syncthreads();
            }
        }
    }
}

template <int kMode>
void launch(ps_store* ps, const SmallArgs& a, cudaStream_t s) {
    const uint32_t strips = div_up_u32(a.F4, 32);
    const uint32_t bx = div_up_u32(a.n, kWarps) + 1;
    // Few rows: a warp per 32 float4, for latency.  Once that is more than about two waves of warps the
    // comparison of the keys, done anew for every stretch of columns, should serve more of the row.
    const bool narrow = strips == 1 || (uint64_t)a.n * strips <= (uint64_t)ps->sm_count * kWarps * 4;
    if (narrow) PS_LAUNCH(ps, (small_push_kernel<kMode, 1>), dim3(bx, strips), kThreads, s, a);
    else if (strips == 2) PS_LAUNCH(ps, (small_push_kernel<kMode, 2>), dim3(bx, 1), kThreads, s, a);
    else if (kMode == kAdaGrad) PS_LAUNCH(ps, (small_push_kernel<kMode, 2>), dim3(bx, div_up_u32(strips, 2)), kThreads, s, a);
    else PS_LAUNCH(ps, (small_push_kernel<kMode, kMode == kAdaGrad ? 2 : 4>), dim3(bx, div_up_u32(strips, 4)), kThreads, s, a);
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
                       cudaStream_t s) {
    SmallArgs a = common(ps, n, d_loss_accum, loss_blocks);
    a.F4 /= 2;
    a.lr = lr;
    a.eps = eps;
    launch<kAdaGrad>(ps, a, s);
}

}  // namespace psb
