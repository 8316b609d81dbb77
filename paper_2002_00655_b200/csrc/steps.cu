// Fused pull -> per-example gradient kernels of the matrix-factorization and
// skip-gram tasks of Section 4.1 / Appendix A of the paper (ComplEx: complex.cu,
// RESCAL: rescal.cu).  One warp handles one example (a matrix cell, a skip-gram
// center word with its window): it looks the example's keys up in the location
// table, gathers their rows with coalesced loads, forms dot products with warp
// shuffles, and writes one additive update row per key occurrence (skip-gram:
// two rows and the occurrences' factors).  The push stage then sums them per key
// and applies them: pull_push.cu on the sorted occurrences, small.cu for calls of
// few, whose keys are written here too.  Every read sees the state from before the
// step: a row is only updated here, in place, if its key occurs once in the batch.
#include "ps_internal.cuh"

namespace psb {

__device__ __forceinline__ float softplusf(float z) { return fmaxf(z, 0.f) + log1pf(expf(-fabsf(z))); }
__device__ __forceinline__ float sigmoidf(float z) {
    const float e = expf(-fabsf(z));
    return (z >= 0.f ? 1.f : e) / (1.f + e);
}

// Sum of the warps' loss terms -> loss_partial[blockIdx.x]; fixed order.
__device__ __forceinline__ void block_loss_out(double loss, double* __restrict__ loss_partial) {
    __shared__ double wl[8];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    if (lane == 0) wl[w] = loss;
    __syncthreads();
    if (threadIdx.x == 0) {
        double t = 0;
        for (int i = 0; i < (int)(blockDim.x >> 5); ++i) t += wl[i];
        loss_partial[blockIdx.x] = t;
    }
}

// blocks_per_sm: how many blocks of the kernel an SM holds.  With exactly the resident number of blocks every warp
// loops over its share of the examples, and the shares differ by at most one example; with more blocks than fit, the
// last wave is partly empty.
static uint32_t step_grid(ps_store* ps, uint64_t n_examples, uint32_t blocks_per_sm = 8) {
    uint64_t g = (n_examples + 7) / 8;
    const uint64_t cap = (uint64_t)ps->sm_count * blocks_per_sm;
    if (g > cap) g = cap;
    if (g > kMaxLossBlocks) g = kMaxLossBlocks;
    return g ? (uint32_t)g : 1u;
}

// ------------------------------------------------------------------ MF ----
// kCh = number of float4 a lane holds per row (row_len <= 128 * kCh); 0 = any
// row length, rows re-read from cache for the second pass.
template <int kCh>
__global__ void __launch_bounds__(256)
mf_step_kernel(const uint32_t* ci, const uint32_t* cj, const float* cv,
               uint64_t n, uint64_t col_base, float lr, float lam, const float4* store,
               const uint2* table, uint64_t S, uint64_t K, uint32_t L4,
               float4* __restrict__ upd, uint32_t* keys_out, double* __restrict__ loss_partial,
               DevStatus* st, unsigned int epoch) {
    const int lane = threadIdx.x & 31;
    const uint64_t warp = ((uint64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const uint64_t n_warps = ((uint64_t)gridDim.x * blockDim.x) >> 5;
    constexpr int kRegs = kCh > 0 ? kCh : 1;
    double loss = 0;
    pdl_trigger();
    pdl_wait();
    for (uint64_t t = warp; t < n; t += n_warps) {
        const uint32_t i = ci[t], j = cj[t];
        const float v = cv[t];
        const uint64_t kw = i, kh = col_base + j;
        const bool bad = kw >= col_base || kh >= K;
        if (keys_out && lane < 2) keys_out[2 * t + lane] = bad ? kSentinelPad : (uint32_t)(lane ? kh : kw);
        if (bad) {
            if (lane == 0) latch_error(st, epoch, PS_ERR_KEY_RANGE);
            continue;
        }
        const float4* W = store + phys_row(table[kw], S) * L4;
        const float4* H = store + phys_row(table[kh], S) * L4;
        float4 w[kRegs], h[kRegs];
        float dot = 0.f, nw = 0.f, nh = 0.f;
        if constexpr (kCh > 0) {
#pragma unroll
            for (int c = 0; c < kCh; ++c) {
                const uint32_t f = lane + 32 * c;
                w[c] = f < L4 ? W[f] : make_float4(0.f, 0.f, 0.f, 0.f);
                h[c] = f < L4 ? H[f] : make_float4(0.f, 0.f, 0.f, 0.f);
            }
#pragma unroll
            for (int c = 0; c < kCh; ++c) {
                dot += w[c].x * h[c].x + w[c].y * h[c].y + w[c].z * h[c].z + w[c].w * h[c].w;
                nw += w[c].x * w[c].x + w[c].y * w[c].y + w[c].z * w[c].z + w[c].w * w[c].w;
                nh += h[c].x * h[c].x + h[c].y * h[c].y + h[c].z * h[c].z + h[c].w * h[c].w;
            }
        } else {
            for (uint32_t f = lane; f < L4; f += 32) {
                const float4 a = W[f], b = H[f];
                dot += a.x * b.x + a.y * b.y + a.z * b.z + a.w * b.w;
                nw += a.x * a.x + a.y * a.y + a.z * a.z + a.w * a.w;
                nh += b.x * b.x + b.y * b.y + b.z * b.z + b.w * b.w;
            }
        }
        dot = warp_sum(dot);
        nw = warp_sum(nw);
        nh = warp_sum(nh);
        const float e = v - dot;
        loss += (double)(0.5f * e * e + 0.5f * lam * (nw + nh));
        float4* UW = upd + (2 * t) * L4;
        float4* UH = upd + (2 * t + 1) * L4;
        auto emit = [&](uint32_t f, const float4& a, const float4& b) {
            float4 dw, dh;
            dw.x = lr * (e * b.x - lam * a.x); dw.y = lr * (e * b.y - lam * a.y);
            dw.z = lr * (e * b.z - lam * a.z); dw.w = lr * (e * b.w - lam * a.w);
            dh.x = lr * (e * a.x - lam * b.x); dh.y = lr * (e * a.y - lam * b.y);
            dh.z = lr * (e * a.z - lam * b.z); dh.w = lr * (e * a.w - lam * b.w);
            UW[f] = dw;
            UH[f] = dh;
        };
        if constexpr (kCh > 0) {
#pragma unroll
            for (int c = 0; c < kCh; ++c) {
                const uint32_t f = lane + 32 * c;
                if (f < L4) emit(f, w[c], h[c]);
            }
        } else {
            for (uint32_t f = lane; f < L4; f += 32) emit(f, W[f], H[f]);
        }
    }
    block_loss_out(loss, loss_partial);
}

// Rows of at most 128 values: one float4 per lane and row.  A warp works on kCells cells at a time so
// that their index, table and row loads are all in flight together (each cell is a chain of three
// dependent loads; one cell per warp leaves the memory system idle most of the time).
template <int kCells>
__global__ void __launch_bounds__(256)
mf_step_small_kernel(const uint32_t* ci, const uint32_t* cj, const float* cv,
                     uint64_t n, uint64_t col_base, float lr, float lam, const float4* store,
                     const uint2* table, uint64_t S, uint64_t K, uint32_t L4,
                     float4* __restrict__ upd, uint32_t* keys_out, double* __restrict__ loss_partial,
                     DevStatus* st, unsigned int epoch) {
    const int lane = threadIdx.x & 31;
    const uint64_t warp = ((uint64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const uint64_t n_warps = ((uint64_t)gridDim.x * blockDim.x) >> 5;
    const bool act = (uint32_t)lane < L4;
    double loss = 0;
    pdl_trigger();
    pdl_wait();
    for (uint64_t t0 = warp * kCells; t0 < n; t0 += n_warps * kCells) {
        uint64_t kw[kCells], kh[kCells];
        float v[kCells];
        bool ok[kCells];
#pragma unroll
        for (int c = 0; c < kCells; ++c) {
            const uint64_t t = t0 + c;
            ok[c] = t < n;
            kw[c] = ok[c] ? ci[t] : 0;
            kh[c] = ok[c] ? col_base + cj[t] : 0;
            v[c] = ok[c] ? cv[t] : 0.f;
            const bool bad = ok[c] && (kw[c] >= col_base || kh[c] >= K);
            if (keys_out && ok[c] && lane < 2) keys_out[2 * t + lane] = bad ? kSentinelPad : (uint32_t)(lane ? kh[c] : kw[c]);
            if (bad) {
                if (lane == 0) latch_error(st, epoch, PS_ERR_KEY_RANGE);
                ok[c] = false;
            }
        }
        uint2 ew[kCells], eh[kCells];
#pragma unroll
        for (int c = 0; c < kCells; ++c) {
            ew[c] = ok[c] ? table[kw[c]] : make_uint2(0, 0);
            eh[c] = ok[c] ? table[kh[c]] : make_uint2(0, 0);
        }
        float4 w[kCells], h[kCells];
#pragma unroll
        for (int c = 0; c < kCells; ++c) {
            const bool ld = ok[c] && act;
            w[c] = ld ? store[phys_row(ew[c], S) * L4 + lane] : make_float4(0.f, 0.f, 0.f, 0.f);
            h[c] = ld ? store[phys_row(eh[c], S) * L4 + lane] : make_float4(0.f, 0.f, 0.f, 0.f);
        }
#pragma unroll
        for (int c = 0; c < kCells; ++c) {
            float dot = w[c].x * h[c].x + w[c].y * h[c].y + w[c].z * h[c].z + w[c].w * h[c].w;
            float nw = w[c].x * w[c].x + w[c].y * w[c].y + w[c].z * w[c].z + w[c].w * w[c].w;
            float nh = h[c].x * h[c].x + h[c].y * h[c].y + h[c].z * h[c].z + h[c].w * h[c].w;
            dot = warp_sum(dot);
            nw = warp_sum(nw);
            nh = warp_sum(nh);
            if (!ok[c]) continue;
            const float e = v[c] - dot;
            loss += (double)(0.5f * e * e + 0.5f * lam * (nw + nh));
            if (act) {
                const uint64_t t = t0 + c;
                float4 dw, dh;
                dw.x = lr * (e * h[c].x - lam * w[c].x); dw.y = lr * (e * h[c].y - lam * w[c].y);
                dw.z = lr * (e * h[c].z - lam * w[c].z); dw.w = lr * (e * h[c].w - lam * w[c].w);
                dh.x = lr * (e * w[c].x - lam * h[c].x); dh.y = lr * (e * w[c].y - lam * h[c].y);
                dh.z = lr * (e * w[c].z - lam * h[c].z); dh.w = lr * (e * w[c].w - lam * h[c].w);
                upd[(2 * t) * L4 + lane] = dw;
                upd[(2 * t + 1) * L4 + lane] = dh;
            }
        }
    }
    block_loss_out(loss, loss_partial);
}

uint32_t launch_step_mf(ps_store* ps, const uint32_t* d_i, const uint32_t* d_j, const float* d_v, uint64_t n,
                        uint64_t col_key_base, float lr, float lambda, uint32_t* keys_out, cudaStream_t s) {
    const uint32_t L4 = ps->cfg.row_len / 4;
    const uint32_t grid = step_grid(ps, n);
    const uint32_t epoch = keys_out ? 0u : ps->epoch;
#define MF_ARGS d_i, d_j, d_v, n, col_key_base, lr, lambda, (const float4*)ps->store, ps->table,                 \
                ps->cfg.slots_per_part, ps->cfg.num_keys, L4, (float4*)ps->upd, keys_out, ps->loss_partial,    \
                ps->status, epoch
    // (a warp per cell for the calls without a sort: they do not fill the chip with four cells a warp)
#define MF_LAUNCH(kernel)                                                                                          \
    do {                                                                                                         \
        if (keys_out) PS_LAUNCH_PDL(ps, #kernel, kernel, dim3(grid), dim3(256), 0, s, MF_ARGS);                    \
        else PS_LAUNCH(ps, kernel, grid, 256, s, MF_ARGS);                                                         \
    } while (0)
    if (L4 <= 32 && keys_out) MF_LAUNCH(mf_step_small_kernel<1>);
    else if (L4 <= 32) MF_LAUNCH(mf_step_small_kernel<4>);
    else if (L4 <= 64) MF_LAUNCH(mf_step_kernel<2>);
    else if (L4 <= 128) MF_LAUNCH(mf_step_kernel<4>);
    else MF_LAUNCH(mf_step_kernel<0>);
#undef MF_LAUNCH
#undef MF_ARGS
    return grid;
}

// ---------------------------------------------------------------- SGNS ----
// number of (center, context) pairs of all centers before position p
__host__ __device__ __forceinline__ uint64_t sgns_pairs_before(uint64_t p, uint64_t T, uint64_t W) {
    // left contexts: sum over q < p of min(q, W)
    const uint64_t m = p < W ? p : W;
    const uint64_t left = m * (m - (m > 0)) / 2 + (p - m) * W;
    // right contexts: sum over q < p of min(T - 1 - q, W)
    const uint64_t full = T > W ? (p < T - W ? p : T - W) : 0;
    const uint64_t rest = p - full;
    const uint64_t first = T - 1 - full;                    // value at q = full (only used if rest > 0)
    const uint64_t right = full * W + (rest ? rest * first - rest * (rest - 1) / 2 : 0);
    return left + right;
}

// rows worked on together: as many as leave 128 registers without spills
__host__ __device__ constexpr int sgns_quad(int kCh) { return kCh == 4 ? 2 : kCh == 1 ? 8 : 4; }

// Occurrence slots of center number c of the batch: slot_base = c * (1 + 2W(1 + n_neg));
// slot_base = the center's input vector; then per context j (ascending position) 1 + n_neg output vectors.
// The update of an output vector is a multiple of the center's input vector, the same vector for all of
// the center's slots, so it is not written out per slot: the kernel writes, per center, two source rows
// (2c: the summed update of the input vector; 2c + 1: a copy of the input vector as it was before the
// batch) and one factor per slot (1 for slot 0); the reduction multiplies as it adds.
// A warp takes one center at a time.  The output-vector slots are handled 32 at a time: every lane first
// resolves one slot (word -> key -> table entry -> row address), so those lookups are in flight together;
// the rows are then read kQuad slots at a time, all their loads before the first dot product.
// kOnce: rows whose key occurs once in the batch (`single`, per slot) are updated here, in place, with the values in hand; a
// third of the skip-gram batch's occurrences, each of which cost the reduction three rows of traffic.
template <int kCh, bool kOnce>
__global__ void __launch_bounds__(256, 2)
sgns_step_kernel(const uint32_t* tokens, uint64_t tok_first, uint64_t first_pos, uint64_t n_centers,
                 uint64_t T, uint32_t window, const uint32_t* negs, uint32_t n_neg, uint64_t out_base,
                 float lr, float4* store, const uint2* table, uint64_t S, uint64_t K, const uint8_t* single,
                 uint32_t L4, float4* __restrict__ upd, float* __restrict__ scales, uint32_t* keys_out,
                 double* __restrict__ loss_partial, DevStatus* st, unsigned int epoch) {
    const unsigned full = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    const uint64_t warp = ((uint64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const uint64_t n_warps = ((uint64_t)gridDim.x * blockDim.x) >> 5;
    const uint32_t per_ctx = 1 + n_neg;
    const uint64_t slots = 1 + (uint64_t)2 * window * per_ctx;
    const uint64_t pairs0 = sgns_pairs_before(first_pos, T, window);
    constexpr int kQuad = sgns_quad(kCh);
    constexpr int kLanes = 32 / kQuad;
    // (rows of more than 128 (kCh - 1) values: the dispatch's rule; only the last column block needs the comparison)
    auto in_row = [&](int c) { return c + 1 < kCh || lane + 32 * c < L4; };
    // Rows of more than 512 bytes arrive in shared memory as bulk copies, two groups of kQuad of them on their way while one
    // is worked on from registers: [warp][2][kQuad][L4].  (With loads straight into the registers one group was on its way, and
    // that only between two groups' arithmetic: 295 us for 32,768 centers of 300 values at 4.6 TB/s of DRAM, now 265.)
    constexpr bool kStage = kCh >= 2;
    extern __shared__ __align__(128) float4 sgns_stage[];
    __shared__ __align__(8) uint64_t bars[8][2];
    const int w = threadIdx.x >> 5;
    float4* const ring = sgns_stage + (size_t)w * (2 * kQuad) * L4;
    if (kStage) {
        if (lane < 2) mbar_init(&bars[w][lane], 1);
        mbar_init_fence();
        __syncwarp();
    }
    unsigned uses = 0;                                          // parity of each stage's barrier
    bool dead = false;
    float4 u[kQuad][kCh];                                       // (elements past the row are never loaded: zero throughout)
#pragma unroll
    for (int a = 0; a < kQuad; ++a)
#pragma unroll
        for (int c = 0; c < kCh; ++c) u[a][c] = make_float4(0.f, 0.f, 0.f, 0.f);
    double loss = 0;
    pdl_trigger();
    pdl_wait();
    if (kOnce && call_failed(st, epoch)) return;        // (the key kernel found an index out of range: nothing may be written)
    // the word of slot t of a center at position p with n_left contexts before it, the first at lo, pairs from z0 on
    auto word_of = [&](uint64_t lo, uint32_t n_left, uint64_t z0, uint32_t t) {
        const uint32_t j = t / per_ctx, i = t - j * per_ctx;
        const uint64_t q = j < n_left ? lo + j : lo + j + 1;                    // skip the center itself
        return i == 0 ? tokens[q - tok_first] : negs[(z0 + j) * n_neg + (i - 1)];
    };
    // Words asked for ahead of their use: this lane's of the coming round and, in a center's last round, the next center's (the
    // negatives come from memory: 265 -> 259 us for 32,768 centers of 300 values, in a form compiled for that shape; 270 without it).
    uint32_t word_next = 0, wtok_next = 0;
    bool have = false;
    for (uint64_t cidx = warp; cidx < n_centers && !dead; cidx += n_warps) {
        const uint64_t p = first_pos + cidx;
        const uint64_t lo = p >= window ? p - window : 0;
        const uint64_t hi = p + window < T ? p + window : T - 1;
        const uint64_t z0 = sgns_pairs_before(p, T, window) - pairs0;
        const uint32_t n_left = (uint32_t)(p - lo);
        const uint32_t n_out = (uint32_t)(hi - lo) * per_ctx;   // contexts (the center itself excluded) x (1 + n_neg)
        float4* U = upd + cidx * 2 * L4;
        float* F = scales + cidx * slots;
        const uint32_t wtok = have ? wtok_next : tokens[p - tok_first];
        bool word_ready = have;
        have = false;
        if (keys_out) {                                         // (slots of contexts cut off at the stream's ends: no key)
            if (lane == 0) keys_out[cidx * slots] = wtok < out_base ? wtok : kSentinelPad;
            for (uint32_t t = n_out + lane; t + 1 < slots; t += 32) keys_out[cidx * slots + 1 + t] = (uint32_t)K;
        }
        if (wtok >= out_base) {
            if (lane == 0) latch_error(st, epoch, PS_ERR_KEY_RANGE);
            continue;
        }
        float4* V = store + phys_row(table[wtok], S) * L4;
        const bool center_once = kOnce && single[cidx * slots];
        float4 v[kCh], dv[kCh];
#pragma unroll
        for (int c = 0; c < kCh; ++c) {
            const uint32_t f = lane + 32 * c;
            v[c] = in_row(c) ? V[f] : make_float4(0.f, 0.f, 0.f, 0.f);
            dv[c] = make_float4(0.f, 0.f, 0.f, 0.f);
        }
        bool bad = false;
        for (uint32_t t0 = 0; t0 < n_out && !dead; t0 += 32) {
            // this lane's slot of the round
            const uint32_t t = t0 + lane;
            uint64_t my_row = 0;
            bool my_ok = false;
            if (t < n_out) {
                const uint64_t ku = out_base + (word_ready ? word_next : word_of(lo, n_left, z0, t));
                if (ku < K) {
                    my_row = phys_row(table[ku], S);
                    my_ok = true;
                } else {
                    bad = true;
                }
                if (keys_out) keys_out[cidx * slots + 1 + t] = my_ok ? (uint32_t)ku : kSentinelPad;
            }
            const unsigned ok_mask = __ballot_sync(full, my_ok);
            const unsigned once_mask = kOnce ? __ballot_sync(full, my_ok && single[cidx * slots + 1 + t]) : 0u;
            const uint32_t in_round = tmin<uint32_t>(32u, n_out - t0);
            word_ready = true;
            if (t0 + 32 < n_out) {
                if (t + 32 < n_out) word_next = word_of(lo, n_left, z0, t + 32);
            } else if (cidx + n_warps < n_centers) {
                const uint64_t p2 = p + n_warps, lo2 = p2 >= window ? p2 - window : 0, hi2 = p2 + window < T ? p2 + window : T - 1;
                wtok_next = tokens[p2 - tok_first];
                if (lane < (uint32_t)(hi2 - lo2) * per_ctx)
                    word_next = word_of(lo2, (uint32_t)(p2 - lo2), sgns_pairs_before(p2, T, window) - pairs0, lane);
                have = true;
            }
            float my_scale = 0.f, my_x = 0.f;                                   // factor and score of this lane's slot
            auto ask = [&](uint32_t b) {                                        // the rows of slots b .. b + kQuad
                const unsigned group = (ok_mask >> b) & ((1u << kQuad) - 1u);
                if (b >= in_round || group == 0) return;
                const uint32_t stage = (b / kQuad) & 1;
                if (lane == (int)b) mbar_expect_tx(&bars[w][stage], __popc(group) * L4 * 16);
                __syncwarp();
                if (my_ok && lane - b < kQuad) bulk_g2s(ring + (stage * kQuad + (lane - b)) * L4, store + my_row * L4, L4 * 16, &bars[w][stage]);
            };
            if (kStage) {
                ask(0);
                ask(kQuad);
            }
            for (uint32_t b = 0; b < in_round; b += kQuad) {
                if (kStage && ((ok_mask >> b) & ((1u << kQuad) - 1u))) {
                    const uint32_t stage = (b / kQuad) & 1;
                    if (!mbar_wait(&bars[w][stage], (uses >> stage) & 1u) && !mbar_wait(&bars[w][stage], (uses >> stage) & 1u)) {
                        if (lane == 0) latch_error(st, epoch, PS_ERR_CUDA);
                        dead = true;                                            // a copy that does not arrive: give the call up
                        break;
                    }
                    uses ^= 1u << stage;
#pragma unroll
                    for (int a = 0; a < kQuad; ++a)                             // (a slot without a row: what was there, skipped below)
#pragma unroll
                        for (int c = 0; c < kCh; ++c)
                            if (in_row(c)) u[a][c] = ring[(stage * kQuad + a) * L4 + lane + 32 * c];
                    __syncwarp();
                }
                if (kStage) ask(b + 2 * kQuad);
#pragma unroll
                for (int a = 0; a < kQuad && !kStage; ++a) {                    // (a slot without a row reads row 0, and is skipped below)
                    const float4* Urow = store + __shfl_sync(full, my_row, (b + a) & 31) * L4;
#pragma unroll
                    for (int c = 0; c < kCh; ++c) {
                        const uint32_t f = lane + 32 * c;
                        if (in_row(c)) u[a][c] = Urow[f];
                    }
                }
                float x[kQuad];
#pragma unroll
                for (int a = 0; a < kQuad; ++a) {
                    x[a] = 0.f;
#pragma unroll
                    for (int c = 0; c < kCh; ++c)
                        x[a] += v[c].x * u[a][c].x + v[c].y * u[a][c].y + v[c].z * u[a][c].z + v[c].w * u[a][c].w;
                }
                // The sums over the lanes by exchanging halves: each step leaves half as many values per lane (6 exchanges for
                // four scores, not 20).  Lanes kLanes a .. kLanes (a + 1) are left with the a-th score, and turn it into the
                // slot's factor.
                int o = 16;
#pragma unroll
                for (int half = kQuad / 2; half >= 1; half >>= 1) {
                    const bool up = lane & o;
#pragma unroll
                    for (int a = 0; a < half; ++a) {
                        const float send = up ? x[a] : x[a + half], keep = up ? x[a + half] : x[a];
                        x[a] = keep + __shfl_xor_sync(full, send, o);
                    }
                    o >>= 1;
                }
                float xa = x[0];
#pragma unroll
                for (int o2 = kLanes / 2; o2 > 0; o2 >>= 1) xa += __shfl_xor_sync(full, xa, o2);
                const bool positive = (t0 + b + lane / kLanes) % per_ctx == 0;
                const float sc_mine = -lr * (sigmoidf(xa) - (positive ? 1.f : 0.f));
#pragma unroll
                for (int a = 0; a < kQuad; ++a) {
                    const float sc = __shfl_sync(full, sc_mine, kLanes * a), xs = __shfl_sync(full, xa, kLanes * a);
                    if (!((ok_mask >> (b + a)) & 1u)) continue;
                    if (lane == (int)(b + a)) {
                        my_scale = sc;
                        my_x = xs;
                    }
#pragma unroll
                    for (int c = 0; c < kCh; ++c) {
                        dv[c].x += sc * u[a][c].x; dv[c].y += sc * u[a][c].y;
                        dv[c].z += sc * u[a][c].z; dv[c].w += sc * u[a][c].w;
                    }
                    if (kOnce && ((once_mask >> (b + a)) & 1u)) {           // nobody else reads this row: its update, in place
                        float4* Urow = store + __shfl_sync(full, my_row, (b + a) & 31) * L4;
#pragma unroll
                        for (int c = 0; c < kCh; ++c) {
                            const uint32_t f = lane + 32 * c;
                            const float4 x = make_float4(fmaf(sc, v[c].x, u[a][c].x), fmaf(sc, v[c].y, u[a][c].y),
                                                         fmaf(sc, v[c].z, u[a][c].z), fmaf(sc, v[c].w, u[a][c].w));
                            if (in_row(c)) Urow[f] = x;
                        }
                    }
                }
            }
            if (my_ok) {
                F[1 + t] = my_scale;
                loss += (double)softplusf(t % per_ctx == 0 ? -my_x : my_x);
            }
        }
        if (__any_sync(full, bad) && lane == 0) latch_error(st, epoch, PS_ERR_KEY_RANGE);
        if (dead) {                                             // (dv is a partial sum: the center's row stays as it is)
            if (keys_out && lane == 0) keys_out[cidx * slots] = kSentinelPad;   // without a sort: the reduction then does nothing
            break;
        }
#pragma unroll
        for (int c = 0; c < kCh; ++c) {
            const uint32_t f = lane + 32 * c;
            if (in_row(c)) {
                if (center_once) V[f] = make_float4(dv[c].x + v[c].x, dv[c].y + v[c].y, dv[c].z + v[c].z, dv[c].w + v[c].w);
                else U[f] = dv[c];
                U[L4 + f] = v[c];
            }
        }
        if (lane == 0) F[0] = 1.f;
    }
    block_loss_out(warp_sum_d(loss), loss_partial);
}

// Keys of the occurrence slots of each center: slot 0 the center's input vector, then per context
// 1 + n_neg output vectors; slots of contexts cut off at the stream's ends get the "no key" mark K.  32-bit divisions
// find a thread's slot (1.34M slots: 18.7 us with 64-bit ones, 17.3 with these, the marks' clearing included).  single, if not
// null: a mark per slot, cleared here for single_kernel.
__global__ void __launch_bounds__(256)
sgns_keys_kernel(const uint32_t* __restrict__ tokens, uint64_t tok_first, uint64_t first_pos, uint64_t n_centers,
                 uint64_t T, uint32_t window, const uint32_t* __restrict__ negs, uint32_t n_neg, uint64_t out_base,
                 uint64_t K, uint64_t pairs_first, uint32_t* __restrict__ keys_out, uint8_t* __restrict__ single,
                 DevStatus* st, unsigned int epoch) {
    const uint32_t per_ctx = 1 + n_neg, slots = 1 + 2 * window * per_ctx;      // (a batch's slots are fewer than 2^32)
    const uint32_t x = blockIdx.x * blockDim.x + threadIdx.x;
    if (x >= (uint32_t)n_centers * slots) return;
    if (single) single[x] = 0;
    const uint32_t cidx = x / slots, slot = x - cidx * slots;
    const uint64_t p = first_pos + cidx;
    uint64_t key = K;
    bool bad = false;
    if (slot == 0) {
        const uint32_t w = tokens[p - tok_first];
        bad = w >= out_base;
        key = w;
    } else {
        const uint64_t lo = p >= window ? p - window : 0;
        const uint64_t hi = p + window < T ? p + window : T - 1;
        const uint32_t j = (slot - 1) / per_ctx, i = slot - 1 - j * per_ctx;
        const uint64_t n_left = p - lo;
        const uint64_t q = j < n_left ? lo + j : lo + j + 1;        // skip the center itself
        if (q <= hi) {
            const uint64_t z = sgns_pairs_before(p, T, window) - pairs_first + j;
            const uint32_t word = i == 0 ? tokens[q - tok_first] : negs[z * n_neg + (i - 1)];
            key = out_base + word;
            bad = key >= K;
        }
    }
    if (bad) {
        latch_error(st, epoch, PS_ERR_KEY_RANGE);
        key = K;
    }
    keys_out[x] = (uint32_t)key;
}

// the per-slot factors follow the 2 n_centers source rows in the update buffer
float* sgns_scales(ps_store* ps, uint64_t n_centers) { return ps->upd + n_centers * 2 * ps->cfg.row_len; }

uint32_t launch_step_sgns(ps_store* ps, const uint32_t* d_tokens, uint64_t tok_first, uint64_t first_pos,
                          uint64_t n_centers, uint64_t corpus_len, uint32_t window, const uint32_t* d_negs,
                          uint32_t n_neg, uint64_t out_key_base, float lr, uint32_t* keys_out, cudaStream_t s, const uint8_t* single) {
    const uint32_t L4 = ps->cfg.row_len / 4;
    const uint32_t epoch = keys_out ? 0u : ps->epoch;
    const uint32_t grid = step_grid(ps, n_centers, 2);      // the kernels are bounded to two blocks per SM
#define SG_ARGS d_tokens, tok_first, first_pos, n_centers, corpus_len, window, d_negs, n_neg, out_key_base, lr,   \
                (float4*)ps->store, ps->table, ps->cfg.slots_per_part, ps->cfg.num_keys, single, L4,            \
                (float4*)ps->upd, sgns_scales(ps, n_centers), keys_out, ps->loss_partial, ps->status, epoch
#define SG_LAUNCH(kCh)                                                                                  \
    do {                                                                                                             \
        const size_t smem = (kCh) >= 2 ? (size_t)8 * 2 * sgns_quad(kCh) * L4 * 16 : 0;                               \
        static std::atomic<unsigned long long> smem_set[2];                                                          \
        const void* fn = single ? (const void*)sgns_step_kernel<kCh, true> : (const void*)sgns_step_kernel<kCh, false>; \
        if ((kCh) >= 2) opt_in_smem(fn, (size_t)8 * 2 * sgns_quad(kCh) * (kCh) * 512, &smem_set[single ? 1 : 0]);    \
        if (keys_out) {                                                                                              \
            PS_LAUNCH_PDL(ps, "sgns_step_kernel<" #kCh ">", (sgns_step_kernel<kCh, false>), dim3(grid), dim3(256), smem, s, SG_ARGS); \
        } else {                                                                                                     \
            if (ps->prof) prof_before(ps, "sgns_step_kernel<" #kCh ">", s);                                          \
            if (single) sgns_step_kernel<kCh, true><<<grid, 256, smem, s>>>(SG_ARGS);                   \
            else sgns_step_kernel<kCh, false><<<grid, 256, smem, s>>>(SG_ARGS);                         \
            if (ps->prof) prof_after(ps, s);                                                                         \
            ps->launches++;                                                                                          \
        }                                                                                                            \
    } while (0)
    if (L4 <= 32) SG_LAUNCH(1);
    else if (L4 <= 64) SG_LAUNCH(2);
    else if (L4 <= 96) SG_LAUNCH(3);
    else SG_LAUNCH(4);
#undef SG_LAUNCH
#undef SG_ARGS
    return grid;
}

void launch_keys_sgns(ps_store* ps, const uint32_t* d_tokens, uint64_t tok_first, uint64_t first_pos,
                      uint64_t n_centers, uint64_t corpus_len, uint32_t window, const uint32_t* d_negs, uint32_t n_neg,
                      uint64_t out_key_base, uint8_t* single, cudaStream_t s) {
    const uint64_t total = n_centers * (1 + (uint64_t)2 * window * (1 + n_neg));
    PS_LAUNCH(ps, sgns_keys_kernel, div_up_u32(total, 256), 256, s, d_tokens, tok_first, first_pos, n_centers,
              corpus_len, window, d_negs, n_neg, out_key_base, ps->cfg.num_keys,
              sgns_pairs_before(first_pos, corpus_len, window), ps->keysA, single, ps->status, ps->epoch);
}

}  // namespace psb
