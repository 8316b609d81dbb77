// Reduction of gradient rows key by key, for the steps with AdaGrad (ComplEx, RESCAL).
//
// Most keys of a batch occur once.  Such a key's row is read by one data point only, so that data point's gradient
// kernel, which has the gradient in registers, can update the row in place; its gradient then never goes through memory.
// They do so but for ComplEx on rows of at most 512 values in ordered mode, where the gradient kernel runs beside the sort
// and does not know yet which keys occur once: there single keys are a case of the reduction here.  The keys that occur
// several times are runs (segments) of the sorted occurrences.
//
// segment_kernel (on the stream of the sort, right after it) looks at every sorted position and writes
//   single[occurrence]     1 iff the occurrence's key occurs once
//   shorts                 {first position, length} of the other segments of fewer than kMediumRun occurrences; from the end of
//                          the array backwards, those of fewer than kWholeRun, which a warp adds alone too, but first
//   longs                  the longer ones, cut into pieces of about kLongPiece
//   pieces, chunks         RESCAL only: the relations' segments (any length), cut into pieces for its two kernels
// The lists' order is the hardware's, the sums' is not: a segment is summed in position order whoever takes it.
#include "ps_internal.cuh"

namespace psb {

namespace {
// Occurrences from which on a block, not a warp, adds a segment.  Where many segments are that long their warps are busy anyway,
// and a block's meetings per segment cost more than they save (8,000 data points of 5,000 uniform entities, 19 occurrences each:
// 125 us for the reduction with all from 12 on added by blocks, 63 now); the warps take those from kMediumRun on first, so
// that no long one is left for the end.
constexpr uint32_t kMediumRun = 12, kWholeRun = 40;
constexpr uint32_t kLongPiece = 96;             // ... and about as many as one block adds of it
constexpr uint32_t kMaxStrips = 64;             // (wider rows, of 16,384 values and more, are not cut: the tickets' room)
}  // namespace

// The first position from `from` on whose key is not k (which the position before it holds), by all lanes: 32 probes at a time,
// 1 apart, then 32, 1,024, ... until one differs, and back down.
__device__ uint32_t run_end(const uint32_t* __restrict__ sk, uint32_t n, uint64_t from, uint32_t k, uint32_t lane) {
    uint64_t apart = 1;
    auto equal = [&]() {
        const uint64_t q = from + apart * lane;
        return (uint32_t)__popc(__ballot_sync(0xffffffffu, q < n && sk[q] == k));
    };
    uint32_t c = equal();
    while (c == 32) {
        apart <<= 5;
        c = equal();
    }
    while (apart > 1) {
        from += apart * (c - 1);
        apart >>= 5;
        c = equal();
    }
    return (uint32_t)(from + c);
}

// A warp looks at 32 positions: the end of a run is the next head among them, or, for the last one, found by run_end, and a
// run cut into many pieces has them written by all lanes.  (A thread per head, with a search by doubling steps and a loop
// over its pieces, took 23 us for 42,000 positions with 11 relations' runs of 600; now 10.)
__global__ void __launch_bounds__(256)
segment_kernel(const uint32_t* __restrict__ sk, const uint32_t* __restrict__ sv, uint32_t n, uint32_t K, uint32_t rel_base,
               uint32_t long_piece, uint32_t rel_piece, uint32_t rel_chunk, SegLists L, const DevStatus* st, unsigned int epoch) {
    const unsigned full = 0xffffffffu;
    if (__any_sync(full, call_failed(st, epoch))) return;
    const uint32_t p = blockIdx.x * blockDim.x + threadIdx.x, lane = threadIdx.x & 31;
    const uint32_t key = p < n ? sk[p] : kSentinelPad;
    const uint32_t prev = p && p - 1 < n ? sk[p - 1] : kSentinelPad, next = p + 1 < n ? sk[p + 1] : kSentinelPad;
    const bool live = key < K, head = live && key != prev, rel = live && key >= rel_base;
    if (live) L.single[sv[p]] = head && key != next && !rel;
    const bool run = head && (key == next || rel);
    const unsigned later = __ballot_sync(full, key != prev) & ~((2u << lane) - 1u);     // boundaries among the positions to come
    uint32_t end = p - lane + (later ? (uint32_t)__ffs(later) - 1u : 32u);
    const unsigned open = __ballot_sync(full, run && !later);
    if (open) {
        const int src = __ffs(open) - 1;
        const uint32_t e = run_end(sk, n, (uint64_t)(p - lane) + 32, __shfl_sync(full, key, src), lane);
        if ((int)lane == src) end = e;
    }
    const uint32_t len = end - p;
    if (run && !rel && len < kMediumRun) L.shorts[atomicAdd(L.counts, 1u)] = make_uint2(p, len);
    else if (run && !rel && len < kWholeRun) L.shorts[L.short_room - 1 - atomicAdd(L.counts + kSegMediums, 1u)] = make_uint2(p, len);
    // pieces of nearly equal length: of a long run, or of a relation's, which also has chunks
    uint32_t np = 0, at = 0, park = 0, nc = 0, at_c = 0, park_c = 0;
    if (run && !rel && len >= kWholeRun) {
        np = tmax<uint32_t>(tmin<uint32_t>((uint32_t)(((uint64_t)len + long_piece / 2) / long_piece), 0xffffu), 1u);
        at = atomicAdd(L.counts + 1, np);
        if (np > 1) {
            park = atomicAdd(L.counts + 5, np);         // where its pieces leave their partial sums
            for (uint32_t i = 0; i < L.strips; ++i) L.long_tickets[(uint64_t)park * L.strips + i] = 0u;
        }
    } else if (run && rel) {
        np = (len + rel_piece - 1) / rel_piece;
        at = atomicAdd(L.counts + 2, np);
        nc = (len + rel_chunk - 1) / rel_chunk;
        at_c = atomicAdd(L.counts + 3, nc);
        if (nc > 1) park_c = atomicAdd(L.counts + 4, nc);       // where its chunks leave their partial sums
    }
    auto cut = [](uint32_t l, uint32_t i, uint32_t of) { return (uint32_t)((uint64_t)l * i / of); };
    auto write = [&](bool r, uint32_t p0, uint32_t l, uint32_t i, uint32_t of, uint32_t to, uint32_t pk) {
        const uint32_t x = cut(l, i, of), y = cut(l, i + 1, of);
        if (r) L.pieces[to + i] = make_uint2(p0 + x, y - x);
        else L.longs[to + i] = make_uint4(p0 + x, y - x, pk, i | of << 16);
    };
    auto write_chunk = [&](uint32_t p0, uint32_t l, uint32_t i, uint32_t of, uint32_t to, uint32_t pk) {
        const uint32_t x = cut(l, i, of), y = cut(l, i + 1, of);
        L.chunks[to + i] = make_uint4(p0 + x, y - x, pk, i | of << 16);
        for (uint32_t t = 0; of > 1 && t < kRelTickets / 4; ++t)
            reinterpret_cast<uint4*>(L.tickets + (uint64_t)(pk + i) * kRelTickets)[t] = make_uint4(0u, 0u, 0u, 0u);
    };
    const bool many = np > 4 || nc > 4;
    if (!many) {
        for (uint32_t i = 0; i < np; ++i) write(rel, p, len, i, np, at, park);
        for (uint32_t i = 0; i < nc; ++i) write_chunk(p, len, i, nc, at_c, park_c);
    }
    for (unsigned m = __ballot_sync(full, many); m; m &= m - 1) {
        const int src = __ffs(m) - 1;
        const bool r = __shfl_sync(full, (int)rel, src) != 0;
        const uint32_t p0 = __shfl_sync(full, p, src), l = __shfl_sync(full, len, src);
        const uint32_t mp = __shfl_sync(full, np, src), ma = __shfl_sync(full, at, src), mk = __shfl_sync(full, park, src);
        const uint32_t mc = __shfl_sync(full, nc, src), mac = __shfl_sync(full, at_c, src), mkc = __shfl_sync(full, park_c, src);
        for (uint32_t i = lane; i < mp; i += 32) write(r, p0, l, i, mp, ma, mk);
        for (uint32_t i = lane; i < mc; i += 32) write_chunk(p0, l, i, mc, mac, mkc);
    }
}

// The flags alone, for the skip-gram step (its other keys go through scaled_reduce_kernel).  The key kernel has cleared them:
// a byte to a random place costs more than the rest of this (1.34M slots: 28.7 us writing all, 21.9 writing the ones).
__global__ void __launch_bounds__(256)
single_kernel(const uint32_t* __restrict__ sk, const uint32_t* __restrict__ sv, uint32_t n, uint32_t K, uint8_t* __restrict__ single,
              const DevStatus* st, unsigned int epoch) {
    if (call_failed(st, epoch)) return;
    const uint32_t p = blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= n) return;
    const uint32_t key = sk[p];
    if (key < K && (p == 0 || sk[p - 1] != key) && (p + 1 == n || sk[p + 1] != key)) single[sv[p]] = 1;
}

const uint8_t* launch_singles(ps_store* ps, uint32_t n, int which, cudaStream_t s) {
    uint8_t* single = (uint8_t*)ps->cellpos;
    PS_LAUNCH(ps, single_kernel, div_up_u32(n, 256), 256, s, which ? ps->keysB : ps->keysA, which ? ps->valsB : ps->valsA, n,
              (uint32_t)ps->cfg.num_keys, single, ps->status, ps->epoch);
    return single;
}

SegLists seg_lists(ps_store* ps) {
    SegLists L;
    L.counts = ps->group_done;                  // (zeroed by the sort)
    L.single = (uint8_t*)ps->cellpos;
    // the records of the matrix-factorization step (16 bytes per key occurrence) are not in use
    L.longs = ps->rec;
    L.shorts = (uint2*)(L.longs + ps->max_keys / kMediumRun + 2);
    L.short_room = (uint32_t)(ps->max_keys / 2 + 1);
    L.pieces = L.shorts + L.short_room;
    L.long_tickets = (unsigned int*)(L.pieces + ps->max_keys / 6 + 1);     // at least six slots per data point of RESCAL
    L.chunks = ps->mf_dup;
    L.tickets = ps->mf_tickets;
    L.strips = 1;
    return L;
}

// stretches of a half row's columns that blocks take separately (blockIdx.y of segment_adagrad_kernel)
static uint32_t seg_strips(uint32_t half_row) {
    const bool quads = half_row % 4 == 0;
    const uint32_t vec = quads ? 4 : 2, ch = half_row <= (quads ? 128u : 64u) ? 1 : 2;
    return div_up_u32(half_row, 32 * vec * ch);
}

uint32_t rel_piece_len(uint32_t d) { return d <= 64 ? kRelPiece / 2 : kRelPiece; }

// Data points per chunk of rescal_matrix_kernel: 64, and fewer (16 at least) while the batch's chunks, a block for each of a
// matrix's strips, would not fill the chip (1,288 data points of 11 relations of dimension 28: 34.7 -> 22.9 us); but the block
// that finishes a relation adds up its groups of kRelGroup chunks one after the other, about twice as long per group as a data
// point takes, so not below half the square root of a relation's share of the batch.  A chunk parks two sums per element, 2 d d doubles, where a
// tile of the push's reductions has room for 4 d, and a relation's chunks may be half empty: at least n d / tiles.
static uint32_t rel_chunk_len(const ps_store* ps, uint32_t n_points, uint64_t n_rel, uint32_t d) {
    const uint64_t strips = div_up_u32((uint64_t)d * d / 8, 256), blocks = (uint64_t)ps->sm_count * 3;
    uint64_t len = tmax<uint64_t>(n_points * strips / blocks, div_up_u32((uint64_t)n_points * d, ps->tile_cap));
    while (len < kRelChunk && 4 * len * len < (uint64_t)n_points / tmax<uint64_t>(n_rel, 1)) ++len;
    len = (len + 7) / 8 * 8;
    return (uint32_t)tmin<uint64_t>(tmax<uint64_t>(len, 16), kRelChunk);
}

void launch_segments(ps_store* ps, uint32_t n, int which, uint32_t half_row, uint64_t rel_key_base, uint32_t n_points, cudaStream_t s) {
    const uint32_t* sk = which ? ps->keysB : ps->keysA;
    const uint32_t* sv = which ? ps->valsB : ps->valsA;
    SegLists L = seg_lists(ps);
    L.strips = seg_strips(half_row);
    PS_LAUNCH(ps, segment_kernel, div_up_u32(n, 256), 256, s, sk, sv, n, (uint32_t)ps->cfg.num_keys, (uint32_t)rel_key_base,
              L.strips <= kMaxStrips ? kLongPiece : kSentinelPad, rel_piece_len(half_row), rel_chunk_len(ps, n_points, (ps->cfg.num_keys - rel_key_base) / half_row, half_row), L, ps->status, ps->epoch);
}

// The segments' sums: AdaGrad per occurrence from the row [parameters | accumulators] as it was before the batch (the
// expression of the gradient kernels), steps and squared gradients added in fp64 in position order, one rounding.  A warp
// takes a short segment, kFly gradient rows in flight; a long one is shared by the block's warps (a stretch of it
// each, partial sums added in order), and one of several pieces leaves each piece's fp64 sum in memory for the block
// that draws its last ticket, which adds them in piece order.  What bounds it is the unit for square roots and
// conversions, four operations per value: the hottest entity of a batch (1,200 of 16,384 subjects and objects on
// Zipf(1) triples) took one block 40 us.  V: float4, or float2 for rows whose halves are not whole float4s; blockIdx.y counts
// stretches of 32 kCh vectors.  Conversions go through the integer pipe (widen_scaled).  The last block adds the loss terms, strided per thread, then a tree.
template <class V> struct Vec;
template <> struct Vec<float4> {
    static constexpr int kN = 4;
    __device__ static float get(const float4& v, int i) { return i == 0 ? v.x : i == 1 ? v.y : i == 2 ? v.z : v.w; }
    __device__ static void set(float4& v, int i, float f) { if (i == 0) v.x = f; else if (i == 1) v.y = f; else if (i == 2) v.z = f; else v.w = f; }
};
template <> struct Vec<float2> {
    static constexpr int kN = 2;
    __device__ static float get(const float2& v, int i) { return i == 0 ? v.x : v.y; }
    __device__ static void set(float2& v, int i, float f) { if (i == 0) v.x = f; else v.y = f; }
};

template <class V, int kCh>
__global__ void __launch_bounds__(256, 2)
segment_adagrad_kernel(const uint32_t* __restrict__ sk, const uint32_t* __restrict__ sv, const V* __restrict__ grad,
                       V* __restrict__ store, const uint2* __restrict__ table, uint64_t S, uint32_t K, uint32_t n_singles,
                       uint32_t GV, float lr, float eps,
                       SegLists L, double* __restrict__ parked, const double* __restrict__ loss_terms, uint32_t n_loss,
                       double* loss_accum, const DevStatus* st, unsigned int epoch) {
    constexpr int kN = Vec<V>::kN, kWarps = 8;
    constexpr int kFly = 4;                     // gradient rows a warp has in flight
    __shared__ double s_part[kWarps][32 * kN];
    __shared__ uint32_t s_ticket;
    // Beside RESCAL's matrix kernel (launched while that one's last blocks run, on other rows): what follows on the stream has
    // to come after both.  Elsewhere nothing is waited for.
    struct AtExit {
        __device__ ~AtExit() { pdl_wait(); }
    } at_exit;
    if (call_failed(st, epoch)) return;
    const unsigned full = 0xffffffffu;
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    if (blockIdx.x == gridDim.x - 1) {
        if (blockIdx.y != 0 || !loss_accum) return;
        double t = 0;
        for (uint32_t i = tid; i < n_loss; i += 256) t += loss_terms[i];
        t = warp_sum_d(t);
        if (lane == 0) s_part[0][w] = t;
        __syncthreads();
        if (tid == 0) {
            double tot = 0;
            for (int i = 0; i < kWarps; ++i) tot += s_part[0][i];
            *loss_accum += tot;
        }
        return;
    }
    const uint32_t f0 = blockIdx.y * (32 * kCh) + lane;
    V th[kCh], G[kCh];
    double a_t[kCh][kN], a_g[kCh][kN];
    auto load_row = [&](const V* row) {
#pragma unroll
        for (int c = 0; c < kCh; ++c)
            if (f0 + 32 * c < GV) {
                th[c] = row[f0 + 32 * c];
                G[c] = row[GV + f0 + 32 * c];
            }
    };
    // occurrences at positions lo .. lo + cnt of one segment
    auto sum = [&](uint32_t lo, uint32_t cnt) {
#pragma unroll
        for (int c = 0; c < kCh; ++c)
#pragma unroll
            for (int i = 0; i < kN; ++i) a_t[c][i] = a_g[c][i] = 0.0;       // (times 2^-896: widen_scaled)
        for (uint32_t j0 = 0; j0 < cnt; j0 += 32) {
            const uint32_t in = cnt - j0 < 32u ? cnt - j0 : 32u;
            const uint32_t occ = (uint32_t)lane < in ? sv[lo + j0 + lane] : 0u;
            for (uint32_t j = 0; j < in; j += kFly) {
                V u[kFly][kCh];
#pragma unroll
                for (int q = 0; q < kFly; ++q) {
                    const uint32_t o = __shfl_sync(full, occ, (j + q) & 31);
#pragma unroll
                    for (int c = 0; c < kCh; ++c)
                        if (j + q < in && f0 + 32 * c < GV) u[q][c] = __ldg(grad + (uint64_t)o * GV + f0 + 32 * c);
                }
#pragma unroll
                for (int q = 0; q < kFly; ++q) {
                    if (j + q >= in) break;
#pragma unroll
                    for (int c = 0; c < kCh; ++c) {
                        if (f0 + 32 * c >= GV) continue;
                        float g[kN], g2[kN], x[kN], step[kN];
#pragma unroll
                        for (int i = 0; i < kN; ++i) {
                            g[i] = Vec<V>::get(u[q][c], i);
                            g2[i] = g[i] * g[i];
                            x[i] = Vec<V>::get(G[c], i) + g2[i];
                        }
                        const bool fine = adagrad_steps<kN>(g, x, lr, eps, step);
#pragma unroll
                        for (int i = 0; i < kN; ++i) {
                            a_t[c][i] += fine ? widen_scaled(step[i]) : kScale * (double)step[i];
                            a_g[c][i] += fine ? widen_scaled(g2[i]) : kScale * (double)g2[i];
                        }
                    }
                }
            }
        }
    };
    auto unscale = [&]() {
#pragma unroll
        for (int c = 0; c < kCh; ++c)
#pragma unroll
            for (int i = 0; i < kN; ++i) {
                a_t[c][i] *= kUnscale;
                a_g[c][i] *= kUnscale;
            }
    };
    auto finish = [&](V* row) {
#pragma unroll
        for (int c = 0; c < kCh; ++c)
            if (f0 + 32 * c < GV) {
#pragma unroll
                for (int i = 0; i < kN; ++i) {
                    Vec<V>::set(th[c], i, (float)((double)Vec<V>::get(th[c], i) + a_t[c][i]));
                    Vec<V>::set(G[c], i, (float)((double)Vec<V>::get(G[c], i) + a_g[c][i]));
                }
                row[f0 + 32 * c] = th[c];
                row[GV + f0 + 32 * c] = G[c];
            }
    };
    // the warps' sums, added in warp order: warp 0 has the total
    auto over_warps = [&]() {
#pragma unroll
        for (int c = 0; c < kCh; ++c)
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                __syncthreads();                // (every warp has read the row; the sums before are taken)
#pragma unroll
                for (int i = 0; i < kN; ++i) s_part[w][i * 32 + lane] = h ? a_g[c][i] : a_t[c][i];
                __syncthreads();
                if (w == 0) {
#pragma unroll
                    for (int i = 0; i < kN; ++i) {
                        double tot = s_part[0][i * 32 + lane];
#pragma unroll
                        for (int k = 1; k < kWarps; ++k) tot += s_part[k][i * 32 + lane];
                        if (h) a_g[c][i] = tot; else a_t[c][i] = tot;
                    }
                }
            }
    };
    const uint32_t n_work = gridDim.x - 1;
    const uint32_t n_longs = L.counts[1], n_mediums = L.counts[kSegMediums], n_shorts = n_mediums + L.counts[0];
    for (uint32_t j = blockIdx.x; j < n_longs; j += n_work) {
        const uint4 seg = L.longs[j];
        V* row = store + phys_row(table[sk[seg.x]], S) * (2 * GV);
        load_row(row);
        const uint32_t a = (uint32_t)((uint64_t)seg.y * w / kWarps), b = (uint32_t)((uint64_t)seg.y * (w + 1) / kWarps);
        sum(seg.x + a, b - a);
        unscale();
        over_warps();
        const uint32_t np = seg.w >> 16, piece = seg.w & 0xffffu;
        if (np > 1) {
            if (w == 0) {
                double* p = parked + (uint64_t)(seg.z + piece) * (2 * GV * kN);
#pragma unroll
                for (int c = 0; c < kCh; ++c)
                    if (f0 + 32 * c < GV)
#pragma unroll
                        for (int i = 0; i < kN; ++i) {
                            p[(f0 + 32 * c) * kN + i] = a_t[c][i];
                            p[(GV + f0 + 32 * c) * kN + i] = a_g[c][i];
                        }
                __threadfence();
            }
            __syncthreads();
            if (tid == 0) s_ticket = atomicAdd(&L.long_tickets[(uint64_t)seg.z * gridDim.y + blockIdx.y], 1u);
            __syncthreads();
            if (s_ticket != np - 1) continue;
            // the last of the segment's blocks: a stretch of the pieces per warp (one warp took 0.7 us for each, 42 of them for a
            // relation that half of 8,000 data points have)
            __threadfence();
#pragma unroll
            for (int c = 0; c < kCh; ++c)
#pragma unroll
                for (int i = 0; i < kN; ++i) a_t[c][i] = a_g[c][i] = 0.0;
            for (uint32_t k = np * w / kWarps; k < np * (w + 1) / kWarps; ++k) {
                const double* q = parked + (uint64_t)(seg.z + k) * (2 * GV * kN);
#pragma unroll
                for (int c = 0; c < kCh; ++c)
                    if (f0 + 32 * c < GV)
#pragma unroll
                        for (int i = 0; i < kN; ++i) {
                            a_t[c][i] += __ldcg(q + (f0 + 32 * c) * kN + i);
                            a_g[c][i] += __ldcg(q + (GV + f0 + 32 * c) * kN + i);
                        }
            }
            over_warps();
            if (w == 0) finish(row);
            continue;
        }
        if (w == 0) finish(row);
    }
    // The warps draw the short ones (the next one's number on its way while one is added), so that blocks that had long segments
    // take fewer: 106,496 occurrences of 400 values 44.8 -> 41.6 us, RESCAL's of 200 30 -> 26.6.  Where single keys follow, those
    // balance it (drawing both costs 25 -> 29 us at 35,000 occurrences of 256 values).
    const bool drawn = gridDim.y <= kMaxStrips && n_singles == 0;
    uint32_t next = blockIdx.x * kWarps + w;
    if (drawn && lane == 0) next = atomicAdd(L.counts + 8 + blockIdx.y, 1u);
    for (;;) {
        const uint32_t j = __shfl_sync(full, next, 0);
        if (j >= n_shorts) break;
        next = j + n_work * kWarps;
        if (drawn && lane == 0) next = atomicAdd(L.counts + 8 + blockIdx.y, 1u);
        const uint2 seg = L.shorts[j < n_mediums ? L.short_room - 1 - j : j - n_mediums];
        V* row = store + phys_row(table[sk[seg.x]], S) * (2 * GV);
        load_row(row);
        sum(seg.x, seg.y);
        unscale();
        finish(row);
    }
    // Keys that occur once, 32 sorted positions per warp at a time: all look-ups together, then kPair rows in flight; row
    // + step in fp32 rounds the exact sum once.
    // They come last and the warps draw them, so that blocks which had long segments take fewer.
    auto draw = [&]() {
        uint32_t v = 0;
        if (lane == 0) v = atomicAdd(L.counts + 6 + blockIdx.y, 1u);
        return __shfl_sync(full, v, 0) * 32;
    };
    for (uint32_t p0 = n_singles ? draw() : 0; p0 < n_singles;) {
        const uint32_t p = p0 + lane;
        p0 = draw();
        const uint32_t key = p < n_singles ? sk[p] : K;
        const bool mine = key < K && (p == 0 || sk[p - 1] != key) && (p + 1 == n_singles || sk[p + 1] != key);
        const uint32_t occ = mine ? sv[p] : 0u;
        const uint64_t row_of = mine ? phys_row(table[key], S) : 0;
        unsigned todo = __ballot_sync(full, mine);
        constexpr int kPair = kCh * kN >= 8 ? 3 : 4;
        while (todo) {
            V u[kPair][kCh], t1[kPair][kCh], g1[kPair][kCh];
            V* row[kPair];
            bool have[kPair];
#pragma unroll
            for (int q = 0; q < kPair; ++q) {
                have[q] = todo != 0;
                const int src = todo ? __ffs(todo) - 1 : 0;
                todo &= todo - 1;                   // 0 stays 0
                const V* g = grad + (uint64_t)__shfl_sync(full, occ, src) * GV;
                row[q] = store + __shfl_sync(full, row_of, src) * (2 * GV);
#pragma unroll
                for (int c = 0; c < kCh; ++c)
                    if (have[q] && f0 + 32 * c < GV) {
                        u[q][c] = __ldg(g + f0 + 32 * c);
                        t1[q][c] = row[q][f0 + 32 * c];
                        g1[q][c] = row[q][GV + f0 + 32 * c];
                    }
            }
#pragma unroll
            for (int q = 0; q < kPair; ++q)
#pragma unroll
                for (int c = 0; c < kCh; ++c) {
                    if (!have[q] || f0 + 32 * c >= GV) continue;
                    float g[kN], x[kN], step[kN];
#pragma unroll
                    for (int i = 0; i < kN; ++i) {
                        g[i] = Vec<V>::get(u[q][c], i);
                        x[i] = __fadd_rn(Vec<V>::get(g1[q][c], i), __fmul_rn(g[i], g[i]));
                    }
                    adagrad_steps<kN>(g, x, lr, eps, step);
#pragma unroll
                    for (int i = 0; i < kN; ++i) {
                        Vec<V>::set(t1[q][c], i, __fadd_rn(Vec<V>::get(t1[q][c], i), step[i]));
                        Vec<V>::set(g1[q][c], i, x[i]);
                    }
                    row[q][f0 + 32 * c] = t1[q][c];
                    row[q][GV + f0 + 32 * c] = g1[q][c];
                }
        }
    }
}

void run_segment_adagrad(ps_store* ps, uint32_t n, int which, uint32_t half_row, bool singles, float lr, float eps,
                         double* parked, const double* loss_terms, uint32_t n_loss, double* d_loss_accum, cudaStream_t s, bool beside) {
    const uint32_t* sk = which ? ps->keysB : ps->keysA;
    const uint32_t* sv = which ? ps->valsB : ps->valsA;
    const SegLists L = seg_lists(ps);
    if (!n_loss) d_loss_accum = nullptr;
#define SEG_ARGS(V) sk, sv, (const V*)ps->upd, (V*)ps->store, (const uint2*)ps->table, ps->cfg.slots_per_part, (uint32_t)ps->cfg.num_keys, \
                 singles ? n : 0u, GV, lr, eps, L, parked, loss_terms, n_loss, d_loss_accum, (const DevStatus*)ps->status, ps->epoch
#define SEG_LAUNCH(V, kCh)                                                                                              \
    do {                                                                                                                \
        const uint32_t GV = half_row / Vec<V>::kN, strips = seg_strips(half_row);                                       \
        /* as many blocks as are resident over all stretches of columns; the warps loop over the lists */               \
        const uint32_t gx = tmax<uint32_t>(1u, tmin<uint32_t>(div_up_u32(n, 32), (uint32_t)ps->sm_count * 2 / strips)); \
        if (ps->prof) prof_before(ps, "segment_adagrad_kernel", s);                                                     \
        if (beside) launch_pdl(segment_adagrad_kernel<V, kCh>, dim3(gx + 1, strips), dim3(256), 0, s, SEG_ARGS(V));     \
        else segment_adagrad_kernel<V, kCh><<<dim3(gx + 1, strips), 256, 0, s>>>(SEG_ARGS(V));                           \
        if (ps->prof) prof_after(ps, s);                                                                                \
        ps->launches++;                                                                                                 \
    } while (0)
    if (half_row % 4 == 0) {
        if (half_row <= 128) SEG_LAUNCH(float4, 1);
        else SEG_LAUNCH(float4, 2);
    } else {
        if (half_row <= 64) SEG_LAUNCH(float2, 1);
        else SEG_LAUNCH(float2, 2);
    }
#undef SEG_LAUNCH
#undef SEG_ARGS
}

}  // namespace psb
