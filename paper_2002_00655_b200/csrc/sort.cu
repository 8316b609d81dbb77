// Stable least-significant-digit radix sort of (key, value) pairs, 8 bits per
// pass, as ONE kernel launch.  It orders the key occurrences of a batch so that
// the push can reduce them segment by segment (cumulative push, Section 2.1 of
// the paper) and so that localize sees each distinct key once, in ascending
// order.
//
// The batches are small (10^5 .. 10^6 keys), so the sort is bound by launch and
// memory latency, not by bandwidth.  All passes therefore run inside one
// cooperative kernel of at most one block per SM; a block owns a contiguous
// chunk of positions in every pass.  Per pass a block needs, for each digit,
// the number of keys with that digit in all chunks before its own.  Those
// counts are gathered while the PREVIOUS pass scatters: a key that goes to
// position pos adds one to counter [next pass][chunk of pos][next digit].  So
// a pass is: grid barrier, read one column of counters per digit, rank the
// chunk's keys tile by tile (warp_rank: stable), scatter.
// The key source of the first pass and the sink of the last pass are functors:
// a step extracts its keys from the batch arrays inside the sort, and the
// matrix-factorization step has the last pass emit, per sorted position, the
// addresses the gradient kernel needs instead of bare (key, index) pairs.
//
// The only waiting is the grid barrier; it is bounded, and a block that gives
// up latches an error and returns.
#include "ps_internal.cuh"

namespace psb {

struct SortParams {
    uint32_t *kA, *vA, *kB, *vB;        // pass p reads (kA, vA) if (start + p) is even, else (kB, vB)
    int start;
    uint32_t n_host;
    const unsigned int* n_dev;
    int n_passes;
    uint32_t tiles_per_block;
    uint32_t* counts;                   // [pass][block][digit]
    unsigned int* bar;
    unsigned int* zero_a;               // words cleared before the first barrier (counters of later kernels)
    uint32_t n_zero_a;
    unsigned int* zero_b;
    DevStatus* st;
    unsigned int epoch;
};

// ---- key sources: what is read for occurrence idx, and its key.  (Two steps, so that a thread's reads are all on their way
// before the first is checked: the check's atomics keep later reads behind them.  One by one, the 16 reads a thread has in a
// sort of 1M keys took 10 us of its 59, now 4.5.)  kFromBuffer: the keys are already in the pass-0 input buffer. ----
struct SrcBuffer {
    static constexpr bool kFromBuffer = true;
    using Raw = uint32_t;
    __device__ __forceinline__ Raw read(uint32_t) const { return 0u; }
    __device__ __forceinline__ uint32_t key(uint32_t, Raw, const SortParams&) const { return 0u; }
};
// 64-bit caller keys, range-checked (push, localize)
struct SrcKeys64 {
    static constexpr bool kFromBuffer = false;
    const uint64_t* keys;
    uint64_t K;
    using Raw = uint64_t;
    __device__ __forceinline__ Raw read(uint32_t idx) const { return keys[idx]; }
    __device__ __forceinline__ uint32_t key(uint32_t, Raw k, const SortParams& P) const {
        if (k >= K) {
            latch_error(P.st, P.epoch, PS_ERR_KEY_RANGE);
            return (uint32_t)K;
        }
        return (uint32_t)k;
    }
};
// occurrences of a batch of matrix cells: 2t = row factor of cell t, 2t + 1 = its column factor
struct SrcMF {
    static constexpr bool kFromBuffer = false;
    const uint32_t *ci, *cj;
    uint64_t col_base, K;
    using Raw = uint2;
    __device__ __forceinline__ Raw read(uint32_t idx) const { return make_uint2(ci[idx >> 1], cj[idx >> 1]); }
    __device__ __forceinline__ uint32_t key(uint32_t idx, Raw c, const SortParams& P) const {
        const uint64_t kw = c.x, kh = col_base + c.y;
        if (kw >= col_base || kh >= K) {
            latch_error(P.st, P.epoch, PS_ERR_KEY_RANGE);
            return (uint32_t)K;
        }
        return (idx & 1u) ? (uint32_t)kh : (uint32_t)kw;
    }
};

// ---- sinks of the last pass ----
struct SinkPairs {
    static constexpr bool kPairs = true;
};
// Matrix factorization: besides the sorted key, one record per sorted position with everything the gradient
// kernel would otherwise have to chase through three dependent loads: {key, value of the cell, physical
// row of the key, physical row of the cell's other factor}.  (It says {cell, ...}: the key is in the sorted key array.)
struct SinkMF {
    static constexpr bool kPairs = false;
    const uint32_t *ci, *cj;
    const float* cv;
    uint32_t col_base, K;
    const uint2* table;
    uint64_t S;
    uint4* rec;
    uint32_t* cellpos;                  // sorted position of each cell's row-factor occurrence
};

// Rank of a lane's digit among the warp's keys so far (stable: item by item, lane by lane), and the warp's counter of the
// digit moved on.  Lanes with equal digits find one another through a word per digit in shared memory (every lane ORs its
// bit in, as in the atomic-OR form of the warp match of CUB's BlockRadixRankMatch); __match_any_sync takes 61 cycles of an SM
// per instruction, the OR and the read 6.  `mask` is all zero before and after.
__device__ __forceinline__ uint32_t warp_rank(volatile uint32_t* mask, volatile uint32_t* hist, uint32_t digit, bool valid,
                                              int lane) {
    if (valid) atomicOr(const_cast<uint32_t*>(mask) + digit, 1u << lane);
    __syncwarp();
    const uint32_t peers = valid ? mask[digit] : 1u << lane;
    const int leader = 31 - __clz(peers);
    uint32_t old = 0;
    if (valid && lane == leader) {
        old = hist[digit];
        hist[digit] = old + __popc(peers);
    }
    old = __shfl_sync(0xffffffffu, old, leader);
    if (valid && lane == leader) mask[digit] = 0u;
    __syncwarp();
    return old + __popc(peers & ((1u << lane) - 1u));
}

// Exclusive scan of one value per digit held by threads 0..255 of a block of kThreads; every thread calls.
template <int kThreads>
__device__ __forceinline__ uint32_t scan_digits(uint32_t v, uint32_t* sm8, uint32_t* total) {
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    uint32_t incl = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t t = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += t;
    }
    if (lane == 31 && w < 8) sm8[w] = incl;
    __syncthreads();
    uint32_t wbase = 0, tot = 0;
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        const uint32_t t = sm8[i];
        if (i < w) wbase += t;
        tot += t;
    }
    __syncthreads();
    *total = tot;
    return wbase + incl - v;
}

// A tile is kThreads x kItems keys: 512 x 4 in small sorts (every phase of a pass is a short chain of dependent steps, and all
// SMs get a tile), 512 x 8 in large ones.
template <class Src, class Sink, int kThreads, int kItems>
__global__ void __launch_bounds__(kThreads, 2)
sort_all_kernel(Src src, Sink sink, SortParams P) {
    constexpr int kTile = kThreads * kItems;
    constexpr int kWarps = kThreads / 32;
    constexpr int kQ = kThreads / 64;                // threads per group of four digits in the counter read
    constexpr int kRowsAtOnce = 16;
    __shared__ uint32_t digit_base[kRadix];          // global position of the tile's first key with each digit
    __shared__ uint32_t local_base[kRadix];          // the same inside the tile
    extern __shared__ __align__(16) uint32_t s_dyn[];  // the tile in digit order, on its way out: keys, then values
    uint32_t* const s_key = s_dyn;
    uint32_t* const s_val = s_dyn + kTile;
    uint32_t (*const warp_hist)[kRadix] = reinterpret_cast<uint32_t (*)[kRadix]>(s_dyn + 2 * kTile);
    uint32_t (*const warp_mask)[kRadix] = warp_hist + kWarps;
    __shared__ uint32_t sm[8];
    __shared__ int s_ok;
    const uint32_t n = P.n_dev ? tmin<uint32_t>(*((const volatile unsigned int*)P.n_dev), P.n_host) : P.n_host;
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    const bool digit_thread = tid < kRadix;
    const uint32_t b = blockIdx.x, G = gridDim.x;
    const uint32_t chunk = P.tiles_per_block * kTile;
    const uint64_t c0_64 = (uint64_t)b * chunk;
    const uint32_t c0 = c0_64 < n ? (uint32_t)c0_64 : n;
    const uint32_t c1 = (uint64_t)c0 + chunk < n ? c0 + chunk : n;
    const uint32_t my_tiles = (c1 - c0 + kTile - 1) / kTile;
    const uint32_t magic = (uint32_t)tmin<uint64_t>(((1ull << 32) + chunk - 1) / chunk, 0xFFFFFFFFull);
    unsigned int barriers = 0;

    // ---- before the first barrier: clear what must start at zero, count the digits of pass 0 ----
    if (digit_thread) {
        for (int p = 1; p < P.n_passes; ++p) P.counts[((size_t)p * G + b) * kRadix + tid] = 0u;
        digit_base[tid] = 0u;
    }
    for (int i = tid; i < kWarps * kRadix; i += kThreads) (&warp_mask[0][0])[i] = 0u;
    if (b == 0) {
        for (uint32_t i = tid; i < P.n_zero_a; i += kThreads) P.zero_a[i] = 0u;
        if (tid == 0 && P.zero_b) P.zero_b[0] = P.zero_b[1] = 0u;     // (the list counter of the coming reduction and its neighbour)
    }
    __syncthreads();
    uint32_t key0[kItems];                           // keys of the chunk's first tile stay in registers for pass 0
#pragma unroll
    for (int it = 0; it < kItems; ++it) key0[it] = 0u;
    uint32_t* kin0 = (P.start & 1) ? P.kB : P.kA;
    for (uint32_t t = 0; t < my_tiles; ++t) {
        const uint32_t tb = c0 + t * kTile + w * (32 * kItems);
        uint32_t kk[kItems];
        if constexpr (Src::kFromBuffer) {
#pragma unroll
            for (int it = 0; it < kItems; ++it) {
                const uint32_t idx = tb + it * 32 + lane;
                kk[it] = idx < c1 ? __ldcg(kin0 + idx) : 0u;
            }
        } else {
            typename Src::Raw raw[kItems];
#pragma unroll
            for (int it = 0; it < kItems; ++it) {
                const uint32_t idx = tb + it * 32 + lane;
                raw[it] = src.read(idx < c1 ? idx : c0);        // (the block has a key: a read that is not used)
            }
#pragma unroll
            for (int it = 0; it < kItems; ++it) {
                const uint32_t idx = tb + it * 32 + lane;
                kk[it] = 0u;
                if (idx < c1) kk[it] = src.key(idx, raw[it], P);
            }
        }
#pragma unroll
        for (int it = 0; it < kItems; ++it) {
            const uint32_t idx = tb + it * 32 + lane;
            if (idx < c1) {
                if (!Src::kFromBuffer && t > 0) kin0[idx] = kk[it];
                atomicAdd(&digit_base[kk[it] & (kRadix - 1)], 1u);
            }
            if (t == 0) key0[it] = kk[it];
        }
    }
    __syncthreads();
    if (digit_thread) P.counts[(size_t)b * kRadix + tid] = digit_base[tid];
    if (!grid_barrier(P.bar, ++barriers * G, &s_ok)) {
        if (tid == 0) atomicCAS(&P.st->sticky, 0u, (unsigned int)PS_ERR_CUDA);
        return;
    }

    for (int p = 0; p < P.n_passes; ++p) {
        const bool from_a = ((P.start + p) & 1) == 0;
        uint32_t* kin = from_a ? P.kA : P.kB;
        uint32_t* vin = from_a ? P.vA : P.vB;
        uint32_t* kout = from_a ? P.kB : P.kA;
        uint32_t* vout = from_a ? P.vB : P.vA;
        const int shift = p * kRadixBits;
        const bool last = p + 1 == P.n_passes;
        uint32_t key[kItems], val[kItems];
        // the keys of the chunk's first tile are asked for now, so that they travel beside the counters below
        auto load_tile = [&](uint32_t t) {
            const uint32_t tb = c0 + t * kTile + w * (32 * kItems);
#pragma unroll
            for (int it = 0; it < kItems; ++it) {
                const uint32_t idx = tb + it * 32 + lane;
                key[it] = 0u;
                val[it] = idx;
                if (idx < c1) {
                    if (p == 0) {
                        key[it] = (t == 0) ? key0[it] : __ldcg(kin + idx);
                    } else {
                        key[it] = __ldcg(kin + idx);
                        val[it] = __ldcg(vin + idx);
                    }
                }
            }
        };
        if (my_tiles > 0) load_tile(0);
        // ---- per digit: keys with that digit in the chunks before this block's, and in all chunks.  Thread
        // (q, d4) adds up four digits over every kQ-th block; the kQ partial sums meet in shared memory.
        {
            const int q = tid >> 6, d4 = tid & 63;
            const uint4* col = reinterpret_cast<const uint4*>(P.counts + (size_t)p * G * kRadix) + d4;
            uint4 before = make_uint4(0u, 0u, 0u, 0u), total = before;
            for (uint32_t r0 = q; r0 < G; r0 += kRowsAtOnce * kQ) {
                uint4 c[kRowsAtOnce];
#pragma unroll
                for (int k = 0; k < kRowsAtOnce; ++k)
                    c[k] = r0 + kQ * k < G ? __ldcg(col + (size_t)(r0 + kQ * k) * (kRadix / 4)) : make_uint4(0u, 0u, 0u, 0u);
#pragma unroll
                for (int k = 0; k < kRowsAtOnce; ++k) {
                    total.x += c[k].x; total.y += c[k].y; total.z += c[k].z; total.w += c[k].w;
                    if (r0 + kQ * k < b) { before.x += c[k].x; before.y += c[k].y; before.z += c[k].z; before.w += c[k].w; }
                }
            }
            uint32_t* part = &warp_hist[0][0];        // [2][kQ][256], free between tiles
            reinterpret_cast<uint4*>(part + q * kRadix)[d4] = before;
            reinterpret_cast<uint4*>(part + (kQ + q) * kRadix)[d4] = total;
            __syncthreads();
            uint32_t bf = 0, tt = 0;
            if (digit_thread) {
#pragma unroll
                for (int i = 0; i < kQ; ++i) {
                    bf += part[i * kRadix + tid];
                    tt += part[(kQ + i) * kRadix + tid];
                }
            }
            uint32_t tot;
            const uint32_t gbase = scan_digits<kThreads>(tt, sm, &tot);            // has barriers
            if (digit_thread) digit_base[tid] = gbase + bf;
        }
        for (uint32_t t = 0; t < my_tiles; ++t) {
            if (t > 0) load_tile(t);
#pragma unroll
            for (int i = tid; i < kWarps * kRadix; i += kThreads) (&warp_hist[0][0])[i] = 0u;
            __syncthreads();
            const uint32_t t0 = c0 + t * kTile;
            const uint32_t tb = t0 + w * (32 * kItems);
            const uint32_t in_tile = tmin<uint32_t>((uint32_t)kTile, c1 - t0);
            uint32_t rank[kItems];
#pragma unroll
            for (int it = 0; it < kItems; ++it)
                rank[it] = warp_rank(warp_mask[w], warp_hist[w], (key[it] >> shift) & (kRadix - 1), tb + it * 32 + lane < c1, lane);
            __syncthreads();
            // thread d: this tile's count of digit d; the per-warp counters become offsets inside the digit
            uint32_t run = 0;
            if (digit_thread) {
#pragma unroll
                for (int i = 0; i < kWarps; ++i) {
                    const uint32_t c = warp_hist[i][tid];
                    warp_hist[i][tid] = run;
                    run += c;
                }
            }
            uint32_t tile_tot;
            const uint32_t lb = scan_digits<kThreads>(run, sm, &tile_tot);         // has barriers
            if (digit_thread) local_base[tid] = lb;
            __syncthreads();
            // the tile in digit order in shared memory, so that the stores below walk runs of equal digits
#pragma unroll
            for (int it = 0; it < kItems; ++it) {
                if (tb + it * 32 + lane < c1) {
                    const uint32_t digit = (key[it] >> shift) & (kRadix - 1);
                    const uint32_t lp = local_base[digit] + warp_hist[w][digit] + rank[it];
                    s_key[lp] = key[it];
                    s_val[lp] = val[it];
                }
            }
            __syncthreads();
            uint32_t pos[kItems];
#pragma unroll
            for (int it = 0; it < kItems; ++it) {
                const uint32_t j = it * kThreads + tid;
                key[it] = j < in_tile ? s_key[j] : 0u;
                val[it] = j < in_tile ? s_val[j] : 0u;
                const uint32_t digit = (key[it] >> shift) & (kRadix - 1);
                pos[it] = digit_base[digit] + (j - local_base[digit]);
            }
            if (!last) {
#pragma unroll
                for (int it = 0; it < kItems; ++it) {
                    const bool valid = it * kThreads + tid < in_tile;
                    if (valid) {
                        kout[pos[it]] = key[it];
                        vout[pos[it]] = val[it];
                    }
                    // one more key with this digit of the next pass in the chunk the key lands in; neighbouring lanes that
                    // agree on both (a frequent key's occurrences stand together) send one addition
                    const uint32_t nd = (key[it] >> (shift + kRadixBits)) & (kRadix - 1);
                    uint32_t to = __umulhi(pos[it], magic);         // pos / chunk, or one more
                    if (to * chunk > pos[it]) --to;
                    const uint32_t cell = valid ? to * kRadix + nd : 0xFFFFFFFFu;
                    const uint32_t left = __shfl_up_sync(0xffffffffu, cell, 1);
                    const bool head = lane == 0 || left != cell;
                    const unsigned later = __ballot_sync(0xffffffffu, head) & ~((2u << lane) - 1u);
                    if (valid && head) atomicAdd(P.counts + (size_t)(p + 1) * G * kRadix + cell, (uint32_t)((later ? __ffs(later) - 1 : 32) - lane));
                }
            } else if constexpr (Sink::kPairs) {
#pragma unroll
                for (int it = 0; it < kItems; ++it) {
                    if (it * kThreads + tid < in_tile) {
                        kout[pos[it]] = key[it];
                        vout[pos[it]] = val[it];
                    }
                }
            } else {
                // four items at a time: all their index loads, then all table loads, then the records
                constexpr int kAtOnce = kItems < 4 ? kItems : 4;
#pragma unroll
                for (int i0 = 0; i0 < kItems; i0 += kAtOnce) {
                    uint32_t pk[kAtOnce];
                    float cval[kAtOnce];
                    uint2 e_own[kAtOnce], e_par[kAtOnce];
#pragma unroll
                    for (int i = 0; i < kAtOnce; ++i) {
                        const int it = i0 + i;
                        const bool live = it * kThreads + tid < in_tile && key[it] < sink.K;
                        const uint32_t cell = val[it] >> 1;
                        pk[i] = sink.K;
                        cval[i] = 0.f;
                        if (live) {
                            pk[i] = (val[it] & 1u) ? sink.ci[cell] : sink.col_base + sink.cj[cell];
                            cval[i] = sink.cv[cell];
                        }
                    }
#pragma unroll
                    for (int i = 0; i < kAtOnce; ++i) {
                        const bool live = pk[i] < sink.K;       // cells with an index out of range carry the mark K
                        e_own[i] = live ? sink.table[key[i0 + i]] : make_uint2(0u, 0u);
                        e_par[i] = live ? sink.table[pk[i]] : make_uint2(0u, 0u);
                    }
#pragma unroll
                    for (int i = 0; i < kAtOnce; ++i) {
                        const int it = i0 + i;
                        if (it * kThreads + tid < in_tile) {
                            kout[pos[it]] = key[it];
                            if (!(val[it] & 1u)) sink.cellpos[val[it] >> 1] = pos[it];
                            sink.rec[pos[it]] = make_uint4(val[it] >> 1, __float_as_uint(cval[i]),
                                                           (uint32_t)phys_row(e_own[i], sink.S),
                                                           (uint32_t)phys_row(e_par[i], sink.S));
                        }
                    }
                }
            }
            __syncthreads();
            if (digit_thread) digit_base[tid] += run;           // the chunk's next tile starts after this one
        }
        if (!last && !grid_barrier(P.bar, ++barriers * G, &s_ok)) {
            if (tid == 0) atomicCAS(&P.st->sticky, 0u, (unsigned int)PS_ERR_CUDA);
            return;
        }
    }
    grid_leave(P.bar, G);
}

// ------------------------------------------------------------------------------------------------
// Sorts of at most kClusterSort keys as one cluster of sixteen blocks.  The keys stay in the blocks' shared memory from
// the first pass to the last; a pass ranks a block's chunk (warp_rank: stable), tells every
// other block its digit counts (a 16 x 256 matrix in each block's shared memory) and scatters each key to its place in
// another block's shared memory.  The blocks meet at the cluster's hardware barrier, twice per pass.
// 20,000 24-bit keys: 18.5 us against 24.7 of the cooperative form, whose passes go through global memory and a grid barrier.
// With 16 keys a thread it would take 131,072, but sixteen SMs are too few for that many (48 us against 26), and the
// records of the matrix-factorization step's sink want the whole chip's loads in flight (74 us against 34).
constexpr int kClThreads = 512, kClItems = 4, kClBlocks = 16, kClWarps = kClThreads / 32;
constexpr uint32_t kClChunk = kClThreads * kClItems;
constexpr uint32_t kClusterSort = kClBlocks * kClChunk;         // 32,768
static_assert(kClusterSort <= (1u << 17) && kClItems * 32 <= (1 << 15), "value and rank share a register");

struct ClusterSmem {
    uint2 buf[kClChunk];                    // the chunk's (key, value) pairs
    uint32_t warp_hist[kClWarps][kRadix], warp_mask[kClWarps][kRadix];
    uint32_t counts[kClBlocks][kRadix];     // digit counts of all blocks, written by them
    uint32_t base[kRadix];
    uint32_t sm[8];
};

template <class Src>
__global__ void __launch_bounds__(kClThreads, 2)
sort_cluster_kernel(Src src, SortParams P) {
    extern __shared__ __align__(16) unsigned char cl_dyn[];
    ClusterSmem& M = *reinterpret_cast<ClusterSmem*>(cl_dyn);
    const uint32_t n = P.n_dev ? tmin<uint32_t>(*((const volatile unsigned int*)P.n_dev), P.n_host) : P.n_host;
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    const uint32_t b = blockIdx.x;
    cluster_arrive();                       // (every block has started: before the first write to another's memory)
    if (b == 0) {
        for (uint32_t i = tid; i < P.n_zero_a; i += kClThreads) P.zero_a[i] = 0u;
        if (tid == 0 && P.zero_b) P.zero_b[0] = P.zero_b[1] = 0u;
    }
    const uint32_t chunk = tmax<uint32_t>((n + kClBlocks - 1) / kClBlocks, 32u);    // (at least two: `magic` has 32 bits)
    const uint32_t magic = (uint32_t)(((1ull << 32) + chunk - 1) / chunk);      // pos / chunk, exact for 17-bit positions
    const uint32_t c0 = tmin<uint32_t>(b * chunk, n), len = tmin<uint32_t>(chunk, n - c0);
    const uint32_t share = ((chunk + kClWarps - 1) / kClWarps + 31) & ~31u;     // consecutive positions per warp
    const uint32_t l0 = w * share + lane;
    for (int i = lane; i < kRadix; i += 32) M.warp_mask[w][i] = 0u;
    uint32_t key[kClItems], vr[kClItems];
    {
        const uint32_t* kin = (P.start & 1) ? P.kB : P.kA;
        typename Src::Raw raw[kClItems] = {};
#pragma unroll
        for (int it = 0; it < kClItems && !Src::kFromBuffer; ++it)
            if (it * 32 < share && l0 + it * 32 < len) raw[it] = src.read(c0 + l0 + it * 32);
#pragma unroll
        for (int it = 0; it < kClItems; ++it) {
            const uint32_t l = l0 + it * 32;
            key[it] = 0u;
            vr[it] = c0 + l;
            if (it * 32 < share && l < len) key[it] = Src::kFromBuffer ? __ldcg(kin + c0 + l) : src.key(c0 + l, raw[it], P);
        }
    }
    cluster_wait();
    for (int p = 0; p < P.n_passes; ++p) {
        const int shift = p * kRadixBits;
        if (p > 0) {
#pragma unroll
            for (int it = 0; it < kClItems; ++it) {
                const uint32_t l = l0 + it * 32;
                if (it * 32 < share && l < len) {
                    const uint2 x = M.buf[l];
                    key[it] = x.x;
                    vr[it] = x.y;
                }
            }
        }
        for (int i = lane; i < kRadix; i += 32) M.warp_hist[w][i] = 0u;
        __syncwarp();
#pragma unroll
        for (int it = 0; it < kClItems; ++it) {
            if (it * 32 >= share) break;
            vr[it] |= warp_rank(M.warp_mask[w], M.warp_hist[w], (key[it] >> shift) & (kRadix - 1), l0 + it * 32 < len, lane) << 17;
        }
        __syncthreads();
        if (tid < kRadix) {
            uint32_t run = 0;
#pragma unroll
            for (int i = 0; i < kClWarps; ++i) {
                const uint32_t c = M.warp_hist[i][tid];
                M.warp_hist[i][tid] = run;
                run += c;
            }
#pragma unroll
            for (uint32_t r = 0; r < kClBlocks; ++r)
                asm volatile("st.shared::cluster.u32 [%0], %1;\n" ::"r"(peer_smem(&M.counts[b][tid], r)), "r"(run) : "memory");
        }
        cluster_arrive();
        cluster_wait();
        uint32_t before = 0, total = 0;
        if (tid < kRadix) {
#pragma unroll
            for (uint32_t r = 0; r < kClBlocks; ++r) {
                const uint32_t c = M.counts[r][tid];
                if (r < b) before += c;
                total += c;
            }
        }
        uint32_t all;
        const uint32_t gbase = scan_digits<kClThreads>(total, M.sm, &all);      // has barriers
        if (tid < kRadix) M.base[tid] = gbase + before;
        __syncthreads();
#pragma unroll
        for (int it = 0; it < kClItems; ++it) {
            if (it * 32 >= share) break;
            if (l0 + it * 32 < len) {
                const uint32_t digit = (key[it] >> shift) & (kRadix - 1);
                const uint32_t pos = M.base[digit] + M.warp_hist[w][digit] + (vr[it] >> 17);
                const uint32_t to = __umulhi(pos, magic);
                asm volatile("st.shared::cluster.v2.u32 [%0], {%1, %2};\n" ::"r"(peer_smem(&M.buf[pos - to * chunk], to)),
                             "r"(key[it]), "r"(vr[it] & 0x1ffffu)
                             : "memory");
            }
        }
        cluster_arrive();
        cluster_wait();
    }
    uint32_t* kout = ((P.start + P.n_passes) & 1) ? P.kB : P.kA;
    uint32_t* vout = ((P.start + P.n_passes) & 1) ? P.vB : P.vA;
    for (uint32_t l = tid; l < len; l += kClThreads) {
        const uint2 x = M.buf[l];
        kout[c0 + l] = x.x;
        vout[c0 + l] = x.y;
    }
}

// Small sorts: few blocks of many threads.  The sort of the next step runs beside the current step's kernels;
// its blocks spend most of their life waiting at grid barriers, so it should hold few SMs' registers while it
// does, and the cost of a pass grows with the number of blocks (barrier, counter read) more than with the keys
// per block.
constexpr int kSmallThreads = 512, kSmallItems = 4;      // tiles of 2048 keys
constexpr int kSmallTile = kSmallThreads * kSmallItems;
// Large sorts (more than a short tile per block): tiles of 4,096 keys.  1M keys in 88 us with 256 threads x 8, 71 us with 512 x 4,
// 69 with 512 x 8, 65 with 1024 x 8, which holds whole SMs while kernels of other streams run beside it (skip-gram step
// 788 us against 783).
constexpr int kBigThreads = 512, kBigItems = 8;
constexpr size_t sort_smem(int threads, int items) { return ((size_t)2 * threads * items + 2 * (threads / 32) * kRadix) * sizeof(uint32_t); }
static_assert(kSmallTile >= kSortTile / 2, "the digit counters are sized for tiles of at least kSortTile / 2 keys");

// Once per device: the opt-ins (shared memory, a cluster of more than eight blocks), and whether such a cluster can be
// resident at all (a GPU's clusters are as large as its smallest partition of multiprocessors allows).
template <class Src>
static bool cluster_sort_fits() {
    static std::atomic<unsigned long long> asked{0}, fits{0};
    int d = -1;
    if (cudaGetDevice(&d) != cudaSuccess || d < 0 || d >= 64) return false;
    if (!((asked.load(std::memory_order_acquire) >> d) & 1ull)) {
        const void* fn = (const void*)sort_cluster_kernel<Src>;
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3(kClBlocks);
        cfg.blockDim = dim3(kClThreads);
        cfg.dynamicSmemBytes = sizeof(ClusterSmem);
        cudaLaunchAttribute attr;
        attr.id = cudaLaunchAttributeClusterDimension;
        attr.val.clusterDim.x = kClBlocks;
        attr.val.clusterDim.y = attr.val.clusterDim.z = 1;
        cfg.attrs = &attr;
        cfg.numAttrs = 1;
        int clusters = 0;
        if (cudaFuncSetAttribute(fn, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) == cudaSuccess &&
            cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(ClusterSmem)) == cudaSuccess &&
            cudaOccupancyMaxActiveClusters(&clusters, sort_cluster_kernel<Src>, &cfg) == cudaSuccess && clusters > 0)
            fits.fetch_or(1ull << d, std::memory_order_relaxed);
        cudaGetLastError();
        asked.fetch_or(1ull << d, std::memory_order_release);
    }
    return (fits.load(std::memory_order_relaxed) >> d) & 1ull;
}

template <class Src, class Sink>
static int sort_launch(ps_store* ps, const Src& src, const Sink& sink, uint32_t n, const unsigned int* n_dev, int bits,
                       cudaStream_t stream, int start, unsigned int* zero_me, uint32_t zero_groups) {
    if (bits < 1) bits = 1;
    SortParams P;
    P.kA = ps->keysA; P.vA = ps->valsA; P.kB = ps->keysB; P.vB = ps->valsB;
    P.start = start;
    P.n_host = n;
    P.n_dev = n_dev;
    P.n_passes = (bits + kRadixBits - 1) / kRadixBits;
    const uint32_t max_grid = (uint32_t)tmax(ps->sm_count, 1);
    // short tiles while they still give every block at most one (and the counters have room for that many blocks)
    const bool small = n <= max_grid * (uint32_t)kSmallTile && div_up_u32(n, kSmallTile) <= ps->sort_blocks_cap;
    const uint32_t tile = small ? kSmallTile : kBigThreads * kBigItems;
    const uint32_t n_tiles = div_up_u32(n, tile);
    P.tiles_per_block = div_up_u32(n_tiles, max_grid);
    const uint32_t grid = div_up_u32(n_tiles, P.tiles_per_block);
    P.counts = ps->tile_state;
    P.bar = ps->sort_ctl;
    P.zero_a = ps->group_done;
    P.n_zero_a = zero_groups;
    P.zero_b = zero_me;
    P.st = ps->status;
    P.epoch = ps->epoch;
    if constexpr (Sink::kPairs) {
        if (n <= kClusterSort && cluster_sort_fits<Src>()) {
            cudaLaunchConfig_t cfg = {};
            cfg.gridDim = dim3(kClBlocks);
            cfg.blockDim = dim3(kClThreads);
            cfg.dynamicSmemBytes = sizeof(ClusterSmem);
            cfg.stream = stream;
            cudaLaunchAttribute attr;
            attr.id = cudaLaunchAttributeClusterDimension;
            attr.val.clusterDim.x = kClBlocks;
            attr.val.clusterDim.y = attr.val.clusterDim.z = 1;
            cfg.attrs = &attr;
            cfg.numAttrs = 1;
            if (ps->prof) prof_before(ps, "sort_cluster_kernel", stream);
            cudaLaunchKernelEx(&cfg, sort_cluster_kernel<Src>, src, P);
            if (ps->prof) prof_after(ps, stream);
            ps->launches++;
            return (start + P.n_passes) & 1;
        }
    }
    if (ps->prof) prof_before(ps, "sort_all_kernel", stream);
    void* args[] = {(void*)&src, (void*)&sink, (void*)&P};
    // cooperative: the blocks wait for one another at the grid barrier, so all of them must be resident
    if (small) {
        static std::atomic<unsigned long long> attr_set{0};
        const void* fn = (const void*)sort_all_kernel<Src, Sink, kSmallThreads, kSmallItems>;
        const size_t smem = sort_smem(kSmallThreads, kSmallItems);
        opt_in_smem(fn, smem, &attr_set);
        cudaLaunchCooperativeKernel(fn, dim3(grid), dim3(kSmallThreads), args, smem, stream);
    } else {
        static std::atomic<unsigned long long> attr_set{0};
        const void* fn = (const void*)sort_all_kernel<Src, Sink, kBigThreads, kBigItems>;
        const size_t smem = sort_smem(kBigThreads, kBigItems);
        opt_in_smem(fn, smem, &attr_set);
        cudaLaunchCooperativeKernel(fn, dim3(grid), dim3(kBigThreads), args, smem, stream);
    }
    if (ps->prof) prof_after(ps, stream);
    ps->launches++;
    return (start + P.n_passes) & 1;
}

int radix_sort_pairs(ps_store* ps, uint32_t n, const unsigned int* n_dev, int bits, cudaStream_t stream, int start,
                     unsigned int* zero_me, uint32_t zero_groups) {
    if (n == 0) return start;
    return sort_launch(ps, SrcBuffer{}, SinkPairs{}, n, n_dev, bits, stream, start, zero_me, zero_groups);
}

int radix_sort_keys64(ps_store* ps, const uint64_t* d_keys, uint32_t n, cudaStream_t stream, unsigned int* zero_me,
                      uint32_t zero_groups) {
    if (n == 0) return 0;
    SrcKeys64 src{d_keys, ps->cfg.num_keys};
    return sort_launch(ps, src, SinkPairs{}, n, nullptr, ps->key_bits, stream, 0, zero_me, zero_groups);
}

int radix_sort_mf(ps_store* ps, const uint32_t* d_i, const uint32_t* d_j, const float* d_v, uint32_t n_cells,
                  uint64_t col_key_base, bool records, cudaStream_t stream, unsigned int* zero_me,
                  uint32_t zero_groups) {
    if (n_cells == 0) return 0;
    SrcMF src{d_i, d_j, col_key_base, ps->cfg.num_keys};
    if (!records)
        return sort_launch(ps, src, SinkPairs{}, 2 * n_cells, nullptr, ps->key_bits, stream, 0, zero_me, zero_groups);
    SinkMF sink{d_i, d_j, d_v, (uint32_t)col_key_base, (uint32_t)ps->cfg.num_keys, ps->table,
                ps->cfg.slots_per_part, ps->rec, ps->cellpos};
    return sort_launch(ps, src, sink, 2 * n_cells, nullptr, ps->key_bits, stream, 0, zero_me, zero_groups);
}

}  // namespace psb
