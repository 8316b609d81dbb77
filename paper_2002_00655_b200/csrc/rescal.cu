// RESCAL (Section 4.1 of the paper names the model; Table 4: entity dimension d, relation dimension d * d): the
// gradient kernels of one minibatch.  Rows of the store have one length, so a relation's d x d matrix is d keys, one per
// matrix row:  key e < rel_base: entity e, row [x | G];  key rel_base + r d + a: row a of R_r, row [R_r[a][.] | G]
// (G: element-wise AdaGrad accumulators, row_len = 2 d).  Score  phi(s, r, o) = x_s^T R_r x_o.
//
// A data point is a positive triple and its negatives (each replaces the subject or the object).  With c_q the
// derivative of softplus(-y phi_q) with respect to phi_q, the gradients of the data point's loss factor through four
// matrix-vector products of the one matrix R = R_r:
//   u = R x_o,  w = R^T x_s                 phi_pos = x_s . u,  phi of a subject-negative k = x_k . u,  of an
//                                           object-negative k = w . x_k
//   a = c_pos x_s + sum over subject-negatives c_k x_k,   b' = sum over object-negatives c_k x_k,  b = c_pos x_o + b'
//   subject slot: R b      object slot: R^T a      subject-negative k: c_k u      object-negative k: c_k w
//   matrix row alpha:  a[alpha] x_o + x_s[alpha] b'
// Slots that hold the same entity are folded into the first of them before anything is written (AdaGrad is taken on
// the gradient with respect to each DISTINCT key), as the key kernel marks the later ones "no key": the gradient of an
// entity slot is c1 (R b) + c2 (R^T a) + c3 u + c4 w with four numbers per slot, and folding adds the numbers.
//
// The data points of a batch that share a relation share its matrix, so the batch is worked on by relation: a data point
// has 2 + n_neg entity slots and ONE slot for its relation in the key sort, the relations' runs of sorted positions are
// its groups (segments.cu), and
//   rescal_points_kernel  takes up to eight data points of one relation per block.  The matrix goes to shared memory once
//                         for all of them and the four products are matrix products on the fp64 tensor instructions
//                         (DMMA, m8n8k4); scores, coefficients and the entities' gradients follow in the same block.
//                         An entity whose key occurs once in the batch is updated in place, the others' gradients go to
//                         the segmented reduction.  Per data point it leaves the vectors a, b', x_o, x_s.
//   rescal_matrix_kernel  updates the matrices: a thread holds a few elements of R and G in registers and walks over
//                         the relation's data points, forming each one's gradient a[alpha] x_o + x_s[alpha] b' from those
//                         vectors (staged in shared memory) and AdaGrad's step from it; sums in fp64, one rounding.
// The d * d gradients of a data point never go through memory (335 MB per 8,192 data points of dimension 100 did, with
// a sort of 112 keys per data point where 13 do now), and a relation's rows are read and written once per batch.
// Before: a warp per data point with two passes over the matrix in L2, 292 us, and the matrix rows through the sorted
// reduction, 278 us, of 577 us per step of 8,192 data points of dimension 100; now 122 + 105 us with the entities' reduction beside the latter, 235 us per step.
// rescal_points_kernel is bound by the latency of its phases (16 warps per SM, issue slots 40 % used, tensor pipe 27 %),
// rescal_matrix_kernel by instruction issue and the special-function unit.
#include <string.h>

#include "ps_internal.cuh"

namespace psb {

namespace {

constexpr int kPoints = 8;                      // columns of one tile: data points of one relation per block at a time, a warp each
constexpr int kMatThreads = 256;                // eight matrix elements each
constexpr int kMatStage = 8;                    // data points whose vectors are staged together

// Row stride of the matrix and of the vectors in shared memory: 4 mod 8 elements, so that the eight rows x four columns a
// warp reads for one tensor instruction fall into different banks (two-way for the transposed read).
__host__ __device__ constexpr uint32_t pad_ld(uint32_t d) { return d % 8 == 4 ? d : d + 4; }

struct RescalArgs {
    const uint32_t *ts, *tr, *to, *neg_ent;
    const uint8_t* neg_side;
    uint32_t n, n_neg, d, K;
    uint64_t rel_base;
    float lr, eps;
    float* store;
    const uint2* table;
    uint64_t S;
    float* grad;                    // a row of d values per slot (2 + n_neg + n_mat per data point)
    double* vec;                    // per data point: a, b', x_o, x_s
    double* loss_of;                // per data point
    const uint32_t *sk, *sv;        // sorted keys and occurrences (null: calls without a sort)
    SegLists L;
    uint32_t* keys_out;             // calls without a sort: keys of all slots, the d matrix rows among them
    DevStatus* st;
    unsigned int epoch;
};

// D += A B, fp64: A 8x4 (lane: row lane / 4, column lane % 4), B 4x8 (row lane % 4, column lane / 4), D 8x8 (row lane / 4,
// columns 2 (lane % 4) and the next)
__device__ __forceinline__ void dmma(double (&c)[2], double a, double b) {
    asm volatile("mma.sync.aligned.m8n8k4.row.col.f64.f64.f64.f64 {%0, %1}, {%2}, {%3}, {%0, %1};"
                 : "+d"(c[0]), "+d"(c[1]) : "d"(a), "d"(b));
}
__device__ __forceinline__ double sum8(double v) {          // over the eight lanes of a group
    v += __shfl_xor_sync(0xffffffffu, v, 1);
    v += __shfl_xor_sync(0xffffffffu, v, 2);
    return v + __shfl_xor_sync(0xffffffffu, v, 4);
}

// kSorted: the blocks take the pieces segment_kernel listed.  Otherwise (calls without a sort): data points one by one,
// every gradient row written (the d matrix rows' too) together with the slots' keys.
// All rows a block needs (the matrix, the points' entities) are asked for at once as bulk copies into shared memory and
// waited for once; with plain loads phase by phase the block's time was a chain of memory latencies (248 us a step).
// kWarps: 8, or 4 (up to four data points at a time) for dimensions up to 64, whose tiles four warps hold: as many warps per
// SM in twice the blocks, so a relation of few data points idles fewer warps (1,288 data points of 573 relations of dimension
// 28: 34.6 -> 23.8 us; 8,000 of 237 of dimension 64: 81 -> 76).
template <bool kSorted, int kWarps>
__global__ void __launch_bounds__(32 * kWarps, 16 / kWarps) rescal_points_kernel(const RescalArgs A) {
    constexpr int kPointThreads = 32 * kWarps;
    extern __shared__ __align__(128) unsigned char dyn[];
    __shared__ __align__(8) uint64_t bar, mat_bar;
    const unsigned full = 0xffffffffu;
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    const uint32_t d = A.d, d4 = d / 4, ld = pad_ld(d), n_neg = A.n_neg, n_ent = 2 + n_neg;
    const uint32_t n_slots = n_ent + (kSorted ? 1u : d);
    const bool slot = lane < (int)n_ent, act = (uint32_t)lane < d4;
    double* const Y = reinterpret_cast<double*>(dyn);           // [8][ld]: x_o, then b, then R b
    double* const X = Y + kPoints * ld;                         // x_s, then a, then R^T a
    double* const U = X + kPoints * ld;                         // R x_o
    double* const W = U + kPoints * ld;                         // R^T x_s
    float* const R = reinterpret_cast<float*>(W + kPoints * ld);        // [d][ld]
    float* const E = R + d * ld;                                // [points][n_ent][d]: the entities' rows
    if (tid < 2) mbar_init(tid ? &mat_bar : &bar, 1);
    mbar_init_fence();
    pdl_trigger();
    pdl_wait();
    if (kSorted && call_failed(A.st, A.epoch)) return;
    const uint64_t L = 2 * (uint64_t)d;
    const uint32_t row_bytes = d * 4;
    const uint32_t n_items = kSorted ? A.L.counts[2] : A.n;
    const uint32_t m_tiles = (d + 7) / 8;
    unsigned parity = 0;
    // Both products of a pass, R Y and R^T X: warp w takes the tiles w, w + kWarps, ... of the 2 m_tiles together
    // (four independent chains of tensor instructions).
    double acc[4][2];
    auto products = [&]() {
        const float* a[4];
        uint32_t step[4];
        bool tr[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const uint32_t job = tmin<uint32_t>(w + kWarps * j, 2 * m_tiles - 1);    // (past the last: computed, not stored)
            tr[j] = job >= m_tiles;
            const uint32_t row = tmin<uint32_t>((tr[j] ? job - m_tiles : job) * 8 + lane / 4, d - 1);
            a[j] = tr[j] ? R + (lane % 4) * ld + row : R + row * ld + lane % 4;
            step[j] = tr[j] ? 4 * ld : 4;
            acc[j][0] = acc[j][1] = 0.0;
        }
        const double* by = Y + (lane / 4) * ld + lane % 4;
        const double* bx = X + (lane / 4) * ld + lane % 4;
#pragma unroll 2
        for (uint32_t k = 0; k < d4; ++k) {
            const double y = by[4 * k], x = bx[4 * k];
#pragma unroll
            for (int j = 0; j < 4; ++j) dmma(acc[j], (double)a[j][k * step[j]], tr[j] ? x : y);
        }
    };
    auto store_products = [&](double* u, double* wt, uint32_t len) {
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const uint32_t job = w + kWarps * j;
            const bool tr = job >= m_tiles;
            const uint32_t row = (tr ? job - m_tiles : job) * 8 + lane / 4, col = 2 * (lane % 4);
            if (job >= 2 * m_tiles || row >= d) continue;
            double* o = (tr ? wt : u) + col * ld + row;
            if (col < len) o[0] = acc[j][0];
            if (col + 1 < len) o[ld] = acc[j][1];
        }
    };
    // kSorted: look-ups of an item, a chain of four (piece, data points, their slots' keys, places of the rows).  With eight warps a
    // link is asked for between the phases of the item before, and the matrix itself once that one's has been read (8,192 data
    // points of dimension 100: 4 of an item's 24 us; the step 238 -> 235; blocks of four warps, of which more share an SM, lose 1 %).
    constexpr bool kAhead = kSorted && kWarps == 8;
    struct {
        uint32_t pos, len, rk, t, key, side;
        bool once;
        uint2 entry, mat_entry;
    } next = {};
    auto find_piece = [&](uint32_t item) {
        const uint2 it = item < n_items ? A.L.pieces[item] : make_uint2(0u, 0u);
        next.pos = it.x;
        next.len = it.y;
    };
    auto find_points = [&]() {
        next.rk = next.len ? A.sk[next.pos] : 0u;
        next.t = w < (int)next.len ? A.sv[next.pos + w] / n_slots : 0u;
    };
    auto key_of = [&](uint64_t t) -> uint32_t { return lane == 0 ? A.ts[t] : lane == 1 ? A.to[t] : A.neg_ent[t * n_neg + (lane - 2)]; };
    auto find_keys = [&]() {
        const bool mine = w < (int)next.len && slot;
        next.key = mine ? key_of(next.t) : 0u;
        next.side = mine && lane >= 2 ? A.neg_side[(uint64_t)next.t * n_neg + (lane - 2)] : 0u;
        next.once = mine && A.L.single[(uint64_t)next.t * n_slots + lane];
        next.mat_entry = next.len && tid < (int)d ? A.table[next.rk + tid] : make_uint2(0u, 0u);
    };
    auto find_rows = [&]() { next.entry = w < (int)next.len && slot ? A.table[next.key] : make_uint2(0u, 0u); };
    auto announce_matrix = [&]() {
        if (tid == 0 && next.len) mbar_expect_tx(&mat_bar, d * row_bytes);
    };
    auto ask_matrix = [&]() {                   // (after the block has met: nobody reads the matrix before)
        if (next.len && tid < (int)d) bulk_g2s(R + tid * ld, A.store + phys_row(next.mat_entry, A.S) * L, row_bytes, &mat_bar);
    };
    auto look_up = [&](uint32_t item) {
        find_piece(item);
        find_points();
        find_keys();
        find_rows();
        if (tid == 0 && next.len) mbar_expect_tx(&bar, next.len * n_ent * row_bytes);
        announce_matrix();
        fence_async_smem();                     // (the rows of the item before have been read)
        __syncthreads();
        ask_matrix();
    };
    if (kAhead) look_up(blockIdx.x);
    for (uint32_t item = blockIdx.x; item < n_items; item += gridDim.x) {
        if (kSorted && !kAhead) look_up(item);
        const uint32_t len = kSorted ? next.len : 1;
        const uint64_t rk = kSorted ? next.rk : A.rel_base + (uint64_t)A.tr[item] * d;
        if (!kSorted) {
            if (tid == 0) mbar_expect_tx(&bar, (d + n_ent) * row_bytes);
            fence_async_smem();                 // (the rows of the item before have been read)
            __syncthreads();
        }
        // ---- the slots of the warp's data point: lane u holds slot u (subject, object, negatives) ----
        const bool mine = w < (int)len;
        const uint64_t t = !mine ? 0 : kSorted ? next.t : item;
        uint32_t key = 0, side = 0;
        int rep = lane;
        bool once = false, bad = !kSorted && rk + d > A.K;
        uint64_t erow = 0;
        if (mine) {
            if (kSorted) {
                key = next.key;
                side = next.side;
            } else if (slot) {
                key = key_of(t);
                if (lane >= 2) side = A.neg_side[t * n_neg + (lane - 2)];
                bad |= key >= A.rel_base;
            }
            const unsigned same = __match_any_sync(full, slot ? key : kSentinelPad);
            if (slot) rep = __ffs(same) - 1;
            if (kSorted && slot) once = rep == lane && next.once;
        }
        if (!kSorted) {                         // (a call with a sort: checked and latched by its key kernel)
            uint32_t* ko = A.keys_out + (uint64_t)item * n_slots;
            if (__syncthreads_or(bad)) {
                if (tid == 0) {
                    latch_error(A.st, 0u, PS_ERR_KEY_RANGE);
                    // nothing is copied for this item: the announced bytes are taken back by starting the barrier anew
                    mbar_inval(&bar);
                    mbar_init(&bar, 1);
                }
                mbar_init_fence();
                parity = 0;
                for (uint32_t u = tid; u < n_slots; u += kPointThreads) ko[u] = kSentinelPad;
                __syncthreads();
                continue;
            }
            if (w == 0 && slot) ko[lane] = rep == lane ? key : A.K;
            for (uint32_t a = tid; a < d; a += kPointThreads) ko[n_ent + a] = (uint32_t)(rk + a);
        }
        if (mine && slot) {
            erow = phys_row(kSorted ? next.entry : A.table[key], A.S);
            bulk_g2s(E + (w * n_ent + lane) * d, A.store + erow * L, row_bytes, &bar);
            if (once)                           // its accumulators are wanted at the end
                for (uint32_t o = 0; o < row_bytes; o += 128)
                    asm volatile("prefetch.global.L2 [%0];" ::"l"((const char*)(A.store + erow * L + d) + o));
        }
        if (!kSorted && tid < (int)d) bulk_g2s(R + tid * ld, A.store + phys_row(A.table[rk + tid], A.S) * L, row_bytes, &bar);
        if (kAhead) find_piece(item + gridDim.x);
        // (both are waited for, also where one does not come: a block that gives up has no copy on its way)
        const bool rows_in = mbar_wait(&bar, parity) || mbar_wait(&bar, parity);
        const bool matrix_in = !kSorted || mbar_wait(&mat_bar, parity) || mbar_wait(&mat_bar, parity);
        if (__syncthreads_or(!rows_in || !matrix_in)) {
            if (tid == 0) {
                latch_error(A.st, kSorted ? A.epoch : 0u, PS_ERR_CUDA);
                if (!kSorted) A.keys_out[(uint64_t)item * n_slots] = kSentinelPad;      // (the reduction then does nothing)
            }
            return;                             // a copy that does not arrive: give the call up
        }
        parity ^= 1;
        const float4* const e4 = reinterpret_cast<const float4*>(E + w * n_ent * d);    // row z of the warp's point: e4 + z d4
        float4 x_s = make_float4(0.f, 0.f, 0.f, 0.f), x_o = x_s;
        if (act) {
            if (mine) {
                x_s = e4[lane];
                x_o = e4[d4 + lane];
            }
            double* y = Y + w * ld + 4 * lane;
            double* x = X + w * ld + 4 * lane;
            y[0] = x_o.x; y[1] = x_o.y; y[2] = x_o.z; y[3] = x_o.w;
            x[0] = x_s.x; x[1] = x_s.y; x[2] = x_s.z; x[3] = x_s.w;
        }
        __syncthreads();
        if (kAhead) find_points();
        products();
        store_products(U, W, len);
        __syncthreads();
        if (kAhead) find_keys();
        // ---- scores, coefficients, a and b ----
        double coef = 0;                        // lane 1: the positive's, lane 2 + q: negative q's
        if (mine) {
            const double *x = X + w * ld, *u = U + w * ld, *wv = W + w * ld;
            const int g = lane >> 3, l8 = lane & 7;
            double phi = 0;
            // eight lanes per triple; slot 1 stands for the positive, u . x_s
            for (uint32_t z0 = 1; z0 < n_ent; z0 += 4) {
                const uint32_t z = z0 + g;
                const uint32_t sd = __shfl_sync(full, side, z & 31);
                double s = 0;
                if (z < n_ent) {
                    const double* m = (z == 1 || sd == 0) ? u : wv;
                    const float4* row = e4 + (z == 1 ? 0 : z * d4);
#pragma unroll 4
                    for (uint32_t e = l8; e < d4; e += 8) {
                        const float4 v = row[e];
                        const double2 m0 = *reinterpret_cast<const double2*>(m + 4 * e), m1 = *reinterpret_cast<const double2*>(m + 4 * e + 2);
                        s += (double)v.x * m0.x + (double)v.y * m0.y + (double)v.z * m1.x + (double)v.w * m1.y;
                    }
                }
                s = sum8(s);
                const double got = __shfl_sync(full, s, ((lane - z0) & 3) * 8);
                if ((uint32_t)lane >= z0 && (uint32_t)lane < z0 + 4) phi = got;
            }
            double loss = 0;
            if (lane >= 1 && slot) {
                const double yl = lane == 1 ? 1.0 : -1.0, z = -yl * phi, e = exp(-fabs(z));
                coef = -yl * ((z >= 0.0 ? 1.0 : e) / (1.0 + e));
                loss = fmax(z, 0.0) + log1p(e);
            }
            loss = warp_sum_d(loss);
            if (lane == 0) A.loss_of[t] = loss;
            const double c_pos = __shfl_sync(full, coef, 1);
            double a[4] = {c_pos * (double)x_s.x, c_pos * (double)x_s.y, c_pos * (double)x_s.z, c_pos * (double)x_s.w};
            double b[4] = {0.0, 0.0, 0.0, 0.0};
#pragma unroll 2
            for (uint32_t z = 2; z < n_ent; ++z) {
                const double c = __shfl_sync(full, coef, z);
                const uint32_t sd = __shfl_sync(full, side, z);
                const float4 v = act ? e4[z * d4 + lane] : make_float4(0.f, 0.f, 0.f, 0.f);
                const double vv[4] = {v.x, v.y, v.z, v.w};
                if (sd == 0) {
#pragma unroll
                    for (int i = 0; i < 4; ++i) a[i] += c * vv[i];
                } else {
#pragma unroll
                    for (int i = 0; i < 4; ++i) b[i] += c * vv[i];
                }
            }
            if (act) {
                const double o[4] = {x_o.x, x_o.y, x_o.z, x_o.w}, sx[4] = {x_s.x, x_s.y, x_s.z, x_s.w};
                // for the matrices: a, b', x_o, x_s (calls without a sort: in columns of U that one data point leaves free)
                double* v = kSorted ? A.vec + t * d * 4 : U + ld;
                const uint32_t vs = kSorted ? d : ld;
#pragma unroll
                for (int i = 0; i < 4; i += 2) {
                    *reinterpret_cast<double2*>(v + 4 * lane + i) = make_double2(a[i], a[i + 1]);
                    *reinterpret_cast<double2*>(v + vs + 4 * lane + i) = make_double2(b[i], b[i + 1]);
                    *reinterpret_cast<double2*>(v + 2 * vs + 4 * lane + i) = make_double2(o[i], o[i + 1]);
                    *reinterpret_cast<double2*>(v + 3 * vs + 4 * lane + i) = make_double2(sx[i], sx[i + 1]);
                }
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    X[w * ld + 4 * lane + i] = a[i];
                    Y[w * ld + 4 * lane + i] = c_pos * o[i] + b[i];
                }
            }
        }
        __syncthreads();
        if (kAhead) find_rows();
        products();
        if (kAhead) {
            fence_async_smem();
            announce_matrix();
        }
        __syncthreads();
        if (kAhead) ask_matrix();
        store_products(Y, X, len);              // R b, R^T a
        __syncthreads();
        // ---- the entities' gradients, folded into the first slot of each key ----
        if (mine) {
            double c3 = 0, c4 = 0;              // lane v: the numbers of slot v
            unsigned roles = 0;                 // ... and what it is: subject, object, negative in the subject's place, in the object's
            for (int z = 0; z < (int)n_ent; ++z) {
                const int rz = __shfl_sync(full, rep, z);
                const double cz = __shfl_sync(full, coef, z);
                const uint32_t sz = __shfl_sync(full, side, z);
                if (rz != lane) continue;
                if (z >= 2 && sz == 0u) c3 += cz;
                else if (z >= 2) c4 += cz;
                roles |= z < 2 ? 1u << z : sz == 0u ? 4u : 8u;
            }
            double gs[4], go[4], u[4], wv[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const uint32_t e = w * ld + 4 * lane + i;
                gs[i] = act ? Y[e] : 0.0;
                go[i] = act ? X[e] : 0.0;
                u[i] = act ? U[e] : 0.0;
                wv[i] = act ? W[e] : 0.0;
            }
            float* out = A.grad + t * n_slots * d;
            const unsigned reps = __ballot_sync(full, slot && rep == lane), in_place = __ballot_sync(full, once);
            // A slot's gradient has the terms of its roles only, nearly always one (a number that is zero does not say that: the
            // score that made it so may be infinite, and zero times that is no number).
            const unsigned as_s = __ballot_sync(full, roles & 1u), as_o = __ballot_sync(full, roles & 2u);
            const unsigned as_3 = __ballot_sync(full, roles & 4u), as_4 = __ballot_sync(full, roles & 8u);
            for (uint32_t v0 = 0; v0 < n_ent; v0 += 4) {        // four slots' accumulators asked for at a time
                float4 G[4];
                float* rows[4];
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    rows[i] = A.store + __shfl_sync(full, erow, (v0 + i) & 31) * L + 4 * lane;
                    if (kSorted && act && ((in_place >> (v0 + i)) & 1u)) G[i] = *reinterpret_cast<const float4*>(rows[i] + d);
                }
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const int v = v0 + i;
                    if (v >= (int)n_ent || !((reps >> v) & 1u)) continue;
                    const double f3 = __shfl_sync(full, c3, v), f4 = __shfl_sync(full, c4, v);
                    double x[4] = {0.0, 0.0, 0.0, 0.0};
                    auto add = [&](unsigned has, double f, const double (&y)[4]) {
                        if (!((has >> v) & 1u)) return;
#pragma unroll
                        for (int k = 0; k < 4; ++k) x[k] += f * y[k];
                    };
                    add(as_s, 1.0, gs);
                    add(as_o, 1.0, go);
                    add(as_3, f3, u);
                    add(as_4, f4, wv);
                    const float4 g = make_float4((float)x[0], (float)x[1], (float)x[2], (float)x[3]);
                    if (!act) continue;
                    if (kSorted && ((in_place >> v) & 1u)) {
                        const float4 s2 = make_float4(g.x * g.x, g.y * g.y, g.z * g.z, g.w * g.w);
                        float4 th = e4[v * d4 + lane], c = G[i];
                        c.x += s2.x; c.y += s2.y; c.z += s2.z; c.w += s2.w;
                        float4 step;
                        adagrad_steps4(g, c, A.lr, A.eps, step);
                        th.x += step.x; th.y += step.y; th.z += step.z; th.w += step.w;
                        *reinterpret_cast<float4*>(rows[i]) = th;
                        *reinterpret_cast<float4*>(rows[i] + d) = c;
                    } else {
                        *reinterpret_cast<float4*>(out + (size_t)v * d + 4 * lane) = g;
                    }
                }
            }
        }
        if (!kSorted) {                         // matrix rows: a[alpha] x_o + x_s[alpha] b'
            const double *a = U + ld, *b = a + ld, *xo = b + ld, *xs = xo + ld;
            float* out = A.grad + ((uint64_t)item * n_slots + n_ent) * d;
            for (uint32_t x = tid; x < d * d4; x += kPointThreads) {
                const uint32_t al = x / d4, e = 4 * (x - al * d4);
                const double aa = a[al], sa = xs[al];
                float4 g;
                g.x = (float)(aa * xo[e] + sa * b[e]);
                g.y = (float)(aa * xo[e + 1] + sa * b[e + 1]);
                g.z = (float)(aa * xo[e + 2] + sa * b[e + 2]);
                g.w = (float)(aa * xo[e + 3] + sa * b[e + 3]);
                *reinterpret_cast<float4*>(out + (size_t)al * d + e) = g;
            }
        }
        if (kAhead) {
            fence_async_smem();                 // (the rows have been read; the next ones come through the async proxy)
            if (tid == 0 && next.len) mbar_expect_tx(&bar, next.len * n_ent * row_bytes);
        }
        __syncthreads();
    }
}

// The matrices' update.  blockIdx.y: which 2,048 (kMatThreads x 8) of a matrix's d * d elements; blocks of one y loop over
// the chunks of at most kRelChunk data points that segment_kernel listed.  Per element and data point: two fp64
// multiply-adds, a rounding to fp32, a reciprocal square root, two fp64 sums.  Bound by the unit that does roundings,
// widenings and roots (16 lanes per clock and SM: each such operation per element is 18 us of a step of 8,192 data points
// of dimension 100), so the vectors are staged in fp64 (widened once per data point, not once per element), the squares
// are summed as fp64 products and the steps widened by integer operations.  A relation of several chunks
// leaves fp64 partial sums of each; the last chunk of a group of kRelGroup to finish (a ticket) adds the group's in chunk order, the
// last group the groups'.
__global__ void __launch_bounds__(kMatThreads, 3) rescal_matrix_kernel(const RescalArgs A, double* __restrict__ parked) {
    extern __shared__ __align__(128) unsigned char dyn[];
    __shared__ __align__(8) uint64_t bars[2];
    __shared__ uint32_t s_t[kRelChunk];
    __shared__ uint32_t s_ticket;
    pdl_trigger();                              // (for the entities' reduction: run_rescal_sorted)
    if (call_failed(A.st, A.epoch)) return;
    const int tid = threadIdx.x;
    if (tid < 2) mbar_init(&bars[tid], 1);
    mbar_init_fence();
    unsigned uses = 0;                          // parity of each stage's barrier
    const uint32_t d = A.d, d4 = d / 4, quads = d * d4, n_slots = 3 + A.n_neg;
    const uint64_t L = 2 * (uint64_t)d;
    const uint32_t n_items = A.L.counts[3];
    for (uint32_t item = blockIdx.x; item < n_items; item += gridDim.x) {
        const uint4 it = A.L.chunks[item];
        const uint32_t pos = it.x, len = it.y, nc = it.w >> 16, chunk = it.w & 0xffffu;
        const uint32_t rk = A.sk[pos];
        if (tid < (int)len) s_t[tid] = A.sv[pos + tid] / n_slots;
        __syncthreads();
        // the vectors of the data points p0 .. p0 + kMatStage: one bulk copy per data point
        auto issue = [&](uint32_t p0) {
            if (p0 >= len) return;
            const uint32_t cnt = tmin<uint32_t>(kMatStage, len - p0), stage = p0 / kMatStage & 1;
            if (tid == 0) {
                mbar_expect_tx(&bars[stage], cnt * 32 * d);
                for (uint32_t p = 0; p < cnt; ++p)
                    bulk_g2s(dyn + (size_t)(stage * kMatStage + p) * 32 * d, A.vec + (uint64_t)s_t[p0 + p] * 4 * d, 32 * d, &bars[stage]);
            }
        };
        issue(0);
        bool dead = false;                      // a copy that does not arrive
        // a thread's two quads are the same four columns of two neighbouring rows
        const uint32_t x = blockIdx.y * kMatThreads + tid;
        const bool act = x < quads / 2;
        const uint32_t al = act ? 2 * (x / d4) : 0u, e = act ? 4 * (x % d4) : 0u;
        float* row[2];
        float4 G[2];
        double at[2][4], ag[2][4];
#pragma unroll
        for (int i = 0; i < 2; ++i) {
            row[i] = A.store + phys_row(A.table[rk + al + i], A.S) * L + e;
            G[i] = *reinterpret_cast<const float4*>(row[i] + d);
            asm volatile("prefetch.global.L2 [%0];" ::"l"(row[i]));     // (the parameters: read at the end)
#pragma unroll
            for (int k = 0; k < 4; ++k) at[i][k] = ag[i][k] = 0.0;
        }
        for (uint32_t p0 = 0; p0 < len; p0 += kMatStage) {
            const uint32_t cnt = tmin<uint32_t>(kMatStage, len - p0), stage = p0 / kMatStage & 1;
            issue(p0 + kMatStage);              // (the stage's readers have met at the end of the round before)
            const bool ok = mbar_wait(&bars[stage], (uses >> stage) & 1u) || mbar_wait(&bars[stage], (uses >> stage) & 1u);
            uses ^= 1u << stage;
            if (!ok) dead = true;
#pragma unroll 1
            for (uint32_t p = 0; p < cnt; ++p) {
                const double* a = reinterpret_cast<const double*>(dyn) + (stage * kMatStage + p) * 4 * d;
                const double2 aa = *reinterpret_cast<const double2*>(a + al), sa = *reinterpret_cast<const double2*>(a + 3 * d + al);
                const double2 b0 = *reinterpret_cast<const double2*>(a + d + e), b1 = *reinterpret_cast<const double2*>(a + d + e + 2);
                const double2 o0 = *reinterpret_cast<const double2*>(a + 2 * d + e), o1 = *reinterpret_cast<const double2*>(a + 2 * d + e + 2);
                const double ov[4] = {o0.x, o0.y, o1.x, o1.y}, bv[4] = {b0.x, b0.y, b1.x, b1.y};
                float gf[8], xf[8];
#pragma unroll
                for (int i = 0; i < 2; ++i) {
                    const double ai = i ? aa.y : aa.x, si = i ? sa.y : sa.x;
                    const float gv[4] = {G[i].x, G[i].y, G[i].z, G[i].w};
#pragma unroll
                    for (int k = 0; k < 4; ++k) {
                        const double g = ai * ov[k] + si * bv[k];
                        gf[4 * i + k] = (float)g;
                        xf[4 * i + k] = fmaf(gf[4 * i + k], gf[4 * i + k], gv[k]);
                        ag[i][k] += g * g;
                    }
                }
                float step[8];
                const bool fine = adagrad_steps<8>(gf, xf, A.lr, A.eps, step);
                if (fine) {
#pragma unroll
                    for (int k = 0; k < 8; ++k) at[k / 4][k % 4] += widen_scaled(step[k]);
                } else {
#pragma unroll
                    for (int k = 0; k < 8; ++k) at[k / 4][k % 4] += kScale * (double)step[k];
                }
            }
            __syncthreads();
        }
        if (__syncthreads_or(dead)) {
            if (tid == 0) latch_error(A.st, A.epoch, PS_ERR_CUDA);
            return;
        }
#pragma unroll
        for (int i = 0; i < 2; ++i)
#pragma unroll
            for (int k = 0; k < 4; ++k) at[i][k] *= kUnscale;
        bool finish = true;
        if (nc > 1) {
            // laid out [chunk][value of the thread's eight][thread]: coalesced either way
            auto park = [&](uint32_t slot) {
                double2* mine = reinterpret_cast<double2*>(parked) + (uint64_t)(it.z + slot) * quads * 4;
                if (act)
#pragma unroll
                    for (int i = 0; i < 2; ++i)
#pragma unroll
                        for (int k = 0; k < 4; ++k) mine[(uint64_t)(4 * i + k) * (quads / 2) + x] = make_double2(at[i][k], ag[i][k]);
            };
            // the last chunk of a group to finish adds the group's sums, the last group the groups' (one after the other, 47 chunks
            // of one relation took 33 us; each is a round trip to memory)
            auto drawn_last = [&](uint32_t word, uint32_t of) {
                __threadfence();
                __syncthreads();
                if (tid == 0) s_ticket = atomicAdd(&A.L.tickets[(uint64_t)(it.z + word) * kRelTickets + blockIdx.y], 1u);
                __syncthreads();
                const bool last = s_ticket == of - 1;
                if (last) __threadfence();
                return last;
            };
            auto add_up = [&](uint32_t first, uint32_t step, uint32_t count) {
#pragma unroll
                for (int i = 0; i < 2; ++i)
#pragma unroll
                    for (int k = 0; k < 4; ++k) at[i][k] = ag[i][k] = 0.0;
                for (uint32_t c = 0; c < count && act; ++c) {
                    const double2* from = reinterpret_cast<const double2*>(parked) + (uint64_t)(it.z + first + c * step) * quads * 4;
#pragma unroll
                    for (int i = 0; i < 2; ++i)
#pragma unroll
                        for (int k = 0; k < 4; ++k) {
                            const double2 v = __ldcg(from + (uint64_t)(4 * i + k) * (quads / 2) + x);
                            at[i][k] += v.x;
                            ag[i][k] += v.y;
                        }
                }
            };
            const uint32_t g0 = chunk / kRelGroup * kRelGroup, groups = (nc + kRelGroup - 1) / kRelGroup;
            const uint32_t in_group = tmin(kRelGroup, nc - g0);
            park(chunk);
            finish = in_group == 1 || drawn_last(g0, in_group);
            if (finish) {
                if (in_group > 1) add_up(g0, 1, in_group);
                if (groups > 1) {
                    if (in_group > 1) park(g0);
                    finish = drawn_last(1, groups);             // (no group begins with chunk 1)
                    if (finish) add_up(0, kRelGroup, groups);
                }
            }
        }
        if (finish && act) {
#pragma unroll
            for (int i = 0; i < 2; ++i) {
                float4 t = *reinterpret_cast<const float4*>(row[i]), g = G[i];
                t.x = (float)((double)t.x + at[i][0]); t.y = (float)((double)t.y + at[i][1]);
                t.z = (float)((double)t.z + at[i][2]); t.w = (float)((double)t.w + at[i][3]);
                g.x = (float)((double)g.x + ag[i][0]); g.y = (float)((double)g.y + ag[i][1]);
                g.z = (float)((double)g.z + ag[i][2]); g.w = (float)((double)g.w + ag[i][3]);
                *reinterpret_cast<float4*>(row[i]) = t;
                *reinterpret_cast<float4*>(row[i] + d) = g;
            }
        }
    }
}

// Keys of the occurrence slots of each data point: 2 + n_neg entity slots (a slot that repeats an earlier slot's key gets the
// "no key" mark K), then one slot for the relation (the key of its matrix's row 0); every slot of a data point with an
// index out of range gets K.
__global__ void __launch_bounds__(256)
rescal_keys_kernel(const uint32_t* __restrict__ ts, const uint32_t* __restrict__ tr, const uint32_t* __restrict__ to,
                   const uint32_t* __restrict__ neg_ent, uint64_t n, uint32_t n_neg, uint64_t rel_base, uint32_t d,
                   uint64_t K, uint32_t* __restrict__ keys_out, DevStatus* st, unsigned int epoch) {
    const uint64_t idx = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const uint32_t n_ent = 2 + n_neg, n_slots = n_ent + 1;
    if (idx >= n * n_slots) return;
    const uint64_t t = idx / n_slots;
    const uint32_t u = (uint32_t)(idx - t * n_slots);
    const uint64_t rk = rel_base + (uint64_t)tr[t] * d;
    bool bad = ts[t] >= rel_base || to[t] >= rel_base || rk + d > K;
    for (uint32_t q = 0; q < n_neg; ++q) bad |= neg_ent[t * n_neg + q] >= rel_base;
    if (bad) {
        if (u == 0) latch_error(st, epoch, PS_ERR_KEY_RANGE);
        keys_out[idx] = (uint32_t)K;
        return;
    }
    if (u == n_ent) {
        keys_out[idx] = (uint32_t)rk;
        return;
    }
    auto key_of = [&](uint32_t z) { return z == 0 ? ts[t] : (z == 1 ? to[t] : neg_ent[t * n_neg + (z - 2)]); };
    const uint32_t mine = key_of(u);
    bool first = true;
    for (uint32_t z = 0; z < u; ++z) first &= key_of(z) != mine;
    keys_out[idx] = first ? mine : (uint32_t)K;
}

RescalArgs rescal_args(ps_store* ps, const RescalBatch& B, uint32_t rows_per_point) {
    RescalArgs A;
    memset(&A, 0, sizeof A);
    A.ts = B.s; A.tr = B.r; A.to = B.o; A.neg_ent = B.neg_ent; A.neg_side = B.neg_side;
    A.n = (uint32_t)B.n; A.n_neg = B.n_neg; A.d = B.dim; A.K = (uint32_t)ps->cfg.num_keys;
    A.rel_base = B.rel_key_base;
    A.lr = B.lr; A.eps = B.eps;
    A.store = ps->store;
    A.table = ps->table;
    A.S = ps->cfg.slots_per_part;
    // the update rows' region (2 dim values for every one of the call's (2 + n_neg + dim) n key occurrences): gradient
    // rows, then the data points' vectors, then their loss terms
    A.grad = ps->upd;
    A.vec = (double*)(ps->upd + B.n * rows_per_point * B.dim);
    A.loss_of = A.vec + B.n * B.dim * 4;
    A.st = ps->status;
    A.epoch = ps->epoch;
    return A;
}

constexpr size_t points_smem(uint32_t d, uint32_t n_neg, int points) {
    return (size_t)4 * kPoints * pad_ld(d) * 8 + (size_t)d * pad_ld(d) * 4 + (size_t)points * (2 + n_neg) * d * 4;
}
constexpr size_t kMaxSmem = points_smem(128, 29, kPoints);
static_assert(kMaxSmem + 1024 <= 227 * 1024, "a block's shared memory");

}  // namespace

void launch_keys_rescal(ps_store* ps, const RescalBatch& B, cudaStream_t s) {
    PS_LAUNCH(ps, rescal_keys_kernel, div_up_u32(B.n * (3 + (uint64_t)B.n_neg), 256), 256, s, B.s, B.r, B.o, B.neg_ent, B.n, B.n_neg,
              B.rel_key_base, B.dim, ps->cfg.num_keys, ps->keysA, ps->status, ps->epoch);
}

const double* run_rescal_small(ps_store* ps, const RescalBatch& B, uint32_t* keys_out, cudaStream_t s) {
    RescalArgs A = rescal_args(ps, B, 2 + B.n_neg + B.dim);
    A.keys_out = keys_out;
    A.loss_of = ps->loss_partial;               // (kSmallOcc key occurrences are fewer data points than it has room for)
    static std::atomic<unsigned long long> smem_set{0};
    opt_in_smem((const void*)rescal_points_kernel<false, 8>, kMaxSmem, &smem_set);
    PS_LAUNCH_PDL(ps, "rescal_points_kernel<false>", (rescal_points_kernel<false, 8>),
                  dim3((uint32_t)tmin<uint64_t>(B.n, (uint64_t)ps->sm_count * 2)), dim3(256),
                  points_smem(B.dim, B.n_neg, 1), s, A);
    return A.loss_of;
}

void run_rescal_sorted(ps_store* ps, const RescalBatch& B, int which, uint32_t n_loss, double* d_loss_accum, cudaStream_t s) {
    RescalArgs A = rescal_args(ps, B, 3 + B.n_neg);
    A.sk = which ? ps->keysB : ps->keysA;
    A.sv = which ? ps->valsB : ps->valsA;
    A.L = seg_lists(ps);
    static std::atomic<unsigned long long> smem_set{0}, smem_set2{0}, smem_set4{0};
    const int points = (int)rel_piece_len(B.dim);
    const size_t p_smem = points_smem(B.dim, B.n_neg, points);
    const uint32_t p_grid = (uint32_t)tmin<uint64_t>(B.n, (uint64_t)ps->sm_count * 2 * (kPoints / points));
    if (ps->prof) prof_before(ps, "rescal_points_kernel<true>", s);
    if (points == kPoints) {
        opt_in_smem((const void*)rescal_points_kernel<true, 8>, kMaxSmem, &smem_set);
        rescal_points_kernel<true, 8><<<p_grid, 256, p_smem, s>>>(A);
    } else {
        opt_in_smem((const void*)rescal_points_kernel<true, 4>, points_smem(64, 29, 4), &smem_set4);
        rescal_points_kernel<true, 4><<<p_grid, 128, p_smem, s>>>(A);
    }
    if (ps->prof) prof_after(ps, s);
    ps->launches++;
    const uint32_t strips = div_up_u32((uint64_t)B.dim * B.dim / 8, kMatThreads);
    static_assert(128 * 128 / 8 / kMatThreads <= (int)kRelTickets, "a ticket per strip of a matrix");
    const size_t smem = (size_t)2 * kMatStage * B.dim * 32;
    opt_in_smem((const void*)rescal_matrix_kernel, (size_t)2 * kMatStage * 128 * 32, &smem_set2);
    PS_LAUNCH_SMEM(ps, rescal_matrix_kernel, dim3((uint32_t)tmin<uint64_t>(B.n, tmax(1, ps->sm_count * 3 / (int)strips)), strips),
                   kMatThreads, smem, s, A, ps->carry);
    // The entities' reduction fills the places that the matrix kernel's blocks leave one after the other: it needs the points
    // kernel, which was complete before the matrix kernel began, and works on other rows (8,192 data points of dimension 100:
    // 262 -> 243 us per step; the entities first, with the matrix kernel beginning beside their longest segments: 265, the
    // data points' vectors have left L2 by then).  Its partial sums lie behind the loss terms: two rows of 2 dim doubles per
    // 96 entity occurrences at most, where the region has 2 dim floats for each occurrence, matrix rows included.
    double* const parked = A.loss_of + ((B.n + 1) & ~1ull);
    run_segment_adagrad(ps, (uint32_t)((3 + (uint64_t)B.n_neg) * B.n), which, B.dim, false, B.lr, B.eps, parked, A.loss_of, n_loss,
                        d_loss_accum, s, true);
}

}  // namespace psb
