// ComplEx with AdaGrad and negative sampling (Section 4.1 / Appendix A of the paper): the gradient kernel of a minibatch.
//
// Slots of a data point: 0 = subject, 1 = relation, 2 = object, 3 + q = the q-th negative entity.  Lane u holds slot
// u's key and row.  Slots that repeat an earlier slot's key emit no update (key mark K): their gradient is folded into
// the first slot with that key, so that AdaGrad sees the gradient of the data point's loss with respect to each DISTINCT
// key.  A row is [Re | Im | G_Re | G_Im].
//
// Scores and gradient sums are formed in fp64 from the fp32 rows.  With a zero accumulator AdaGrad's step is
// -lr * g / (|g| + eps), which near g = 0 turns rounding noise of g into a visible change of the parameter; fp64 sums
// keep that noise far below the fp32 resolution of the result.  The final AdaGrad expression is evaluated in fp32 on
// the rounded gradient.
//
// What becomes of a slot's gradient (2 d values, Re then Im):
//   key occurs once in the batch   the row is updated in place: this data point is the only one that reads it, and it
//                                  has row and gradient in registers.  That is most keys (negatives are drawn uniformly).
//   other keys                     the gradient is written out for the segmented reduction (segments.cu)
//   calls without a sort           every gradient is written out, with the slot's key
// Before, every gradient went through memory (and for rows of more than 512 values the finished (step, square) pair, twice
// that): 6.8 GB of traffic per step of 2,048 data points of 4,000 dimensions whose rows are 2.9 GB.
#include "ps_internal.cuh"

namespace psb {

namespace {

struct KgeArgs {
    const uint32_t *ts, *tr, *to, *neg_ent;
    const uint8_t* neg_side;
    uint64_t n, rel_base, K;
    uint32_t n_neg, d;
    float lr, eps;
    float* store;
    const uint2* table;
    uint64_t S;
    float* upd;                     // a row of 2 d values per slot (finished: 4 d)
    const uint8_t* single;          // per slot: the key occurs once in the batch (null: calls without a sort)
    uint32_t* keys_out;             // calls without a sort: the slots' keys
    bool finished;                  // write (step, squared gradient) rows instead of gradients
    double* loss_partial;
    DevStatus* st;
    unsigned int epoch;
};

// A bulk copy that does not arrive: the call is given up.  What follows it on the stream sees that by the call's number or, in calls
// without a sort, by a key out of range among the slots' keys (lane 0 wrote slot 0's).
__device__ __forceinline__ void give_up(const KgeArgs& A, uint64_t t, int lane) {
    if (lane != 0) return;
    latch_error(A.st, A.keys_out ? 0u : A.epoch, PS_ERR_CUDA);
    if (A.keys_out) A.keys_out[t * (3 + A.n_neg)] = kSentinelPad;
}

// Sums over the 32 lanes of NP values each, NP a power of two: halves are exchanged, so that each step leaves half as many
// values per lane to add (NP + 5 - log2 NP exchanges in place of 5 NP).  Lane l is left with value l / (32 / NP).
template <int NP>
__device__ __forceinline__ double lane_sums(double (&v)[NP], int lane) {
    int o = 16;
#pragma unroll
    for (int w = NP / 2; w >= 1; w >>= 1) {
        const bool up = lane & o;
#pragma unroll
        for (int i = 0; i < w; ++i) {
            const double send = up ? v[i] : v[i + w], keep = up ? v[i + w] : v[i];
            v[i] = keep + __shfl_xor_sync(0xffffffffu, send, o);
        }
        o >>= 1;
    }
    for (; o; o >>= 1) v[0] += __shfl_xor_sync(0xffffffffu, v[0], o);
    return v[0];
}

// Rows of at most 128 complex dimensions: a warp per data point.  The embeddings of its rows arrive in the warp's shared
// memory as bulk copies asked for all at once, the next data point's keys and table entries are looked up meanwhile, and
// both passes over the dimensions read from there: no load inside a pass.  (With loads into registers before each block of
// dimensions the passes were chains of memory latencies at 16 warps per SM: 66 us for 8,192 data points of dimension 100,
// 113 us where it also updated the rows whose key occurs once, with 84 and 45 us for the reduction; this one takes 89 with
// those updates, 43 instead of 78 at 3,000 data points of dimension 60 with 20 negatives.  Four dimensions per lane at a time
// spill: 100 us.)
// A lane has two dimensions at a time.  kV2: consecutive ones, as pairs (d even); otherwise 32 apart.
constexpr int kShortWarps = 4;

template <bool kV2> struct Dims {                               // dimensions at and at + kStep
    static constexpr uint32_t kStep = kV2 ? 1 : 32;
    __device__ static __forceinline__ void load(const float* row, uint32_t at, uint32_t d, float (&v)[2]) {
        if constexpr (kV2) {
            const float2 x = *reinterpret_cast<const float2*>(row + at);
            v[0] = x.x; v[1] = x.y;
        } else {
            v[0] = row[at];
            v[1] = at + kStep < d ? row[at + kStep] : 0.f;
        }
    }
    __device__ static __forceinline__ void store(float* row, uint32_t at, uint32_t d, const float (&v)[2]) {
        if constexpr (kV2) {
            *reinterpret_cast<float2*>(row + at) = make_float2(v[0], v[1]);
        } else {
            row[at] = v[0];
            if (at + kStep < d) row[at + kStep] = v[1];
        }
    }
};

// kAcc: some slots need their accumulators here (rows updated in place, finished rows); otherwise gradients are all it writes.
template <int kMaxNeg, bool kV2, bool kAcc>
__global__ void __launch_bounds__(32 * kShortWarps, kMaxNeg <= 10 ? 4 : 2) kge_short_kernel(const KgeArgs A) {
    constexpr int NP = kMaxNeg < 8 ? 8 : kMaxNeg < 16 ? 16 : 32;
    using D = Dims<kV2>;
    extern __shared__ __align__(128) float row_mem[];           // [warp][slot][row_len]
    __shared__ __align__(8) uint64_t bars[kShortWarps];
    __shared__ double s_w[kShortWarps][3][32];                  // coefficient of negative q; weights of a slot's two directions
    __shared__ uint64_t s_off[kShortWarps][32];
    __shared__ double s_loss[kShortWarps];
    const unsigned full = 0xffffffffu;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const uint32_t d = A.d, n_neg = A.n_neg;
    const int n_slots = 3 + (int)n_neg;
    const bool slot = lane < n_slots;
    const uint64_t L = 4 * (uint64_t)d, K = A.K;
    const uint32_t rl = (2 * d + 3) & ~3u;                      // floats copied per row: the embedding, to a multiple of 16 bytes
    float* const rows = row_mem + (size_t)w * n_slots * rl;
    if (lane == 0) mbar_init(&bars[w], 1);
    mbar_init_fence();
    pdl_trigger();
    pdl_wait();
    if (A.single && call_failed(A.st, A.epoch)) return;
    const uint64_t n_warps = (uint64_t)gridDim.x * kShortWarps;
    uint64_t t = (uint64_t)blockIdx.x * kShortWarps + w;
    // a data point's slots, lane u slot u: key (K: no slot; all ones: out of range) and side
    auto key_of = [&](uint64_t t2, int& side) -> uint64_t {
        side = 0;
        if (!slot || t2 >= A.n) return K;
        if (lane == 1) {
            const uint64_t k = A.rel_base + A.tr[t2];
            return k < K ? k : ~0ull;
        }
        const uint32_t e = lane == 0 ? A.ts[t2] : (lane == 2 ? A.to[t2] : A.neg_ent[t2 * n_neg + (lane - 3)]);
        if (lane >= 3) side = A.neg_side[t2 * n_neg + (lane - 3)] != 0;
        return e < A.rel_base ? e : ~0ull;
    };
    auto entry_of = [&](uint64_t k) { return k < K ? A.table[k] : make_uint2(0u, 0u); };
    auto once_of = [&](uint64_t t2) { return slot && A.single && t2 < A.n && A.single[t2 * n_slots + lane]; };
    int side, next_side = 0;
    uint64_t key = key_of(t, side);
    uint2 entry = entry_of(key);
    bool alone = once_of(t);
    unsigned parity = 0;
    double loss = 0;
    for (; t < A.n; t += n_warps) {
        const bool bad = __any_sync(full, key == ~0ull);
        const unsigned same = __match_any_sync(full, slot ? (uint32_t)key : kSentinelPad);
        const int rep = slot ? __ffs(same) - 1 : lane;
        const bool once = alone && rep == lane;
        const uint64_t off = phys_row(entry, A.S) * L;
        const int my_side = side;
        if (!bad && lane == 0) mbar_expect_tx(&bars[w], (uint32_t)n_slots * rl * 4);
        __syncwarp();
        if (!bad && slot) {
            bulk_g2s(rows + lane * rl, A.store + off, rl * 4, &bars[w]);
            if (once)                                           // its accumulators are wanted at the end
                for (uint32_t o = 0; o < 2 * d; o += 32) asm volatile("prefetch.global.L2 [%0];" ::"l"(A.store + off + 2 * d + o));
        }
        s_off[w][lane] = off;
        if (A.keys_out && slot) A.keys_out[t * n_slots + lane] = bad ? kSentinelPad : rep == lane ? (uint32_t)key : (uint32_t)K;
        // the next data point's look-ups travel beside this one's rows
        const uint64_t next_key = key_of(t + n_warps, next_side);
        const bool next_alone = once_of(t + n_warps);
        const unsigned subj_mask = __ballot_sync(full, lane >= 3 && slot && my_side == 0) >> 3;
        const unsigned rep_mask = __ballot_sync(full, slot && rep == lane), once_mask = __ballot_sync(full, once);
        const unsigned acc_mask = !kAcc ? 0u : A.finished ? rep_mask : once_mask;   // slots whose accumulators are needed here
        const int rep_o = __shfl_sync(full, rep, 2);            // 0 if object == subject
        const uint2 next_entry = entry_of(next_key);
        if (bad) {                                              // (the same decision in every lane)
            if (lane == 0) latch_error(A.st, A.keys_out ? 0u : A.epoch, PS_ERR_KEY_RANGE);
            key = next_key; entry = next_entry; alone = next_alone; side = next_side;
            continue;
        }
        if (!mbar_wait(&bars[w], parity) && !mbar_wait(&bars[w], parity)) {
            give_up(A, t, lane);
            break;                                              // a copy that does not arrive: give the call up
        }
        parity ^= 1;
        auto emb = [&](int u, int part, uint32_t at, float (&v)[2]) { D::load(rows + u * rl + part * d, at, d, v); };
        // ---- pass A: partial scores of the 1 + n_neg triples over this lane's dimensions ----
        double part[NP];
#pragma unroll
        for (int q = 0; q < NP; ++q) part[q] = 0.0;
        for (uint32_t c0 = 0; c0 < d; c0 += 64) {
            const uint32_t at = c0 + (kV2 ? 2 * lane : lane);
            if (at >= d) continue;
            float av[2], bv[2], crv[2], civ[2], ev[2], fv[2];
            emb(0, 0, at, av); emb(0, 1, at, bv); emb(1, 0, at, crv); emb(1, 1, at, civ); emb(2, 0, at, ev); emb(2, 1, at, fv);
            double re_o[2], im_o[2], re_s[2], im_s[2];
#pragma unroll
            for (int i = 0; i < 2; ++i) {
                const double a = av[i], b = bv[i], cr = crv[i], ci = civ[i], e = ev[i], f = fv[i];
                part[0] += cr * (a * e + b * f) + ci * (a * f - b * e);
                // (n, r, o): cr (na e + nb f) + ci (na f - nb e);   (s, r, n): cr (a na + b nb) + ci (a nb - b na)
                re_o[i] = cr * e + ci * f; im_o[i] = cr * f - ci * e;       // multiplies (na, nb) in the subject's place
                re_s[i] = cr * a - ci * b; im_s[i] = cr * b + ci * a;       // ... in the object's place
            }
#pragma unroll
            for (int q = 0; q < kMaxNeg; ++q) {
                if (q >= (int)n_neg) break;
                float na[2], nb[2];
                emb(3 + q, 0, at, na); emb(3 + q, 1, at, nb);
                if ((subj_mask >> q) & 1u)
                    part[q + 1] += ((double)na[0] * re_o[0] + (double)nb[0] * im_o[0]) + ((double)na[1] * re_o[1] + (double)nb[1] * im_o[1]);
                else
                    part[q + 1] += ((double)na[0] * re_s[0] + (double)nb[0] * im_s[0]) + ((double)na[1] * re_s[1] + (double)nb[1] * im_s[1]);
            }
        }
        const double sum = lane_sums<NP>(part, lane);
        const double phi_mine = __shfl_sync(full, sum, (lane * (32 / NP)) & 31);
        // lane q: loss term and d loss / d phi of triple q (label +1 for the positive, -1 for negatives)
        double coef = 0, loss_q = 0;
        if (lane <= (int)n_neg) {
            const double y = lane == 0 ? 1.0 : -1.0, z = -y * phi_mine, ez = exp(-fabs(z));
            loss_q = fmax(z, 0.0) + log1p(ez);
            coef = -y * ((z >= 0.0 ? 1.0 : ez) / (1.0 + ez));
        }
        loss += loss_q;                                         // (lane q's share)
        // ---- weights with which each entity slot receives the two "negative role" directions ----
        // A negative with side 0 stands in the subject's place: its gradient is coef * dphi/dS(r, o).  With side 1 it stands in
        // the object's place: coef * dphi/dO(s, r).  Summed over the negatives whose key's first slot is this lane.
        if (lane >= 1 && lane <= (int)n_neg) s_w[w][0][lane - 1] = coef;
        __syncwarp();
        double wS = 0, wO = 0;
        if (slot && rep == lane) {
            for (unsigned m = (same >> 3) & ((1u << n_neg) - 1u); m; m &= m - 1) {
                const int q = __ffs(m) - 1;
                if ((subj_mask >> q) & 1u) wS += s_w[w][0][q]; else wO += s_w[w][0][q];
            }
        }
        s_w[w][1][lane] = wS;
        s_w[w][2][lane] = wO;
        const double cf0 = __shfl_sync(full, coef, 0);
        __syncwarp();
        const double *cf = s_w[w][0], *ws = s_w[w][1], *wo = s_w[w][2];
        // ---- pass B: gradients ----
        const uint32_t LU = kAcc && A.finished ? 4 * d : 2 * d; // values per update row
        float* const U = A.upd + t * n_slots * (uint64_t)LU;
        for (uint32_t c0 = 0; c0 < d; c0 += 64) {
            const uint32_t at = c0 + (kV2 ? 2 * lane : lane);
            if (at >= d) continue;
            // the accumulators of slot u, where they are needed
            auto ask = [&](int u, float (&re)[2], float (&im)[2]) {
                re[0] = re[1] = im[0] = im[1] = 0.f;
                if (kAcc && ((acc_mask >> u) & 1u)) {
                    D::load(A.store + s_off[w][u] + 2 * d, at, d, re);
                    D::load(A.store + s_off[w][u] + 3 * d, at, d, im);
                }
            };
            auto out = [&](int u, const double (&re)[2], const double (&im)[2], const float (&G_re)[2], const float (&G_im)[2]) {
                const float g[4] = {(float)re[0], (float)re[1], (float)im[0], (float)im[1]};
                float* o = U + (uint64_t)u * LU;
                auto put = [&](int part, float x0, float x1) {
                    const float v[2] = {x0, x1};
                    D::store(o + part * d, at, d, v);
                };
                if (!kAcc || !((acc_mask >> u) & 1u)) {
                    put(0, g[0], g[1]);
                    put(1, g[2], g[3]);
                    return;
                }
                float g2[4], x[4], step[4];
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    g2[i] = __fmul_rn(g[i], g[i]);
                    x[i] = __fadd_rn(i < 2 ? G_re[i] : G_im[i - 2], g2[i]);
                }
                adagrad_steps<4>(g, x, A.lr, A.eps, step);
                if ((once_mask >> u) & 1u) {
                    o = A.store + s_off[w][u];
                    float r[2], m[2];
                    emb(u, 0, at, r);
                    emb(u, 1, at, m);
                    put(0, __fadd_rn(r[0], step[0]), __fadd_rn(r[1], step[1]));
                    put(1, __fadd_rn(m[0], step[2]), __fadd_rn(m[1], step[3]));
                    put(2, x[0], x[1]);
                    put(3, x[2], x[3]);
                } else {
                    put(0, step[0], step[1]);
                    put(1, step[2], step[3]);
                    put(2, g2[0], g2[1]);
                    put(3, g2[2], g2[3]);
                }
            };
            float G_re[3][2], G_im[3][2];
#pragma unroll
            for (int u = 0; u < 3; ++u) ask(u, G_re[u], G_im[u]);
            // The negatives enter the gradients of subject, relation and object only through their weighted sums:
            // (A0, B0) over those in the subject's place (triples (n, r, o)), (A1, B1) over those in the object's
            // place (triples (s, r, n)).
            double A0[2] = {0.0, 0.0}, B0[2] = {0.0, 0.0}, A1[2] = {0.0, 0.0}, B1[2] = {0.0, 0.0};
#pragma unroll
            for (int q = 0; q < kMaxNeg; ++q) {
                if (q >= (int)n_neg) break;
                float na[2], nb[2];
                emb(3 + q, 0, at, na); emb(3 + q, 1, at, nb);
                const double wq = cf[q];
                if ((subj_mask >> q) & 1u) {
                    A0[0] += wq * (double)na[0]; A0[1] += wq * (double)na[1];
                    B0[0] += wq * (double)nb[0]; B0[1] += wq * (double)nb[1];
                } else {
                    A1[0] += wq * (double)na[0]; A1[1] += wq * (double)na[1];
                    B1[0] += wq * (double)nb[0]; B1[1] += wq * (double)nb[1];
                }
            }
            float av[2], bv[2], crv[2], civ[2], ev[2], fv[2];
            emb(0, 0, at, av); emb(0, 1, at, bv); emb(1, 0, at, crv); emb(1, 1, at, civ); emb(2, 0, at, ev); emb(2, 1, at, fv);
            // directions that do not depend on the negative: d phi / d subject (object = o), d phi / d object (subject = s)
            double dS_re[2], dS_im[2], dO_re[2], dO_im[2], gs_re[2], gs_im[2], gr_re[2], gr_im[2], go_re[2], go_im[2];
#pragma unroll
            for (int i = 0; i < 2; ++i) {
                const double a = av[i], b = bv[i], cr = crv[i], ci = civ[i], e = ev[i], f = fv[i];
                dS_re[i] = cr * e + ci * f; dS_im[i] = cr * f - ci * e;
                dO_re[i] = cr * a - ci * b; dO_im[i] = cr * b + ci * a;
                gr_re[i] = cf0 * (a * e + b * f) + (A0[i] * e + B0[i] * f) + (a * A1[i] + b * B1[i]);
                gr_im[i] = cf0 * (a * f - b * e) + (A0[i] * f - B0[i] * e) + (a * B1[i] - b * A1[i]);
                // (negatives that coincide with the subject or the object: the slots' weights)
                go_re[i] = cf0 * dO_re[i] + (cr * A0[i] - ci * B0[i]) + ws[2] * dS_re[i] + wo[2] * dO_re[i];
                go_im[i] = cf0 * dO_im[i] + (cr * B0[i] + ci * A0[i]) + ws[2] * dS_im[i] + wo[2] * dO_im[i];
                gs_re[i] = cf0 * dS_re[i] + (cr * A1[i] + ci * B1[i]) + ws[0] * dS_re[i] + wo[0] * dO_re[i];
                gs_im[i] = cf0 * dS_im[i] + (cr * B1[i] - ci * A1[i]) + ws[0] * dS_im[i] + wo[0] * dO_im[i];
                if (rep_o == 0) { gs_re[i] += go_re[i]; gs_im[i] += go_im[i]; }
            }
            out(0, gs_re, gs_im, G_re[0], G_im[0]);
            out(1, gr_re, gr_im, G_re[1], G_im[1]);
            if (rep_o == 2) out(2, go_re, go_im, G_re[2], G_im[2]);
            auto negative = [&](int u, const float (&G_re2)[2], const float (&G_im2)[2]) {
                const double wSq = ws[u], wOq = wo[u];
                const double x[2] = {wSq * dS_re[0] + wOq * dO_re[0], wSq * dS_re[1] + wOq * dO_re[1]};
                const double y[2] = {wSq * dS_im[0] + wOq * dO_im[0], wSq * dS_im[1] + wOq * dO_im[1]};
                out(u, x, y, G_re2, G_im2);
            };
            if (!kAcc) {
                const float none[2] = {0.f, 0.f};
#pragma unroll
                for (int q = 0; q < kMaxNeg; ++q)
                    if ((rep_mask >> (3 + q)) & 1u) negative(3 + q, none, none);
                continue;
            }
            // one negative after the other (the code of one, not of ten: the instruction cache; 103 -> 89 us), the accumulators
            // of the next two on their way
            float Gq[3][2][2];
            ask(tmin(3, n_slots - 1), Gq[0][0], Gq[0][1]);
            ask(tmin(4, n_slots - 1), Gq[1][0], Gq[1][1]);
#pragma unroll 1
            for (int u = 3; u < n_slots; ++u) {
                ask(tmin(u + 2, n_slots - 1), Gq[2][0], Gq[2][1]);
                if ((rep_mask >> u) & 1u) negative(u, Gq[0][0], Gq[0][1]);
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    Gq[0][i / 2][i % 2] = Gq[1][i / 2][i % 2];
                    Gq[1][i / 2][i % 2] = Gq[2][i / 2][i % 2];
                }
            }
        }
        fence_async_smem();                                     // (the rows have been read; the next ones come through the async proxy)
        __syncwarp();
        key = next_key; entry = next_entry; alone = next_alone; side = next_side;
    }
    // per-block loss partial, fixed order
    loss = warp_sum_d(loss);
    if (lane == 0) s_loss[w] = loss;
    __syncthreads();
    if (threadIdx.x == 0) {
        double tot = 0;
        for (int i = 0; i < kShortWarps; ++i) tot += s_loss[i];
        A.loss_partial[blockIdx.x] = tot;
    }
}

// Rows of more than 128 complex dimensions that kge_resident_kernel does not take (launch_resident; odd dimensions in calls without a
// sort): a block per data point (batches of few data points: a
// cluster of up to four, which meets to add up the scores), the rows streamed through shared memory in stretches of 256
// dimensions as bulk copies, what the next job needs on its way while one is worked on, across the two passes and across
// data points.  (Measured on 2,048 data points of 4,000 dimensions with 10 negatives, whose rows take 440 us; they go to
// kge_resident_kernel now, 743.  With loads into registers, one stretch after the other, the memory system was idle three quarters
// of the time: 1,199 us; streamed 808 us; with two stretches per job
// in the first pass, which has little to do on them and waits for their arrival, and the two kinds of update row compiled
// apart, 747.)  It is bound by the second pass's instructions (1,300 per warp and stretch, half of them AdaGrad's, issued at
// 16 warps per SM in chains) and by those arrivals.  Filling a stage when its last reader leaves, without a barrier per
// job, gained nothing; asking L2 for the rows two jobs earlier cost 200 us.  A stretch of a part (Re, Im, G_Re or G_Im) of a
// row starts at a multiple of 16 bytes only if d is a multiple of four: the copy starts at the boundary before it, and
// `shift` floats are skipped.
//
// kGroups = 2 (more than ten negatives): a stretch is 128 dimensions, and the block's halves share the negatives, so that a
// thread's score sums stay in registers and two blocks' stages fit an SM (up to 20 negatives).  The first half, which also
// has the subject, the relation and the object, gets fewer of them; the second hands it its weighted sums.  1,000 data points
// of 400 dimensions with 20 negatives, which this kernel had then: 287 us with a block per data point and loads into registers at 8
// warps per SM, so 146.
template <int kMaxNeg>
struct Wide {
    static constexpr int kGroups = kMaxNeg > 10 ? 2 : 1, kSlots = 3 + kMaxNeg;
    static constexpr uint32_t kStretch = 256 / kGroups, kPad = kStretch + 4;
    static constexpr int kFirst = kGroups == 1 ? kMaxNeg : (kMaxNeg - 2) / 2;          // negatives of the first half
    static constexpr int kMine = kGroups == 1 ? kMaxNeg : kMaxNeg - kFirst;            // of either, at most
    static constexpr size_t kSmem = (size_t)2 * kSlots * 4 * kPad * sizeof(float);     // [2 stages][slot][part][kPad]
    static constexpr int kPerSm = kMaxNeg > 20 ? 1 : 2;
};

template <int kMaxNeg, bool kFinished>
__global__ void __launch_bounds__(256, Wide<kMaxNeg>::kPerSm) kge_wide_kernel(const KgeArgs A) {
    constexpr int kGroups = Wide<kMaxNeg>::kGroups, kSlots = Wide<kMaxNeg>::kSlots, kMine = Wide<kMaxNeg>::kMine;
    constexpr uint32_t kStretch = Wide<kMaxNeg>::kStretch, kStretchPad = Wide<kMaxNeg>::kPad;
    constexpr int kWarps = 8, kGroupWarps = kWarps / kGroups;
    extern __shared__ __align__(128) float stage_mem[];
    __shared__ __align__(8) uint64_t bars[2];
    __shared__ double s_part[kWarps][kMine + 1];
    __shared__ double s_sum[4][kGroups == 1 ? 1 : kStretch];        // the second half's weighted sums
    __shared__ double s_tot[2][kMaxNeg + 1];                    // the block's share of the scores, by the data point's parity
    __shared__ int s_failed;
    __shared__ double s_w[3][32];
    __shared__ uint64_t s_off[32];
    const unsigned full = 0xffffffffu;
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    const uint32_t d = A.d, n_neg = A.n_neg;
    const int group = kGroups == 1 ? 0 : w / kGroupWarps, q0 = group ? Wide<kMaxNeg>::kFirst : 0;
    const int n_mine = group ? tmax(0, (int)n_neg - q0) : tmin((int)n_neg, Wide<kMaxNeg>::kFirst);
    const uint32_t gtid = tid % kStretch;                       // the thread's dimension in a stretch
    const int n_slots = 3 + (int)n_neg;
    const bool slot = lane < n_slots;
    const uint64_t L = 4 * (uint64_t)d, K = A.K;
    if (tid < 2) mbar_init(&bars[tid], 1);
    mbar_init_fence();
    pdl_trigger();
    pdl_wait();
    uint32_t rank, C;
    asm("mov.u32 %0, %%cluster_ctarank;" : "=r"(rank));
    asm("mov.u32 %0, %%cluster_nctaid.x;" : "=r"(C));
    if (A.single) {
        bool failed = call_failed(A.st, A.epoch);
        if (C > 1) {                                            // a block that started later may see more: one decision
            if (tid == 0) s_failed = failed;
            cluster_arrive();
            cluster_wait();
            for (uint32_t r = 0; r < C; ++r) failed |= peer_i32(&s_failed, r) != 0;
            cluster_arrive();
            cluster_wait();
        }
        if (failed) return;
    }
    __syncthreads();
    const uint32_t n_str = ((d + kStretch - 1) / kStretch - rank + C - 1) / C;         // stretches rank, rank + C, ... are the block's
    const uint64_t stride = gridDim.x / C;
    double loss = 0;
    // what a warp knows of a data point: lane u its slot u
    struct Point {
        uint64_t off;
        uint32_t key;
        int rep;
        unsigned subj, reps, once;
        bool bad;
    };
    auto look_up = [&](uint64_t t) {
        Point P;
        uint64_t key = K;
        int side = 0;
        bool bad = false;
        if (slot) {
            if (lane == 1) {
                key = A.rel_base + A.tr[t];
                bad = key >= K;
            } else {
                const uint32_t e = lane == 0 ? A.ts[t] : (lane == 2 ? A.to[t] : A.neg_ent[t * n_neg + (lane - 3)]);
                key = e;
                bad = e >= A.rel_base;
                if (lane >= 3) side = A.neg_side[t * n_neg + (lane - 3)] != 0;
            }
        }
        P.bad = __any_sync(full, bad);
        P.key = (uint32_t)key;
        const unsigned same = __match_any_sync(full, slot ? P.key : kSentinelPad);
        P.rep = slot ? __ffs(same) - 1 : lane;
        const bool once = slot && !P.bad && A.single && P.rep == lane && A.single[t * n_slots + lane];
        P.off = (slot && !P.bad) ? phys_row(A.table[key], A.S) * L : 0;
        P.subj = __ballot_sync(full, lane >= 3 && slot && side == 0) >> 3;
        P.reps = __ballot_sync(full, slot && P.rep == lane);
        P.once = __ballot_sync(full, once);
        return P;
    };
    // Warp 0 asks for what a job of a data point reads.  First pass: the next two stretches of its rows' Re and Im (as many
    // bytes as a job of the second pass: there is little to do on them, so it is their arrival that counts).  Second pass: one
    // stretch, and of the accumulators too where they are needed.
    const uint32_t n_first = (n_str + 1) / 2, n_jobs = n_first + n_str;
    auto issue = [&](const Point& P, uint32_t job, int stage) {
        const bool second = job >= n_first;
        const uint32_t str = second ? job - n_first : 2 * job;
        const uint32_t c0 = (str * C + rank) * kStretch, c1 = c0 + C * kStretch;        // c1: the stretch after it
        const uint32_t len0 = tmin(d - c0, kStretch), len1 = second || str + 1 == n_str ? 0u : tmin(d - c1, kStretch);
        const unsigned acc = !second ? 0u : kFinished ? P.reps : P.once;
        uint32_t bytes[4], total = 0;
#pragma unroll
        for (int p = 0; p < 4; ++p) {
            const uint32_t q = second ? p : p & 1, len = second || p < 2 ? len0 : len1;
            bytes[p] = len ? ((len + ((q * d) & 3) + 3) & ~3u) * 4 : 0u;
            total += bytes[p] * (second && p >= 2 ? (uint32_t)__popc(acc) : (uint32_t)n_slots);
        }
        if (lane == 0) mbar_expect_tx(&bars[stage], total);
        __syncwarp();
        if (!slot) return;
        const int parts = (second ? (acc >> lane) & 1u : len1 != 0) ? 4 : 2;
        for (int p = 0; p < parts; ++p)
            bulk_g2s(stage_mem + (((size_t)stage * kSlots + lane) * 4 + p) * kStretchPad,
                     A.store + P.off + (second ? (p * d + c0) & ~3u : ((p & 1) * d + (p < 2 ? c0 : c1)) & ~3u), bytes[p], &bars[stage]);
    };
    uint64_t t = blockIdx.x / C;
    Point P = {}, N = {};
    // the first data point (from `from` on) whose indexes are all valid; marks the others (the same in every warp)
    auto next_valid = [&](uint64_t from, Point& Q) {
        for (; from < A.n; from += stride) {
            Q = look_up(from);
            if (A.keys_out && slot && w == 0 && rank == 0)
                A.keys_out[from * n_slots + lane] = Q.bad ? kSentinelPad : Q.rep == lane ? Q.key : (uint32_t)K;
            if (!Q.bad) break;
            if (tid == 0) latch_error(A.st, A.keys_out ? 0u : A.epoch, PS_ERR_KEY_RANGE);
        }
        return from;
    };
    t = next_valid(t, P);
    unsigned uses = 0;
    int stage = 0;
    bool dead = false;
    int parity = 0;
    if (t < A.n && w == 0) issue(P, 0, 0);
    while (t < A.n) {
        const uint64_t tn = next_valid(t + stride, N);
        const unsigned subj_mask = P.subj, rep_mask = P.reps, acc_mask = kFinished ? P.reps : P.once;
        double part[kMine + 1];                                 // scores of the triple (first half) and of the thread's negatives
#pragma unroll
        for (int q = 0; q <= kMine; ++q) part[q] = 0.0;
        double cf0 = 0;
        int rep_o = 2;
        const uint32_t LU = kFinished ? 4 * d : 2 * d;         // values per update row
        float* const U = A.upd + t * n_slots * (uint64_t)LU;
        for (uint32_t job = 0; job < n_jobs; ++job) {
            const bool pass_b = job >= n_first;
            const uint32_t str = pass_b ? job - n_first : 2 * job;
            // the job after this one; its stage was read two jobs ago (and the warps have met since)
            if (w == 0) {
                if (job + 1 < n_jobs) issue(P, job + 1, stage ^ 1);
                else if (tn < A.n) issue(N, 0, stage ^ 1);
            }
            if (!mbar_wait(&bars[stage], (uses >> stage) & 1u) && !mbar_wait(&bars[stage], (uses >> stage) & 1u)) dead = true;
            uses ^= 1u << stage;
            const float* base = stage_mem + (size_t)stage * kSlots * 4 * kStretchPad + gtid;
            const uint32_t sh1 = d & 3, sh2 = (2 * d) & 3, sh3 = (3 * d) & 3;
            auto re = [&](int u) { return base[u * 4 * kStretchPad]; };
            auto im = [&](int u) { return base[(u * 4 + 1) * kStretchPad + sh1]; };
            auto gre = [&](int u) { return base[(u * 4 + 2) * kStretchPad + sh2]; };
            auto gim = [&](int u) { return base[(u * 4 + 3) * kStretchPad + sh3]; };
            uint32_t c = (str * C + rank) * kStretch + gtid;
            // the values of the triple's rows in dimension c, and the directions that do not depend on the negative:
            // d phi / d subject (object = o), d phi / d object (subject = s)
            struct Triple {
                double a, b, cr, ci, e, f, dS_re, dS_im, dO_re, dO_im;
            };
            auto triple = [&]() {
                Triple T;
                const float a_f = re(0), b_f = im(0), cr_f = re(1), ci_f = im(1), e_f = re(2), f_f = im(2);
                T.a = a_f; T.b = b_f; T.cr = cr_f; T.ci = ci_f; T.e = e_f; T.f = f_f;
                T.dS_re = T.cr * T.e + T.ci * T.f; T.dS_im = T.cr * T.f - T.ci * T.e;
                T.dO_re = T.cr * T.a - T.ci * T.b; T.dO_im = T.cr * T.b + T.ci * T.a;
                return T;
            };
            if (!pass_b) {
                for (int half = 0; half < 2 && c < d; ++half, c += C * kStretch, base += 2 * kStretchPad) {
                    const Triple T = triple();
                    if (group == 0) part[0] += T.cr * (T.a * T.e + T.b * T.f) + T.ci * (T.a * T.f - T.b * T.e);
#pragma unroll
                    for (int i = 0; i < kMine; ++i) {
                        if (i >= n_mine) break;
                        const int q = q0 + i;
                        const double na = re(3 + q), nb = im(3 + q);
                        part[i + 1] += ((subj_mask >> q) & 1u) ? (na * T.dS_re + nb * T.dS_im) : (na * T.dO_re + nb * T.dO_im);
                    }
                }
            } else {
                const double *cf = s_w[0], *ws = s_w[1], *wo = s_w[2];
                auto out = [&](int u, double gd_re, double gd_im) {
                    const float g[2] = {(float)gd_re, (float)gd_im};
                    float* o = U + (uint64_t)u * LU + c;
                    if (!((acc_mask >> u) & 1u)) {
                        o[0] = g[0];
                        o[d] = g[1];
                        return;
                    }
                    const float g2[2] = {g[0] * g[0], g[1] * g[1]}, x[2] = {gre(u) + g2[0], gim(u) + g2[1]};
                    float step[2];
                    adagrad_steps<2>(g, x, A.lr, A.eps, step);
                    if (!kFinished) o = A.store + s_off[u] + c;     // in place
                    o[0] = kFinished ? step[0] : re(u) + step[0];
                    o[d] = kFinished ? step[1] : im(u) + step[1];
                    o[2 * d] = kFinished ? g2[0] : x[0];
                    o[3 * d] = kFinished ? g2[1] : x[1];
                };
                double A0 = 0.0, B0 = 0.0, A1 = 0.0, B1 = 0.0;      // weighted sums of the negatives in either place
                // subject, relation and object
                auto triple_out = [&](const Triple& T) {
                    double gs_re = cf0 * T.dS_re, gs_im = cf0 * T.dS_im;
                    double go_re = cf0 * T.dO_re, go_im = cf0 * T.dO_im;
                    double gr_re = cf0 * (T.a * T.e + T.b * T.f), gr_im = cf0 * (T.a * T.f - T.b * T.e);
                    gr_re += (A0 * T.e + B0 * T.f) + (T.a * A1 + T.b * B1); gr_im += (A0 * T.f - B0 * T.e) + (T.a * B1 - T.b * A1);
                    go_re += T.cr * A0 - T.ci * B0; go_im += T.cr * B0 + T.ci * A0;
                    gs_re += T.cr * A1 + T.ci * B1; gs_im += T.cr * B1 - T.ci * A1;
                    // negatives that coincide with the subject or the object
                    gs_re += ws[0] * T.dS_re + wo[0] * T.dO_re; gs_im += ws[0] * T.dS_im + wo[0] * T.dO_im;
                    go_re += ws[2] * T.dS_re + wo[2] * T.dO_re; go_im += ws[2] * T.dS_im + wo[2] * T.dO_im;
                    if (rep_o == 0) { gs_re += go_re; gs_im += go_im; }
                    out(0, gs_re, gs_im);
                    out(1, gr_re, gr_im);
                    if (rep_o == 2) out(2, go_re, go_im);
                };
                if (c < d) {
                    const Triple T = triple();
#pragma unroll
                    for (int i = 0; i < kMine; ++i) {
                        if (i >= n_mine) break;
                        const int q = q0 + i;
                        const double na = re(3 + q), nb = im(3 + q), wq = cf[q];
                        if ((subj_mask >> q) & 1u) { A0 += wq * na; B0 += wq * nb; }
                        else { A1 += wq * na; B1 += wq * nb; }
                    }
                    if (kGroups == 1) {
                        triple_out(T);
                    } else if (group == 1) {
                        s_sum[0][gtid] = A0; s_sum[1][gtid] = B0; s_sum[2][gtid] = A1; s_sum[3][gtid] = B1;
                    }
#pragma unroll
                    for (int i = 0; i < kMine; ++i) {
                        if (i >= n_mine) break;
                        const int q = q0 + i;
                        if (!((rep_mask >> (3 + q)) & 1u)) continue;
                        const double wSq = ws[3 + q], wOq = wo[3 + q];
                        out(3 + q, wSq * T.dS_re + wOq * T.dO_re, wSq * T.dS_im + wOq * T.dO_im);
                    }
                }
                if (kGroups > 1) {
                    __syncthreads();
                    if (group == 0 && c < d) {
                        A0 += s_sum[0][gtid]; B0 += s_sum[1][gtid]; A1 += s_sum[2][gtid]; B1 += s_sum[3][gtid];
                        triple_out(triple());
                    }
                }
            }
            stage ^= 1;
            if (job + 1 == n_first) {           // the scores are complete: coefficients and weights
#pragma unroll
                for (int o = 16; o > 0; o >>= 1)
#pragma unroll
                    for (int q = 0; q <= kMine; ++q) part[q] += __shfl_xor_sync(full, part[q], o);
                if (lane == 0)
#pragma unroll
                    for (int q = 0; q <= kMine; ++q) s_part[w][q] = part[q];
                __syncthreads();
                double phi = 0, coef = 0, loss_q = 0;           // lane q + 1: negative q; lane 0: the triple
                if (lane <= kMaxNeg) {
                    const bool later = lane > Wide<kMaxNeg>::kFirst;
                    const int from = later ? kWarps - kGroupWarps : 0, at = later ? lane - Wide<kMaxNeg>::kFirst : lane;
                    for (int i = 0; i < kGroupWarps; ++i) phi += s_part[from + i][at];
                }
                if (C > 1) {                    // the blocks' shares, in rank order
                    if (w == 0 && lane <= kMaxNeg) s_tot[parity][lane] = phi;
                    cluster_arrive();
                    cluster_wait();
                    phi = 0;
                    if (lane <= kMaxNeg)
                        for (uint32_t r = 0; r < C; ++r) phi += peer_f64(&s_tot[parity][lane], r);
                    parity ^= 1;                // (two data points on, all have met again: the reads above are done)
                }
                if (lane <= (int)n_neg) {
                    const double y = lane == 0 ? 1.0 : -1.0, z = -y * phi, ez = exp(-fabs(z));
                    loss_q = fmax(z, 0.0) + log1p(ez);
                    coef = -y * ((z >= 0.0 ? 1.0 : ez) / (1.0 + ez));
                }
                loss_q = warp_sum_d(loss_q);
                if (w == 0) loss += loss_q;
                double wS = 0, wO = 0;
                for (int q = 0; q < (int)n_neg; ++q) {
                    const int rq = __shfl_sync(full, P.rep, 3 + q);
                    const double cfq = __shfl_sync(full, coef, q + 1);
                    if (rq == lane) {
                        if ((subj_mask >> q) & 1u) wS += cfq; else wO += cfq;
                    }
                }
                cf0 = __shfl_sync(full, coef, 0);
                rep_o = __shfl_sync(full, P.rep, 2);            // 0 if object == subject
                if (w == 0) {
                    if (lane >= 1 && lane <= (int)n_neg) s_w[0][lane - 1] = coef;
                    s_w[1][lane] = wS;
                    s_w[2][lane] = wO;
                    s_off[lane] = P.off;
                }
            }
            if (__syncthreads_or(dead)) {
                if (C == 1) {
                    give_up(A, t, tid);
                    return;
                }
                if (tid == 0) latch_error(A.st, A.keys_out ? 0u : A.epoch, PS_ERR_CUDA);
                // the cluster's other blocks go on: meet them as often as they will, with nothing done in between
                if (job + 1 < n_first) {
                    cluster_arrive();
                    cluster_wait();
                }
                for (uint64_t r = tn; r < A.n; r = next_valid(r + stride, N)) {
                    cluster_arrive();
                    cluster_wait();
                }
                cluster_arrive();
                cluster_wait();
                give_up(A, t, tid);                             // (after the block that writes the keys has written them all)
                return;
            }
        }
        P = N;
        t = tn;
    }
    if (tid == 0) A.loss_partial[blockIdx.x] = rank == 0 ? loss : 0.0;
    if (C > 1) {                                // (nobody reads a block's shared memory after it has left)
        cluster_arrive();
        cluster_wait();
    }
}

// Rows of more than 128 dimensions, and some of 65 to 128 (launch_points_kge), whose data point fits the shared memory of a block or of a
// cluster of two or four (13 rows: 2,112, 4,224 and 8,448 dimensions, 2,047, 3,839 and 7,679 where they are no multiple of four;
// launch_resident): the embeddings stay there from the first pass to the second.  A
// warp has chunks of 64 dimensions to itself (chunk (s C + rank) warps + w of the row is the s-th of warp w), with their own
// places in shared memory and their own barrier words: it asks for its part of the next data point's rows when it is done
// with this one's, and meets the others once per data point, to add up the scores.  In kge_wide_kernel, which streams stretches
// of 256 dimensions through a block, the warps meet after every stretch (a third of their stalls), a last stretch idles some
// of them, and the rows are read twice.  us per launch, streamed and now: 4,000 data points of 200 dimensions with 10 negatives
// 148 and 86, 1,600 of 500 105 and 86, 800 of 1,000 98 and 86, 1,500 of 300 with 20 negatives 171 and 92, 600 of 600 with 29 248 and
// 121, 8,000 of 141 with one 140 and 76; clusters of two, 2,048 of 4,000 753 and 743.  On shorter rows the warp per data point of
// kge_short_kernel is better in large calls, 89 and 115 us for 8,192 data points of 100 dimensions, but for its form for more than ten
// negatives that updates rows in place (8 warps per SM; 6,000 of 70 with 20 negatives 123 and 102).  Bound by the latency of its
// instructions at 16 warps per SM, which 128 registers fix (96 registers and 20 warps spill: 87 and 101 us at 500 dimensions).
template <int kMaxNeg> struct Resident {
    static constexpr uint32_t kNumbers = 3 + kMaxNeg <= 16 ? 16 : 32;                   // places per table of slots
    __host__ __device__ static constexpr uint32_t pad(int kVec) { return kVec == 4 ? 64 : 68; }             // floats of a chunk of a row's Re or Im
    static constexpr size_t smem(int kVec, uint32_t slots, uint32_t warps, uint32_t bufs, uint32_t C) {
        return (size_t)warps * bufs * (slots * 2 * pad(kVec) * sizeof(float) + 8) + (size_t)2 * C * warps * (kMaxNeg + 1) * 8 +
               (size_t)warps * 3 * kNumbers * 8 + 2 * 32 * 8 + 16;
    }
};

template <int kMaxNeg, int kVec>
__global__ void __launch_bounds__(512, 1) kge_resident_kernel(const KgeArgs A, const uint32_t n_str, const bool twice) {
    constexpr int NP = kMaxNeg < 8 ? 8 : kMaxNeg < 16 ? 16 : 32;
    constexpr uint32_t kPad = Resident<kMaxNeg>::pad(kVec), kNumbers = Resident<kMaxNeg>::kNumbers;
    constexpr uint32_t kStep = kVec > 1 ? 1 : 32;               // a lane's two dimensions: neighbours, or 32 apart (odd d)
    extern __shared__ __align__(128) float chunk_mem[];
    const unsigned full = 0xffffffffu;
    const uint32_t tid = threadIdx.x, lane = tid & 31, w = tid >> 5, n_warps = blockDim.x >> 5;
    const uint32_t d = A.d, shift = kVec == 4 ? 0 : d & 3, n_neg = A.n_neg, n_slots = 3 + n_neg, n_bufs = twice ? 2 * n_str : n_str;
    const bool slot = lane < n_slots;
    const uint64_t L = 4 * (uint64_t)d, K = A.K;
    uint32_t rank, C;
    asm("mov.u32 %0, %%cluster_ctarank;" : "=r"(rank));
    asm("mov.u32 %0, %%cluster_nctaid.x;" : "=r"(C));
    float* const mine = chunk_mem + (size_t)w * n_bufs * n_slots * 2 * kPad;            // [buffer][slot][Re, Im][kPad]
    double* const s_part = reinterpret_cast<double*>(chunk_mem + (size_t)n_warps * n_bufs * n_slots * 2 * kPad);  // [parity][rank][warp][1 + kMaxNeg]
    double* const s_w = s_part + 2 * C * n_warps * (kMaxNeg + 1) + w * 3 * kNumbers;    // the warp's: coefficients, weights of a slot's directions
    uint64_t* const s_off = reinterpret_cast<uint64_t*>(s_part + 2 * C * n_warps * (kMaxNeg + 1) + n_warps * 3 * kNumbers);   // [parity][slot]
    uint64_t* const bars = s_off + 64 + w * n_bufs;
    int* const s_dead = reinterpret_cast<int*>(s_off + 64 + n_warps * n_bufs);          // [parity]; then s_failed
    if (lane < n_bufs) mbar_init(&bars[lane], 1);
    if (tid < 3) s_dead[tid] = 0;
    mbar_init_fence();
    pdl_trigger();
    pdl_wait();
    __syncthreads();
    if (C > 1) {                                                // (all blocks have started, their words are zero)
        cluster_arrive();
        cluster_wait();
    }
    if (A.single) {
        bool failed = call_failed(A.st, A.epoch);
        if (C > 1) {                                            // a block that started later may see more: one decision
            if (tid == 0) s_dead[2] = failed;
            cluster_arrive();
            cluster_wait();
            for (uint32_t r = 0; r < C; ++r) failed |= peer_i32(&s_dead[2], r) != 0;
            cluster_arrive();
            cluster_wait();
        }
        if (failed) return;
    }
    const uint64_t stride = gridDim.x / C;
    // what a warp knows of a data point: lane u its slot u
    struct Point {
        uint64_t off;
        uint32_t key;
        int rep;
        unsigned same, subj, reps, once;
        bool bad;
    };
    auto look_up = [&](uint64_t t) {
        Point P;
        uint64_t key = K;
        int side = 0;
        bool bad = false;
        if (slot) {
            if (lane == 1) {
                key = A.rel_base + A.tr[t];
                bad = key >= K;
            } else {
                key = lane == 0 ? A.ts[t] : (lane == 2 ? A.to[t] : A.neg_ent[t * n_neg + (lane - 3)]);
                bad = key >= A.rel_base;
                if (lane >= 3) side = A.neg_side[t * n_neg + (lane - 3)] != 0;
            }
        }
        P.bad = __any_sync(full, bad);
        P.key = (uint32_t)key;
        P.same = __match_any_sync(full, slot ? P.key : kSentinelPad);
        P.rep = slot ? __ffs(P.same) - 1 : (int)lane;
        const bool once = slot && !P.bad && A.single && P.rep == (int)lane && A.single[t * n_slots + lane];
        P.off = (slot && !P.bad) ? phys_row(A.table[key], A.S) * L : 0;
        P.subj = __ballot_sync(full, lane >= 3 && slot && side == 0) >> 3;
        P.reps = __ballot_sync(full, slot && P.rep == (int)lane);
        P.once = __ballot_sync(full, once);
        return P;
    };
    // the first data point (from `from` on) whose indexes are all valid; marks the others (the same in every warp)
    auto next_valid = [&](uint64_t from, Point& Q) {
        for (; from < A.n; from += stride) {
            Q = look_up(from);
            if (A.keys_out && slot && w == 0 && rank == 0)
                A.keys_out[from * n_slots + lane] = Q.bad ? kSentinelPad : Q.rep == (int)lane ? Q.key : (uint32_t)K;
            if (!Q.bad) break;
            if (tid == 0) latch_error(A.st, A.keys_out ? 0u : A.epoch, PS_ERR_KEY_RANGE);
        }
        return from;
    };
    // the lane's two dimensions at row + its first (the second may lie past the row: zero)
    auto get = [&](const float* row, bool both) {
        if constexpr (kVec > 1) return *reinterpret_cast<const float2*>(row);
        else return make_float2(row[0], both ? row[32] : 0.f);
    };
    auto put = [&](float* row, bool both, float x, float y) {
        if constexpr (kVec > 1) {
            *reinterpret_cast<float2*>(row) = make_float2(x, y);
        } else {
            row[0] = x;
            if (both) row[32] = y;
        }
    };
    const uint32_t first = kVec > 1 ? 2 * lane : lane;
    auto chunk_at = [&](uint32_t s) { return ((s * C + rank) * n_warps + w) * 64; };
    auto buffer_of = [&](uint32_t j, uint32_t s) { return twice ? (j & 1) * n_str + s : s; };      // j: the block's j-th data point
    auto parity_of = [&](uint32_t j) { return (twice ? j >> 1 : j) & 1; };
    // lane u asks for the chunk of slot u's row (and has its accumulators brought to L2, where they are wanted)
    auto ask = [&](const Point& Q, uint32_t j, uint32_t s) {
        const uint32_t c0 = chunk_at(s);
        if (c0 >= d) return;
        const uint32_t len = tmin(64u, d - c0), buf = buffer_of(j, s);
        const uint32_t re_bytes = ((len + 3) & ~3u) * 4, im_bytes = ((len + shift + 3) & ~3u) * 4;   // (Im may start between two 16-byte boundaries)
        if (lane == 0) mbar_expect_tx(&bars[buf], n_slots * (re_bytes + im_bytes));
        __syncwarp();
        if (!slot) return;
        float* to = mine + (size_t)(buf * n_slots + lane) * 2 * kPad;
        const float* row = A.store + Q.off + c0;
        bulk_g2s(to, row, re_bytes, &bars[buf]);
        bulk_g2s(to + kPad, row + d - shift, im_bytes, &bars[buf]);
        if ((Q.once >> lane) & 1u) {
            // (as prefetches of lines: as bulk prefetches, each as dear as a copy, 3 % slower)
            const float *g0 = row + 2 * d, *g1 = row + 3 * d;
#pragma unroll
            for (uint32_t o = 0; o < 64; o += 32)
                if (o < len) {
                    asm volatile("prefetch.global.L2 [%0];" ::"l"(g0 + o));
                    asm volatile("prefetch.global.L2 [%0];" ::"l"(g1 + o));
                }
            asm volatile("prefetch.global.L2 [%0];" ::"l"(g0 + len - 1));           // (a part need not start on a line)
            asm volatile("prefetch.global.L2 [%0];" ::"l"(g1 + len - 1));
        }
    };
    Point P = {}, N = {};
    uint64_t t = next_valid(blockIdx.x / C, P);
    double loss = 0;
    if (t < A.n)
        for (uint32_t s = 0; s < n_str; ++s) ask(P, 0, s);
    uint32_t j = 0;
    uint64_t tn = A.n;
    bool dead = false;
    for (; t < A.n; ++j) {
        tn = next_valid(t + stride, N);
        if (twice && tn < A.n) {
            fence_async_smem();                                 // (the data point before this one has been read from there)
            __syncwarp();
            for (uint32_t s = 0; s < n_str; ++s) ask(N, j + 1, s);
        }
        const unsigned subj_mask = P.subj, rep_mask = P.reps, acc_mask = P.once;
        const int rep_o = __shfl_sync(full, P.rep, 2);          // 0 if object == subject
        // ---- pass A: scores of the 1 + n_neg triples over the warp's dimensions, two per lane at a time ----
        double part[NP];
#pragma unroll
        for (int q = 0; q < NP; ++q) part[q] = 0.0;
        for (uint32_t s = 0; s < n_str; ++s) {
            const uint32_t c0 = chunk_at(s), buf = buffer_of(j, s);
            if (c0 >= d) break;
            if (!mbar_wait(&bars[buf], parity_of(j)) && !mbar_wait(&bars[buf], parity_of(j))) dead = true;
            if (c0 + first >= d) continue;
            const bool both = c0 + first + kStep < d;
            const float *at = mine + (size_t)buf * n_slots * 2 * kPad + first, *at_im = at + kPad + shift;
            auto re = [&](int u) { return get(at + u * 2 * kPad, both); };
            auto im = [&](int u) { return get(at_im + u * 2 * kPad, both); };
            const float2 av = re(0), bv = im(0), crv = re(1), civ = im(1), ev = re(2), fv = im(2);
            double re_o[2], im_o[2], re_s[2], im_s[2];
#pragma unroll
            for (int i = 0; i < 2; ++i) {
                const double a = i ? av.y : av.x, b = i ? bv.y : bv.x, cr = i ? crv.y : crv.x, ci = i ? civ.y : civ.x;
                const double e = i ? ev.y : ev.x, f = i ? fv.y : fv.x;
                part[0] += cr * (a * e + b * f) + ci * (a * f - b * e);
                re_o[i] = cr * e + ci * f; im_o[i] = cr * f - ci * e;           // multiplies a negative in the subject's place
                re_s[i] = cr * a - ci * b; im_s[i] = cr * b + ci * a;           // ... in the object's place
            }
#pragma unroll
            for (int q = 0; q < kMaxNeg; ++q) {
                if (q >= (int)n_neg) break;
                const float2 na = re(3 + q), nb = im(3 + q);
                if ((subj_mask >> q) & 1u)
                    part[q + 1] += ((double)na.x * re_o[0] + (double)nb.x * im_o[0]) + ((double)na.y * re_o[1] + (double)nb.y * im_o[1]);
                else
                    part[q + 1] += ((double)na.x * re_s[0] + (double)nb.x * im_s[0]) + ((double)na.y * re_s[1] + (double)nb.y * im_s[1]);
            }
        }
        // ---- the warps' sums meet in every block of the cluster, and are added in the order of the row ----
        const uint32_t parity = j & 1;                          // (two data points on, all have met again: what is read below has been read)
        {
            const double sum = lane_sums<NP>(part, lane);
            const uint32_t q = lane / (32 / NP);
            double* const to = s_part + ((size_t)(parity * C + rank) * n_warps + w) * (kMaxNeg + 1) + q;
            const bool writes = lane % (32 / NP) == 0 && q <= kMaxNeg;
            if (w == 0) s_off[parity * 32 + lane] = P.off;
            if (C == 1) {
                if (writes) *to = sum;
                if (dead) s_dead[parity] = 1;
                __syncthreads();
            } else {
                for (uint32_t r = 0; r < C; ++r) {
                    if (writes) asm volatile("st.shared::cluster.f64 [%0], %1;\n" ::"r"(peer_smem(to, r)), "d"(sum) : "memory");
                    if (dead) asm volatile("st.shared::cluster.u32 [%0], %1;\n" ::"r"(peer_smem(&s_dead[parity], r)), "r"(1) : "memory");
                }
                cluster_arrive();
                cluster_wait();
            }
        }
        dead = *(volatile int*)&s_dead[parity] != 0;            // the same decision in every warp of the cluster
        if (dead) break;
        double coef = 0, loss_q = 0;                            // lane q + 1: negative q; lane 0: the triple
        if (lane <= n_neg) {
            const double* from = s_part + (size_t)parity * C * n_warps * (kMaxNeg + 1) + lane;
            double phi = 0;
            for (uint32_t i = 0; i < C * n_warps; ++i) phi += from[i * (kMaxNeg + 1)];
            const double y = lane == 0 ? 1.0 : -1.0, z = -y * phi, ez = exp(-fabs(z));
            loss_q = fmax(z, 0.0) + log1p(ez);
            coef = -y * ((z >= 0.0 ? 1.0 : ez) / (1.0 + ez));
        }
        loss += loss_q;                                         // (lane q's share)
        // ---- weights with which each entity slot receives the two "negative role" directions (see kge_short_kernel) ----
        double *const cf = s_w, *const ws = s_w + kNumbers, *const wo = s_w + 2 * kNumbers;
        if (lane >= 1 && lane <= n_neg) cf[lane - 1] = coef;
        __syncwarp();
        double wS = 0, wO = 0;
        if (slot && P.rep == (int)lane) {
            for (unsigned m = (P.same >> 3) & ((1u << n_neg) - 1u); m; m &= m - 1) {
                const int q = __ffs(m) - 1;
                if ((subj_mask >> q) & 1u) wS += cf[q]; else wO += cf[q];
            }
        }
        if (lane < kNumbers) {
            ws[lane] = wS;
            wo[lane] = wO;
        }
        const double cf0 = __shfl_sync(full, coef, 0);
        __syncwarp();
        // ---- pass B: gradients ----
        const uint32_t LU = 2 * d;                              // values per update row
        float* const U = A.upd + t * n_slots * (uint64_t)LU;
        const uint64_t* const off = s_off + parity * 32;
        for (uint32_t s = 0; s < n_str; ++s) {
            const uint32_t c0 = chunk_at(s), buf = buffer_of(j, s), at0 = c0 + first;
            if (c0 >= d) break;
            if (at0 < d) {
                const bool both = at0 + kStep < d;
                const float *at = mine + (size_t)buf * n_slots * 2 * kPad + first, *at_im = at + kPad + shift;
                auto re = [&](int u) { return get(at + u * 2 * kPad, both); };
                auto im = [&](int u) { return get(at_im + u * 2 * kPad, both); };
                struct Acc { float2 re, im; };
                // the accumulators of slot u, where they are needed
                auto acc_of = [&](int u) {
                    Acc G = {make_float2(0.f, 0.f), make_float2(0.f, 0.f)};
                    if ((acc_mask >> u) & 1u) {
                        const float* g = A.store + off[u] + 2 * d + at0;
                        G.re = get(g, both);
                        G.im = get(g + d, both);
                    }
                    return G;
                };
                auto out = [&](int u, const double (&gd)[4], const Acc& G) {    // gd: Re, Re, Im, Im
                    const float g[4] = {(float)gd[0], (float)gd[1], (float)gd[2], (float)gd[3]};
                    if (!((acc_mask >> u) & 1u)) {
                        float* o = U + (uint64_t)u * LU + at0;
                        put(o, both, g[0], g[1]);
                        put(o + d, both, g[2], g[3]);
                        return;
                    }
                    const float x[4] = {__fadd_rn(G.re.x, __fmul_rn(g[0], g[0])), __fadd_rn(G.re.y, __fmul_rn(g[1], g[1])),
                                        __fadd_rn(G.im.x, __fmul_rn(g[2], g[2])), __fadd_rn(G.im.y, __fmul_rn(g[3], g[3]))};
                    float step[4];
                    adagrad_steps<4>(g, x, A.lr, A.eps, step);
                    const float2 r = re(u), m = im(u);
                    float* o = A.store + off[u] + at0;          // in place
                    put(o, both, r.x + step[0], r.y + step[1]);
                    put(o + d, both, m.x + step[2], m.y + step[3]);
                    put(o + 2 * d, both, x[0], x[1]);
                    put(o + 3 * d, both, x[2], x[3]);
                };
                const Acc G0 = acc_of(0), G1 = acc_of(1), G2 = acc_of(2);
                Acc Ga = acc_of(tmin(3u, n_slots - 1)), Gb = acc_of(tmin(4u, n_slots - 1));
                // the negatives' weighted sums: in the subject's place, in the object's
                double A0[2] = {0.0, 0.0}, B0[2] = {0.0, 0.0}, A1[2] = {0.0, 0.0}, B1[2] = {0.0, 0.0};
#pragma unroll
                for (int q = 0; q < kMaxNeg; ++q) {
                    if (q >= (int)n_neg) break;
                    const float2 na = re(3 + q), nb = im(3 + q);
                    const double wq = cf[q];
                    if ((subj_mask >> q) & 1u) {
                        A0[0] += wq * (double)na.x; A0[1] += wq * (double)na.y;
                        B0[0] += wq * (double)nb.x; B0[1] += wq * (double)nb.y;
                    } else {
                        A1[0] += wq * (double)na.x; A1[1] += wq * (double)na.y;
                        B1[0] += wq * (double)nb.x; B1[1] += wq * (double)nb.y;
                    }
                }
                double dS[4], dO[4];                            // d phi / d subject (object = o), d phi / d object (subject = s)
                {
                    const float2 av = re(0), bv = im(0), crv = re(1), civ = im(1), ev = re(2), fv = im(2);
                    double gs[4], gr[4], go[4];
#pragma unroll
                    for (int i = 0; i < 2; ++i) {
                        const double a = i ? av.y : av.x, b = i ? bv.y : bv.x, cr = i ? crv.y : crv.x, ci = i ? civ.y : civ.x;
                        const double e = i ? ev.y : ev.x, f = i ? fv.y : fv.x;
                        dS[i] = cr * e + ci * f; dS[2 + i] = cr * f - ci * e;
                        dO[i] = cr * a - ci * b; dO[2 + i] = cr * b + ci * a;
                        gr[i] = cf0 * (a * e + b * f) + (A0[i] * e + B0[i] * f) + (a * A1[i] + b * B1[i]);
                        gr[2 + i] = cf0 * (a * f - b * e) + (A0[i] * f - B0[i] * e) + (a * B1[i] - b * A1[i]);
                        // (negatives that coincide with the subject or the object: the slots' weights)
                        go[i] = cf0 * dO[i] + (cr * A0[i] - ci * B0[i]) + ws[2] * dS[i] + wo[2] * dO[i];
                        go[2 + i] = cf0 * dO[2 + i] + (cr * B0[i] + ci * A0[i]) + ws[2] * dS[2 + i] + wo[2] * dO[2 + i];
                        gs[i] = cf0 * dS[i] + (cr * A1[i] + ci * B1[i]) + ws[0] * dS[i] + wo[0] * dO[i];
                        gs[2 + i] = cf0 * dS[2 + i] + (cr * B1[i] - ci * A1[i]) + ws[0] * dS[2 + i] + wo[0] * dO[2 + i];
                        if (rep_o == 0) { gs[i] += go[i]; gs[2 + i] += go[2 + i]; }
                    }
                    out(0, gs, G0);
                    out(1, gr, G1);
                    if (rep_o == 2) out(2, go, G2);
                }
                // one negative after the other, the accumulators of the next two on their way
#pragma unroll 1
                for (uint32_t u = 3; u < n_slots; ++u) {
                    const Acc Gc = acc_of(tmin(u + 2, n_slots - 1));
                    if ((rep_mask >> u) & 1u) {
                        const double wSq = ws[u], wOq = wo[u];
                        const double g[4] = {wSq * dS[0] + wOq * dO[0], wSq * dS[1] + wOq * dO[1], wSq * dS[2] + wOq * dO[2], wSq * dS[3] + wOq * dO[3]};
                        out(u, g, Ga);
                    }
                    Ga = Gb;
                    Gb = Gc;
                }
            }
            if (!twice && tn < A.n) {
                fence_async_smem();                             // (the rows have been read; the next ones come through the async proxy)
                __syncwarp();
                ask(N, j + 1, s);
            }
        }
        P = N;
        t = tn;
    }
    if (dead) {                                                 // a copy did not arrive: the call is given up
        if (w == 0 && rank == 0) give_up(A, t, lane);
        else if (tid == 0) latch_error(A.st, A.keys_out ? 0u : A.epoch, PS_ERR_CUDA);
        if (twice && tn < A.n)                          // copies still on their way to this block
            for (uint32_t s = 0; s < n_str && chunk_at(s) < d; ++s) mbar_wait(&bars[buffer_of(j + 1, s)], parity_of(j + 1));
    }
    loss = warp_sum_d(loss);
    if (tid == 0) A.loss_partial[blockIdx.x] = rank == 0 ? loss : 0.0;
}

// Keys of the occurrence slots of each data point; a slot that repeats an earlier slot's key, and every
// slot of a data point with an index out of range, gets the "no key" mark K.
__global__ void __launch_bounds__(256)
kge_keys_kernel(const uint32_t* __restrict__ ts, const uint32_t* __restrict__ tr, const uint32_t* __restrict__ to,
                const uint32_t* __restrict__ neg_ent, uint64_t n, uint32_t n_neg, uint64_t rel_base, uint64_t K,
                uint32_t* __restrict__ keys_out, DevStatus* st, unsigned int epoch) {
    // a warp per data point, lane u its slot u
    const int lane = threadIdx.x & 31;
    const uint64_t t = ((uint64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    if (t >= n) return;
    const int n_slots = 3 + (int)n_neg;
    const bool slot = lane < n_slots;
    uint64_t key = K;
    bool bad = false;
    if (slot) {
        key = lane == 0 ? ts[t] : lane == 1 ? rel_base + tr[t] : lane == 2 ? to[t] : neg_ent[t * n_neg + (lane - 3)];
        bad = lane == 1 ? key >= K : key >= rel_base;
    }
    const bool any_bad = __any_sync(0xffffffffu, bad);
    if (any_bad && lane == 0) latch_error(st, epoch, PS_ERR_KEY_RANGE);
    const unsigned same = __match_any_sync(0xffffffffu, slot ? (uint32_t)key : kSentinelPad);
    if (slot) keys_out[t * n_slots + lane] = (!any_bad && __ffs(same) - 1 == lane) ? (uint32_t)key : (uint32_t)K;
}

// A cluster of several blocks per data point where the data points alone would leave blocks' places empty (60 data points of
// 4,000 dimensions: 77 us with one block each, 46 with two, 32 with four, 36 with eight).  Not otherwise, although fewer data
// points in flight would keep more of their rows in L2 between the passes: the meetings cost more than the 0.4 of 1.7 GB
// fewer reads save (2,048 data points: 747 us with one block, 791 with two, 950 with four).
template <int kMaxNeg, bool kFinished>
uint32_t launch_wide(ps_store* ps, const KgeArgs& A, cudaStream_t s) {
    const size_t smem = Wide<kMaxNeg>::kSmem;
    const uint32_t places = (uint32_t)ps->sm_count * Wide<kMaxNeg>::kPerSm;
    static std::atomic<unsigned long long> smem_set{0};
    static std::atomic<int> fit[64][3];                         // clusters resident at once, by device and size (0: not asked yet)
    opt_in_smem((const void*)kge_wide_kernel<kMaxNeg, kFinished>, smem, &smem_set);
    const uint32_t stretches = (A.d + Wide<kMaxNeg>::kStretch - 1) / Wide<kMaxNeg>::kStretch;
    int lg = 0;
    while (lg < 2 && ((uint64_t)A.n << (lg + 1)) <= places && (2u << lg) <= stretches) ++lg;
    cudaLaunchConfig_t cfg = {};
    cfg.blockDim = dim3(256);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = 1u << lg;
    attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    int clusters = ps->cfg.device < 64 ? fit[ps->cfg.device][lg].load(std::memory_order_relaxed) : 0;
    if (clusters == 0) {
        cfg.gridDim = dim3(1u << lg);
        cfg.numAttrs = 1;
        if (cudaOccupancyMaxActiveClusters(&clusters, kge_wide_kernel<kMaxNeg, kFinished>, &cfg) != cudaSuccess || clusters < 1)
            clusters = tmax(1, (int)(places >> lg));
        if (ps->cfg.device < 64) fit[ps->cfg.device][lg].store(clusters, std::memory_order_relaxed);
    }
    const uint32_t grid = (uint32_t)tmin<uint64_t>(A.n, (uint64_t)clusters) << lg;
    cfg.gridDim = dim3(grid);
    cfg.numAttrs = A.keys_out ? 2 : 1;                          // (the pdl form: kernels of small calls)
    if (ps->prof) prof_before(ps, "kge_wide_kernel", s);
    cudaLaunchKernelEx(&cfg, kge_wide_kernel<kMaxNeg, kFinished>, A);
    if (ps->prof) prof_after(ps, s);
    ps->launches++;
    return grid;
}

// 0: not with this kernel (a data point does not fit four blocks, or only in blocks of few warps).  The number of warps per block: as many
// warps per SM as 128 registers a thread allow (16), in blocks whose chunks go evenly, several chunks per warp where that costs none (a
// warp's work per data point is about a quarter of a chunk's); no blocks of one warp, whose waits nothing covers (9,000 data points of 170
// dimensions with 4 negatives: 160 us a step with those, 152).
// Few data points have an SM to themselves: what counts then are the warps of one block, and its rows may take all the shared memory
// (us per step, ordered, in blocks that could share an SM / so / kge_wide_kernel: 12 data points of 3,000 dimensions with one negative
// 20.3, 13.8, 16.3, 12 of 1,000 with 4 15.8, 13.2, 14.0, 30 of 900 with 4 19.4, 15.9, 15.9, 90 of 130 with 20 28.3, 24.3, 25.4).
// Near the most that fits, the only blocks may be a few warps with many chunks each (2,000 dimensions with 11 negatives: two warps of 16),
// and an SM with so few waits most of the time.  A wider cluster, or in the end kge_wide_kernel, is better from `least` warps per SM on:
// us per step with any number of warps, with these limits, with kge_wide_kernel: 300 data points of 2,000 dimensions with 11 negatives 403,
// 122, 225; 148 of 3,902 with 10 170, 113, 94; 300 of 1,102 with 20 259, 130, 176; 111 of 4,102 with 20 338, 183, 183; 60 of 13,900 with
// 5 136, 96, 96.  In clusters of four there is only kge_wide_kernel left to take, which is slow with more than ten negatives: 60 of 15,900
// with 4 (seven warps) 108, 93, 93; 60 of 7,001 with 11 (seven) 108, 108, 125; 60 of 2,902 with 29 (six) 111, 111, 152; 60 of 3,700 with
// 25 (five) 135, 135, 172; 60 of 5,800 with 15 (four) 155, 120, 120; and where every data point has its cluster at once: 30 of 15,900
// with 4 58, 58, 76, 30 of 13,900 with 5 (five) 74, 74, 78, 30 of 5,800 with 15 86, 86, 106.
template <int kMaxNeg, int kVec>
uint32_t launch_resident(ps_store* ps, const KgeArgs& A, cudaStream_t s) {
    using R = Resident<kMaxNeg>;
    const uint32_t chunks = (A.d + 63) / 64, slots = 3 + A.n_neg, sms = (uint32_t)ps->sm_count;
    constexpr uint32_t kMost = 227 * 1024, kPerSm = 228 * 1024;
    uint32_t warps = 0, n_str = 0, resident = 0, C = 1;
    bool twice = false;
    for (;; C *= 2) {
        const uint32_t per = (chunks + C - 1) / C;
        const bool alone = A.n * C * 8 <= (uint64_t)sms * 7;    // (clusters do not come by all SMs)
        uint32_t most = 0;                                      // warps that an SM has room for
        double best = 0;
        for (uint32_t w = tmin(2u, per); w <= tmin(16u, per); ++w) {
            const uint32_t str = (per + w - 1) / w;
            const size_t once = R::smem(kVec, slots, w, str, C), both = R::smem(kVec, slots, w, 2 * str, C);
            if (once > kMost || 2 * str > 32) continue;        // (32 barrier words per warp; so many chunks go with few warps)
            const uint32_t fit = tmin<uint32_t>(16 / w, (uint32_t)(kPerSm / (once + 1024))), blocks = alone ? 1 : fit;
            const double score = (double)blocks * per / str * (4 * str) / (4 * str + 1);
            if (score > best) {
                best = score;
                warps = w;
                n_str = str;
                resident = blocks;
                most = w * fit;
                twice = both <= kMost && blocks * (both + 1024) <= kPerSm;
            }
        }
        const bool at_once = A.n * C <= (uint64_t)sms * (most / tmax(warps, 1u));
        const uint32_t least = C < 4 ? 7 : A.n_neg <= 10 ? (at_once ? 5 : 8) : (at_once ? 4 : 5);
        if (most < least) {
            if (C == 4) return 0;
            warps = 0;
            continue;
        }
        // few data points: a cluster of two or four blocks for each, as long as none has to wait (16 data points of 600 dimensions
        // and their reduction: 24 -> 20 us)
        if (C == 4 || A.n * 2 * C > (uint64_t)sms * resident || chunks < 4 * C) break;
    }
    const void* fn = (const void*)kge_resident_kernel<kMaxNeg, kVec>;
    const size_t smem = R::smem(kVec, slots, warps, twice ? 2 * n_str : n_str, C);
    static std::atomic<unsigned long long> smem_set{0};
    opt_in_smem(fn, kMost, &smem_set);
    cudaLaunchConfig_t cfg = {};
    cfg.blockDim = dim3(32 * warps);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = C;
    attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    uint64_t places = (uint64_t)sms * resident;
    if (C > 1) {                                                // clusters resident at once: asked for when the shape is not the last one (shapes in turn: no slower)
        ClusterFit& f = ps->kge_fit;
        if (f.fn != fn || f.smem != smem || f.threads != 32 * warps || f.blocks != C) {
            int clusters = 0;
            cfg.gridDim = dim3(C);
            cfg.numAttrs = 1;
            if (cudaOccupancyMaxActiveClusters(&clusters, fn, &cfg) != cudaSuccess) cudaGetLastError();
            f.fn = fn; f.smem = smem; f.threads = 32 * warps; f.blocks = C;
            f.clusters = (uint32_t)tmax(clusters, 0);
        }
        places = f.clusters;
        if (places == 0) return 0;
    }
    const uint32_t grid = (uint32_t)tmin<uint64_t>(A.n, places) * C;
    cfg.gridDim = dim3(grid);
    cfg.numAttrs = A.keys_out ? 2 : 1;                          // (the pdl form: kernels of small calls)
    if (ps->prof) prof_before(ps, "kge_resident_kernel", s);
    cudaLaunchKernelEx(&cfg, kge_resident_kernel<kMaxNeg, kVec>, A, n_str, twice);
    if (ps->prof) prof_after(ps, s);
    ps->launches++;
    return grid;
}

}  // namespace

uint32_t launch_points_kge(ps_store* ps, const KgeBatch& B, const uint8_t* single, bool finished, uint32_t* keys_out, cudaStream_t s) {
    KgeArgs A;
    A.ts = B.s; A.tr = B.r; A.to = B.o; A.neg_ent = B.neg_ent; A.neg_side = B.neg_side;
    A.n = B.n; A.rel_base = B.rel_key_base; A.K = ps->cfg.num_keys;
    A.n_neg = B.n_neg; A.d = B.dim; A.lr = B.lr; A.eps = B.eps;
    A.store = ps->store; A.table = ps->table; A.S = ps->cfg.slots_per_part;
    A.upd = ps->upd; A.single = single; A.keys_out = keys_out; A.finished = finished;
    A.loss_partial = ps->loss_partial; A.st = ps->status; A.epoch = ps->epoch;
    // as many blocks as are resident at once, or one per example (the pdl form: kernels of small calls)
#define KGE_LAUNCH(name, kernel, threads, smem, per_block, per_sm)                                               \
    do {                                                                                                         \
        static std::atomic<unsigned long long> smem_set{0};                                                      \
        opt_in_smem((const void*)kernel, 200 * 1024, &smem_set);                                                 \
        const uint32_t grid = (uint32_t)tmin<uint64_t>((B.n + per_block - 1) / per_block, (uint64_t)ps->sm_count * (per_sm)); \
        if (keys_out) {                                                                                          \
            PS_LAUNCH_PDL(ps, name, kernel, dim3(grid), dim3(threads), smem, s, A);                              \
        } else {                                                                                                 \
            if (ps->prof) prof_before(ps, name, s);                                                              \
            kernel<<<grid, threads, smem, s>>>(A);                                                               \
            if (ps->prof) prof_after(ps, s);                                                                     \
            ps->launches++;                                                                                      \
        }                                                                                                        \
        return grid;                                                                                             \
    } while (0)
    // 65 to 128 dimensions: with more than 10 negatives in calls with a sort; in calls without one with 5 to 10 negatives and more than
    // 40 data points.  A step with kge_resident_kernel over one with kge_short_kernel, 8 dimensions from 66 to 128 by 10 numbers of data
    // points from 7 to 500: 10 negatives 1.01 to 1.04 at 7 and 16 data points, 0.98 to 1.03 at 30 and 41, 0.87 to 0.98 from 60 on; 8
    // negatives 0.93 to 1.03 from 41 on; 5 and 6 negatives 1.00 to 1.06 up to 30, 0.96 to 1.04 from 41 to 100 (a limit of 100 for 5 to 7:
    // 0.2 % slower over 270 sizes), 0.92 to 0.99 from 160 on; with few relations single sizes up to 1.10.  Outside: 4 negatives 0.92 to
    // 1.06, 1 and 3 0.95 to 1.10, 11 to 20 up to 1.13.
    const bool narrow = keys_out ? B.n_neg > 4 && B.n_neg <= 10 && B.n > 40 : B.n_neg > 10 && single;
    if (!finished && (B.dim > 128 || (B.dim > 64 && narrow))) {
#define KGE_RESIDENT(kMaxNeg)                                                                                     \
    (B.dim % 4 == 0 ? launch_resident<kMaxNeg, 4>(ps, A, s) : B.dim % 2 == 0 ? launch_resident<kMaxNeg, 2>(ps, A, s) \
                    : launch_resident<kMaxNeg, 1>(ps, A, s))
        const uint32_t grid = B.n_neg <= 4    ? KGE_RESIDENT(4)
                              : B.n_neg <= 10 ? KGE_RESIDENT(10)
                              : B.n_neg <= 20 ? KGE_RESIDENT(20) : KGE_RESIDENT(29);
#undef KGE_RESIDENT
        if (grid) return grid;
    }
    if (B.dim > 128) {
#define KGE_WIDE(kMaxNeg) return finished ? launch_wide<kMaxNeg, true>(ps, A, s) : launch_wide<kMaxNeg, false>(ps, A, s)
        if (B.n_neg <= 4) KGE_WIDE(4);
        if (B.n_neg <= 10) KGE_WIDE(10);
        if (B.n_neg <= 20) KGE_WIDE(20);
        KGE_WIDE(29);
#undef KGE_WIDE
    }
    const size_t smem = (size_t)kShortWarps * (3 + B.n_neg) * ((2 * B.dim + 3) & ~3u) * sizeof(float);
    const uint32_t fit = tmax<uint32_t>(1u, (uint32_t)((220 * 1024) / (smem + 4096)));
#define KGE_SHORT(kMaxNeg, resident)                                                                             \
    do {                                                                                                         \
        const bool even = B.dim % 2 == 0, acc = single || finished;                                              \
        if (even && acc) KGE_LAUNCH("kge_short_kernel<acc>", (kge_short_kernel<kMaxNeg, true, true>), 32 * kShortWarps, smem, kShortWarps, tmin<uint32_t>(fit, resident)); \
        if (even) KGE_LAUNCH("kge_short_kernel", (kge_short_kernel<kMaxNeg, true, false>), 32 * kShortWarps, smem, kShortWarps, tmin<uint32_t>(fit, resident)); \
        if (acc) KGE_LAUNCH("kge_short_kernel<acc>", (kge_short_kernel<kMaxNeg, false, true>), 32 * kShortWarps, smem, kShortWarps, tmin<uint32_t>(fit, resident)); \
        KGE_LAUNCH("kge_short_kernel", (kge_short_kernel<kMaxNeg, false, false>), 32 * kShortWarps, smem, kShortWarps, tmin<uint32_t>(fit, resident)); \
    } while (0)
    if (B.n_neg <= 4) KGE_SHORT(4, 4u);
    if (B.n_neg <= 10) KGE_SHORT(10, 4u);
    KGE_SHORT(29, 2u);
#undef KGE_SHORT
#undef KGE_LAUNCH
}

void launch_keys_kge(ps_store* ps, const KgeBatch& B, cudaStream_t s) {
    PS_LAUNCH(ps, kge_keys_kernel, div_up_u32(B.n, 8), 256, s, B.s, B.r, B.o, B.neg_ent, B.n, B.n_neg, B.rel_key_base,
              ps->cfg.num_keys, ps->keysA, ps->status, ps->epoch);
}

}  // namespace psb
