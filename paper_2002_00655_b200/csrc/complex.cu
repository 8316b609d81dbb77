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

// kMaxNeg bounds n_neg at compile time so that a data point's values live in registers: for every block of 32
// dimensions the Re and Im of all its rows are requested together, before any is used.  kDim / kExact: the complex
// dimension and "n_neg equals kMaxNeg" known at compile time (0 / false: taken from the arguments).
// kAcc: some slots need their accumulators here (rows updated in place, finished rows).
// kW: warps per data point.  One for rows of up to 128 complex dimensions (eight data points per block); eight for
// longer ones: a data point's rows are then read by one block within a short time, so that the second pass over them
// finds them in L2 (13 rows of 32 KB per block, one or two blocks per SM, fit; a data point per warp does not).
template <int kMaxNeg, int kDim, bool kExact, int kW, bool kAcc>
__global__ void __launch_bounds__(256, kMaxNeg <= 10 ? 2 : 1) kge_points_kernel(const KgeArgs A) {
    constexpr int kGroups = 8 / kW;                             // data points per block at a time
    __shared__ double s_part[kW > 1 ? kW : 1][kMaxNeg + 1];
    __shared__ double s_w[kGroups][3][32];                      // per slot: coefficient of negative q; weights of the two directions
    __shared__ double s_loss[8];
    const unsigned full = 0xffffffffu;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int group = w / kW, wg = w % kW;
    const uint32_t d = kDim ? (uint32_t)kDim : A.d;
    const uint32_t n_neg = kExact ? (uint32_t)kMaxNeg : A.n_neg;
    const int n_slots = 3 + (int)n_neg;
    const uint64_t L = 4 * (uint64_t)d, K = A.K;
    pdl_trigger();
    pdl_wait();
    if (A.single && call_failed(A.st, A.epoch)) return;
    double loss = 0;
    for (uint64_t t = (uint64_t)blockIdx.x * kGroups + group; t < A.n; t += (uint64_t)gridDim.x * kGroups) {
        // ---- keys, validity, rows, first slot with the same key (lane u holds slot u) ----
        uint64_t key = K;
        int side = 0;
        bool bad = false;
        const bool slot = lane < n_slots;
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
        if (__any_sync(full, bad)) {                            // (the same decision in every warp of the data point)
            if (lane == 0 && wg == 0) latch_error(A.st, A.keys_out ? 0u : A.epoch, PS_ERR_KEY_RANGE);
            if (A.keys_out && slot && wg == 0) A.keys_out[t * n_slots + lane] = kSentinelPad;
            continue;
        }
        const unsigned same = __match_any_sync(full, slot ? (uint32_t)key : kSentinelPad);
        const int rep = slot ? __ffs(same) - 1 : lane;
        if (A.keys_out && slot && wg == 0) A.keys_out[t * n_slots + lane] = rep == lane ? (uint32_t)key : (uint32_t)K;
        const bool once = slot && A.single && rep == lane && A.single[t * n_slots + lane];
        uint64_t off = 0;
        if (slot) off = phys_row(A.table[key], A.S) * L;
        float* const Srow = A.store + __shfl_sync(full, off, 0);
        float* const Rrow = A.store + __shfl_sync(full, off, 1);
        float* const Orow = A.store + __shfl_sync(full, off, 2);
        float* Nrow[kMaxNeg];
#pragma unroll
        for (int q = 0; q < kMaxNeg; ++q) Nrow[q] = A.store + __shfl_sync(full, off, (3 + q) & 31);
        // bit q: negative q stands in the subject's place; bit u: slot u is the first with its key / its key occurs once
        const unsigned subj_mask = __ballot_sync(full, lane >= 3 && slot && side == 0) >> 3;
        const unsigned rep_mask = __ballot_sync(full, slot && rep == lane), once_mask = __ballot_sync(full, once);
        const unsigned acc_mask = !kAcc ? 0u : A.finished ? rep_mask : once_mask;       // slots whose accumulators are needed here

        // ---- pass A: partial scores of the 1 + n_neg triples over this lane's dimensions ----
        double part[kMaxNeg + 1];
#pragma unroll
        for (int q = 0; q <= kMaxNeg; ++q) part[q] = 0.0;
        for (uint32_t c = wg * 32 + lane; c < d; c += 32 * kW) {
            const float a_f = Srow[c], b_f = Srow[d + c], cr_f = Rrow[c], ci_f = Rrow[d + c];
            const float e_f = Orow[c], f_f = Orow[d + c];
            float na_f[kMaxNeg], nb_f[kMaxNeg];
#pragma unroll
            for (int q = 0; q < kMaxNeg; ++q) {
                na_f[q] = q < (int)n_neg ? Nrow[q][c] : 0.f;
                nb_f[q] = q < (int)n_neg ? Nrow[q][d + c] : 0.f;
            }
            const double a = a_f, b = b_f, cr = cr_f, ci = ci_f, e = e_f, f = f_f;
            part[0] += cr * (a * e + b * f) + ci * (a * f - b * e);
            // (n, r, o): cr (na e + nb f) + ci (na f - nb e);   (s, r, n): cr (a na + b nb) + ci (a nb - b na)
            const double re_o = cr * e + ci * f, im_o = cr * f - ci * e;        // multiplies (na, nb) for side 0
            const double re_s = cr * a - ci * b, im_s = cr * b + ci * a;        // multiplies (na, nb) for side 1
#pragma unroll
            for (int q = 0; q < kMaxNeg; ++q) {
                const double na = na_f[q], nb = nb_f[q];
                part[q + 1] += ((subj_mask >> q) & 1u) ? (na * re_o + nb * im_o) : (na * re_s + nb * im_s);
            }
        }
        // the sums over the lanes, all triples' chains interleaved; lane q keeps triple q's score
#pragma unroll
        for (int o = 16; o > 0; o >>= 1)
#pragma unroll
            for (int q = 0; q <= kMaxNeg; ++q) part[q] += __shfl_xor_sync(full, part[q], o);
        double phi_mine = 0;
        if (kW > 1) {
            __syncthreads();                                    // (the data point before has been read)
            if (lane == 0)
#pragma unroll
                for (int q = 0; q <= kMaxNeg; ++q) s_part[wg][q] = part[q];
            __syncthreads();
            if (lane <= kMaxNeg)
                for (int i = 0; i < kW; ++i) phi_mine += s_part[i][lane];
        } else {
#pragma unroll
            for (int q = 0; q <= kMaxNeg; ++q)
                if (lane == q) phi_mine = part[q];
        }
        // lane q: loss term and d loss / d phi of triple q (label +1 for the positive, -1 for negatives)
        double coef = 0, loss_q = 0;
        if (lane <= (int)n_neg) {
            const double y = lane == 0 ? 1.0 : -1.0, z = -y * phi_mine, ez = exp(-fabs(z));
            loss_q = fmax(z, 0.0) + log1p(ez);
            coef = -y * ((z >= 0.0 ? 1.0 : ez) / (1.0 + ez));
        }
        loss_q = warp_sum_d(loss_q);
        if (wg == 0) loss += loss_q;

        // ---- weights with which each entity slot receives the two "negative role" directions ----
        // A negative with side 0 stands in the subject's place: its gradient is coef * dphi/dS(r, o).
        // With side 1 it stands in the object's place: coef * dphi/dO(s, r).  Summed over the
        // negatives whose key's first slot is this lane.
        double wS = 0, wO = 0;
#pragma unroll
        for (int q = 0; q < kMaxNeg; ++q) {
            const int rq = __shfl_sync(full, rep, (3 + q) & 31);
            const double cfq = __shfl_sync(full, coef, (q + 1) & 31);
            if (q < (int)n_neg && rq == lane) {
                if ((subj_mask >> q) & 1u) wS += cfq; else wO += cfq;
            }
        }
        const double cf0 = __shfl_sync(full, coef, 0);
        const int rep_o = __shfl_sync(full, rep, 2);            // 0 if object == subject
        // (read back as broadcasts; the warps of a data point write the same values)
        if (lane >= 1 && lane <= (int)n_neg) s_w[group][0][lane - 1] = coef;
        s_w[group][1][lane] = wS;
        s_w[group][2][lane] = wO;
        __syncwarp();
        const double* const cf = s_w[group][0];
        const double* const ws = s_w[group][1];
        const double* const wo = s_w[group][2];

        // ---- pass B: gradients per block of 32 complex dimensions ----
        const uint32_t LU = kAcc && A.finished ? 4 * d : 2 * d; // values per update row
        float* const U = A.upd + t * n_slots * (uint64_t)LU;
        auto out = [&](int u, float* row, uint32_t c, double gd_re, double gd_im, float x_re, float x_im, float G_re, float G_im) {
            const float g[2] = {(float)gd_re, (float)gd_im};
            if (!kAcc || !((acc_mask >> u) & 1u)) {
                U[(uint64_t)u * LU + c] = g[0];
                U[(uint64_t)u * LU + d + c] = g[1];
                return;
            }
            const float g2[2] = {g[0] * g[0], g[1] * g[1]}, x[2] = {G_re + g2[0], G_im + g2[1]};
            float step[2];
            adagrad_steps<2>(g, x, A.lr, A.eps, step);
            if ((once_mask >> u) & 1u) {
                row[c] = x_re + step[0];
                row[d + c] = x_im + step[1];
                row[2 * d + c] = x[0];
                row[3 * d + c] = x[1];
            } else {
                float* o = U + (uint64_t)u * LU;
                o[c] = step[0];
                o[d + c] = step[1];
                o[2 * d + c] = g2[0];
                o[3 * d + c] = g2[1];
            }
        };
        for (uint32_t c = wg * 32 + lane; c < d; c += 32 * kW) {
            // every value this block of dimensions needs, requested before the first use
            const float a_f = Srow[c], b_f = Srow[d + c], cr_f = Rrow[c], ci_f = Rrow[d + c];
            const float e_f = Orow[c], f_f = Orow[d + c];
            float na_f[kMaxNeg], nb_f[kMaxNeg];
#pragma unroll
            for (int q = 0; q < kMaxNeg; ++q) {
                const bool live = q < (int)n_neg;
                na_f[q] = live ? Nrow[q][c] : 0.f;
                nb_f[q] = live ? Nrow[q][d + c] : 0.f;
            }
            float G_re[3] = {0.f, 0.f, 0.f}, G_im[3] = {0.f, 0.f, 0.f};
            if (kAcc && (acc_mask & 1u)) { G_re[0] = Srow[2 * d + c]; G_im[0] = Srow[3 * d + c]; }
            if (kAcc && (acc_mask & 2u)) { G_re[1] = Rrow[2 * d + c]; G_im[1] = Rrow[3 * d + c]; }
            if (kAcc && (acc_mask & 4u)) { G_re[2] = Orow[2 * d + c]; G_im[2] = Orow[3 * d + c]; }
            const double a = a_f, b = b_f, cr = cr_f, ci = ci_f, e = e_f, f = f_f;
            // directions that do not depend on the negative
            const double dS_re = cr * e + ci * f, dS_im = cr * f - ci * e;      // d phi / d subject, object = o
            const double dO_re = cr * a - ci * b, dO_im = cr * b + ci * a;      // d phi / d object, subject = s
            // The negatives enter the gradients of subject, relation and object only through their weighted sums:
            // (A0, B0) over those in the subject's place (triples (n, r, o)), (A1, B1) over those in the object's
            // place (triples (s, r, n)).
            double A0 = 0.0, B0 = 0.0, A1 = 0.0, B1 = 0.0;
#pragma unroll
            for (int q = 0; q < kMaxNeg; ++q) {
                if (q >= (int)n_neg) break;
                const double na = na_f[q], nb = nb_f[q], wq = cf[q];
                if ((subj_mask >> q) & 1u) { A0 += wq * na; B0 += wq * nb; }
                else { A1 += wq * na; B1 += wq * nb; }
            }
            double gs_re = cf0 * dS_re, gs_im = cf0 * dS_im;
            double go_re = cf0 * dO_re, go_im = cf0 * dO_im;
            double gr_re = cf0 * (a * e + b * f), gr_im = cf0 * (a * f - b * e);
            gr_re += (A0 * e + B0 * f) + (a * A1 + b * B1); gr_im += (A0 * f - B0 * e) + (a * B1 - b * A1);
            go_re += cr * A0 - ci * B0; go_im += cr * B0 + ci * A0;
            gs_re += cr * A1 + ci * B1; gs_im += cr * B1 - ci * A1;
            // negatives that coincide with the subject or the object
            gs_re += ws[0] * dS_re + wo[0] * dO_re; gs_im += ws[0] * dS_im + wo[0] * dO_im;
            go_re += ws[2] * dS_re + wo[2] * dO_re; go_im += ws[2] * dS_im + wo[2] * dO_im;
            if (rep_o == 0) { gs_re += go_re; gs_im += go_im; }
            out(0, Srow, c, gs_re, gs_im, a_f, b_f, G_re[0], G_im[0]);
            out(1, Rrow, c, gr_re, gr_im, cr_f, ci_f, G_re[1], G_im[1]);
            if (rep_o == 2) out(2, Orow, c, go_re, go_im, e_f, f_f, G_re[2], G_im[2]);
            constexpr int kB = kMaxNeg < 5 ? kMaxNeg : 5;       // accumulators of so many negatives asked for together
#pragma unroll
            for (int q0 = 0; q0 < kMaxNeg; q0 += kB) {
                float Gq_re[kB], Gq_im[kB];
#pragma unroll
                for (int i = 0; i < kB; ++i) {
                    const int q = q0 + i;
                    Gq_re[i] = Gq_im[i] = 0.f;
                    if (kAcc && q < kMaxNeg && ((acc_mask >> (3 + q)) & 1u)) {
                        Gq_re[i] = Nrow[q][2 * d + c];
                        Gq_im[i] = Nrow[q][3 * d + c];
                    }
                }
#pragma unroll
                for (int i = 0; i < kB; ++i) {
                    const int q = q0 + i;
                    if (q >= kMaxNeg || !((rep_mask >> (3 + q)) & 1u)) continue;
                    const double wSq = ws[3 + q], wOq = wo[3 + q];
                    out(3 + q, Nrow[q], c, wSq * dS_re + wOq * dO_re, wSq * dS_im + wOq * dO_im, na_f[q], nb_f[q], Gq_re[i], Gq_im[i]);
                }
            }
        }
        __syncwarp();
    }
    // per-block loss partial, fixed order
    if (lane == 0) s_loss[w] = loss;
    __syncthreads();
    if (threadIdx.x == 0) {
        double tot = 0;
        for (int i = 0; i < 8; ++i) tot += s_loss[i];
        A.loss_partial[blockIdx.x] = tot;
    }
}

// Rows of more than 128 complex dimensions and up to ten negatives: a block per data point, the rows streamed through
// shared memory 256 dimensions at a time as bulk copies, the next stretch on its way while one is worked on, across the two
// passes and across data points.  (With loads into registers, one stretch after the other, the memory system was idle
// three quarters of the time: 1,199 us for 2,048 data points of 4,000 dimensions whose rows take 440 us.)  A stretch of a part
// (Re, Im, G_Re or G_Im) of a row starts at a multiple of 16 bytes only if d is a multiple of four: the copy starts at the
// boundary before it, and `shift` floats are skipped.
constexpr uint32_t kStretch = 256, kStretchPad = kStretch + 4;

template <int kMaxNeg>
__global__ void __launch_bounds__(256, 2) kge_wide_kernel(const KgeArgs A) {
    constexpr int kSlots = 3 + kMaxNeg, kWarps = 8;
    extern __shared__ __align__(128) float stage_mem[];         // [2 stages][slot][part][kStretchPad]
    __shared__ __align__(8) uint64_t bars[2];
    __shared__ double s_part[kWarps][kMaxNeg + 1];
    __shared__ double s_w[3][32];
    __shared__ uint64_t s_off[32];
    const unsigned full = 0xffffffffu;
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    const uint32_t d = A.d, n_neg = A.n_neg;
    const int n_slots = 3 + (int)n_neg;
    const bool slot = lane < n_slots;
    const uint64_t L = 4 * (uint64_t)d, K = A.K;
    if (tid < 2) mbar_init(&bars[tid], 1);
    mbar_init_fence();
    pdl_trigger();
    pdl_wait();
    if (A.single && call_failed(A.st, A.epoch)) return;
    __syncthreads();
    const uint32_t n_str = (d + kStretch - 1) / kStretch;
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
    // warp 0 asks for stretch number `str` of a data point's rows; with_acc: of their accumulators too where they are needed
    auto issue = [&](const Point& P, uint32_t str, bool with_acc, int stage) {
        const uint32_t c0 = str * kStretch, len = d - c0 < kStretch ? d - c0 : kStretch;
        const unsigned acc = with_acc ? (A.finished ? P.reps : P.once) : 0u;
        uint32_t bytes[4], total = 0;
#pragma unroll
        for (int p = 0; p < 4; ++p) {
            bytes[p] = ((len + ((p * d) & 3) + 3) & ~3u) * 4;
            total += bytes[p] * (p < 2 ? (uint32_t)n_slots : (uint32_t)__popc(acc));
        }
        if (lane == 0) mbar_expect_tx(&bars[stage], total);
        __syncwarp();
        if (!slot) return;
        const int parts = ((acc >> lane) & 1u) ? 4 : 2;
        for (int p = 0; p < parts; ++p)
            bulk_g2s(stage_mem + (((size_t)stage * kSlots + lane) * 4 + p) * kStretchPad, A.store + P.off + ((p * d + c0) & ~3u),
                     bytes[p], &bars[stage]);
    };
    uint64_t t = blockIdx.x;
    Point P = {}, N = {};
    // the first data point (from `from` on) whose indexes are all valid; marks the others (the same in every warp)
    auto next_valid = [&](uint64_t from, Point& Q) {
        for (; from < A.n; from += gridDim.x) {
            Q = look_up(from);
            if (A.keys_out && slot && w == 0)
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
    if (t < A.n && w == 0) issue(P, 0, false, 0);
    while (t < A.n) {
        const uint64_t tn = next_valid(t + gridDim.x, N);
        const unsigned subj_mask = P.subj, rep_mask = P.reps, once_mask = P.once, acc_mask = A.finished ? P.reps : P.once;
        double part[kMaxNeg + 1];
#pragma unroll
        for (int q = 0; q <= kMaxNeg; ++q) part[q] = 0.0;
        double cf0 = 0;
        int rep_o = 2;
        const uint32_t LU = A.finished ? 4 * d : 2 * d;         // values per update row
        float* const U = A.upd + t * n_slots * (uint64_t)LU;
        for (uint32_t job = 0; job < 2 * n_str; ++job) {
            const bool pass_b = job >= n_str;
            const uint32_t str = pass_b ? job - n_str : job;
            // the job after this one; its stage was read two jobs ago (and the warps have met since)
            if (w == 0) {
                if (job + 1 < 2 * n_str) issue(P, job + 1 >= n_str ? job + 1 - n_str : job + 1, job + 1 >= n_str, stage ^ 1);
                else if (tn < A.n) issue(N, 0, false, stage ^ 1);
            }
            if (!mbar_wait(&bars[stage], (uses >> stage) & 1u) && !mbar_wait(&bars[stage], (uses >> stage) & 1u)) dead = true;
            uses ^= 1u << stage;
            const float* const base = stage_mem + (size_t)stage * kSlots * 4 * kStretchPad + tid;
            const uint32_t sh1 = d & 3, sh2 = (2 * d) & 3, sh3 = (3 * d) & 3;
            auto re = [&](int u) { return base[u * 4 * kStretchPad]; };
            auto im = [&](int u) { return base[(u * 4 + 1) * kStretchPad + sh1]; };
            auto gre = [&](int u) { return base[(u * 4 + 2) * kStretchPad + sh2]; };
            auto gim = [&](int u) { return base[(u * 4 + 3) * kStretchPad + sh3]; };
            const uint32_t c = str * kStretch + tid;
            if (c < d) {
                const float a_f = re(0), b_f = im(0), cr_f = re(1), ci_f = im(1), e_f = re(2), f_f = im(2);
                const double a = a_f, b = b_f, cr = cr_f, ci = ci_f, e = e_f, f = f_f;
                // directions that do not depend on the negative: d phi / d subject (object = o), d phi / d object (subject = s)
                const double dS_re = cr * e + ci * f, dS_im = cr * f - ci * e;
                const double dO_re = cr * a - ci * b, dO_im = cr * b + ci * a;
                if (!pass_b) {
                    part[0] += cr * (a * e + b * f) + ci * (a * f - b * e);
#pragma unroll
                    for (int q = 0; q < kMaxNeg; ++q) {
                        if (q >= (int)n_neg) break;
                        const double na = re(3 + q), nb = im(3 + q);
                        part[q + 1] += ((subj_mask >> q) & 1u) ? (na * dS_re + nb * dS_im) : (na * dO_re + nb * dO_im);
                    }
                } else {
                    const double *cf = s_w[0], *ws = s_w[1], *wo = s_w[2];
                    double A0 = 0.0, B0 = 0.0, A1 = 0.0, B1 = 0.0;      // weighted sums of the negatives in either place
#pragma unroll
                    for (int q = 0; q < kMaxNeg; ++q) {
                        if (q >= (int)n_neg) break;
                        const double na = re(3 + q), nb = im(3 + q), wq = cf[q];
                        if ((subj_mask >> q) & 1u) { A0 += wq * na; B0 += wq * nb; }
                        else { A1 += wq * na; B1 += wq * nb; }
                    }
                    double gs_re = cf0 * dS_re, gs_im = cf0 * dS_im;
                    double go_re = cf0 * dO_re, go_im = cf0 * dO_im;
                    double gr_re = cf0 * (a * e + b * f), gr_im = cf0 * (a * f - b * e);
                    gr_re += (A0 * e + B0 * f) + (a * A1 + b * B1); gr_im += (A0 * f - B0 * e) + (a * B1 - b * A1);
                    go_re += cr * A0 - ci * B0; go_im += cr * B0 + ci * A0;
                    gs_re += cr * A1 + ci * B1; gs_im += cr * B1 - ci * A1;
                    // negatives that coincide with the subject or the object
                    gs_re += ws[0] * dS_re + wo[0] * dO_re; gs_im += ws[0] * dS_im + wo[0] * dO_im;
                    go_re += ws[2] * dS_re + wo[2] * dO_re; go_im += ws[2] * dS_im + wo[2] * dO_im;
                    if (rep_o == 0) { gs_re += go_re; gs_im += go_im; }
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
                        const bool in_place = (once_mask >> u) & 1u;
                        if (in_place) o = A.store + s_off[u] + c;
                        o[0] = in_place ? re(u) + step[0] : step[0];
                        o[d] = in_place ? im(u) + step[1] : step[1];
                        o[2 * d] = in_place ? x[0] : g2[0];
                        o[3 * d] = in_place ? x[1] : g2[1];
                    };
                    out(0, gs_re, gs_im);
                    out(1, gr_re, gr_im);
                    if (rep_o == 2) out(2, go_re, go_im);
#pragma unroll
                    for (int q = 0; q < kMaxNeg; ++q) {
                        if (q >= (int)n_neg) break;
                        if (!((rep_mask >> (3 + q)) & 1u)) continue;
                        const double wSq = ws[3 + q], wOq = wo[3 + q];
                        out(3 + q, wSq * dS_re + wOq * dO_re, wSq * dS_im + wOq * dO_im);
                    }
                }
            }
            stage ^= 1;
            if (job + 1 == n_str) {             // the scores are complete: coefficients and weights, as in kge_points_kernel
#pragma unroll
                for (int o = 16; o > 0; o >>= 1)
#pragma unroll
                    for (int q = 0; q <= kMaxNeg; ++q) part[q] += __shfl_xor_sync(full, part[q], o);
                if (lane == 0)
#pragma unroll
                    for (int q = 0; q <= kMaxNeg; ++q) s_part[w][q] = part[q];
                __syncthreads();
                double phi = 0, coef = 0, loss_q = 0;
                if (lane <= kMaxNeg)
                    for (int i = 0; i < kWarps; ++i) phi += s_part[i][lane];
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
                if (tid == 0) latch_error(A.st, A.epoch, PS_ERR_CUDA);
                return;
            }
        }
        P = N;
        t = tn;
    }
    if (tid == 0) A.loss_partial[blockIdx.x] = loss;
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

}  // namespace

uint32_t launch_points_kge(ps_store* ps, const KgeBatch& B, const uint8_t* single, bool finished, uint32_t* keys_out, cudaStream_t s) {
    KgeArgs A;
    A.ts = B.s; A.tr = B.r; A.to = B.o; A.neg_ent = B.neg_ent; A.neg_side = B.neg_side;
    A.n = B.n; A.rel_base = B.rel_key_base; A.K = ps->cfg.num_keys;
    A.n_neg = B.n_neg; A.d = B.dim; A.lr = B.lr; A.eps = B.eps;
    A.store = ps->store; A.table = ps->table; A.S = ps->cfg.slots_per_part;
    A.upd = ps->upd; A.single = single; A.keys_out = keys_out; A.finished = finished;
    A.loss_partial = ps->loss_partial; A.st = ps->status; A.epoch = ps->epoch;
    const bool wide = B.dim > 128;
    if (wide && B.n_neg <= 10) {
        const uint32_t grid = (uint32_t)tmin<uint64_t>(B.n, (uint64_t)ps->sm_count * 2);
#define KGE_WIDE(kMaxNeg)                                                                                        \
        do {                                                                                                     \
            static std::atomic<unsigned long long> smem_set{0};                                                  \
            const size_t smem = (size_t)2 * (3 + kMaxNeg) * 4 * kStretchPad * sizeof(float);                     \
            opt_in_smem((const void*)kge_wide_kernel<kMaxNeg>, smem, &smem_set);                                 \
            if (keys_out) PS_LAUNCH_PDL(ps, "kge_wide_kernel<" #kMaxNeg ">", kge_wide_kernel<kMaxNeg>, dim3(grid), dim3(256), smem, s, A); \
            else PS_LAUNCH_SMEM(ps, kge_wide_kernel<kMaxNeg>, grid, 256, smem, s, A);                            \
        } while (0)
        if (B.n_neg <= 4) KGE_WIDE(4);
        else KGE_WIDE(10);
#undef KGE_WIDE
        return grid;
    }
    uint64_t g = wide ? B.n : (B.n + 7) / 8;
    g = tmin<uint64_t>(g, tmin<uint64_t>((uint64_t)ps->sm_count * (wide ? 2 : 8), kMaxLossBlocks));
    const uint32_t grid = (uint32_t)g;
#define KGE_LAUNCH(kMaxNeg, kDim, kExact, kW, kAcc)                                                                   \
    do {                                                                                                         \
        const char* name = kW > 1 ? "kge_points_kernel<wide>" : "kge_points_kernel";                             \
        if (keys_out) {                                                                                          \
            PS_LAUNCH_PDL(ps, name, (kge_points_kernel<kMaxNeg, kDim, kExact, kW, kAcc>), dim3(grid), dim3(256), 0, s, A); \
        } else {                                                                                                 \
            if (ps->prof) prof_before(ps, name, s);                                                              \
            kge_points_kernel<kMaxNeg, kDim, kExact, kW, kAcc><<<grid, 256, 0, s>>>(A);                          \
            if (ps->prof) prof_after(ps, s);                                                                     \
            ps->launches++;                                                                                      \
        }                                                                                                        \
    } while (0)
    if (wide) KGE_LAUNCH(29, 0, false, 8, true);
    else if (finished) {
        if (B.n_neg <= 10) KGE_LAUNCH(10, 0, false, 1, true);
        else KGE_LAUNCH(29, 0, false, 1, true);
    } else {
        if (B.n_neg == 10 && B.dim == 100) KGE_LAUNCH(10, 100, true, 1, false);
        else if (B.n_neg <= 4) KGE_LAUNCH(4, 0, false, 1, false);
        else if (B.n_neg <= 10) KGE_LAUNCH(10, 0, false, 1, false);
        else KGE_LAUNCH(29, 0, false, 1, false);
    }
#undef KGE_LAUNCH
    return grid;
}

void launch_keys_kge(ps_store* ps, const KgeBatch& B, cudaStream_t s) {
    PS_LAUNCH(ps, kge_keys_kernel, div_up_u32(B.n, 8), 256, s, B.s, B.r, B.o, B.neg_ent, B.n, B.n_neg, B.rel_key_base,
              ps->cfg.num_keys, ps->keysA, ps->status, ps->epoch);
}

}  // namespace psb
