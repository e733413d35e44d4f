// Active set and extrapolation grade of Sec. 2.3 (D-optimality, MaxVol of Goreinov et al. 2010).
//
// k_maxvol (cooperative, double precision, all loops and waits bounded):
//   0. columns are scaled by 1 / max |column| (the grades and the selection are invariant under
//      B -> B D, and the scaled matrix is far better conditioned);
//   1. start rows: the pivot rows of Gaussian elimination with partial pivoting on the tall
//      matrix B (n_rows x m); ties go to the smaller current row position (or, for the select-add
//      update, the first m rows: the current active set stacked above the candidates);
//   2. A^-1 of A = B[sel] by Gauss-Jordan elimination with partial pivoting;
//   3. C = B A^-1 for every row;
//   4. repeat at most max_iter times: (k, j) = argmax |C_kj| (ties: smallest k, then smallest j);
//      stop when |C_kj| <= 1 + tol (tol = 1e-3); otherwise row k replaces active row j, and C follows
//      by the rank-one (Sherman-Morrison) update  C <- C - C[:,j] (C[k,:] - e_j) / C_kj.
//   A^-1 is computed from scratch at the end.
//
// Every phase is a chain of dependent steps (m pivots, or one swap), each a rank-one update of all rows.
// A block owns a fixed set of rows and keeps them in shared memory for a whole phase, so that a step
// exchanges only what the others need: every block publishes its best candidate (value, position) with
// the candidate's row, waits for the others' and takes the same winner (Exchange).  Rows are never
// moved: a row's current position is a number beside it.  The inverse runs in place (the column that a
// pivot eliminates is replaced by the column of the inverse that it creates).  Pivots, factors and
// inverse are the same operations in the same order as elimination by one block with explicit
// interchanges, so the selection does not depend on the number of blocks.
// Bound: one exchange per step (a trip to the L2 for the records and one for the winner's row) and the
// step's FMAs and the swaps' divisions on the double-precision pipe (~2 FMAs per clock and SM).  Measured with
// all grades of the rows: 232 x 116 in 1.68 ms, 920 x 460 in 8.2 ms; with flags and fences instead of tagged
// words (and without the divisions) 2.81 and 13.7; one block with every matrix in global memory 10.8 and 451.
// k_grade: gamma_r = max_j |(b_r A^-1)_j| for many rows; 64x64 output tiles through shared memory,
//   the row maxima are combined with an atomic max on the bit pattern (gamma >= 0); a NaN in a row
//   of b A^-1 gives gamma = +inf, so a broken configuration reads as extrapolating.
#include <cuda_runtime.h>
#include <stdint.h>
#include <algorithm>
#include <mutex>
#include "../../include/mtp.h"
#include "mtp_common.cuh"

namespace mtp {

namespace {

constexpr int kMvThreads = 512;

// One round of all blocks: each publishes a candidate (a non-negative value and a 32-bit payload, ties
// to the smaller payload) and its row; everyone gets the winner.  Every word that another block reads
// travels with the round's number in one 128-bit store, and a reader polls until the number is there, so
// that neither the record nor the row waits for a fence: a round costs one trip to the L2 for the records
// and one for the winner's row.  Two alternating sets of records and rows: a block publishes round t + 1
// only after it has read all that it needs of round t, and nobody publishes t + 2 before that, so nobody
// can still be reading what is overwritten.
constexpr unsigned kNone = 0xffffffffu;
constexpr long kMvSpins = 4l << 20;  // a poll takes the better part of a microsecond: gives up after seconds

// (generic addresses: the exchange lies in shared memory when there is one block)
__device__ __forceinline__ void put_tagged(void* p, unsigned long long v, unsigned long long tag) {
    asm volatile("{ .reg .b128 q; mov.b128 q, {%1, %2}; st.relaxed.gpu.b128 [%0], q; }" ::"l"(p), "l"(v), "l"(tag)
                 : "memory");
}
__device__ __forceinline__ unsigned long long get_tagged(const void* p, unsigned long long* tag) {
    unsigned long long v;
    asm volatile("{ .reg .b128 q; ld.relaxed.gpu.b128 q, [%2]; mov.b128 {%0, %1}, q; }"
                 : "=l"(v), "=l"(*tag)
                 : "l"(p)
                 : "memory");
    return v;
}

// The warp's best (value bits, payload): the largest value, ties to the smaller payload, kNone loses to
// everything.  Every lane gets it, and the lane that holds it (payloads are distinct).
__device__ __forceinline__ int warp_best(unsigned long long& v, unsigned& p) {
    const unsigned hi = p == kNone ? 0u : (unsigned)(v >> 32), lo = p == kNone ? 0u : (unsigned)v;
    const unsigned mh = __reduce_max_sync(0xffffffffu, hi);
    const unsigned ml = __reduce_max_sync(0xffffffffu, hi == mh ? lo : 0u);
    const bool top = hi == mh && lo == ml;
    const unsigned mp = __reduce_min_sync(0xffffffffu, top ? p : kNone);
    v = ((unsigned long long)mh << 32) | ml;
    const unsigned who = __ballot_sync(0xffffffffu, top && p == mp);
    p = mp;
    return __ffs(who) - 1;
}

// A block's own rows: w [R][m], their positions, and R numbers for a column of them.
struct Rows {
    double* w;
    int* pos;
    double* col;
    int first, R, m;          // rows first .. first + R - 1 of the matrix
    double* prow;             // shared [m]: the winner's row
    unsigned long long* s_v;  // shared [32]: candidates of the warps
    unsigned* s_p;
    int* s_r;
};

struct Exchange {
    unsigned long long* rec;    // [2][G][2]: (value bits, round | payload)
    unsigned long long* slots;  // [2][G][m + 2][2]: the candidates' rows, the row's number, 1 / pivot
    int G, m;
    unsigned t;
    int* err;
    unsigned long long* s_win;  // shared [3]: the winner's value, payload, block (-1: none, -2: gave up)

    __device__ unsigned long long* slot(int q) const {
        return slots + ((size_t)(t & 1) * G + q) * (m + 2) * 2;
    }
    __device__ void send(int c, double v) const {
        put_tagged(slot(blockIdx.x) + 2 * c, (unsigned long long)__double_as_longlong(v), t);
    }
    // entry c of block q's row; *bad if it never comes
    __device__ double receive(int q, int c, bool* bad) const {
        unsigned long long tag, v;
        long spins = 0;
        do {
            v = get_tagged(slot(q) + 2 * c, &tag);
        } while (tag != t && ++spins < kMvSpins);
        if (tag != t) *bad = true;
        return __longlong_as_double((long long)v);
    }
    // the same, or a negative number if it is not there yet
    __device__ double peek(int q, int c) const {
        unsigned long long tag;
        const unsigned long long v = get_tagged(slot(q) + 2 * c, &tag);
        return tag == t ? __longlong_as_double((long long)v) : -1.0;
    }
    // (one thread) this block's record of the round
    __device__ void publish(unsigned long long v, unsigned payload) const {
        put_tagged(rec + ((size_t)(t & 1) * G + blockIdx.x) * 2, v, ((unsigned long long)t << 32) | payload);
    }
    // (one warp) all blocks' records: the winner into s_win
    __device__ void poll() const {
        unsigned long long bv = 0;
        unsigned bp = kNone;
        int bq = -1;
        bool bad = false;
        constexpr int kEach = 8;  // records a lane polls at once (256 blocks; more take turns)
        for (int q0 = threadIdx.x & 31; q0 < G; q0 += 32 * kEach) {
            unsigned long long v[kEach], w[kEach];
            long spins = 0;
            bool missing;
            do {  // all loads are on their way before the first is looked at
                missing = false;
#pragma unroll
                for (int u = 0; u < kEach; ++u)
                    if (q0 + 32 * u < G) v[u] = get_tagged(rec + ((size_t)(t & 1) * G + q0 + 32 * u) * 2, &w[u]);
#pragma unroll
                for (int u = 0; u < kEach; ++u)
                    if (q0 + 32 * u < G) missing = missing || (unsigned)(w[u] >> 32) != t;
            } while (missing && ++spins < kMvSpins);
            bad = bad || missing;
#pragma unroll
            for (int u = 0; u < kEach; ++u) {
                const unsigned p = (unsigned)w[u];
                if (q0 + 32 * u < G && p != kNone && (bq < 0 || v[u] > bv || (v[u] == bv && p < bp))) {
                    bv = v[u];
                    bp = p;
                    bq = q0 + 32 * u;
                }
            }
        }
        bad = __any_sync(0xffffffffu, bad);
        const int who = warp_best(bv, bp);
        bq = __shfl_sync(0xffffffffu, bq, who);
        if ((threadIdx.x & 31) == 0) {
            s_win[0] = bv;
            s_win[1] = bp;
            s_win[2] = (unsigned long long)(long long)(bad ? -2 : bq);
            if (bad) atomicOr(err, kErrTimeout);
        }
    }
    // The round's end for the block, after warp 0 published: the winner's block, or -1, or -2.
    __device__ int winner(double* value, unsigned* payload) const {
        if ((threadIdx.x >> 5) == 1) poll();
        __syncthreads();
        *value = __longlong_as_double((long long)s_win[0]);
        *payload = (unsigned)s_win[1];
        return (int)(long long)s_win[2];
    }
    // Waits until every block has come here; what the blocks wrote before is visible after.
    __device__ bool barrier() {
        ++t;
        __syncthreads();
        if (threadIdx.x == 0) {
            __threadfence();
            publish(0, kNone);
        }
        double v;
        unsigned p;
        const int q = winner(&v, &p);
        __threadfence();
        __syncthreads();
        return q != -2;
    }
};

// The candidate of a pivot step: largest |w[r][k]| among the block's rows at positions >= k (ties to the
// smaller position; NaN is no candidate).  Warp 0 publishes it with its row from column c0 on and, if asked
// to, while the record travels, the reciprocal of the pivot.  The block is in step before and after is not.
__device__ void publish_pivot(Exchange& x, const Rows& a, int k, int c0, bool reciprocal) {
    ++x.t;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    unsigned long long bv = 0;
    unsigned bp = kNone;
    int br = -1;
    auto scan = [&](int from, int step) {
        for (int r = from; r < a.R; r += step) {
            const int p = a.pos[r];
            const unsigned long long v =
                (unsigned long long)__double_as_longlong(a.w[(size_t)r * a.m + k]) & 0x7fffffffffffffffull;
            if (p >= k && v <= 0x7ff0000000000000ull && (br < 0 || v > bv || (v == bv && (unsigned)p < bp))) {
                bv = v;
                bp = (unsigned)p;
                br = r;
            }
        }
    };
    if (a.R > 64) {  // many rows: every warp takes a share first
        scan(threadIdx.x, blockDim.x);
        const int who = warp_best(bv, bp);
        br = __shfl_sync(0xffffffffu, br, who);
        if (lane == 0) {
            a.s_v[warp] = bv;
            a.s_p[warp] = bp;
            a.s_r[warp] = br;
        }
        __syncthreads();
        if (warp == 0) {
            bv = lane < nw ? a.s_v[lane] : 0;
            bp = lane < nw ? a.s_p[lane] : kNone;
            br = lane < nw ? a.s_r[lane] : -1;
        }
    } else if (warp == 0) {
        scan(lane, 32);
    }
    if (warp == 0) {
        const int who = warp_best(bv, bp);
        br = __shfl_sync(0xffffffffu, br, who);
        if (lane == 0) x.publish(bv, bp);
        if (bp != kNone) {
            const double* row = a.w + (size_t)br * a.m;
            for (int c = c0 + lane; c < a.m; c += 32) x.send(c, row[c]);
            if (lane == 0) x.send(a.m, (double)(a.first + br));
            if (reciprocal && lane == 1) x.send(a.m + 1, 1.0 / row[k]);
        }
    }
}

// w[r][c] <- update(w[r][c], col[r], prow[c]) for the block's rows that keep(r) takes and columns c0 <= c < m;
// seen(value, r, c) gets every new value.  Warps take rows, and parts of a row where there are more warps
// than rows.
template <class Keep, class Update, class Seen>
__device__ __forceinline__ void rank_one(const Rows& a, int c0, Keep keep, Update update, Seen seen) {
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nw = blockDim.x >> 5;
    if (a.R < 1) return;
    const int parts = a.R < nw ? nw / a.R : 1;
    const int part = a.R < nw ? warp / a.R : 0;
    if (part >= parts) return;
    for (int r = a.R < nw ? warp % a.R : warp; r < a.R; r += nw) {
        if (!keep(r)) continue;
        const double l = a.col[r];
        double* w = a.w + (size_t)r * a.m;
        for (int c = c0 + part * 32 + lane; c < a.m; c += parts * 32) {
            const double v = update(w[c], l, a.prow[c]);
            w[c] = v;
            seen(v, r, c);
        }
    }
}
__device__ __forceinline__ double eliminate(double w, double l, double p) { return fma(-l, p, w); }

// NR rows of C = B A^-1 (chunk: NR rows of B, scaled): a thread per column, k in order.
template <int NR, class Put>
__device__ __forceinline__ void product_rows(const double* chunk, const double* Ai, int m, Put put) {
    for (int c = threadIdx.x; c < m; c += blockDim.x) {
        double s[NR];
#pragma unroll
        for (int r = 0; r < NR; ++r) s[r] = 0.0;
#pragma unroll 8
        for (int k = 0; k < m; ++k) {
            const double ai = __ldcg(Ai + (size_t)k * m + c);
#pragma unroll
            for (int r = 0; r < NR; ++r) s[r] = fma(chunk[r * m + k], ai, s[r]);
        }
#pragma unroll
        for (int r = 0; r < NR; ++r) put(s[r], r, c);
    }
}

// Inverse of the m x m matrix whose row j is load(j, c), in place with partial pivoting; its row at
// position q goes to Ai[q][.], scaled by scale(q).  False: a zero (or no finite) pivot, or a wait that
// gave up (then *err is set).  orig: shared [m].
template <class Load, class Scale>
__device__ bool invert_rows(Exchange& x, Rows& a, int* orig, double* Ai, int* status, Load load, Scale scale) {
    const int m = a.m, tid = threadIdx.x, nt = blockDim.x;
    for (int e = tid; e < a.R * m; e += nt) a.w[e] = load(a.first + e / m, e % m);
    for (int r = tid; r < a.R; r += nt) a.pos[r] = a.first + r;
    __syncthreads();
    for (int k = 0; k < m; ++k) {
        publish_pivot(x, a, k, 0, true);
        double v;
        unsigned p;
        const int q = x.winner(&v, &p);
        if (q < 0 || v == 0.0) {
            if (q != -2 && tid == 0 && blockIdx.x == 0) atomicOr(status, kErrSingular);
            return false;
        }
        bool bad = false;
        const double inv = x.receive(q, m + 1, &bad);
        for (int c = tid; c < m; c += nt) a.prow[c] = c == k ? inv : x.receive(q, c, &bad) * inv;
        if (tid == nt - 1) orig[k] = (int)x.receive(q, m, &bad);
        for (int r = tid; r < a.R; r += nt) {
            if (a.pos[r] == (int)p)
                a.pos[r] = k;
            else if (a.pos[r] == k)
                a.pos[r] = (int)p;
            a.col[r] = a.w[(size_t)r * m + k];
            a.w[(size_t)r * m + k] = 0.0;  // the eliminated column; the new column of the inverse grows here
        }
        if (__syncthreads_or(bad)) {
            if (bad) atomicOr(x.err, kErrTimeout);
            return false;
        }
        rank_one(a, 0, [&](int r) { return a.pos[r] != k; }, eliminate, [](double, int, int) {});
        if (q == (int)blockIdx.x)
            for (int r = 0; r < a.R; ++r)
                if (a.pos[r] == k)
                    for (int c = tid; c < m; c += nt) a.w[(size_t)r * m + c] = a.prow[c];
        __syncthreads();
    }
    for (int e = tid; e < a.R * m; e += nt) {
        const int row = a.pos[e / m];
        Ai[(size_t)row * m + orig[e % m]] = a.w[e] * scale(row);
    }
    return true;
}

// Shared memory of the cooperative kernels, in order: the winner, the warps' candidates,
// (G == 1: records and rows of the exchange), prow [m], orig [m], then for k_maxvol D [m], sel [m] and a chunk of B, and
// the block's rows with their positions and column when those fit.
struct Layout {
    int G, R, br;          // blocks, rows of a block at most, rows of B in a chunk
    bool rows_in, col_in;  // rows, positions and column in shared memory
    size_t bytes;
};
constexpr size_t kMvSharedMost = 200 * 1024;

__host__ __device__ inline int mv_rows(int n, int G) { return (n + G - 1) / G; }

inline Layout mv_layout(int n, int m, int G, bool full) {
    Layout l{};
    l.G = G;
    l.R = mv_rows(n > m ? n : m, G);
    l.br = full ? (m <= 1024 ? 8 : 1) : 0;
    size_t b = 32 + 32 * 16 + (G == 1 ? 32 + 32 * (size_t)(m + 2) : 0);
    const size_t ints = 8 * ((size_t)(m + 1) / 2);                    // m ints in 8-byte slots
    b += 8 * (size_t)m + ints;                                        // prow, orig
    if (full) b += 8 * (size_t)m + ints + 8 * (size_t)m * l.br;       // D, sel, chunk
    l.col_in = b + 16 * (size_t)l.R <= kMvSharedMost;
    if (l.col_in) b += 16 * (size_t)l.R;
    l.rows_in = b + 8 * (size_t)l.R * m <= kMvSharedMost;
    if (l.rows_in) b += 8 * (size_t)l.R * m;
    l.bytes = b;
    return l;
}

struct Carve {
    unsigned char* p;
    template <class T>
    __device__ T* take(size_t count) {  // 8-byte slots
        T* r = reinterpret_cast<T*>(p);
        p += 8 * ((count * sizeof(T) + 7) / 8);
        return r;
    }
};

__device__ void carve_common(Carve& s, Exchange& x, Rows& a, int** orig) {
    x.s_win = s.take<unsigned long long>(4);
    a.s_v = s.take<unsigned long long>(32);
    a.s_p = s.take<unsigned>(32);
    a.s_r = s.take<int>(32);
    if (x.G == 1) {  // (16-byte aligned: everything before is a multiple of 32 bytes)
        x.rec = s.take<unsigned long long>(4);
        x.slots = s.take<unsigned long long>(4 * (size_t)(x.m + 2));
        for (int e = threadIdx.x; e < 4 + 4 * (x.m + 2); e += blockDim.x) x.rec[e] = 0;
    }
    a.prow = s.take<double>(x.m);
    *orig = s.take<int>(x.m);
}

struct MaxvolArgs {
    int n, m, G, br;
    bool rows_in, col_in;
    const double* B;           // [n][m]
    double* rows;              // [max(n, m)][m] when the rows do not fit in shared memory
    double* col;               // [max(n, m)], likewise
    int* pos;                  // [n], likewise
    unsigned long long* rec;   // [2][G][2], zero at the start (G > 1)
    unsigned long long* slots; // [2][G][m + 2][2], zero at the start (G > 1)
    int* sel;                  // [m]
    double* A;                 // [m][m]
    double* Ai;                // [m][m]
    double tol;
    int max_iter, start_given;
    int *status, *swaps;
    double* gmax;
};

__global__ void __launch_bounds__(kMvThreads) k_maxvol(const MaxvolArgs g) {
    extern __shared__ __align__(16) unsigned char smem[];
    const int tid = threadIdx.x, nt = blockDim.x, n = g.n, m = g.m;
    Carve sh{smem};
    Exchange x{g.rec, g.slots, g.G, m, 0u, g.status, nullptr};
    Rows a{};
    int* orig;
    carve_common(sh, x, a, &orig);
    double* D = sh.take<double>(m);
    int* sel = sh.take<int>(m);
    double* chunk = sh.take<double>((size_t)m * g.br);
    const int Rn = mv_rows(n, g.G), Rm = mv_rows(m, g.G), Rmost = Rn > Rm ? Rn : Rm;
    double* col_s = g.col_in ? sh.take<double>(Rmost) : nullptr;
    int* pos_s = g.col_in ? sh.take<int>(2 * Rmost) : nullptr;
    double* rows_s = g.rows_in ? sh.take<double>((size_t)Rmost * m) : nullptr;
    a.m = m;
    auto own = [&](int total, int each) {  // the block's share of `total` rows
        a.first = min(total, (int)blockIdx.x * each);
        a.R = min(total, a.first + each) - a.first;
        a.w = g.rows_in ? rows_s : g.rows + (size_t)a.first * m;
        a.col = g.col_in ? col_s : g.col + a.first;
        a.pos = g.col_in ? pos_s : g.pos + a.first;
    };
    own(n, Rn);
    __syncthreads();
    // 0. column equilibration: the largest |column| of the block's rows, then of all blocks'
    ++x.t;
    for (int c = tid; c < m; c += nt) {
        double mx = 0.0;
        for (int r = 0; r < a.R; ++r) mx = fmax(mx, fabs(g.B[(size_t)(a.first + r) * m + c]));
        x.send(c, mx);
    }
    if (tid == 0) x.publish(0, kNone);
    {
        double v;
        unsigned p;
        if (x.winner(&v, &p) == -2) return;
    }
    bool zero = false, late = false;
    for (int c = tid; c < m; c += nt) {
        double mx = 0.0;
        for (int q0 = 0; q0 < g.G; q0 += 8) {  // eight on their way at once
            double each[8];
#pragma unroll
            for (int u = 0; u < 8; ++u) each[u] = x.peek(min(q0 + u, g.G - 1), c);
#pragma unroll
            for (int u = 0; u < 8; ++u)
                mx = fmax(mx, each[u] >= 0.0 ? each[u] : x.receive(min(q0 + u, g.G - 1), c, &late));
        }
        D[c] = mx > 0.0 ? 1.0 / mx : 0.0;
        zero = zero || D[c] == 0.0;
    }
    if (__syncthreads_or(late)) {
        if (late) atomicOr(g.status, kErrTimeout);
        return;
    }
    if (__syncthreads_or(zero)) {
        if (tid == 0 && blockIdx.x == 0) atomicOr(g.status, kErrSingular);
        return;
    }
    if (g.start_given) {  // select-add: start from the first m rows (the current active set)
        for (int j = tid; j < m; j += nt) sel[j] = j;
    } else {
        // 1. pivot rows of LU with partial pivoting
        for (int e = tid; e < a.R * m; e += nt) a.w[e] = g.B[(size_t)a.first * m + e] * D[e % m];
        for (int r = tid; r < a.R; r += nt) a.pos[r] = a.first + r;
        __syncthreads();
        for (int k = 0; k < m; ++k) {
            publish_pivot(x, a, k, k, false);
            double v;
            unsigned p;
            const int q = x.winner(&v, &p);
            if (q < 0 || v == 0.0) {
                if (q != -2 && tid == 0 && blockIdx.x == 0) atomicOr(g.status, kErrSingular);
                return;
            }
            bool bad = false;
            for (int c = k + 1 + tid; c < m; c += nt) a.prow[c] = x.receive(q, c, &bad);
            if (tid == nt / 2) sel[k] = (int)x.receive(q, m, &bad);
            // (the last warps: the division, over a thousand clocks, runs beside the row's arrival)
            const int rt = nt - 1 - tid;
            const double pivot = rt < a.R ? x.receive(q, k, &bad) : 1.0;
            for (int r = rt; r < a.R; r += nt) {
                if (a.pos[r] == (int)p)
                    a.pos[r] = k;
                else if (a.pos[r] == k)
                    a.pos[r] = (int)p;
                a.col[r] = a.w[(size_t)r * m + k] / pivot;
            }
            if (__syncthreads_or(bad)) {
                if (bad) atomicOr(g.status, kErrTimeout);
                return;
            }
            rank_one(a, k + 1, [&](int r) { return a.pos[r] > k; }, eliminate, [](double, int, int) {});
            __syncthreads();
        }
    }
    __syncthreads();
    // The shares of A's rows begin elsewhere than those of B's.  In global memory (matrices of some 10,000
    // rows and more) a block's first rows of A lie among another's rows of B, so everyone finishes first: one
    // round of the exchange, a few microseconds of such a phase's milliseconds.
    const bool shared = g.rows_in && g.col_in;
    if (!shared && !x.barrier()) return;
    // 2. the inverse of A = B[sel]
    const auto load = [&](int j, int c) { return g.B[(size_t)sel[j] * m + c] * D[c]; };
    own(m, Rm);
    if (!invert_rows(x, a, orig, g.Ai, g.status, load, [](int) { return 1.0; })) return;
    if (!x.barrier()) return;  // every block's rows of A^-1 are written
    // 3. C = B A^-1 for the block's rows, a few rows at a time (a thread per column)
    own(n, Rn);
    double best = -1.0;
    int at = 0;
    auto track = [&](double v, int e) {
        v = fabs(v);
        if (v > best || (v == best && e < at)) {
            best = v;
            at = e;
        }
    };
    for (int r0 = 0; r0 < a.R; r0 += g.br) {
        const int nr = min(g.br, a.R - r0);
        __syncthreads();
        for (int e = tid; e < nr * m; e += nt) chunk[e] = g.B[(size_t)(a.first + r0) * m + e] * D[e % m];
        __syncthreads();
        const auto put = [&](double v, int r, int c) {
            a.w[(size_t)(r0 + r) * m + c] = v;
            track(v, (a.first + r0 + r) * m + c);
        };
        switch (nr) {
            case 8: product_rows<8>(chunk, g.Ai, m, put); break;
            case 7: product_rows<7>(chunk, g.Ai, m, put); break;
            case 6: product_rows<6>(chunk, g.Ai, m, put); break;
            case 5: product_rows<5>(chunk, g.Ai, m, put); break;
            case 4: product_rows<4>(chunk, g.Ai, m, put); break;
            case 3: product_rows<3>(chunk, g.Ai, m, put); break;
            case 2: product_rows<2>(chunk, g.Ai, m, put); break;
            default: product_rows<1>(chunk, g.Ai, m, put); break;
        }
    }
    // 4. swaps
    int swaps = 0;
    double gm = -1.0;
    for (int it = 0; it <= g.max_iter; ++it) {
        // the block's largest |C| (ties: the smallest element), with its row
        {
            unsigned long long bv = best >= 0.0 ? (unsigned long long)__double_as_longlong(best) : 0;
            unsigned bp = best >= 0.0 ? (unsigned)at : kNone;
            warp_best(bv, bp);
            ++x.t;
            if ((tid & 31) == 0) {
                a.s_v[tid >> 5] = bv;
                a.s_p[tid >> 5] = bp;
            }
            __syncthreads();  // (and the rows are up to date)
            if (tid < 32) {
                bv = tid < nt >> 5 ? a.s_v[tid] : 0;
                bp = tid < nt >> 5 ? a.s_p[tid] : kNone;
                warp_best(bv, bp);
                if (tid == 0) x.publish(bv, bp);
                if (bp != kNone) {
                    const double* row = a.w + (size_t)((int)bp / m - a.first) * m;
                    for (int c = tid; c < m; c += 32) x.send(c, row[c]);
                }
            }
        }
        unsigned e;
        double v;
        const int q = x.winner(&v, &e);
        if (q == -2) return;
        gm = q < 0 ? -1.0 : v;
        if (gm <= 1.0 + g.tol) break;
        if (it == g.max_iter) {
            if (tid == 0 && blockIdx.x == 0) atomicOr(g.status, kErrTimeout);
            break;
        }
        const int j = (int)e % m;
        bool bad = false;
        const double ckj = x.receive(q, j, &bad);
        for (int c = tid; c < m; c += nt) a.prow[c] = x.receive(q, c, &bad) - (c == j ? 1.0 : 0.0);
        for (int r = tid; r < a.R; r += nt) a.col[r] = a.w[(size_t)r * m + j];
        if (tid == 0) sel[j] = (int)e / m;
        if (__syncthreads_or(bad)) {
            if (bad) atomicOr(g.status, kErrTimeout);
            return;
        }
        best = -1.0;
        at = 0;
        // (product, then quotient, then difference: with the factor divided beforehand ties fall differently)
        rank_one(a, 0, [](int) { return true; }, [&](double w, double l, double p) { return w - l * p / ckj; },
                 [&](double v, int r, int c) { track(v, (a.first + r) * m + c); });
        ++swaps;
    }
    __syncthreads();
    // A^-1 = D (A D)^-1, computed from scratch, and the unscaled A
    if (!shared && !x.barrier()) return;
    own(m, Rm);
    if (!invert_rows(x, a, orig, g.Ai, g.status, load, [&](int row) { return D[row]; })) return;
    for (int e = tid; e < a.R * m; e += nt)
        g.A[(size_t)a.first * m + e] = g.B[(size_t)sel[a.first + e / m] * m + e % m];
    if (blockIdx.x == 0) {
        for (int j = tid; j < m; j += nt) g.sel[j] = sel[j];
        if (tid == 0) {
            *g.swaps = swaps;
            *g.gmax = gm;
        }
    }
}

// gamma_r = max_j |sum_k B[r][k] Ai[k][j]|, accumulated as an atomic max of the bit pattern.
template <class T>
__global__ void __launch_bounds__(256) k_grade(int n, int m, const T* __restrict__ B, int ldb,
                                               const T* __restrict__ Ai, unsigned long long* gbits) {
    __shared__ T sb[16][64 + 1];
    __shared__ T sa[16][64 + 1];
    const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;  // 16 x 16 threads, 4 x 4 outputs each
    const int row0 = blockIdx.y * 64, col0 = blockIdx.x * 64;
    T acc[4][4];
#pragma unroll
    for (int a = 0; a < 4; ++a)
#pragma unroll
        for (int b = 0; b < 4; ++b) acc[a][b] = T(0);
    for (int k0 = 0; k0 < m; k0 += 16) {
        for (int e = threadIdx.x; e < 16 * 64; e += 256) {
            const int kk = e / 64, rr = e % 64;
            const int r = row0 + rr, k = k0 + kk;
            sb[kk][rr] = (r < n && k < m) ? B[(size_t)r * ldb + k] : T(0);
            const int c = col0 + rr;
            sa[kk][rr] = (c < m && k < m) ? Ai[(size_t)k * m + c] : T(0);
        }
        __syncthreads();
#pragma unroll
        for (int kk = 0; kk < 16; ++kk) {
            T bv[4], av[4];
#pragma unroll
            for (int a = 0; a < 4; ++a) bv[a] = sb[kk][ty * 4 + a];
#pragma unroll
            for (int b = 0; b < 4; ++b) av[b] = sa[kk][tx * 4 + b];
#pragma unroll
            for (int a = 0; a < 4; ++a)
#pragma unroll
                for (int b = 0; b < 4; ++b) acc[a][b] += bv[a] * av[b];
        }
        __syncthreads();
    }
#pragma unroll
    for (int a = 0; a < 4; ++a) {
        double mx = 0.0;
#pragma unroll
        for (int b = 0; b < 4; ++b)
            if (col0 + tx * 4 + b < m) {
                // a NaN entry counts as an infinite grade (fmax would drop it and report a row
                // of NaN as interpolating)
                const double v = fabs((double)acc[a][b]);
                mx = fmax(mx, v != v ? (double)INFINITY : v);
            }
        // combine the 16 threads that share this row (consecutive lanes)
        for (int o = 8; o > 0; o >>= 1) mx = fmax(mx, __shfl_xor_sync(0xffffffffu, mx, o, 16));
        const int r = row0 + ty * 4 + a;
        if (tx == 0 && r < n) atomicMax(&gbits[r], (unsigned long long)__double_as_longlong(mx));
    }
}

struct InvertArgs {
    int m, G;
    bool rows_in, col_in;
    const double* A;
    double* Ai;
    double* rows;             // [m][m] when the rows do not fit in shared memory
    double* col;              // (col_in is always set for m rows)
    unsigned long long* slots;  // [2][G][m + 2][2], zero at the start
    unsigned long long* rec;  // [2][G][2], zero at the start
    int* status;
};

__global__ void __launch_bounds__(kMvThreads) k_invert(const InvertArgs g) {
    extern __shared__ __align__(16) unsigned char smem[];
    const int m = g.m, R = mv_rows(m, g.G);
    Carve sh{smem};
    Exchange x{g.rec, g.slots, g.G, m, 0u, g.status, nullptr};
    Rows a{};
    int* orig;
    carve_common(sh, x, a, &orig);
    a.m = m;
    a.first = min(m, (int)blockIdx.x * R);
    a.R = min(m, a.first + R) - a.first;
    a.col = sh.take<double>(R);
    a.pos = sh.take<int>(2 * R);
    a.w = g.rows_in ? sh.take<double>((size_t)R * m) : g.rows + (size_t)a.first * m;
    __syncthreads();
    invert_rows(x, a, orig, g.Ai, g.status, [&](int j, int c) { return g.A[(size_t)j * m + c]; },
                [](int) { return 1.0; });
}

int mv_sm_count() {
    int dev = 0, n = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev);
    return n > 0 ? n : 1;
}

// Blocks of a cooperative kernel: as many as have room for their exchange rows and two rows of A or 16 rows of B
// each, one for two of three SMs at most if a block then has no more than 64 rows and shared memory holds them, else
// one for every SM.  More blocks take longer over the exchange and shorter over their rows: with 76, 101, 128 and 152 of them 920 x 460 takes 9.0,
// 8.7, 8.5 and 8.6 ms on one box, 101 8.8 against 9.3 with 152 on another, but 2000 x 1000 70, 63, 49 and 33 (in
// shared memory at last), 3000 x 2000 308, 270, 206 and 195, 20000 x 460 92, 73, 65 and 65; 232 x 116 1.48 with 57,
// 1.51 with 50.  Rows of B count for tall, narrow matrices (a block for 16, 64, 256 and 1024 of them): 1000 x 9 0.24,
// 0.28, 0.52, 0.51 ms, 3000 x 17 0.47, 0.49, 1.01, 1.27, 100000 x 9 1.27, 1.26, 1.27, 1.75 (1.69 with 101 blocks at
// most; by the rows of A alone, one block, 113).  Where the exchange rows lie in memory moves 920 x 460 by up to 15%.
size_t mv_exchange(int m) { return 4 * (size_t)m + 12; }  // doubles of a block: two records, two rows
int mv_blocks(int n, int m, size_t room, bool full) {
    const long sms = mv_sm_count(), by_room = (long)(room / mv_exchange(m));
    const auto most = [&](long limit) {
        return (int)std::max(1l, std::min({limit, std::max((long)m / 2, (long)n / 16), by_room}));
    };
    const int few = most(sms * 2 / 3);
    const Layout l = mv_layout(n, m, few, full);
    return l.rows_in && l.col_in && l.R <= 64 ? few : most(sms);
}
size_t mv_slot_bytes(int m, int G) { return 32 * (size_t)G * (m + 2); }

template <class K, class Args>
int mv_launch(K kernel, Args& g, int G, size_t smem, cudaStream_t st) {
    void* args[] = {&g};
    const bool ok =
        (G == 1 || (cudaMemsetAsync(g.rec, 0, 32 * (size_t)G, st) == cudaSuccess &&
                    cudaMemsetAsync(g.slots, 0, mv_slot_bytes(g.m, G), st) == cudaSuccess)) &&
        cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kMvSharedMost) == cudaSuccess &&
        cudaLaunchCooperativeKernel((void*)kernel, dim3(G), dim3(kMvThreads), args, smem, st) == cudaSuccess;
    if (!ok) cudaGetLastError();
    return ok ? 1 : -1;
}

}  // namespace

// The launchers return the number of kernels launched, or -1 if the launch itself failed (the
// error is taken off cudaGetLastError, so the caller reports it instead of reading stale results).
// W: 2 m^2 + 4 doubles, 16-byte aligned.
int launch_invert(int m, const double* A, double* Ai, double* W, int* status, cudaStream_t st) {
    // W = [records 4 G | slots 4 G (m + 2) | rows m^2 if they do not fit in shared memory]
    const size_t mm = (size_t)m * m;
    int G = mv_blocks(m, m, 2 * mm, false);
    Layout l = mv_layout(m, m, G, false);
    if (!l.rows_in) {
        G = mv_blocks(m, m, mm, false);
        l = mv_layout(m, m, G, false);
    }
    if (!l.col_in || l.bytes > kMvSharedMost) return -1;  // above m = 16,000
    auto* rec = reinterpret_cast<unsigned long long*>(W);
    InvertArgs g{m, G, l.rows_in, l.col_in, A, Ai, W + mm, nullptr, rec + 4 * (size_t)G, rec, status};
    return mv_launch(k_invert, g, G, l.bytes, st);
}

size_t maxvol_exchange_doubles(int n, int m) { return mv_exchange(m) * (size_t)mv_blocks(n, m, ~(size_t)0 / 2, true); }

// W: n m + n doubles; X: x_doubles doubles (any number: fewer give fewer blocks), 16-byte aligned; pos: n ints.
int launch_maxvol(int n, int m, const double* B, double* W, double* X, size_t x_doubles, int* pos, int* sel, double* A,
                  double* Ai, double tol, int max_iter, int* status, int* swaps, double* gmax, cudaStream_t st,
                  int start_given) {
    const int G = mv_blocks(n, m, x_doubles, true);
    const Layout l = mv_layout(n, m, G, true);
    if (l.bytes > kMvSharedMost) return -1;  // above m = 6382; a model's widest active set is 5580 columns
    auto* rec = reinterpret_cast<unsigned long long*>(X);
    MaxvolArgs g{n, m, G, l.br, l.rows_in, l.col_in, B, W, W + (size_t)n * m, pos, rec, rec + 4 * (size_t)G, sel, A, Ai, tol,
                 max_iter, start_given, status, swaps, gmax};
    return mv_launch(k_maxvol, g, G, l.bytes, st);
}

__global__ void k_gather_columns(int rows, int w_in, const double* in, int w_out, const int* cols, double* out) {
    const size_t total = (size_t)rows * w_out;
    for (size_t e = blockIdx.x * (size_t)blockDim.x + threadIdx.x; e < total; e += (size_t)gridDim.x * blockDim.x) {
        const size_t r = e / w_out, q = e - r * w_out;
        out[e] = in[r * w_in + cols[q]];
    }
}

int launch_gather_columns(int rows, int w_in, const double* in, int w_out, const int* cols, double* out,
                          cudaStream_t st) {
    const size_t total = (size_t)rows * w_out;
    if (total == 0) return 0;
    const int blocks = (int)std::min<size_t>((total + 255) / 256, 152 * 32);
    k_gather_columns<<<blocks, 256, 0, st>>>(rows, w_in, in, w_out, cols, out);
    return cudaGetLastError() == cudaSuccess ? 1 : -1;
}

template <class T>
int launch_grade(int n, int m, const T* B, int ldb, const T* Ai, unsigned long long* gbits, cudaStream_t st) {
    if (n <= 0) return 0;
    cudaMemsetAsync(gbits, 0, sizeof(unsigned long long) * (size_t)n, st);
    dim3 grid((m + 63) / 64, (n + 63) / 64);
    k_grade<T><<<grid, 256, 0, st>>>(n, m, B, ldb, Ai, gbits);
    return 1;
}
template int launch_grade<float>(int, int, const float*, int, const float*, unsigned long long*, cudaStream_t);
template int launch_grade<double>(int, int, const double*, int, const double*, unsigned long long*, cudaStream_t);

}  // namespace mtp

// ------------------------------------------------------------------------------------------------
// Active-set selection without any allocation (mtp_select_active_set_noalloc in include/mtp.h).
//
// Some callers cannot let a library allocate device memory: a simulation loop that checks the
// extrapolation grade inside its time step must not pay for cudaMalloc (which may synchronise the
// whole device and stall the other streams), and applications that hand all device memory to
// their own pool allocator have nothing left for a library to take.  This entry point therefore
// runs the same MaxVol kernel with all of its scratch in one fixed array compiled into the library.
// Every GPU that loads the library holds this array (kNoAllocScratchDoubles doubles, 4 MiB) until
// the process exits.  Calls share it and it keeps the last call's contents, so calls that overlap
// on the GPU (two streams, or two host threads) race; the status word is cleared at every call.
// ------------------------------------------------------------------------------------------------
namespace mtp {
namespace {

constexpr size_t kNoAllocScratchDoubles = (size_t)1 << 19;  // 4 MiB
constexpr int kNoAllocMaxDevices = 64;

static __device__ __align__(256) double g_noalloc_scratch[kNoAllocScratchDoubles];

std::mutex g_noalloc_mutex;
double* g_noalloc_ptr[kNoAllocMaxDevices] = {};

// Device address of the scratch array on the current device, looked up once per device.
cudaError_t noalloc_scratch(double** out) {
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= kNoAllocMaxDevices) return cudaErrorInvalidDevice;
    std::lock_guard<std::mutex> lock(g_noalloc_mutex);
    if (!g_noalloc_ptr[dev]) {
        void* p = nullptr;
        e = cudaGetSymbolAddress(&p, g_noalloc_scratch);
        if (e != cudaSuccess) return e;
        g_noalloc_ptr[dev] = static_cast<double*>(p);
    }
    *out = g_noalloc_ptr[dev];
    return cudaSuccess;
}

}  // namespace
}  // namespace mtp

extern "C" mtp_status mtp_select_active_set_noalloc(int n_rows, int m, const double* b_rows, int32_t* selected,
                                                    double* a_inv, int* n_swaps, void* stream) {
    using namespace mtp;
    if (m < 1 || n_rows < m || !b_rows || !selected) return MTP_EINVAL;
    // the documented limit; layout inside the fixed array (in doubles): W [max(n m, 2 m m) + 2 m + n]; A,
    // A^-1 [m m]; then ints: pos [n], sel [m], status, swaps; then the exchange (2 n m + m); then gmax.
    const size_t nm = (size_t)n_rows * m, mm = (size_t)m * m;
    const size_t w = (nm > 2 * mm ? nm : 2 * mm) + 2 * (size_t)m + n_rows;
    const size_t ints = (size_t)n_rows + m + 2;
    const size_t need = 2 * nm + w + m + 2 * mm + (ints + 1) / 2 + 1;
    if (need > kNoAllocScratchDoubles) return MTP_EINVAL;  // larger than the fixed scratch array
    double* base = nullptr;
    if (noalloc_scratch(&base) != cudaSuccess) return MTP_ECUDA;
    double* W = base;
    double* A = W + w;
    double* Ai = A + mm;
    int* pos = reinterpret_cast<int*>(Ai + mm);
    int* sel = pos + n_rows;
    int* status = sel + m;
    int* swaps = status + 1;
    const size_t x0 = (w + 2 * mm + (ints + 1) / 2 + 1) & ~(size_t)1;  // 16-byte aligned
    const size_t x_doubles = x0 < need - 1 ? need - 1 - x0 : 0;
    double* gmax = reinterpret_cast<double*>(base + (need - 1));
    cudaStream_t st = (cudaStream_t)stream;
    if (cudaMemsetAsync(status, 0, 2 * sizeof(int), st) != cudaSuccess) return MTP_ECUDA;
    if (launch_maxvol(n_rows, m, b_rows, W, base + x0, x_doubles, pos, sel, A, Ai, 1e-3, 100 * m, status, swaps, gmax, st, 0) < 0)
        return MTP_ECUDA;
    int h[2] = {0, 0};
    if (cudaMemcpyAsync(h, status, sizeof h, cudaMemcpyDeviceToHost, st) != cudaSuccess) return MTP_ECUDA;
    if (cudaStreamSynchronize(st) != cudaSuccess) return MTP_ECUDA;
    if (h[0] & kErrSingular) return MTP_ESINGULAR;
    if (h[0] & kErrTimeout) return MTP_ETIMEOUT;
    if (cudaMemcpyAsync(selected, sel, sizeof(int) * m, cudaMemcpyDeviceToDevice, st) != cudaSuccess) return MTP_ECUDA;
    if (a_inv && cudaMemcpyAsync(a_inv, Ai, sizeof(double) * mm, cudaMemcpyDeviceToDevice, st) != cudaSuccess)
        return MTP_ECUDA;
    if (n_swaps) *n_swaps = h[1];
    return cudaStreamSynchronize(st) == cudaSuccess ? MTP_OK : MTP_ECUDA;
}
