// mm64.cu -- FP64 contraction with T_l and T_l^T on the tensor cores
// (mm64.cuh: exact FP16 digits of 64-bit fixed-point operands), dense and, for
// plans with DSBT_PLAN_FAST64, through the interval bases of fast64.cu.
//
// Every step is rows times lines: a CTA of four warps takes a block of 16, 32 or
// 64 output rows of one group and a tile of its lines, and adds up segments
// (A rows, K range, B lines):
//   dense forward   rows r of T_l over columns <= r (completion rows: all)
//   dense inverse   rows c of T_l^T over the completion rows and r >= c
//   moments         rows k of Q_j^T (forward) or beta_j^T (inverse) over the
//                   columns of a used interval, or the rows of its sibling
//   fast forward    rows r of leaf J: the leaf's diagonal block, then beta_{r,j}
//                   against the moments of each interval J takes; completion
//                   rows of leaf 0 over all columns
//   fast inverse    rows c of leaf J: completion rows, the transposed diagonal
//                   block, then Q_j against the weights of each interval
//                   that holds the leaf
// (see fast64.cu for the scheme).  All operands are stored with K contiguous.
//
// A thread loads 32-byte pieces of two A rows straight into registers and
// forms their digits there (each A entry is used by one warp): from doubles, or
// for the interval scheme's operands from fixed-point words made at plan
// creation.  The lines are copied to shared memory and turned into digits there,
// once per CTA, 128 (wide) or 512 (narrow) columns at a time.
// Each line's scale is its largest exponent over the K range of the tile, found
// in a first pass over the (cached) lines, so no scale travels between kernels.
// The range depends on the row's block of 64 only and the sums are exact, so a
// channel's result does not depend on the other channels of a call, the rows per
// CTA or the form below.
//
// Two forms by the number of real lines of a group:
//   wide    16 lines a tile, one matrix instruction of 8 lines per digit pair:
//           held by the matrix instructions (72 clocks per 16 x 16 x 8 lines, 28 to
//           39 % of the tensor pipe's cycles) and the conversions beside them
//   narrow  2 lines a tile, the 8 digits of both lines as 16 columns, so one
//           digit of A meets all digits of the lines in two instructions (12
//           instead of 36): bound by turning A into digits and by reading it
// A 16 x 16 block of A costs a warp about 300 issue slots and 12 matrix
// instructions per two lines (narrow), 250 and 72 per sixteen (wide): groups of up to 4
// lines take the narrow form, and groups of up to 16 while the call leaves SMs idle
// (5 lines of 1280 points: 49 us wide).
//
// Measured on a GB300, forward + inverse contraction of one call (before: FP64
// multiply-adds on the same schemes):
//   interval scheme, N = 2048, l < 32 all m (2048 lines)   4.66 -> 0.71 ms
//   interval scheme, N = 2048, l < 40, 34 lines each       1.88 -> 0.55 ms
//   interval scheme, N = 2048, l < 64, 2 lines each        374 -> 233 us
//   dense, N = 1280, l <= 20 all m (882 lines)             7.25 -> 0.61 ms
#include <algorithm>

#include "mm64.cuh"
#include "plan.cuh"

namespace dsbt {

namespace {

using namespace mm64;

constexpr int THREADS = 128;
constexpr int FB = 64;          // leaf of the interval scheme
constexpr int KM = 64;          // stored basis width
constexpr int MAX_SEG = 12;

// Row tiles of a moment CTA over K = len columns: a warp has a latency of its own
// per 16 columns, so long intervals share K between the warps (8 to 16 units each)
// instead of giving each warp its own rows (64 units at 1024 columns made the
// longest CTAs half of the launch's time).  Wide tiles keep their rows together:
// there the digits of the lines cost more than a warp's latency.
__host__ __device__ inline int moment_mt(int most, int len, int narrow) {
    const int mt = !narrow ? 4 : (len >= 512 ? 1 : (len == 256 ? 2 : 4));
    return mt < most ? mt : most;
}

enum Kind { kDense = 0, kMoments = 1, kFastRows = 2 };

struct MmArgs {
    const double* T64;
    const double* Tt64;
    const double* Q;        // interval scheme (fast64.cu), else null
    const double* QT;
    const double* Qw;       // odd l: the first leaf of each level's Q, row 0 times sqrt(w_0) ...
    const double* QTw;      // ... and QT, column 0 times sqrt(w_0) (weights outside the inner loops: see fast64.cu)
    const double* beta;
    const double* betaT;
    const double* near;
    const double* nearT;
    double* M;              // moments / weights of this launch sequence
    const double* in;
    double* out;
    const double2* phase;
    const double* row_scale;   // real factor per output row, or null
    int N, nleaf, levels, R;
    int dir, in_cplx, out_cplx, per_l;
    int mt;                 // 16-row tiles per CTA at most: 1, 2 or 4
    int kind;
    int narrow;             // this launch's form ...
    int narrow_max;         // ... and the most lines of a group that the narrow one takes
    int npos;
    int gidx[kMaxGroups];        // groups of this launch, largest l first
    // CTAs: first (kFastRows forward) the completion tiles of all groups, comp0 the
    // prefix; then `reps` rounds over the groups' row blocks x line tiles, unit0 the
    // prefix: a round is one row block (or interval, longest first) of every group,
    // so the longest K ranges start first
    int comp0[kMaxGroups + 1];
    int unit0[3][kMaxGroups + 1];   // at 1, 2 and 4 row tiles per CTA
};

// A strided set of lines: line j, index k at base + (j >> 1) pair + (j & 1) odd + k step.
struct LineSet {
    const double* base;
    int pair, odd, step;
    __device__ __forceinline__ const double* at(int j, int k) const {
        return base + (size_t)(j >> 1) * pair + (size_t)(j & 1) * odd + (size_t)k * step;
    }
};

__device__ __forceinline__ void prefetch_l2(const void* p) { asm volatile("prefetch.global.L2 [%0];" ::"l"(p)); }

// A range of the tile's K axis: columns [k0, next segment's k0).
struct Seg {
    const double* A;   // row 0 of the block, first column
    LineSet B;         // first line of the tile, first column
    int lda, k0;
    int fixed;         // A holds biased fixed-point words, not doubles
};

struct Tile {
    Seg seg[MAX_SEG];
    int nseg, K;
    int mt, row0, nrow, phase_row;
    LineSet out;
};

// First entry of level j in the bases: levels below hold 64, 128, ... points of 64 functions.
__device__ __forceinline__ size_t level_offset(int j) { return (size_t)KM * FB * ((1 << j) - 1); }

// Moments of level j, interval i: levels below hold nleaf, nleaf / 2, ... intervals (a power of two).
__device__ __forceinline__ double* moments_at(const MmArgs& a, int j, int i, int line) {
    return a.M + ((size_t)(2 * (a.nleaf - (a.nleaf >> j)) + i) * a.R + line) * KM;
}

__device__ __forceinline__ LineSet line_set(const GroupTable& g, int gi, int line, int cplx, const double* base, int N) {
    if (cplx) return {base + ((size_t)(g.chan0[gi] + (line >> 1)) * N) * 2, 2 * N, 1, 2};
    return {base + (size_t)(g.line0[gi] + line) * N, 2 * N, N, 1};
}

// Fills the tile (called by warp 0; lane j < levels looks at level j).
__device__ void make_tile(const MmArgs& a, const GroupTable& g, int gi, int level, int round, int local, int line, int lane,
                          Tile& t) {
    const int l = g.l[gi], N = a.N, ne = n_extra(l), ne16 = (ne + 15) & ~15, l16 = (l + 15) & ~15;
    const LineSet in = line_set(g, gi, line, a.in_cplx, a.in, N);
    auto shifted = [](const LineSet& s, int k) { return LineSet{s.base + (size_t)k * s.step, s.pair, s.odd, s.step}; };
    const LineSet full = line_set(g, gi, line, a.out_cplx, a.out, N);
    int mt = a.mt, row0 = 0, nrow = 16 * mt, K = 0, n = 0;
    // segments that every lane knows are written by lane 0
    auto add = [&](const double* A, int lda, int len, int fixed, const LineSet& B) {
        if (len <= 0) return;
        if (lane == 0) t.seg[n] = Seg{A, B, lda, K, fixed};
        ++n;
        K += len;
    };
    // level segments: one per lane with `on`, in order of level
    auto add_levels = [&](bool on, const double* A, const LineSet& B) {
        const unsigned m = __ballot_sync(0xffffffffu, on && l16 > 0);
        const int q = __popc(m & ((1u << lane) - 1));
        if (on && l16 > 0) t.seg[n + q] = Seg{A, B, KM, K + q * l16, 1};
        n += __popc(m);
        K += __popc(m) * l16;
    };
    LineSet out = full;
    if (a.kind == kMoments) {
        // level and round: the interval; local: row block
        const int mtiles = l16 >> 4, j = level, i = 2 * round, len = FB << j;
        mt = min(moment_mt(a.mt, len, a.narrow), mtiles > 2 ? 4 : mtiles);
        const size_t qoff = level_offset(j);
        row0 = local * mt * 16;
        nrow = min(mt * 16, l16 - row0);
        if (a.dir > 0)
            add(((l & 1) && i == 0 ? a.QTw : a.QT) + qoff + (size_t)row0 * len, len, len, 1, shifted(in, i * len));
        else
            add(a.betaT + (((size_t)l * a.levels + j) * KM + row0) * N + (size_t)(i + 1) * len, N, len, 1,
                shifted(in, (i + 1) * len));
        out = LineSet{moments_at(a, j, i, g.line0[gi] + line) + row0, 2 * KM, KM, 1};
    } else if (round < 0) {   // completion rows, 16 at a time over all columns
        mt = 1;
        row0 = local * 16;
        nrow = 16;
        add(a.T64 + ((size_t)l * N + row0) * N, N, N, 0, in);
    } else {
        // dense forward rows are longest at the end, dense inverse rows at the start
        const int nrb = N / (16 * mt), rb = a.dir > 0 ? nrb - 1 - round : round;
        row0 = rb * 16 * mt;
        if (a.kind == kDense) {
            // K ranges by blocks of 64 rows, whatever the rows of this CTA (the zeros of
            // the triangle add nothing): a line's scale, the largest exponent over the
            // range, and with it every bit of the result, then do not depend on mt
            const double* A = (a.dir > 0 ? a.T64 : a.Tt64) + ((size_t)l * N + row0) * N;
            const int b0 = row0 & ~(FB - 1);
            if (b0 == 0) {   // the block of the completion rows
                add(A, N, a.dir > 0 && ne == 0 ? FB : N, 0, in);
            } else if (a.dir > 0) {
                add(A, N, b0 + FB, 0, in);
            } else {
                add(A, N, ne16, 0, in);
                add(A + b0, N, N - b0, 0, shifted(in, b0));
            }
        } else {
            const int J = row0 / FB, jb = J * FB, j = min(lane, a.levels - 1), i = J >> j;
            if (a.dir > 0) {
                const int skip = max(0, min(nrow, ne16 - row0));   // rows below ne16 are done by the completion tiles
                row0 += skip;
                nrow -= skip;
                add(a.near + (((size_t)l * a.nleaf + J) * FB + (row0 - jb)) * FB, FB, FB, 1, shifted(in, jb));
                add_levels(lane < a.levels && (i & 1), a.beta + (((size_t)l * a.levels + j) * N + row0) * KM,
                           LineSet{moments_at(a, j, i - 1, g.line0[gi] + line), 2 * KM, KM, 1});
            } else {
                if (J > 0) add(a.Tt64 + ((size_t)l * N + row0) * N, N, ne16, 0, in);
                add(a.nearT + (((size_t)l * a.nleaf + J) * FB + (row0 - jb)) * FB, FB, FB, 1, shifted(in, jb));
                add_levels(lane < a.levels && !(i & 1) && i + 1 < (a.nleaf >> j),
                           (l & 1) && J == 0 ? a.Qw + ((size_t)j * FB + row0) * KM
                                             : a.Q + level_offset(j) + (size_t)(row0 - i * (FB << j)) * KM,
                           LineSet{moments_at(a, j, i, g.line0[gi] + line), 2 * KM, KM, 1});
            }
        }
    }
    if (lane == 0) {
        if (a.kind != kMoments) out = LineSet{full.base + (size_t)row0 * full.step, full.pair, full.odd, full.step};
        t.nseg = n;
        t.K = K;
        t.mt = mt;
        t.row0 = row0;
        t.nrow = nrow;
        t.phase_row = row0;
        t.out = out;
    }
}

// Form of a kernel: NL lines a tile, KR columns a round, KSM groups of warps over K at most.
template <int NL_>
struct Form {
    static constexpr int NL = NL_;
    static constexpr bool NARROW = NL == 2;
    static constexpr int KR = NARROW ? 512 : 128;
    static constexpr int KSM = 4;
    static constexpr int BS = KR + 16;                     // halfs per digit row: 32 bytes past a multiple of 128, so
                                                           // the eight rows of a fragment fall on different banks
    static constexpr int DIG_BYTES = ND * NL * BS * 2;
    static constexpr int NO = NARROW ? 4 : NL / 2;         // results per thread
    static constexpr int RED_BYTES = 3 * NO * 32 * 16;     // K groups 1 .. 3 of a row tile
    static constexpr size_t SMEM = DIG_BYTES > RED_BYTES ? DIG_BYTES : RED_BYTES;
};

template <int NL_>
__global__ void __launch_bounds__(THREADS, NL_ == 2 ? 4 : 3) k_mm64(const __grid_constant__ MmArgs a,
                                                                   const __grid_constant__ GroupTable g) {
    using F = Form<NL_>;
    constexpr int NL = F::NL, KR = F::KR, BS = F::BS, NO = F::NO;
    constexpr bool NARROW = F::NARROW;
    constexpr int NT = NL / 8;                         // wide: n8 tiles
    __shared__ Tile t;
    __shared__ int ef[NL];
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __half* dig = reinterpret_cast<__half*>(smem_raw);   // [ND][NL][BS]
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, gr = lane >> 2, tq = lane & 3;

    int level = 0, round = -1, b = blockIdx.x;
    const int* pre = a.comp0;
    if (b >= a.comp0[a.npos]) {
        b -= a.comp0[a.npos];
        int mt = a.mt;
        if (a.kind == kMoments) {   // the level, longest intervals first
            for (level = a.levels - 1;; --level) {
                mt = moment_mt(a.mt, FB << level, a.narrow);
                const int n = (a.nleaf >> (level + 1)) * a.unit0[mt >> 1][a.npos];
                if (b < n || level == 0) break;
                b -= n;
            }
        }
        pre = a.unit0[mt >> 1];
        round = b / pre[a.npos];
        b -= round * pre[a.npos];
    }
    int lo = 0, hi = a.npos;
    while (hi - lo > 1) {
        const int mid = (lo + hi) >> 1;
        if (pre[mid] <= b) lo = mid;
        else hi = mid;
    }
    const int gi = a.gidx[lo];
    const int nl = g.line0[gi + 1] - g.line0[gi], lt = (nl + NL - 1) / NL;
    const int rel = b - pre[lo];
    const int line = (rel % lt) * NL, nline = min(NL, nl - line);
    if (warp == 0) make_tile(a, g, gi, level, round, rel / lt, line, lane, t);
    if (tid < NL) ef[tid] = 0;
    __syncthreads();
    const int mt = t.mt, nrow = t.nrow, K = t.K, nseg = t.nseg;
    if (nrow <= 0) return;
    const int ks_n = min(F::KSM, 4 / mt), m = warp % mt, ks = warp / mt;
    const bool active = m * 16 < nrow;

    float acc[NARROW ? 12 : NT * ND][4];
    long long shi[NO], slo[NO];
#pragma unroll
    for (int c = 0; c < NO; ++c) shi[c] = slo[c] = 0;
    // Sums stay exact in FP32 up to K = 1024 of one digit pair (narrow: a round is
    // 512) and K = 128 of the eight pairs of s = 7 (wide: a round): drained after
    // every round.
    auto drain = [&]() {
        if (NARROW) {
            // acc[i]: digit i of A, digit tq of the lines; acc[8 + i]: digit 4 + tq.
            // Without the products of i + j > 7 the sums in units of digit 0 of the
            // lines are multiples of 256^tq, so shifting them to the common unit is exact.
            const int sh = 8 * tq;
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                long long h = 0, w = 0, w1 = 0;
#pragma unroll
                for (int i = 0; i < 8; ++i) {
                    const long long v = __float2int_rn(i > 4 && i + tq > 7 ? 0.f : acc[i][c]);
                    if (i < 4) h += v * (1ll << (8 * (3 - i)));
                    else w += v * (1ll << (8 * (7 - i)));
                }
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const long long v = __float2int_rn(i > 0 && i + tq > 3 ? 0.f : acc[8 + i][c]);
                    w1 += v * (1ll << (8 * (3 - i)));
                }
                shi[c] += h >> sh;
                slo[c] += ((w + w1) >> sh) + ((h & ((1ll << sh) - 1)) << (32 - sh));
            }
        } else {
#pragma unroll
            for (int n = 0; n < NT; ++n) drain8(acc + n * ND, shi + n * 4, slo + n * 4);
        }
    };

    // A task is four consecutive columns of one line; a round has KR / 4 per line.
    constexpr int TASKS = NL * (KR / 4) / THREADS;   // per thread
    constexpr int LSTEP = THREADS / (KR / 4);        // lines between a thread's tasks
    const int tk = 4 * (tid % (KR / 4)), tline = tid / (KR / 4);
    auto seg_at = [&](int k) {
        int s = 0;
        while (s + 1 < nseg && t.seg[s + 1].k0 <= k) ++s;
        return s;
    };
    // the largest exponent of each line over all of K, unless one round holds it
    if (K > KR) {
        for (int r0 = 0; r0 < K; r0 += KR) {
            const int k = r0 + tk;
            if (k >= K) continue;
            const Seg& sg = t.seg[seg_at(k)];
            const double* p = sg.B.at(0, k - sg.k0);
            const int step = sg.B.step, pair = sg.B.pair, odd = sg.B.odd;
#pragma unroll
            for (int i = 0; i < TASKS; ++i) {
                const int j = tline + i * LSTEP;
                int e = 0;
                if (j < nline) {
                    const double* q = p + (size_t)(j >> 1) * pair + (size_t)(j & 1) * odd;
                    e = max(max(exponent_of(q[0]), exponent_of(q[step])),
                            max(exponent_of(q[2 * step]), exponent_of(q[3 * step])));
                }
                if (e > ef[j]) atomicMax(&ef[j], e);
            }
        }
        __syncthreads();
    }

    // The A entries of a narrow tile come from HBM (each is used by one or two
    // lines): ask for the first columns of every segment now, and for the rest in
    // load, eight units ahead.
    constexpr int AHEAD = 8 * 16;
    if (NARROW) {
        const int r = tid % (16 * mt);
        for (int q = 0; q < nseg; ++q) {
            const Seg& sg = t.seg[q];
            const int len = min(AHEAD, (q + 1 < nseg ? t.seg[q + 1].k0 : K) - sg.k0);
            for (int k = 16 * (tid / (16 * mt)); k < len; k += 16 * (THREADS / (16 * mt)))
                if (r < nrow) prefetch_l2(sg.A + (size_t)r * sg.lda + k);
        }
    }
    const double* ap = nullptr;
    int lda = 0, fixed = 0, aseg = 0, aend = 0;
    // Row g: columns 4t .. 4t + 3; row g + 8.  (Two units ahead, at three CTAs an SM
    // instead of four, was 10 % slower for the narrow form.)
    ulonglong2 raw[4];
    // loads this thread's A entries of the unit at column k (units of a warp come in increasing k)
    auto load = [&](int k) {
        if (k >= aend) {
            while (aseg + 1 < nseg && t.seg[aseg + 1].k0 <= k) ++aseg;
            const Seg& sg = t.seg[aseg];
            aend = aseg + 1 < nseg ? t.seg[aseg + 1].k0 : K;
            lda = sg.lda;
            fixed = sg.fixed;
            ap = sg.A + (size_t)(m * 16 + gr) * lda + 4 * tq - sg.k0;
        }
        const ulonglong2* r0 = reinterpret_cast<const ulonglong2*>(ap + k);
        const ulonglong2* r1 = reinterpret_cast<const ulonglong2*>(ap + k + (size_t)8 * lda);
        raw[0] = __ldg(r0);
        raw[1] = __ldg(r0 + 1);
        raw[2] = __ldg(r1);
        raw[3] = __ldg(r1 + 1);
        if (NARROW && k + AHEAD < aend) {
            prefetch_l2(ap + k + AHEAD);
            prefetch_l2(ap + k + AHEAD + (size_t)8 * lda);
        }
    };
    if (active && ks * 16 < K) load(ks * 16);
    for (int r0 = 0; r0 < K; r0 += KR) {
        const int kr = min(KR, K - r0);
        const bool on = tk < kr;
        auto put_digits = [&](int j, int e, const double* v) { put_digits4(dig + (size_t)j * BS + tk, NL * BS, v, e); };
        const double* p = nullptr;
        int step = 0, pair = 0, odd = 0;
        if (!NARROW && on) {
            const Seg& sg = t.seg[seg_at(r0 + tk)];
            p = sg.B.at(0, r0 + tk - sg.k0);
            step = sg.B.step, pair = sg.B.pair, odd = sg.B.odd;
        }
        auto fetch = [&](int j, double* v) {
            const double* q = p + (size_t)(j >> 1) * pair + (size_t)(j & 1) * odd;
#pragma unroll
            for (int c = 0; c < 4; ++c) v[c] = on && j < nline ? q[c * step] : 0.0;
        };
        if (NARROW) {   // the round's kr / 4 tasks of each line, spread over all threads
            double v[TASKS][4];
            const int per = kr / 4;
            int tj[TASKS], tkk[TASKS];
#pragma unroll
            for (int i = 0; i < TASKS; ++i) {
                const int idx = tid + i * THREADS;
                tj[i] = idx >= per;
                tkk[i] = idx < 2 * per ? 4 * (idx - (idx >= per ? per : 0)) : -1;
#pragma unroll
                for (int c = 0; c < 4; ++c) v[i][c] = 0.0;
                if (tkk[i] >= 0 && tj[i] < nline) {
                    const Seg& sg = t.seg[seg_at(r0 + tkk[i])];
                    const double* q = sg.B.at(tj[i], r0 + tkk[i] - sg.k0);
                    const int step = sg.B.step;
#pragma unroll
                    for (int c = 0; c < 4; ++c) v[i][c] = q[c * step];
                }
            }
            if (K <= KR) {   // the scales from these values
                int e[2] = {0, 0};
#pragma unroll
                for (int i = 0; i < TASKS; ++i) {
                    const int x = exponent4(v[i]);
                    e[0] = max(e[0], tj[i] ? 0 : x);
                    e[1] = max(e[1], tj[i] ? x : 0);
                }
#pragma unroll
                for (int q = 0; q < 2; ++q) {
                    e[q] = __reduce_max_sync(0xffffffffu, e[q]);
                    if (lane == 0) atomicMax(&ef[q], e[q]);
                }
                __syncthreads();
            }
#pragma unroll
            for (int i = 0; i < TASKS; ++i)
                if (tkk[i] >= 0) put_digits4(dig + (size_t)tj[i] * BS + tkk[i], NL * BS, v[i], ef[tj[i]]);
        } else {
#pragma unroll
            for (int i = 0; i < TASKS; i += 2) {
                double v[2][4];
                fetch(tline + i * LSTEP, v[0]);
                fetch(tline + (i + 1) * LSTEP, v[1]);
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const int j = tline + (i + h) * LSTEP;
                    int e;
                    if (K <= KR) {   // a warp holds the whole line
                        e = __reduce_max_sync(0xffffffffu, exponent4(v[h]));
                        if (lane == 0) ef[j] = e;
                    } else {
                        e = ef[j];
                    }
                    if (on) put_digits(j, e, v[h]);
                }
            }
        }
        __syncthreads();
        if (active) {
#pragma unroll
            for (int i = 0; i < (NARROW ? 12 : NT * ND); ++i)
#pragma unroll
                for (int c = 0; c < 4; ++c) acc[i][c] = 0.f;
            const __half* sub = dig + 4 * tq + (size_t)gr * BS;
            for (int k = ks * 16; k < kr; k += ks_n * 16) {
                uint32_t wl[8], wh[8];
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    const unsigned long long x = raw[q].x, y = raw[q].y;
                    wl[2 * q] = (uint32_t)x; wh[2 * q] = (uint32_t)(x >> 32);
                    wl[2 * q + 1] = (uint32_t)y; wh[2 * q + 1] = (uint32_t)(y >> 32);
                }
                if (!fixed) {
#pragma unroll
                    for (int q = 0; q < 8; ++q) fixed_a(__hiloint2double((int)wh[q], (int)wl[q]), wl[q], wh[q]);
                }
                // the next unit of this warp (KR is a multiple of 16 ks_n, so rounds join up)
                const int kn = r0 + k + ks_n * 16;
                if (kn < K) load(kn);
                Digits4 d0, d1;
                d0.set(wl, wh);
                d1.set(wl + 4, wh + 4);
                const __half* bp = sub + k;
                if (NARROW) {
                    const uint2 b0 = *reinterpret_cast<const uint2*>(bp), b1 = *reinterpret_cast<const uint2*>(bp + 8 * BS);
#pragma unroll
                    for (int i = 0; i < ND; ++i) {
                        mma16816(acc[i], d0.d[i][0], d1.d[i][0], d0.d[i][1], d1.d[i][1], b0.x, b0.y);
                        if (i < 4) mma16816(acc[8 + (i & 3)], d0.d[i][0], d1.d[i][0], d0.d[i][1], d1.d[i][1], b1.x, b1.y);
                    }
                } else {
#pragma unroll
                    for (int j = 0; j < ND; ++j) {
#pragma unroll
                        for (int n = 0; n < NT; ++n) {
                            const uint2 bb = *reinterpret_cast<const uint2*>(bp + (size_t)(j * NL + n * 8) * BS);
#pragma unroll
                            for (int i = 0; i + j < ND; ++i)
                                mma16816(acc[n * ND + i + j], d0.d[i][0], d1.d[i][0], d0.d[i][1], d1.d[i][1], bb.x, bb.y);
                        }
                    }
                }
            }
            drain();
        }
        __syncthreads();   // the digits are used up
    }

    // ---- add the K groups of warps, through the digit buffer
    if (NARROW) {
        // first the digits of the lines, held by the four lanes of a row: lane tq ends
        // with result tq (row g + 8 (tq / 2), line tq & 1) in place 0
        const bool up = tq & 2, odd = tq & 1;
#pragma unroll
        for (int c = 0; c < 2; ++c) {
            const long long h = __shfl_xor_sync(0xffffffffu, up ? shi[c] : shi[c + 2], 2);
            const long long w = __shfl_xor_sync(0xffffffffu, up ? slo[c] : slo[c + 2], 2);
            shi[c] = (up ? shi[c + 2] : shi[c]) + h;
            slo[c] = (up ? slo[c + 2] : slo[c]) + w;
        }
        const long long h = __shfl_xor_sync(0xffffffffu, odd ? shi[0] : shi[1], 1);
        const long long w = __shfl_xor_sync(0xffffffffu, odd ? slo[0] : slo[1], 1);
        shi[0] = (odd ? shi[1] : shi[0]) + h;
        slo[0] = (odd ? slo[1] : slo[0]) + w;
    }
    constexpr int NR = NARROW ? 1 : NO;   // results left per thread
    if (ks_n > 1) {
        longlong2* red = reinterpret_cast<longlong2*>(smem_raw);   // [warp - mt][result][lane]
        if (active && ks > 0)
#pragma unroll
            for (int c = 0; c < NR; ++c) red[((warp - mt) * NR + c) * 32 + lane] = make_longlong2(shi[c], slo[c]);
        __syncthreads();
        if (active && ks == 0)
            for (int q = 1; q < ks_n; ++q)
#pragma unroll
                for (int c = 0; c < NR; ++c) {
                    const longlong2 v = red[(((q - 1) * mt + m) * NR + c) * 32 + lane];
                    shi[c] += v.x;
                    slo[c] += v.y;
                }
    }
    if (!active || ks > 0) return;

    // ---- store: wide threads hold lines (2t, 2t + 1) of rows g and g + 8
    const LineSet out = t.out;
    const int l = g.l[gi];
    const double2* ph = a.kind == kMoments ? nullptr : a.phase;
    const double* rs = a.kind == kMoments ? nullptr : a.row_scale;
    auto phase_of = [&](int r) {
        const int row = t.phase_row + r;
        return a.per_l ? ph[(size_t)l * a.N + row] : ph[(size_t)(l & 1) * a.N + phase_entry(l, row, a.N)];
    };
    auto put = [&](int j, int r, double re, double im) {
        if (j >= nline) return;
        if (ph) {   // lines (j, j + 1) are the parts of one channel
            const double2 w = phase_of(r);
            const double s = re * w.x - im * w.y;
            im = re * w.y + im * w.x;
            re = s;
        }
        if (rs) {
            const double f = rs[t.phase_row + r];
            re *= f;
            im *= f;
        }
        double* o = const_cast<double*>(out.at(j, r));
        *o = re;
        if (j + 1 < nline) *const_cast<double*>(out.at(j + 1, r)) = im;
    };
    if (NARROW) {
        const int j = tq & 1, r = m * 16 + gr + 4 * (tq & 2);
        double v = to_double_once(shi[0], slo[0], ef[j]);
        if (ph) {   // the lane's neighbour holds the channel's other part
            const double o = __shfl_xor_sync(0xffffffffu, v, 1);
            const double2 w = phase_of(r);
            v = j ? o * w.y + v * w.x : v * w.x - o * w.y;
        }
        if (rs) v *= rs[t.phase_row + r];
        if (j < nline) *const_cast<double*>(out.at(j, r)) = v;
    } else {
#pragma unroll
        for (int n = 0; n < NT; ++n) {
            const int j = n * 8 + 2 * tq;
            if (j >= nline) continue;
            const int e0 = ef[j], e1 = ef[j + 1];
            put(j, m * 16 + gr, to_double_once(shi[n * 4], slo[n * 4], e0), to_double_once(shi[n * 4 + 1], slo[n * 4 + 1], e1));
            put(j, m * 16 + gr + 8, to_double_once(shi[n * 4 + 2], slo[n * 4 + 2], e0),
                to_double_once(shi[n * 4 + 3], slo[n * 4 + 3], e1));
        }
    }
}

template <int NL>
int launch(MmArgs a, const GroupTable& g, cudaStream_t st) {
    a.narrow = NL == 2;
    // groups of this form, largest l first; returns the CTAs at a.mt row tiles each
    auto fill = [&]() {
        a.npos = 0;
        a.comp0[0] = a.unit0[0][0] = a.unit0[1][0] = a.unit0[2][0] = 0;
        for (int gi = g.ngroups - 1; gi >= 0; --gi) {
            const int nl = g.line0[gi + 1] - g.line0[gi], l = g.l[gi], lt = (nl + NL - 1) / NL, n = a.npos;
            if ((nl <= a.narrow_max) != (NL == 2)) continue;
            const int mtiles = (l + 15) / 16;
            if (a.kind == kMoments && mtiles == 0) continue;
            a.gidx[n] = gi;
            a.comp0[n + 1] = a.comp0[n] + (a.kind == kFastRows && a.dir > 0 ? lt * ((n_extra(l) + 15) / 16) : 0);
            for (int q = 0; q < 3; ++q) {   // row blocks of a round at 1, 2, 4 row tiles
                const int mt = std::min(1 << q, mtiles > 2 ? 4 : std::max(1, mtiles));
                a.unit0[q][n + 1] = a.unit0[q][n] + lt * (a.kind == kMoments ? (mtiles + mt - 1) / mt : 1);
            }
            ++a.npos;
        }
        int n = a.comp0[a.npos];
        if (a.kind == kMoments)
            for (int j = 0; j < a.levels; ++j)
                n += (a.nleaf >> (j + 1)) * a.unit0[moment_mt(a.mt, FB << j, a.narrow) >> 1][a.npos];
        else
            n += a.N / (16 * a.mt) * a.unit0[a.mt >> 1][a.npos];
        return n;
    };
    // rows per CTA: 64, or 32 or 16 (the warps then share the K range) until
    // every SM has two CTAs
    for (a.mt = 4; a.mt > 1 && fill() < 2 * kSMs; a.mt >>= 1) {}
    const int tiles = fill();
    if (tiles == 0) return DSBT_OK;
    constexpr size_t smem = Form<NL>::SMEM;
    k_mm64<NL><<<tiles, THREADS, smem, st>>>(a, g);
    DSBT_CUDA_TRY(cudaGetLastError());
    return DSBT_OK;
}

int launch_both(MmArgs a, const GroupTable& g, cudaStream_t st) {
    int wide = 0;   // CTAs of the wide form at 64 rows each
    for (int i = 0; i < g.ngroups; ++i) wide += (g.line0[i + 1] - g.line0[i] + 15) / 16 * (a.N / 64);
    a.narrow_max = wide <= kSMs / 2 ? 16 : 4;
    int rc = launch<16>(a, g, st);
    if (rc == DSBT_OK) rc = launch<2>(a, g, st);
    return rc;
}

}  // namespace

// The digits replace FP64 multiply-adds in every call: measured faster from one
// line of 256 points (N = 256, l <= 9) to 2048 lines of 2048; for the errors of both see
// mm64.cuh.
int contract_f64(const dsbt_plan* p, const GroupTable& g, int dir, const double* in, int in_cplx, double* out,
                 int out_cplx, const double2* phase, cudaStream_t st, double* fast_scratch, const double* row_scale) {
    if (!p->T64) {
        set_error("FP64 path needs a plan built with DSBT_PLAN_FP64");
        return DSBT_ERR_UNSUPPORTED;
    }
    if (dir < 0 && phase) {
        set_error("contract_f64: phase only on the forward contraction");
        return DSBT_ERR_INVALID;
    }
    if (g.ngroups == 0) return DSBT_OK;
    MmArgs a{};
    a.T64 = p->T64;
    a.Tt64 = p->Tt64;
    a.in = in;
    a.out = out;
    a.phase = phase;
    a.row_scale = row_scale;
    a.N = p->N;
    a.R = g.total_lines;
    a.dir = dir;
    a.in_cplx = in_cplx;
    a.out_cplx = out_cplx;
    a.per_l = p->knl != nullptr;   // phase table rows per l (corrected momenta) or by parity
    ProfScope ps(kKContract64, st);
    if (p->fast && fast_scratch) {
        fast_operands(p, &a.Q, &a.QT, &a.Qw, &a.QTw, &a.beta, &a.betaT, &a.near, &a.nearT, &a.nleaf, &a.levels);
        a.M = fast_scratch;
        a.kind = kMoments;
        if (int rc = launch_both(a, g, st)) return rc;
        a.kind = kFastRows;
        return launch_both(a, g, st);
    }
    a.kind = kDense;
    return launch_both(a, g, st);
}

}  // namespace dsbt
