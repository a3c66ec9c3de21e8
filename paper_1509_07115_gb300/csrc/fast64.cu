// fast64.cu -- FP64 multiplication by T_l and T_l^T in O(N l log N) work,
// for plans built with DSBT_PLAN_FAST64 (the stable counterpart of the fast
// scheme of Sec. 2.6).
//
// On a regular row n of T_l the entries left of the diagonal are
// T_nm = alpha_n P'_l(n - m, 2n) sqrt(w_m): a polynomial of degree l - 1 in m
// times sqrt(w_m) (w_0 = 1/2 for odd l).  Columns are cut into leaves of B = 64
// points and a binary tree of intervals above them.  Row r (leaf J = r / B)
// takes its own leaf's columns up to the diagonal directly (near field) and
// every other column through the intervals of the dyadic decomposition of
// leaves 0..J-1 (one interval per set bit j of J, index (J >> j) - 1): on such
// an interval I of length L_j = B 2^j the row is exactly
//     T_{r,I} = sqrt(w_I) (Q_j beta_{r,j}),
// with Q_j an orthonormal basis [L_j][K] of the polynomials of degree < K on
// the interval's points (K = the plan's l_max; the first l columns suffice for
// T_l), beta_{r,j} = Q_j^T (T_{r,I} / sqrt(w_I)) computed from the FP64 T_l at
// plan creation.  Forward: moments M_I = Q_j^T (sqrt(w) f)_I of every used
// interval (one with a right sibling), projected directly from f, then
// b_r = near + sum_j beta_{r,j} . M.  Inverse: W_I = sum_{r using I}
// beta_{r,j} b_r, then f_c = sqrt(w_c) sum_j (Q_j W_{I_j(c)})_c + near, over
// the used intervals I_j(c) holding c.  Direct projection costs about as many
// multiply-adds as the leaf-to-root merge through K x K transfer matrices
// would for K near 64, and has no chain of dependent levels.  The completion
// rows (n < n0_l) are dense and applied directly.  The bases are built on the
// host by Arnoldi on the point grid with two Gram-Schmidt passes, so every
// coefficient is a bounded projection (no monomial cancellation).
//
// This file builds the operands (double); mm64.cu multiplies with them.
#include <math.h>

#include <algorithm>
#include <thread>
#include <utility>
#include <vector>

#include "mm64.cuh"
#include "plan.cuh"

namespace dsbt {

namespace {

constexpr int FB = 64;    // leaf size
constexpr int KM = 64;    // basis width stored (>= l_max)

__host__ __device__ inline double sqrt_w(int l, int c) { return ((l & 1) && c == 0) ? 0.70710678118654752440 : 1.0; }

// Orthonormal polynomial basis Q[t][k], t < len, k < KM, on x_t = (2t+1)/len - 1.
void basis(int len, std::vector<double>& Q) {
    const int K = std::min(KM, len);
    Q.assign((size_t)len * KM, 0.0);
    std::vector<double> v(len), x(len);
    for (int t = 0; t < len; ++t) x[t] = (2.0 * t + 1.0) / len - 1.0;
    for (int t = 0; t < len; ++t) Q[(size_t)t * KM] = 1.0 / sqrt((double)len);
    for (int k = 1; k < K; ++k) {
        for (int t = 0; t < len; ++t) v[t] = x[t] * Q[(size_t)t * KM + k - 1];
        for (int pass = 0; pass < 2; ++pass)
            for (int q = 0; q < k; ++q) {
                double d = 0.0;
                for (int t = 0; t < len; ++t) d += v[t] * Q[(size_t)t * KM + q];
                for (int t = 0; t < len; ++t) v[t] -= d * Q[(size_t)t * KM + q];
            }
        double nrm = 0.0;
        for (int t = 0; t < len; ++t) nrm += v[t] * v[t];
        nrm = 1.0 / sqrt(nrm);
        for (int t = 0; t < len; ++t) Q[(size_t)t * KM + k] = v[t] * nrm;
    }
}

// beta[l][j][r][k]: projection of row r of T_l on level j's interval of its
// decomposition (zero where unused).  Block: KM threads (k); grid (r, j, l).
__global__ void k_fast_beta(const double* __restrict__ T64, const double* __restrict__ Q,
                            const size_t* __restrict__ qoff, double* __restrict__ beta, int N, int levels) {
    const int r = blockIdx.x, j = blockIdx.y, l = blockIdx.z, k = threadIdx.x;
    const int J = r / FB;
    double s = 0.0;
    if (r >= n_extra(l) && ((J >> j) & 1) && k < l) {
        const int len = FB << j;
        const int lo = ((J >> j) - 1) * len;
        const double* row = T64 + ((size_t)l * N + r) * N + lo;
        const double* Qj = Q + qoff[j];
        for (int t = 0; t < len; ++t) s = fma(row[t] / sqrt_w(l, lo + t), Qj[(size_t)t * KM + k], s);
    }
    beta[(((size_t)l * levels + j) * N + r) * KM + k] = s;
}

// Build-time layouts: betaT[l][j][k][r] = beta[l][j][r][k] and the transposed
// diagonal leaf blocks nearT[l][J][c][t] = T_l[J B + t][J B + c].
__global__ void k_fast_transpose_beta(const double* __restrict__ beta, double* __restrict__ betaT, int N) {
    const size_t lj = blockIdx.y;
    const int r = blockIdx.x, k = threadIdx.x;
    betaT[(lj * KM + k) * N + r] = beta[(lj * N + r) * KM + k];
}

// near[l][J][t][c] the blocks themselves.
__global__ void k_fast_near(const double* __restrict__ T64, double* __restrict__ near, double* __restrict__ nearT, int N,
                            int nleaf) {
    const int J = blockIdx.x, l = blockIdx.y, c = threadIdx.x;
    const size_t blk = ((size_t)l * nleaf + J) * FB * FB;
    for (int t = 0; t < FB; ++t) {
        const double v = T64[((size_t)l * N + J * FB + t) * N + J * FB + c];
        nearT[blk + (size_t)c * FB + t] = v;
        near[blk + (size_t)t * FB + c] = v;
    }
}

// Doubles (|v| < 2) to the biased fixed-point words that the contraction takes
// apart into digits (mm64.cuh), in place.
__global__ void k_fast_fixed(double* p, size_t n) {
    const size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    uint32_t lo, hi;
    mm64::fixed_a(p[i], lo, hi);
    reinterpret_cast<uint2*>(p)[i] = make_uint2(lo, hi);
}

}  // namespace

struct FastData {
    int nleaf = 0, levels = 0;
    double* Q = nullptr;
    double* QT = nullptr;
    double* Qw = nullptr;    // [level][FB][KM]: the first leaf of Q_j with row 0 times sqrt(w_0) = 1/sqrt(2) (odd l)
    double* QTw = nullptr;   // QT with column 0 of every level times sqrt(w_0) (odd l, intervals holding column 0)
    size_t* qoff = nullptr;
    double* beta = nullptr;
    double* betaT = nullptr;
    double* near = nullptr;
    double* nearT = nullptr;
    // every operand above holds biased fixed-point words once the plan is built
};

void poly_basis(int len, std::vector<double>& Q) { basis(len, Q); }

bool fast_supported(int N) {
    const int nleaf = N / FB;
    return N % FB == 0 && nleaf >= 2 && (nleaf & (nleaf - 1)) == 0;
}

int fast_build(dsbt_plan* p, cudaStream_t st) {
    const int N = p->N;
    DSBT_CHECK_ARG(fast_supported(N), "DSBT_PLAN_FAST64 needs N / 64 a power of two (N = %d)", N);
    DSBT_CHECK_ARG(p->l_max <= KM, "DSBT_PLAN_FAST64: l_max %d above %d", p->l_max, KM);
    FastData* f = new (std::nothrow) FastData();
    if (!f) return DSBT_ERR_NOMEM;
    p->fast = f;
    f->nleaf = N / FB;
    f->levels = 0;
    while ((1 << f->levels) < f->nleaf) ++f->levels;   // levels j = 0 .. levels-1, intervals up to N / 2
    const int levels = f->levels;
    // orthonormal bases of the levels (host, one thread per level), both layouts
    std::vector<std::vector<double>> Qh(levels);
    std::vector<std::thread> pool;
    for (int j = 0; j < levels; ++j) pool.emplace_back([&, j]() { basis(FB << j, Qh[j]); });
    for (auto& t : pool) t.join();
    std::vector<size_t> qoff(levels);
    size_t qtot = 0;
    for (int j = 0; j < levels; ++j) {
        qoff[j] = qtot;
        qtot += Qh[j].size();
    }
    std::vector<double> Qall(qtot), QTall(qtot), Qwall((size_t)levels * FB * KM), QTwall;
    for (int j = 0; j < levels; ++j) {
        const int len = FB << j;
        for (int t = 0; t < len; ++t)
            for (int k = 0; k < KM; ++k) {
                Qall[qoff[j] + (size_t)t * KM + k] = Qh[j][(size_t)t * KM + k];
                QTall[qoff[j] + (size_t)k * len + t] = Qh[j][(size_t)t * KM + k];
            }
    }
    QTwall = QTall;
    const double w0 = sqrt_w(1, 0);
    for (int j = 0; j < levels; ++j)
        for (int k = 0; k < KM; ++k) {
            QTwall[qoff[j] + (size_t)k * (FB << j)] *= w0;
            for (int t = 0; t < FB; ++t)
                Qwall[((size_t)j * FB + t) * KM + k] = Qall[qoff[j] + (size_t)t * KM + k] * (t == 0 ? w0 : 1.0);
        }
    const size_t L = (size_t)p->l_max + 1;
    const size_t nbeta = L * levels * N * KM;
    bool ok = cudaMalloc((void**)&f->Q, qtot * sizeof(double)) == cudaSuccess &&
              cudaMalloc((void**)&f->QT, qtot * sizeof(double)) == cudaSuccess &&
              cudaMalloc((void**)&f->Qw, Qwall.size() * sizeof(double)) == cudaSuccess &&
              cudaMalloc((void**)&f->QTw, qtot * sizeof(double)) == cudaSuccess &&
              cudaMalloc((void**)&f->qoff, levels * sizeof(size_t)) == cudaSuccess &&
              cudaMalloc((void**)&f->beta, nbeta * sizeof(double)) == cudaSuccess &&
              cudaMalloc((void**)&f->betaT, nbeta * sizeof(double)) == cudaSuccess &&
              cudaMalloc((void**)&f->near, L * N * FB * sizeof(double)) == cudaSuccess &&
              cudaMalloc((void**)&f->nearT, L * N * FB * sizeof(double)) == cudaSuccess;
    ok = ok && cudaMemcpy(f->Q, Qall.data(), qtot * sizeof(double), cudaMemcpyHostToDevice) == cudaSuccess &&
         cudaMemcpy(f->QT, QTall.data(), qtot * sizeof(double), cudaMemcpyHostToDevice) == cudaSuccess &&
         cudaMemcpy(f->Qw, Qwall.data(), Qwall.size() * sizeof(double), cudaMemcpyHostToDevice) == cudaSuccess &&
         cudaMemcpy(f->QTw, QTwall.data(), qtot * sizeof(double), cudaMemcpyHostToDevice) == cudaSuccess &&
         cudaMemcpy(f->qoff, qoff.data(), levels * sizeof(size_t), cudaMemcpyHostToDevice) == cudaSuccess;
    if (!ok) {
        cudaGetLastError();
        set_error("DSBT_PLAN_FAST64: device allocation or copy failed");
        return DSBT_ERR_NOMEM;
    }
    k_fast_beta<<<dim3(N, levels, (unsigned)L), KM, 0, st>>>(p->T64, f->Q, f->qoff, f->beta, N, levels);
    k_fast_transpose_beta<<<dim3(N, (unsigned)(L * levels)), KM, 0, st>>>(f->beta, f->betaT, N);
    k_fast_near<<<dim3(f->nleaf, (unsigned)L), FB, 0, st>>>(p->T64, f->near, f->nearT, N, f->nleaf);
    for (const auto& [ptr, n] : {std::make_pair(f->Q, qtot), std::make_pair(f->QT, qtot), std::make_pair(f->QTw, qtot),
                                 std::make_pair(f->Qw, Qwall.size()), std::make_pair(f->beta, nbeta),
                                 std::make_pair(f->betaT, nbeta), std::make_pair(f->near, L * N * FB),
                                 std::make_pair(f->nearT, L * N * FB)})
        k_fast_fixed<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(ptr, n);
    DSBT_CUDA_TRY(cudaGetLastError());
    return DSBT_OK;
}

void fast_free(dsbt_plan* p) {
    if (!p || !p->fast) return;
    cudaFree(p->fast->Q);
    cudaFree(p->fast->QT);
    cudaFree(p->fast->Qw);
    cudaFree(p->fast->QTw);
    cudaFree(p->fast->qoff);
    cudaFree(p->fast->beta);
    cudaFree(p->fast->betaT);
    cudaFree(p->fast->near);
    cudaFree(p->fast->nearT);
    delete p->fast;
    p->fast = nullptr;
}

size_t fast_scratch_bytes(const dsbt_plan* p, int lines) {
    if (!p->fast) return 0;
    size_t n = 0;
    for (int j = 0; j < p->fast->levels; ++j) n += (size_t)(p->fast->nleaf >> j) * lines * KM;
    return n * sizeof(double);
}

void fast_operands(const dsbt_plan* p, const double** Q, const double** QT, const double** Qw, const double** QTw,
                   const double** beta,
                   const double** betaT, const double** near, const double** nearT, int* nleaf, int* levels) {
    const FastData* f = p->fast;
    *Q = f->Q;
    *QT = f->QT;
    *Qw = f->Qw;
    *QTw = f->QTw;
    *beta = f->beta;
    *betaT = f->betaT;
    *near = f->near;
    *nearT = f->nearT;
    *nleaf = f->nleaf;
    *levels = f->levels;
}

}  // namespace dsbt
