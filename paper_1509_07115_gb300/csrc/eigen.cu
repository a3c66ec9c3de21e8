// eigen.cu -- bound states of one l channel by imaginary-time evolution
// (Sec. 4.4): the paper substitutes t -> -i t in the split-step propagator and
// orthogonalises every state against the lower ones after each step.
//
// One step on nstates real FP64 states psi[s][i] (channel l, spherical
// potential U(r_i)), five kernels: the factors come from tables, exp(-k^2 tau/2) goes
// with the forward contraction and both half steps of the potential with the
// Gram-Schmidt:
//   psi *= exp(-U tau/2);  b = T_l F_l psi;  b *= exp(-k^2 tau/2);
//   psi = F_l^T T_l^T b;   psi *= exp(-U tau/2);
//   modified Gram-Schmidt over s (R_ss = the norm before normalising).
// This is orthogonal iteration with S = exp(-U tau/2) B^T exp(-K tau) B
// exp(-U tau/2), so state s converges to S's s-th eigenvector and
// -ln(R_ss)/tau to its level.  The momenta are the plan's (dsbt_plan_get_k).
#include <math.h>

#include <vector>

#include "plan.cuh"

namespace dsbt {


namespace {

constexpr int kThreads = 1024;

// The factors of a step: pot[i] = exp(-U_i ht) and kin[j] = exp(-k_j^2 ht) with the
// plan's momenta of channel l.
__global__ void k_eig_factors(double* pot, double* kin, const double* __restrict__ U, const double* __restrict__ knl,
                              double dk, int l, int N, double ht) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= N) return;
    pot[i] = exp(-U[i] * ht);
    const double km = knl ? knl[(size_t)l * N + i] : k_index(l, i, N) * dk;
    kin[i] = exp(-km * km * ht);
}

// y[s][i] = pot_i psi[s][i]
__global__ void k_eig_scale(const double* __restrict__ psi, double* __restrict__ y, const double* __restrict__ pot, int N,
                            long long total) {
    const long long k = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (k < total) y[k] = psi[k] * pot[k % N];
}

__device__ double block_sum(double v, double* red) {
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    __syncthreads();
    if (lane == 0) red[w] = v;
    __syncthreads();
    if (w == 0) {
        v = (lane < (int)(blockDim.x >> 5)) ? red[lane] : 0.0;
        for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
        if (lane == 0) red[32] = v;
    }
    __syncthreads();
    return red[32];
}

constexpr int kOrthoThreads = 128;   // one warp per quarter of an SM
constexpr int kOrthoMax = 64;   // states

__device__ __forceinline__ void cluster_sync() {
    asm volatile("barrier.cluster.arrive.release.aligned;\nbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}

// Sums of four values over the warp; lane q < 4 (of every 8 lanes) gets value q.  Six
// FP64 additions instead of twenty (one holds a quarter of the SM for 76 clocks).
__device__ __forceinline__ double warp_sum4(const double* v) {
    const int lane = threadIdx.x & 31;
    const bool b = lane & 2, c = lane & 1;
    const double x = (b ? v[2] : v[0]) + __shfl_xor_sync(0xffffffffu, b ? v[0] : v[2], 2);
    const double y = (b ? v[3] : v[1]) + __shfl_xor_sync(0xffffffffu, b ? v[1] : v[3], 2);
    double s = (c ? y : x) + __shfl_xor_sync(0xffffffffu, c ? x : y, 1);
    for (int o = 4; o < 32; o <<= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    return s;
}

// Modified Gram-Schmidt of the ns states x_s = pot in_s (pot may be null) by one cluster of CL
// CTAs, each holding N / CL columns in shared memory (`in_smem`) or working in `psi`
// directly: rdiag[s] = norm of state s after removing the lower states, before
// normalising; psi takes the states and next (may be null) pot times them, the input
// of the next step.  Right-looking: round t takes <x_t, x_s> of all s >= t at once, so
// a round has one reduction over the cluster (the left-looking form on one CTA took
// ns (ns + 1) / 2 reductions of four barriers: 46 us for 4 states of 1024 points; now
// 21 us, the latency of four rounds of FP64 sums and a cluster barrier).
template <int CL>
__global__ void __launch_bounds__(kOrthoThreads) k_eig_orthonormalise(const double* in, double* psi, double* next,
                                                                       const double* __restrict__ pot, int N, int ns,
                                                                       int in_smem, double* rdiag) {
    extern __shared__ __align__(16) double cols[];   // [ns][N / CL]
    __shared__ double part[2][CL][kOrthoMax];         // by round parity and CTA: its sums
    __shared__ double warps[kOrthoThreads / 32][kOrthoMax];
    unsigned rank;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(rank));
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, W = N / CL, c0 = (int)rank * W;
    double* x = in_smem ? cols : psi + c0;
    const size_t ld = in_smem ? W : N;
    for (int s = 0; s < ns; ++s)
        for (int i = tid; i < W; i += kOrthoThreads) {
            const double v = in[(size_t)s * N + c0 + i];
            x[s * ld + i] = pot ? v * pot[c0 + i] : v;
        }
    cluster_sync();   // every CTA runs before its memory is written
    for (int t = 0; t < ns; ++t) {   // a thread's columns are its own: no barrier before the sums
        for (int s = t; s < ns; s += 4) {
            double v[4] = {0.0, 0.0, 0.0, 0.0};
            for (int i = tid; i < W; i += kOrthoThreads) {
                const double y = x[t * ld + i];
#pragma unroll
                for (int q = 0; q < 4; ++q)
                    if (s + q < ns) v[q] = fma(x[(s + q) * ld + i], y, v[q]);
            }
            const double r = warp_sum4(v);
            if (lane < 4 && s + lane < ns) warps[warp][s + lane] = r;
        }
        __syncthreads();
        for (int s = t + tid; s < ns; s += kOrthoThreads) {   // this CTA's sums to every CTA of the cluster
            double r = 0.0;
            for (int w = 0; w < kOrthoThreads / 32; ++w) r += warps[w][s];
            for (unsigned q = 0; q < CL; ++q) {
                uint32_t a = (uint32_t)__cvta_generic_to_shared(&part[t & 1][rank][s]), ra;
                asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(ra) : "r"(a), "r"(q));
                asm volatile("st.shared::cluster.f64 [%0], %1;" ::"r"(ra), "d"(r) : "memory");
            }
        }
        cluster_sync();
        auto total = [&](int s) {
            double r = 0.0;
#pragma unroll
            for (int q = 0; q < CL; ++q) r += part[t & 1][q][s];
            return r;
        };
        const double sq = total(t), inv = sq > 0.0 ? rsqrt(sq) : 0.0;
        if (rank == 0 && tid == 0) rdiag[t] = sqrt(sq);
        for (int i = tid; i < W; i += kOrthoThreads) {
            const double y = x[t * ld + i] * inv;
            x[t * ld + i] = y;
        }
        for (int s = t + 1; s < ns; ++s) {
            const double d = total(s) * inv;
            for (int i = tid; i < W; i += kOrthoThreads) x[s * ld + i] = fma(-d, x[t * ld + i], x[s * ld + i]);
        }
    }
    cluster_sync();   // no CTA leaves while others store to it
    // global stores last: in a round they would be waited for by its barrier
    for (int s = 0; s < ns; ++s)
        for (int i = tid; i < W; i += kOrthoThreads) {
            const double y = x[s * ld + i];
            if (in_smem) psi[(size_t)s * N + c0 + i] = y;
            if (next) next[(size_t)s * N + c0 + i] = pot ? y * pot[c0 + i] : y;
        }
}

template <int CL>
int orthonormalise(const double* in, double* psi, double* next, const double* pot, int N, int ns, double* rdiag,
                   cudaStream_t st) {
    size_t smem = (size_t)ns * (N / CL) * sizeof(double);
    const int in_smem = smem <= 160 * 1024;
    if (!in_smem) smem = 0;
    if (smem > 32 * 1024)   // 12 KB more are static
        if (int rc = ensure_smem((const void*)k_eig_orthonormalise<CL>, smem)) return rc;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(CL);
    cfg.blockDim = dim3(kOrthoThreads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = CL;
    at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    ProfScope ps(kKTdseReduce, st);
    DSBT_CUDA_TRY(cudaLaunchKernelEx(&cfg, k_eig_orthonormalise<CL>, in, psi, next, pot, N, ns, in_smem, rdiag));
    return DSBT_OK;
}

// CTAs by the columns: 256 or more each.
int orthonormalise(const double* in, double* psi, double* next, const double* pot, int N, int ns, double* rdiag,
                   cudaStream_t st) {
    if (N >= 2048) return orthonormalise<8>(in, psi, next, pot, N, ns, rdiag, st);
    if (N >= 1024) return orthonormalise<4>(in, psi, next, pot, N, ns, rdiag, st);
    return orthonormalise<2>(in, psi, next, pot, N, ns, rdiag, st);
}

// E[s] = sum_j (k_j^2/2) b[s][j]^2 + sum_i U_i psi[s][i]^2 for normalised psi.
__global__ void __launch_bounds__(kThreads) k_eig_energy(const double* __restrict__ psi,
                                                         const double* __restrict__ b,
                                                         const double* __restrict__ U,
                                                         const double* __restrict__ knl, double dk, int l,
                                                         int N, double* E) {
    __shared__ double red[33];
    const int s = blockIdx.x;
    double e = 0.0;
    for (int i = threadIdx.x; i < N; i += blockDim.x) {
        const double km = knl ? knl[(size_t)l * N + i] : k_index(l, i, N) * dk;
        const double bv = b[(size_t)s * N + i], pv = psi[(size_t)s * N + i];
        e += 0.5 * km * km * bv * bv + U[i] * pv * pv;
    }
    e = block_sum(e, red);
    if (threadIdx.x == 0) E[s] = e;
}

inline size_t a256(size_t x) { return (x + 255) & ~(size_t)255; }

}  // namespace
}  // namespace dsbt

using namespace dsbt;

extern "C" size_t dsbt_radial_states_workspace_size(const dsbt_plan* plan, int nstates) {
    if (!plan || nstates < 1 || nstates > 64) return 0;
    return 2 * a256((size_t)nstates * plan->N * sizeof(double)) + a256(3 * 64 * sizeof(double)) +
           2 * a256(plan->N * sizeof(double)) + dsbt_workspace_size(plan, nstates, DSBT_F64) + 512;
}

extern "C" int dsbt_radial_states(const dsbt_plan* plan, int l, const double* U, int nstates, double tau,
                                  int nsteps, double* psi, double* levels, double* energies, void* workspace,
                                  size_t workspace_bytes, void* stream) {
    DSBT_CHECK_ARG(plan != nullptr && U != nullptr && psi != nullptr, "dsbt_radial_states: NULL argument");
    DSBT_CHECK_ARG(plan->T64 != nullptr, "dsbt_radial_states: the plan needs DSBT_PLAN_FP64");
    DSBT_CHECK_ARG(l >= 0 && l <= plan->l_max, "dsbt_radial_states: l=%d outside 0..%d", l, plan->l_max);
    DSBT_CHECK_ARG(nstates >= 1 && nstates <= 64, "dsbt_radial_states: nstates=%d not in 1..64", nstates);
    DSBT_CHECK_ARG(tau > 0.0 && isfinite(tau), "dsbt_radial_states: tau must be positive");
    DSBT_CHECK_ARG(nsteps >= 1, "dsbt_radial_states: nsteps must be >= 1");
    const size_t need = dsbt_radial_states_workspace_size(plan, nstates);
    DSBT_CHECK_ARG(workspace != nullptr && workspace_bytes >= need,
                   "dsbt_radial_states: workspace too small (need %zu bytes)", need);
    cudaStream_t st = (cudaStream_t)stream;
    const int N = plan->N, ns = nstates;
    unsigned char* base = (unsigned char*)(((uintptr_t)workspace + 255) & ~(uintptr_t)255);
    auto take = [&](size_t n) {
        double* q = (double*)base;
        base += a256(n * sizeof(double));
        return q;
    };
    double* b = take((size_t)ns * N);
    double* y = take((size_t)ns * N);    // exp(-U tau/2) psi, then the step's result before its half step
    double* small = take(3 * 64);        // rdiag, E
    double* pot = take(N);
    double* kin = take(N);
    void* gws = base;
    const size_t gws_b = dsbt_workspace_size(plan, ns, DSBT_F64);
    int rc;
    {
        ProfScope ps(kKTdsePot, st);
        k_eig_factors<<<(N + 255) / 256, 256, 0, st>>>(pot, kin, U, plan->knl, plan->dk, l, N, 0.5 * tau);
        DSBT_CUDA_TRY(cudaGetLastError());
    }
    rc = orthonormalise(psi, psi, nullptr, nullptr, N, ns, small, st);
    if (rc) return rc;
    {
        ProfScope ps(kKTdsePot, st);
        const long long tot = (long long)ns * N;
        k_eig_scale<<<(unsigned)((tot + 255) / 256), 256, 0, st>>>(psi, y, pot, N, tot);
        DSBT_CUDA_TRY(cudaGetLastError());
    }
    for (int step = 0; step < nsteps; ++step) {
        rc = real_step(plan, l, ns, y, b, y, kin, gws, gws_b, st);   // F, T, exp(-K tau), T^T, F^T
        if (rc) return rc;
        rc = orthonormalise(y, psi, y, pot, N, ns, small, st);
        if (rc) return rc;
    }
    std::vector<int> counts(plan->l_max + 1, 0);
    counts[l] = ns;
    // energies <psi|H|psi> of the final (normalised) states
    rc = grouped_device_call(0, plan, counts.data(), DSBT_F64, 0.0, psi, b, gws, gws_b, st);
    if (rc) return rc;
    {
        ProfScope ps(kKTdseReduce, st);
        k_eig_energy<<<ns, kThreads, 0, st>>>(psi, b, U, plan->knl, plan->dk, l, N, small + 64);
        DSBT_CUDA_TRY(cudaGetLastError());
    }
    std::vector<double> h(128);
    DSBT_CUDA_TRY(cudaMemcpyAsync(h.data(), small, 128 * sizeof(double), cudaMemcpyDeviceToHost, st));
    DSBT_CUDA_TRY(cudaStreamSynchronize(st));
    for (int s = 0; s < ns; ++s) {
        if (levels) levels[s] = -log(h[s]) / tau;
        if (energies) energies[s] = h[64 + s];
    }
    return DSBT_OK;
}
