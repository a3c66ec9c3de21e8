// tdse.cu -- split-operator TDSE step through the DSBT (m = 0, length gauge)
// and its adjoint.
//
// State: psi[l][i], l = 0..L-1, i = 0..N-1, complex128, in the l representation
// (channel l is the radial function of angular momentum l; the DSBT layout).
// One step of length tau (Sec. 4.1, Eq. (81), vector potential A = 0, so the two
// kinetic half steps merge):
//     psi <- Q_s Kin Q_s psi,
//     Q_s = P diag_j exp(-i [V(r_i) + E_s r_i eta_j] tau/2) P^T       (angular grid)
//     Kin = B^T exp(-i K tau) B,  B = T_l F_l per l,  K = k~_n^2 / 2    (dsbt_kinetic)
// with eta_j, w_j the L-point Gauss-Legendre rule and P[l][j] =
// Pbar_l(eta_j) sqrt(w_j) the orthonormal angular transform of Sec. 4.1
// (associated Legendre functions for m = 0), V(r) = -Z / sqrt(r^2 + a2).
//
// Adjacent half steps share the angular grid and P is orthogonal, so Q_{s+1} Q_s =
// P diag_j exp(-i [2 V(r_i) + (E_s + E_{s+1}) r_i eta_j] tau/2) P^T is one pass: a
// propagation alternates Kin with such merged passes and has single ones at its
// ends only.
//
// Adjoint: every factor is unitary and B, P are real orthogonal (Eq. (25),
// T^{-1} = T^T), so U_s^H = Q_s^H Kin^H Q_s^H is the same step with tau -> -tau.
// For the observable O = sum_{r_i > r_cut} |psi_S|^2 and lambda_S = Pi psi_S:
//     nu_s = Kin^H Q_s^H lambda_{s+1},  lambda_s = Q_s^H nu_s,
//     dO/dE_s = tau Im( <lambda_{s+1}, R psi_{s+1}> + <nu_s, R a_s> ),  a_s = Q_s psi_s,
// where R = diag(r_i eta_j) on the angular grid (the field coupling r cos(theta)).
// R commutes with Q_s, so <nu_s, R a_s> = <lambda_s, R psi_s> = g_s and
//     dO/dE_s = tau (Im g_s + Im g_{s+1}),   g_S real (lambda_S = Pi psi_S),
// with g_s = <P^T nu_s, R P^T a_s> from grid values that the merged passes hold:
// the forward pass of a segment stores P^T a_s, the adjoint pass meets P^T nu_s.
#include <math.h>

#include <new>
#include <algorithm>
#include <vector>

#include "mm64.cuh"
#include "plan.cuh"

struct dsbt_tdse {
    const dsbt_plan* plan;
    int L, N;
    int m0;         // |m|: channels are l = m0 .. m0 + L - 1
    double dr, tau, Z, a2;
    double* P;      // [L][L] angular transform
    uint2* Pw;      // its fixed-point words (mm64.cuh): [64][64] P^T by node pairs, then [64][64] P
    double* V;      // [N] potential
    double* rr;     // [N] radii
    double* eta;    // [L] nodes
    std::vector<double> eta_h, w_h;
};

namespace dsbt {

namespace {

constexpr int TI = 8;           // radial points per tile of the angular kernels: 16 real columns
constexpr int kLMax = 64;
constexpr int AB = kLMax + 16;  // halfs per digit row of a tile (mm64.cuh)

// Gauss-Legendre nodes and weights by Newton's method on P_L (three-term
// recurrence for P_L and its derivative).
void gauss_legendre(int L, std::vector<double>& x, std::vector<double>& w) {
    x.assign(L, 0.0);
    w.assign(L, 0.0);
    for (int j = 0; j < L; ++j) {
        double z = cos(M_PI * (j + 0.75) / (L + 0.5));
        double dp = 1.0;
        for (int it = 0; it < 100; ++it) {
            double p0 = 1.0, p1 = z;
            for (int k = 2; k <= L; ++k) {
                const double p2 = ((2.0 * k - 1.0) * z * p1 - (k - 1.0) * p0) / k;
                p0 = p1;
                p1 = p2;
            }
            double pL = (L == 1) ? z : p1, pLm1 = (L == 1) ? 1.0 : p0;
            if (L == 1) { pL = z; pLm1 = 1.0; }
            dp = L * (z * pL - pLm1) / (z * z - 1.0);
            const double dz = pL / dp;
            z -= dz;
            if (fabs(dz) < 1e-16) break;
        }
        // final derivative at the converged node
        double p0 = 1.0, p1 = z;
        for (int k = 2; k <= L; ++k) {
            const double p2 = ((2.0 * k - 1.0) * z * p1 - (k - 1.0) * p0) / k;
            p0 = p1;
            p1 = p2;
        }
        dp = (L == 1) ? 1.0 : L * (z * p1 - p0) / (z * z - 1.0);
        x[j] = z;
        w[j] = 2.0 / ((1.0 - z * z) * dp * dp);
    }
}

// P[l][j] = sqrt((2l+1)/2) P_l(eta_j) sqrt(w_j).
void angular_matrix(int L, const std::vector<double>& x, const std::vector<double>& w,
                    std::vector<double>& P) {
    P.assign((size_t)L * L, 0.0);
    for (int j = 0; j < L; ++j) {
        double p0 = 1.0, p1 = x[j];
        for (int l = 0; l < L; ++l) {
            double pl;
            if (l == 0) pl = 1.0;
            else if (l == 1) pl = x[j];
            else {
                const double p2 = ((2.0 * l - 1.0) * x[j] * p1 - (l - 1.0) * p0) / l;
                p0 = p1;
                p1 = p2;
                pl = p2;
            }
            P[(size_t)l * L + j] = sqrt((2.0 * l + 1.0) / 2.0) * pl * sqrt(w[j]);
        }
    }
}

// m != 0: rows l = m .. m + L - 1 of the normalised associated Legendre
// functions Pbar_l^m(eta_j) sqrt(w_j) (recurrence in l from Pbar_m^m), then
// orthonormalised on the L-point rule by modified Gram-Schmidt in order of l
// (the L-point rule integrates their products exactly only for m = 0).
void angular_matrix_m(int L, int m, const std::vector<double>& x, const std::vector<double>& w,
                      std::vector<double>& P) {
    P.assign((size_t)L * L, 0.0);
    for (int j = 0; j < L; ++j) {
        const double z = x[j], sq = sqrt(std::max(0.0, 1.0 - z * z));
        // Pbar_m^m = sqrt((2m+1)!! / (2 (2m)!!)) (1 - z^2)^(m/2) (Condon-Shortley sign dropped)
        double pmm = sqrt(0.5);
        for (int k = 1; k <= m; ++k) pmm *= sqrt((2.0 * k + 1.0) / (2.0 * k)) * sq;
        double pa = pmm, pb = (L > 1) ? sqrt(2.0 * m + 3.0) * z * pmm : 0.0;   // Pbar_m^m, Pbar_{m+1}^m
        for (int i = 0; i < L; ++i) {
            const int l = m + i;
            double pl;
            if (i == 0) pl = pa;
            else if (i == 1) pl = pb;
            else {
                const double a = sqrt((4.0 * l * l - 1.0) / ((double)l * l - (double)m * m));
                const double b = sqrt(((l - 1.0) * (l - 1.0) - (double)m * m) / (4.0 * (l - 1.0) * (l - 1.0) - 1.0));
                pl = a * (z * pb - b * pa);
                pa = pb;
                pb = pl;
            }
            P[(size_t)i * L + j] = pl * sqrt(w[j]);
        }
    }
    // Modified Gram-Schmidt of the rows.  One pass loses orthogonality as the rows
    // approach dependence on the rule (5e-10 at L = 32, m = 8; 2e-5 at m = 12); with
    // the row normalised and projected twice more P P^T = 1 holds to rounding, which
    // the merged half steps and the adjoint below rely on.
    for (int i = 0; i < L; ++i) {
        double* ri = P.data() + (size_t)i * L;
        for (int pass = 0; pass < 3; ++pass) {
            for (int k = 0; k < i; ++k) {
                const double* rk = P.data() + (size_t)k * L;
                double d = 0.0;
                for (int j = 0; j < L; ++j) d += ri[j] * rk[j];
                for (int j = 0; j < L; ++j) ri[j] -= d * rk[j];
            }
            double q = 0.0;
            for (int j = 0; j < L; ++j) q += ri[j] * ri[j];
            const double inv = 1.0 / sqrt(q);
            for (int j = 0; j < L; ++j) ri[j] *= inv;
        }
    }
}

__device__ __forceinline__ double2 cmul2(double2 a, double2 b) {
    return make_double2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);
}

// The angular kernels take TI radial points (16 real columns) through P^T, a
// diagonal and P.  Both products run on the tensor cores through exact digits
// (mm64.cuh): as FP64 multiply-adds they took 80 us per pass at L = 64, N = 2048,
// the FP64 pipe's whole rate.  What is left on that pipe are the phases, so the
// nodes go in pairs: row g of a 16-row block is node j = 8 m + g and row g + 8 its
// mirror L - 1 - j (eta_{L-1-j} = -eta_j), both in one thread, and one sine and
// cosine serve both.
struct AngularShared {
    __half dig[mm64::ND][2 * TI][AB];
    double2 grid[kLMax][TI];
    int ef[2][2 * TI];
    double2 vph[TI];
};

// Digits of v[c] = rows 4 kq + c of column pair t (re, im); every thread of the CTA.
__device__ __forceinline__ void angular_digits(AngularShared& sh, int pass, int kq, int t, const double2* v) {
    const double re[4] = {v[0].x, v[1].x, v[2].x, v[3].x}, im[4] = {v[0].y, v[1].y, v[2].y, v[3].y};
    int er = mm64::exponent4(re), ei = mm64::exponent4(im);
#pragma unroll
    for (int o = TI; o < 32; o <<= 1) {   // lanes of one point
        er = max(er, __shfl_xor_sync(0xffffffffu, er, o));
        ei = max(ei, __shfl_xor_sync(0xffffffffu, ei, o));
    }
    if ((threadIdx.x & 31) < TI) {
        atomicMax(&sh.ef[pass][2 * t], er);
        atomicMax(&sh.ef[pass][2 * t + 1], ei);
    }
    __syncthreads();
    mm64::put_digits4(&sh.dig[0][2 * t][4 * kq], 2 * TI * AB, re, sh.ef[pass][2 * t]);
    mm64::put_digits4(&sh.dig[0][2 * t + 1][4 * kq], 2 * TI * AB, im, sh.ef[pass][2 * t + 1]);
    __syncthreads();
}

// y = P diag(exp(-i [w V + (E_e1 + E_e2) r eta] ht)) P^T x (w = 2, or w = 1 and no
// second sample for e2 < 0; ht = +tau/2 forward, -tau/2 adjoint).  x and y may
// alias; y may be null (no way back).  grid_out: also stores the grid values
// [L][N] after the phase.  grid_in: adds gscale * sum Im(conj(P^T x) r eta grid_in)
// into *g1 and, unless null, *g2.
__global__ void __launch_bounds__(128) k_tdse_potential(const double2* x, double2* y, const uint2* __restrict__ Pw,
                                                        const double* __restrict__ V, const double* __restrict__ rr,
                                                        const double* __restrict__ eta, int L, int N,
                                                        const double* __restrict__ E, int e1, int e2, double ht,
                                                        double2* grid_out, const double2* __restrict__ grid_in,
                                                        double gscale, double* g1, double* g2) {
    __shared__ AngularShared sh;
    __shared__ double red[4];
    const int i0 = blockIdx.x * TI, tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int t = tid % TI, kq = tid / TI, i = i0 + t;   // N is a multiple of 256
    const int L16 = (L + 15) & ~15, half = (L + 1) / 2;
    double2 v[4];
#pragma unroll
    for (int c = 0; c < 4; ++c) v[c] = 4 * kq + c < L ? x[(size_t)(4 * kq + c) * N + i] : make_double2(0.0, 0.0);
    if (tid < 4 * TI) sh.ef[tid / (2 * TI)][tid % (2 * TI)] = 0;
    if (tid < TI) {
        double sn, cs;
        sincos(-V[i] * (e2 >= 0 ? 2.0 * ht : ht), &sn, &cs);   // 2 V may pass the largest number
        sh.vph[t] = make_double2(cs, sn);
    }
    for (int k = tid; k < (L16 - L) * TI; k += blockDim.x) sh.grid[L + k / TI][k % TI] = make_double2(0.0, 0.0);
    __syncthreads();
    angular_digits(sh, 0, kq, t, v);
    const double Ev = (E ? E[e1] : 0.0) + (E && e2 >= 0 ? E[e2] : 0.0);
    double gim = 0.0;
    if (8 * warp < half) {   // to the angular grid
        long long hi[2][4], lo[2][4];
        mm64::block_product<2>(Pw + (size_t)warp * 16 * kLMax, kLMax, L16 / 16, &sh.dig[0][0][0], AB, lane, hi, lo);
        const int g = lane >> 2, tq = lane & 3, j = 8 * warp + g, jm = L - 1 - j;
        if (j < half) {
            const double ej = eta[j];
#pragma unroll
            for (int n = 0; n < 2; ++n) {
                const int tp = 4 * n + tq, ip = i0 + tp, er = sh.ef[0][2 * tp], ei = sh.ef[0][2 * tp + 1];
                const double re = rr[ip] * ej;
                double2 a = make_double2(mm64::to_double(hi[n][0], lo[n][0], er), mm64::to_double(hi[n][1], lo[n][1], ei));
                double2 b = make_double2(mm64::to_double(hi[n][2], lo[n][2], er), mm64::to_double(hi[n][3], lo[n][3], ei));
                if (grid_in) {   // the middle node of an odd L is its own mirror
                    const double2 ga = grid_in[(size_t)j * N + ip];
                    gim += re * (a.x * ga.y - a.y * ga.x);
                    if (jm != j) {
                        const double2 gb = grid_in[(size_t)jm * N + ip];
                        gim -= re * (b.x * gb.y - b.y * gb.x);
                    }
                }
                double sn, cs;
                sincos(-Ev * re * ht, &sn, &cs);
                const double2 w = sh.vph[tp];
                a = cmul2(cmul2(a, w), make_double2(cs, sn));
                b = cmul2(cmul2(b, w), make_double2(cs, -sn));
                sh.grid[j][tp] = a;
                if (grid_out) grid_out[(size_t)j * N + ip] = a;
                if (jm != j) {
                    sh.grid[jm][tp] = b;
                    if (grid_out) grid_out[(size_t)jm * N + ip] = b;
                }
            }
        }
    }
    if (grid_in) {
        for (int o = 16; o > 0; o >>= 1) gim += __shfl_xor_sync(0xffffffffu, gim, o);
        if (lane == 0) red[warp] = gim;
    }
    __syncthreads();
    if (grid_in && tid == 0) {
        const double sum = gscale * (red[0] + red[1] + red[2] + red[3]);
        atomicAdd(g1, sum);
        if (g2) atomicAdd(g2, sum);
    }
    if (!y) return;
#pragma unroll
    for (int c = 0; c < 4; ++c) v[c] = 4 * kq + c < L16 ? sh.grid[4 * kq + c][t] : make_double2(0.0, 0.0);
    angular_digits(sh, 1, kq, t, v);
    if (16 * warp < L) {   // back to l
        long long hi[2][4], lo[2][4];
        mm64::block_product<2>(Pw + (size_t)(kLMax + warp * 16) * kLMax, kLMax, L16 / 16, &sh.dig[0][0][0], AB, lane, hi,
                               lo);
        const int l = 16 * warp + (lane >> 2);
#pragma unroll
        for (int n = 0; n < 2; ++n) {
            const int tp = 4 * n + (lane & 3), er = sh.ef[1][2 * tp], ei = sh.ef[1][2 * tp + 1];
            if (l < L)
                y[(size_t)l * N + i0 + tp] =
                    make_double2(mm64::to_double(hi[n][0], lo[n][0], er), mm64::to_double(hi[n][1], lo[n][1], ei));
            if (l + 8 < L)
                y[(size_t)(l + 8) * N + i0 + tp] =
                    make_double2(mm64::to_double(hi[n][2], lo[n][2], er), mm64::to_double(hi[n][3], lo[n][3], ei));
        }
    }
}

// The momentum-space middle of the velocity-gauge step (Eq. (81)) on a tile of
// TI momentum slots n = 1..N (k~_n = n dk, Eq. (65)), in place on the DSBT
// coefficients c[l][s] (storage s = n - 1 for even l; s = n for odd l, with
// n = N stored at s = 0):
//   half kinetic phase exp(-i k^2 tau/4)  (k = the plan's momentum of (l, s)),
//   phi = Ytilde^dagger c  (phi_j = sum_l (-i)^l s_l P[l][j] c_l),
//   phi_j *= exp(i A k~_n eta_j tau),
//   c = Ytilde phi  (c_l = i^l s_l sum_j P[l][j] phi_j),  half kinetic phase.
// s_l = (-1)^ceil(l/2) converts this library's sine/cosine sign convention to
// the spherical-wave coefficients of Ytilde, so (-i)^l s_l = 1 (even l) or i
// (odd l).  A is the vector potential sample of this step.
// half: exp(-i k^2 tau/4) by storage row, as the kinetic phase table of tau / 2.
__global__ void __launch_bounds__(128) k_tdse_velocity(double2* c, const uint2* __restrict__ Pw,
                                                       const double* __restrict__ eta,
                                                       const double2* __restrict__ half_phase, int per_l, double dk, int L,
                                                       int N, const double* __restrict__ A, int aidx, double tau, int m0) {
    __shared__ AngularShared sh;
    const int n0 = 1 + blockIdx.x * TI, tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int t = tid % TI, kq = tid / TI, L16 = (L + 15) & ~15, half = (L + 1) / 2;
    auto slot = [&](int ch, int n, double2& ph) {   // storage of momentum n of channel ch, and its half kinetic phase
        const int l = m0 + ch, sidx = (l & 1) ? (n % N) : n - 1;
        ph = per_l ? half_phase[(size_t)l * N + sidx] : half_phase[(size_t)(l & 1) * N + phase_entry(l, sidx, N)];
        return (size_t)ch * N + sidx;
    };
    double2 v[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {   // gather, half kinetic phase, (-i)^l s_l
        const int ch = 4 * kq + q;
        v[q] = make_double2(0.0, 0.0);
        if (ch < L) {
            double2 ph;
            const size_t at = slot(ch, n0 + t, ph);
            v[q] = cmul2(c[at], ph);
            if ((m0 + ch) & 1) v[q] = make_double2(-v[q].y, v[q].x);   // times i
        }
    }
    if (tid < 4 * TI) sh.ef[tid / (2 * TI)][tid % (2 * TI)] = 0;
    for (int k = tid; k < (L16 - L) * TI; k += blockDim.x) sh.grid[L + k / TI][k % TI] = make_double2(0.0, 0.0);
    __syncthreads();
    angular_digits(sh, 0, kq, t, v);
    const double Av = A ? A[aidx] : 0.0;
    if (8 * warp < half) {   // to the angular grid, A . P phase (node pairs as in k_tdse_potential)
        long long hi[2][4], lo[2][4];
        mm64::block_product<2>(Pw + (size_t)warp * 16 * kLMax, kLMax, L16 / 16, &sh.dig[0][0][0], AB, lane, hi, lo);
        const int g = lane >> 2, tq = lane & 3, j = 8 * warp + g, jm = L - 1 - j;
        if (j < half) {
            const double ej = eta[j];
#pragma unroll
            for (int n = 0; n < 2; ++n) {
                const int tp = 4 * n + tq, er = sh.ef[0][2 * tp], ei = sh.ef[0][2 * tp + 1];
                const double2 a = make_double2(mm64::to_double(hi[n][0], lo[n][0], er), mm64::to_double(hi[n][1], lo[n][1], ei));
                const double2 b = make_double2(mm64::to_double(hi[n][2], lo[n][2], er), mm64::to_double(hi[n][3], lo[n][3], ei));
                double sn, cs;
                sincos(Av * ((n0 + tp) * dk) * ej * tau, &sn, &cs);
                sh.grid[j][tp] = cmul2(a, make_double2(cs, sn));
                if (jm != j) sh.grid[jm][tp] = cmul2(b, make_double2(cs, -sn));
            }
        }
    }
    __syncthreads();
#pragma unroll
    for (int q = 0; q < 4; ++q) v[q] = 4 * kq + q < L16 ? sh.grid[4 * kq + q][t] : make_double2(0.0, 0.0);
    angular_digits(sh, 1, kq, t, v);
    if (16 * warp < L) {   // back to l, i^l s_l, half kinetic phase, scatter
        long long hi[2][4], lo[2][4];
        mm64::block_product<2>(Pw + (size_t)(kLMax + warp * 16) * kLMax, kLMax, L16 / 16, &sh.dig[0][0][0], AB, lane, hi,
                               lo);
#pragma unroll
        for (int n = 0; n < 2; ++n) {
            const int tp = 4 * n + (lane & 3), er = sh.ef[1][2 * tp], ei = sh.ef[1][2 * tp + 1];
#pragma unroll
            for (int q = 0; q < 2; ++q) {
                const int ch = 16 * warp + (lane >> 2) + 8 * q;
                if (ch >= L) continue;
                double2 s = make_double2(mm64::to_double(hi[n][2 * q], lo[n][2 * q], er),
                                         mm64::to_double(hi[n][2 * q + 1], lo[n][2 * q + 1], ei));
                if ((m0 + ch) & 1) s = make_double2(s.y, -s.x);   // times -i
                double2 ph;
                const size_t at = slot(ch, n0 + tp, ph);
                c[at] = cmul2(s, ph);
            }
        }
    }
}

// out += sum_{r_i > rc} sum_l |x[l][i]|^2 ; with lam != nullptr also writes
// lam = x on r_i > rc and 0 elsewhere (the projector Pi).
__global__ void k_tdse_observable(const double2* __restrict__ x, double2* __restrict__ lam,
                                  const double* __restrict__ rr, int L, int N, double rc,
                                  double* __restrict__ out) {
    const long long k = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    double v = 0.0;
    if (k < (long long)L * N) {
        const int i = (int)(k % N);
        const double2 a = x[k];
        const bool in = rr[i] > rc;
        if (in) v = a.x * a.x + a.y * a.y;
        if (lam) lam[k] = in ? a : make_double2(0.0, 0.0);
    }
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    if ((threadIdx.x & 31) == 0 && v != 0.0) atomicAdd(out, v);
}

size_t state_bytes(const dsbt_tdse* t) { return (size_t)t->L * t->N * sizeof(double2); }

}  // namespace

void tdse_gauss_legendre(int L, std::vector<double>& x, std::vector<double>& w) { gauss_legendre(L, x, w); }
void tdse_angular_rows(int L, int m, const std::vector<double>& x, const std::vector<double>& w,
                       std::vector<double>& P) {
    angular_matrix_m(L, m, x, w, P);
}

namespace {

inline size_t a256(size_t x) { return (x + 255) & ~(size_t)255; }

// One angular pass with the samples e1 and (merged half steps) e2 >= 0; see k_tdse_potential.
int potential(const dsbt_tdse* t, const double2* x, double2* y, const double* E, int e1, int e2, double ht,
              cudaStream_t st, double2* grid_out = nullptr, const double2* grid_in = nullptr, double gscale = 0.0,
              double* g1 = nullptr, double* g2 = nullptr) {
    ProfScope ps(kKTdsePot, st);
    k_tdse_potential<<<t->N / TI, 128, 0, st>>>(x, y, t->Pw, t->V, t->rr, t->eta, t->L, t->N, E, e1, e2, ht, grid_out,
                                                grid_in, gscale, g1, g2);
    DSBT_CUDA_TRY(cudaGetLastError());
    return DSBT_OK;
}

int observable(const dsbt_tdse* t, const double2* x, double2* lam, double rc, double* out, cudaStream_t st) {
    const long long n = (long long)t->L * t->N;
    ProfScope ps(kKTdseReduce, st);
    k_tdse_observable<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(x, lam, t->rr, t->L, t->N, rc, out);
    DSBT_CUDA_TRY(cudaGetLastError());
    return DSBT_OK;
}

// The kinetic step of one state with the phase table already in the workspace.
int kinetic(const dsbt_tdse* t, const int* counts, const double2* x, double2* y, void* kws, size_t kws_b,
            cudaStream_t st) {
    return grouped_device_call(kKineticReady, t->plan, counts, DSBT_C128, 0.0, x, y, kws, kws_b, st);
}

// The momentum-space part of a velocity-gauge step (Eq. (81)): forward DSBT,
// k_tdse_velocity, inverse DSBT (c: one state of scratch for the coefficients; the
// workspace's phase table holds tau / 2).
int momentum_part(const dsbt_tdse* t, const int* counts, const double2* x, double2* y, double2* c, const double* A,
                  int idx, double tau, void* kws, size_t kws_b, cudaStream_t st) {
    int rc = grouped_device_call(0, t->plan, counts, DSBT_C128, 0.0, x, c, kws, kws_b, st);
    if (rc) return rc;
    {
        ProfScope ps(kKTdseAng, st);
        k_tdse_velocity<<<t->N / TI, 128, 0, st>>>(c, t->Pw, t->eta, kinetic_phase_table(t->plan, kws, t->L), t->plan->knl != nullptr,
                                                   t->plan->dk, t->L, t->N, A, idx, tau, t->m0);
        DSBT_CUDA_TRY(cudaGetLastError());
    }
    return grouped_device_call(1, t->plan, counts, DSBT_C128, 0.0, c, y, kws, kws_b, st);
}

struct TdseWs {
    double2* ckpt;     // [nck][L][N]
    double2* seg;      // [K+1][L][N]
    double2* a;
    double2* mu;
    double2* nu;
    double2* lam;
    double2* tmp;
    void* kws;         // DSBT kinetic workspace
    size_t kws_b;
};

// K >= 1: gradient layout with nsteps/K + 1 checkpoints and a K+1 segment;
// K == 0: propagation only (no checkpoint storage).
size_t ws_layout(const dsbt_tdse* t, int nsteps, int K, TdseWs* w, void* base) {
    const size_t sb = a256(state_bytes(t));
    const int nck = (K >= 1) ? nsteps / K + 1 : 0;
    const size_t kws_b = dsbt_workspace_size(t->plan, t->L, DSBT_C128);
    size_t off = 0;
    unsigned char* p = (unsigned char*)(((uintptr_t)base + 255) & ~(uintptr_t)255);
    auto take = [&](size_t b) { unsigned char* q = p + off; off += a256(b); return q; };
    double2* ck = (double2*)take(sb * nck);
    double2* sg = (K >= 1) ? (double2*)take(sb * (K + 1)) : nullptr;
    double2* a = (double2*)take(sb);
    double2* mu = (double2*)take(sb);
    double2* nu = (double2*)take(sb);
    double2* lam = (double2*)take(sb);
    double2* tmp = (double2*)take(sb);
    void* kws = take(kws_b);
    if (w) *w = TdseWs{ck, sg, a, mu, nu, lam, tmp, kws, kws_b};
    return off + 256;
}

}  // namespace
}  // namespace dsbt

using namespace dsbt;

extern "C" int dsbt_tdse_create(const dsbt_plan* plan, int L, double tau, double Z, double a2,
                                dsbt_tdse** out) {
    return dsbt_tdse_create_m(plan, L, 0, tau, Z, a2, out);
}

extern "C" int dsbt_tdse_create_m(const dsbt_plan* plan, int L, int m, double tau, double Z, double a2,
                                  dsbt_tdse** out) {
    DSBT_CHECK_ARG(plan != nullptr && out != nullptr, "dsbt_tdse_create: NULL argument");
    *out = nullptr;
    const int m0 = m < 0 ? -m : m;
    DSBT_CHECK_ARG(L >= 1 && L <= kLMax && m0 + L - 1 <= plan->l_max,
                   "dsbt_tdse_create: L=%d, |m|=%d need L <= 64 and |m| + L - 1 <= l_max", L, m0);
    DSBT_CHECK_ARG(plan->T64 != nullptr, "dsbt_tdse_create: the plan needs DSBT_PLAN_FP64");
    DSBT_CHECK_ARG(isfinite(tau) && isfinite(Z) && a2 > 0.0, "dsbt_tdse_create: bad tau/Z/a2");
    dsbt_tdse* t = new (std::nothrow) dsbt_tdse();
    if (!t) return DSBT_ERR_NOMEM;
    t->plan = plan;
    t->L = L;
    t->m0 = m0;
    t->N = plan->N;
    t->dr = plan->r_max / plan->N;
    t->tau = tau;
    t->Z = Z;
    t->a2 = a2;
    gauss_legendre(L, t->eta_h, t->w_h);
    std::vector<double> Ph;
    if (m0 == 0) angular_matrix(L, t->eta_h, t->w_h, Ph);
    else angular_matrix_m(L, m0, t->eta_h, t->w_h, Ph);
    std::vector<double> Vh(t->N), rh(t->N);
    for (int i = 0; i < t->N; ++i) {
        rh[i] = (i + 0.5) * t->dr;
        Vh[i] = -Z / sqrt(rh[i] * rh[i] + a2);
    }
    // words of P^T with the nodes in mirror pairs (row 16 m + g: node 8 m + g, row
    // 16 m + 8 + g: its mirror; the middle node of an odd L once), then of P
    std::vector<uint2> Pw((size_t)2 * kLMax * kLMax, mm64::fixed_a_host(0.0));
    for (int r = 0; r < kLMax; ++r) {
        const int j = 8 * (r / 16) + r % 8, node = (r & 8) ? L - 1 - j : j;
        const bool on = j < (L + 1) / 2 && !((r & 8) && node == j);
        for (int k = 0; k < L; ++k) {
            if (on) Pw[(size_t)r * kLMax + k] = mm64::fixed_a_host(Ph[(size_t)k * L + node]);
            if (r < L) Pw[(size_t)(kLMax + r) * kLMax + k] = mm64::fixed_a_host(Ph[(size_t)r * L + k]);
        }
    }
    bool ok = cudaMalloc((void**)&t->P, Ph.size() * sizeof(double)) == cudaSuccess &&
              cudaMalloc((void**)&t->Pw, Pw.size() * sizeof(uint2)) == cudaSuccess &&
              cudaMalloc((void**)&t->V, t->N * sizeof(double)) == cudaSuccess &&
              cudaMalloc((void**)&t->rr, t->N * sizeof(double)) == cudaSuccess &&
              cudaMalloc((void**)&t->eta, L * sizeof(double)) == cudaSuccess;
    ok = ok && cudaMemcpy(t->P, Ph.data(), Ph.size() * sizeof(double), cudaMemcpyHostToDevice) == cudaSuccess &&
         cudaMemcpy(t->Pw, Pw.data(), Pw.size() * sizeof(uint2), cudaMemcpyHostToDevice) == cudaSuccess &&
         cudaMemcpy(t->V, Vh.data(), t->N * sizeof(double), cudaMemcpyHostToDevice) == cudaSuccess &&
         cudaMemcpy(t->rr, rh.data(), t->N * sizeof(double), cudaMemcpyHostToDevice) == cudaSuccess &&
         cudaMemcpy(t->eta, t->eta_h.data(), L * sizeof(double), cudaMemcpyHostToDevice) == cudaSuccess;
    if (!ok) {
        cudaGetLastError();
        cudaFree(t->P);
        cudaFree(t->Pw);
        cudaFree(t->V);
        cudaFree(t->rr);
        cudaFree(t->eta);
        delete t;
        set_error("dsbt_tdse_create: device allocation or copy failed");
        return DSBT_ERR_NOMEM;
    }
    *out = t;
    return DSBT_OK;
}

extern "C" int dsbt_tdse_set_potential(dsbt_tdse* t, const double* V, int n) {
    DSBT_CHECK_ARG(t != nullptr && V != nullptr, "dsbt_tdse_set_potential: NULL argument");
    DSBT_CHECK_ARG(n == t->N, "dsbt_tdse_set_potential: %d values for a grid of %d points", n, t->N);
    for (int i = 0; i < n; ++i) DSBT_CHECK_ARG(isfinite(V[i]), "dsbt_tdse_set_potential: V[%d] not finite", i);
    DSBT_CUDA_TRY(cudaMemcpy(t->V, V, n * sizeof(double), cudaMemcpyHostToDevice));
    return DSBT_OK;
}

extern "C" int dsbt_tdse_destroy(dsbt_tdse* t) {
    if (!t) return DSBT_OK;
    cudaDeviceSynchronize();
    cudaFree(t->P);
    cudaFree(t->Pw);
    cudaFree(t->V);
    cudaFree(t->rr);
    cudaFree(t->eta);
    delete t;
    return DSBT_OK;
}

extern "C" int dsbt_tdse_angular(const dsbt_tdse* t, double* eta, double* w, double* P) {
    DSBT_CHECK_ARG(t != nullptr, "dsbt_tdse_angular: NULL tdse");
    if (eta) for (int j = 0; j < t->L; ++j) eta[j] = t->eta_h[j];
    if (w) for (int j = 0; j < t->L; ++j) w[j] = t->w_h[j];
    if (P) DSBT_CUDA_TRY(cudaMemcpy(P, t->P, (size_t)t->L * t->L * sizeof(double), cudaMemcpyDeviceToHost));
    return DSBT_OK;
}

extern "C" size_t dsbt_tdse_workspace_size(const dsbt_tdse* t, int nsteps, int checkpoint_every) {
    if (!t || nsteps < 0 || checkpoint_every < 0) return 0;
    return ws_layout(t, nsteps, checkpoint_every, nullptr, nullptr);
}

static int check_run(const dsbt_tdse* t, const void* psi, const double* E, int nsteps, int hold, void* ws,
                     size_t ws_b, int K) {
    DSBT_CHECK_ARG(t != nullptr && psi != nullptr, "tdse: NULL argument");
    DSBT_CHECK_ARG(nsteps >= 0 && hold >= 1, "tdse: nsteps >= 0 and hold >= 1 required");
    DSBT_CHECK_ARG(nsteps == 0 || E != nullptr, "tdse: field samples E is NULL");
    DSBT_CHECK_ARG(ws != nullptr && ws_b >= dsbt_tdse_workspace_size(t, nsteps, K),
                   "tdse: workspace too small (need %zu bytes)", dsbt_tdse_workspace_size(t, nsteps, K));
    return DSBT_OK;
}

extern "C" int dsbt_tdse_propagate(const dsbt_tdse* t, void* psi, const double* E, int nsteps, int hold,
                                   double tau_sign, void* workspace, size_t workspace_bytes, void* stream) {
    int rc = check_run(t, psi, E, nsteps, hold, workspace, workspace_bytes, 0);
    if (rc) return rc;
    DSBT_CHECK_ARG(tau_sign == 1.0 || tau_sign == -1.0, "tdse: tau_sign must be +1 or -1");
    cudaStream_t st = (cudaStream_t)stream;
    TdseWs w;
    ws_layout(t, nsteps, 0, &w, workspace);
    std::vector<int> counts(t->plan->l_max + 1, 0);
    for (int l = 0; l < t->L; ++l) counts[t->m0 + l] = 1;
    double2* x = (double2*)psi;
    const double tau = tau_sign * t->tau;
    if (nsteps == 0) return DSBT_OK;
    rc = kinetic_phase_fill(t->plan, w.kws, t->L, tau, st);
    // forward in time: sample s / hold; backward (tau < 0): the samples in reverse
    auto sample = [&](int s) { return (tau_sign > 0 ? s : nsteps - 1 - s) / hold; };
    if (!rc) rc = potential(t, x, w.a, E, sample(0), -1, 0.5 * tau, st);
    for (int s = 0; s < nsteps && !rc; ++s) {
        rc = kinetic(t, counts.data(), w.a, w.tmp, w.kws, w.kws_b, st);
        if (rc) break;
        if (s + 1 < nsteps) rc = potential(t, w.tmp, w.a, E, sample(s), sample(s + 1), 0.5 * tau, st);
        else rc = potential(t, w.tmp, x, E, sample(s), -1, 0.5 * tau, st);
    }
    return rc;
}

extern "C" int dsbt_tdse_propagate_velocity(const dsbt_tdse* t, void* psi, const double* E, const double* A,
                                            int nsteps, int hold, double tau_sign, void* workspace,
                                            size_t workspace_bytes, void* stream) {
    DSBT_CHECK_ARG(t != nullptr && psi != nullptr, "tdse: NULL argument");
    DSBT_CHECK_ARG(nsteps >= 0 && hold >= 1, "tdse: nsteps >= 0 and hold >= 1 required");
    DSBT_CHECK_ARG(workspace != nullptr && workspace_bytes >= dsbt_tdse_workspace_size(t, nsteps, 0),
                   "tdse: workspace too small (need %zu bytes)", dsbt_tdse_workspace_size(t, nsteps, 0));
    DSBT_CHECK_ARG(tau_sign == 1.0 || tau_sign == -1.0, "tdse: tau_sign must be +1 or -1");
    cudaStream_t st = (cudaStream_t)stream;
    TdseWs w;
    ws_layout(t, nsteps, 0, &w, workspace);
    std::vector<int> counts(t->plan->l_max + 1, 0);
    for (int l = 0; l < t->L; ++l) counts[t->m0 + l] = 1;
    double2* x = (double2*)psi;
    const double tau = tau_sign * t->tau;
    if (nsteps == 0) return DSBT_OK;
    int rc = kinetic_phase_fill(t->plan, w.kws, t->L, 0.5 * tau, st);
    auto sample = [&](int s) { return (tau_sign > 0 ? s : nsteps - 1 - s) / hold; };
    if (!rc) rc = potential(t, x, w.a, E, sample(0), -1, 0.5 * tau, st);
    for (int s = 0; s < nsteps && !rc; ++s) {
        rc = momentum_part(t, counts.data(), w.a, w.tmp, w.mu, A, sample(s), tau, w.kws, w.kws_b, st);
        if (rc) break;
        if (s + 1 < nsteps) rc = potential(t, w.tmp, w.a, E, sample(s), sample(s + 1), 0.5 * tau, st);
        else rc = potential(t, w.tmp, x, E, sample(s), -1, 0.5 * tau, st);
    }
    return rc;
}

extern "C" int dsbt_tdse_observable(const dsbt_tdse* t, const void* psi, double r_cut, double* out,
                                    void* stream) {
    DSBT_CHECK_ARG(t != nullptr && psi != nullptr && out != nullptr, "tdse: NULL argument");
    cudaStream_t st = (cudaStream_t)stream;
    DSBT_CUDA_TRY(cudaMemsetAsync(out, 0, sizeof(double), st));
    return observable(t, (const double2*)psi, nullptr, r_cut, out, st);
}

extern "C" int dsbt_tdse_gradient(const dsbt_tdse* t, const void* psi0, const double* E, int nsamples,
                                  int nsteps, int hold, double r_cut, int checkpoint_every, double* O,
                                  double* dOdE, void* workspace, size_t workspace_bytes, void* stream) {
    const int K = checkpoint_every;
    DSBT_CHECK_ARG(K >= 1, "tdse: checkpoint_every must be >= 1");
    int rc = check_run(t, psi0, E, nsteps, hold, workspace, workspace_bytes, K);
    if (rc) return rc;
    DSBT_CHECK_ARG(O != nullptr && dOdE != nullptr, "tdse: NULL output");
    DSBT_CHECK_ARG(nsamples >= (nsteps + hold - 1) / hold, "tdse: nsamples < ceil(nsteps / hold)");
    cudaStream_t st = (cudaStream_t)stream;
    TdseWs w;
    ws_layout(t, nsteps, K, &w, workspace);
    const size_t sb = state_bytes(t);
    const size_t sstride = a256(sb) / sizeof(double2);
    std::vector<int> counts(t->plan->l_max + 1, 0);
    for (int l = 0; l < t->L; ++l) counts[t->m0 + l] = 1;
    const double tau = t->tau, ht = 0.5 * tau;
    DSBT_CUDA_TRY(cudaMemsetAsync(O, 0, sizeof(double), st));
    DSBT_CUDA_TRY(cudaMemsetAsync(dOdE, 0, (size_t)nsamples * sizeof(double), st));
    if (nsteps == 0) return observable(t, (const double2*)psi0, nullptr, r_cut, O, st);
    auto smp = [&](int s) { return s / hold; };
    auto kin = [&](const double2* x, double2* y) { return kinetic(t, counts.data(), x, y, w.kws, w.kws_b, st); };
    // forward sweep: a_s = Q_s psi_s, b_s = Kin a_s = psi_{s+1} before its half step;
    // checkpoint k holds b_{kK-1} (k = 0: psi_0)
    rc = kinetic_phase_fill(t->plan, w.kws, t->L, tau, st);
    if (rc) return rc;
    DSBT_CUDA_TRY(cudaMemcpyAsync(w.ckpt, psi0, sb, cudaMemcpyDeviceToDevice, st));
    rc = potential(t, (const double2*)psi0, w.a, E, smp(0), -1, ht, st);
    const double2* b = w.tmp;   // b_s of the latest step
    for (int s = 0; s < nsteps && !rc; ++s) {
        double2* to = (s + 1 < nsteps && (s + 1) % K == 0) ? w.ckpt + (size_t)((s + 1) / K) * sstride : w.tmp;
        rc = kin(w.a, to);
        b = to;
        if (!rc && s + 1 < nsteps) rc = potential(t, b, w.a, E, smp(s), smp(s + 1), ht, st);
    }
    // psi_S, the observable, lambda_S = Pi psi_S and mu = Q_{S-1}^H lambda_S
    if (!rc) rc = potential(t, b, w.lam, E, smp(nsteps - 1), -1, ht, st);
    if (!rc) rc = observable(t, w.lam, w.mu, r_cut, O, st);
    if (!rc) rc = potential(t, w.mu, w.mu, E, smp(nsteps - 1), -1, -ht, st);
    if (rc) return rc;
    // backward sweep, one checkpoint segment at a time
    const int nseg = (nsteps + K - 1) / K;
    for (int seg = nseg - 1; seg >= 0; --seg) {
        const int s0 = seg * K, s1 = (s0 + K < nsteps) ? s0 + K : nsteps;
        auto grid = [&](int s) { return w.seg + (size_t)(s - s0) * sstride; };   // P^T a_s
        const double2* ck = w.ckpt + (size_t)seg * sstride;
        if (seg < nseg - 1) rc = kinetic_phase_fill(t->plan, w.kws, t->L, tau, st);   // (the adjoint's table is in place)
        if (!rc)
            rc = s0 == 0 ? potential(t, ck, w.a, E, smp(0), -1, ht, st, grid(0))
                         : potential(t, ck, w.a, E, smp(s0 - 1), smp(s0), ht, st, grid(s0));
        for (int s = s0; s + 1 < s1 && !rc; ++s) {
            rc = kin(w.a, w.tmp);
            if (!rc) rc = potential(t, w.tmp, w.a, E, smp(s), smp(s + 1), ht, st, grid(s + 1));
        }
        if (!rc) rc = kinetic_phase_fill(t->plan, w.kws, t->L, -tau, st);
        for (int s = s1 - 1; s >= s0 && !rc; --s) {
            rc = kin(w.mu, w.nu);   // nu_s
            if (rc) break;
            // g_s into dO/dE_s and dO/dE_{s-1}; mu = Q_{s-1}^H Q_s^H nu_s
            double* g = dOdE + smp(s);
            rc = s > 0 ? potential(t, w.nu, w.mu, E, smp(s), smp(s - 1), -ht, st, nullptr, grid(s), tau, g,
                                   dOdE + smp(s - 1))
                       : potential(t, w.nu, nullptr, E, 0, -1, -ht, st, nullptr, grid(0), tau, g, nullptr);
        }
        if (rc) return rc;
    }
    return DSBT_OK;
}
