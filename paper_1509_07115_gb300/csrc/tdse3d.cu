// tdse3d.cu -- the full DSBT-DVR split-operator step (Sec. 4.1): all m at once,
// angular transform Y = P Phi over a (theta, phi) grid, length gauge with a
// field of any direction.
//
// Channels (l, m): m = -M .. M and, for each m, l = |m| .. |m| + L - 1 (the
// per-m range of the fixed-m propagator, so every P^m below is square),
// stored l-major as the DSBT's grouped calls want them (channel c -> line c).
// Angular grid: the L-point Gauss-Legendre nodes eta_j = cos(theta_j) and
// NM = 2M + 1 uniform angles phi_q = 2 pi q / NM.  The transform of Sec. 4.1
// in two factors:
//     G_m(eta_j)      = sum_l P^m[l - |m|][j] psi_lm          (P^m: Pbar_l^|m| sqrt(w_j),
//                                                               orthonormalised on the rule)
//     g(eta_j, phi_q) = sum_m Phi[m][q] G_m(eta_j),   Phi[m][q] = exp(i m phi_q) / sqrt(NM)
// Both factors are orthogonal / unitary, so Y is unitary on the channel space.
// One step of length tau (vector potential 0, the kinetic half steps merged):
//     psi <- Q Kin Q psi,   Q = Y^H diag exp(-i [V(r) + r F.n(theta, phi)] tau/2) Y,
//     Kin = the grouped DSBT kinetic step (each channel with its own l),
// with n = (sin theta cos phi, sin theta sin phi, cos theta) and F the field
// sample of the step (three components).  A field along z couples no m, and the
// step then equals the fixed-m propagator's for every m.
//
// Adjacent half steps share the grid and Y is unitary, so Q_{s+1} Q_s = Y^H diag
// exp(-i [2 V + r (F_s + F_{s+1}).n] tau/2) Y is one pass; a propagation has single
// passes at its ends only.
//
// Adjoint (the gradient of O = sum_{r_i > r_cut} |psi_S|^2 over the field samples):
// with a_s = Q_s psi_s, lambda_S = Pi psi_S (Pi the mask r_i > r_cut), nu_s =
// Kin^H Q_s^H lambda_{s+1} and lambda_s = Q_s^H nu_s, the derivative by the
// component F_c is
//     dO/dF_{s,c} = tau Im <Y lambda_{s+1}, r n_c Y psi_{s+1}> + tau Im <Y nu_s, r n_c Y a_s>.
// The diagonal r n_c commutes with Q_s on the grid, so the second term is g_{s,c} =
// Im <Y lambda_s, r n_c Y psi_s> and the first g_{s+1,c} (g_S = 0: lambda_S = Pi
// psi_S): dO/dF_s = tau (g_s + g_{s+1}), with g_s = Im <Y nu_s, r n_c Y a_s> from the
// grid values of a_s that the forward pass of a segment stores.
#include <math.h>

#include <algorithm>
#include <new>
#include <vector>

#include "mm64.cuh"
#include "plan.cuh"

struct dsbt_tdse3d {
    const dsbt_plan* plan;
    int L, M, NM, N, nchan;
    double tau;
    uint2* Pw;        // [M + 1][2][32][32] fixed-point words (mm64.cuh) of P^|m| (row i = l - |m|, column j):
                      // P^T by node pairs, then P
    int* map;         // [NM][L]: channel of (l = |m| + i, m)
    int* lch;         // [nchan]: l of each channel
    double* V;        // [N]
    double* rr;       // [N]
    double* eta;      // [L]
    std::vector<int> counts;            // channels per l, l = 0 .. plan l_max
    std::vector<int> chan_l, chan_m;    // per channel
};

namespace dsbt {
namespace {

constexpr int TI3 = 4;    // radial points per block of the angular kernels: 8 real columns
constexpr int L3 = 32;     // the largest L
constexpr int AB3 = L3 + 16;   // halfs per digit row (mm64.cuh)
constexpr int DIG3 = mm64::ND * 2 * TI3 * AB3;   // halfs of one warp's digits

struct Angular3 {
    const uint2* Pw;
    const int* map;     // [NM][L]: channel of (l = |m| + i, m)
    const double* eta;
    int L, M, N;
};

// Shared memory: G[NM][L][TI3] and g[L][NM][TI3] complex (the warps' digits in place of g),
// cos and sin of 2 pi k / NM, and per node pair and point the phase of all but the field
// across z.
__host__ __device__ inline size_t grid3(int L, int NM) { return (size_t)NM * L * TI3 * sizeof(double2); }
__host__ __device__ inline size_t second3(int L, int NM) {
    const size_t d = 4 * (size_t)DIG3 * sizeof(__half), g = grid3(L, NM);
    return d > g ? d : g;
}
inline size_t smem3d(int L, int NM) {
    return grid3(L, NM) + second3(L, NM) + (size_t)NM * sizeof(double2) + (size_t)L3 * TI3 * sizeof(double2);
}

__device__ __forceinline__ double2 cmul3(double2 a, double2 b) {
    return make_double2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);
}

// One m block: digits of the warp's values (lane = 4 kq + t holds rows 4 kq .. 4 kq + 3 of
// point t) and the product with the words A[32][32]; put(row, t, value) takes the results.
template <class Put>
__device__ __forceinline__ void m_block(const double2* v, const uint2* A, __half* dig, int L, int lane, Put&& put) {
    const int t = lane & 3, kq = lane >> 2;
    const double re[4] = {v[0].x, v[1].x, v[2].x, v[3].x}, im[4] = {v[0].y, v[1].y, v[2].y, v[3].y};
    int er = mm64::exponent4(re), ei = mm64::exponent4(im);
#pragma unroll
    for (int o = 4; o < 32; o <<= 1) {
        er = max(er, __shfl_xor_sync(0xffffffffu, er, o));
        ei = max(ei, __shfl_xor_sync(0xffffffffu, ei, o));
    }
    __syncwarp();   // the digits of the block before are used up
    mm64::put_digits4(dig + (2 * t) * AB3 + 4 * kq, 2 * TI3 * AB3, re, er);
    mm64::put_digits4(dig + (2 * t + 1) * AB3 + 4 * kq, 2 * TI3 * AB3, im, ei);
    __syncwarp();
    const int units = (L + 15) / 16, tq = lane & 3, g = lane >> 2;
    // lane tq's columns 2 tq, 2 tq + 1 are point tq: its scales are this lane's own
    for (int b = 0; b < units; ++b) {
        long long hi[1][4], lo[1][4];
        mm64::block_product<1>(A + (size_t)b * 16 * L3, L3, units, dig, AB3, lane, hi, lo);
        put(16 * b + g, tq, make_double2(mm64::to_double(hi[0][0], lo[0][0], er), mm64::to_double(hi[0][1], lo[0][1], ei)));
        put(16 * b + g + 8, tq, make_double2(mm64::to_double(hi[0][2], lo[0][2], er), mm64::to_double(hi[0][3], lo[0][3], ei)));
    }
}

// Node of row r of the P^T words (rows g and g + 8 of a 16-row block: node 8 b + g and its
// mirror), or -1.
__host__ __device__ inline int pair_node(int r, int L) {
    const int j = 8 * (r / 16) + r % 8;
    if (j >= (L + 1) / 2) return -1;
    const int node = (r & 8) ? L - 1 - j : j;
    return (r & 8) && node == j ? -1 : node;
}

// G -> G = Y^H D Y G on the block's points, with the phi sums written out in real
// arithmetic: the DFT of NM = 2M + 1 angles works on the sums and differences of m and -m
// (and of the angles q and -q), a quarter of the products of complex sums, and one sine
// and cosine of each of a = r st Fx cos phi_q +- r st Fy sin phi_q serves a node and its
// mirror.  zph[j][t]: exp(-i u) / NM with u the phase of everything that does not depend on
// phi.  ab = (ax, ay): the phase of an angle is rad[t] st (ax cos phi + ay sin phi).
// grid_out / grid_in: as in k_tdse3d_potential; returns the thread's part of the sums.
__device__ __forceinline__ void phi_part(const Angular3& a, double2* G, double2* g, const double2* cs, const double2* zph,
                                         const double* rad, double ax, double ay, int i0, double2* grid_out,
                                         const double2* __restrict__ grid_in, double* gsum) {
    const int L = a.L, M = a.M, NM = 2 * M + 1, tid = threadIdx.x, half = (L + 1) / 2;
    // sums and differences of m and -m (in place: m takes the sum, -m the difference)
    for (int k = tid; k < M * L * TI3; k += blockDim.x) {
        const int m = 1 + k / (L * TI3), c = k % (L * TI3);
        double2 &p = G[(M + m) * L * TI3 + c], &n = G[(M - m) * L * TI3 + c];
        const double2 x = p, y = n;
        p = make_double2(x.x + y.x, x.y + y.y);
        n = make_double2(x.x - y.x, x.y - y.y);
    }
    __syncthreads();
    // task: a node pair, a point and q in 0 .. M (angles q and -q)
    for (int k = tid; k < half * TI3 * (M + 1); k += blockDim.x) {
        const int t = k % TI3, j = (k / TI3) % half, q = k / (TI3 * half), jm = L - 1 - j;
        double2 v[2][2];   // [node, mirror][q, -q]
#pragma unroll
        for (int s = 0; s < 2; ++s) {
            const double2* col = G + (s ? jm : j) * TI3 + t;
            double2 A = col[M * L * TI3], B = make_double2(0.0, 0.0);
            int e = 0;
            for (int m = 1; m <= M; ++m) {   // A += (G_m + G_-m) cos, B += (G_m - G_-m) sin (times i)
                e += q;
                if (e >= NM) e -= NM;
                const double2 w = cs[e], p = col[(M + m) * L * TI3], d = col[(M - m) * L * TI3];
                A.x = fma(w.x, p.x, A.x);
                A.y = fma(w.x, p.y, A.y);
                B.x = fma(w.y, d.x, B.x);
                B.y = fma(w.y, d.y, B.y);
            }
            v[s][0] = make_double2(A.x - B.y, A.y + B.x);
            v[s][1] = make_double2(A.x + B.y, A.y - B.x);
        }
        const double ct = a.eta[j], st = sqrt(fmax(0.0, 1.0 - ct * ct)), cp = cs[q].x, sp = cs[q].y;
        const size_t at = ((size_t)j * NM + q) * a.N + i0 + t, atm = ((size_t)jm * NM + q) * a.N + i0 + t,
                     neg = (size_t)(q ? NM - 2 * q : 0) * a.N;   // from angle q to -q
        if (grid_in) {
            const double r = rad[t];
            auto part = [&](double2 x, double2 y) { return r * (x.x * y.y - x.y * y.x); };
            const double w0 = part(v[0][0], grid_in[at]), w1 = q ? part(v[0][1], grid_in[at + neg]) : 0.0;
            const double u0 = jm != j ? part(v[1][0], grid_in[atm]) : 0.0,
                         u1 = jm != j && q ? part(v[1][1], grid_in[atm + neg]) : 0.0;
            gsum[0] += st * cp * ((w0 + w1) + (u0 + u1));
            gsum[1] += st * sp * ((w0 - w1) + (u0 - u1));
            gsum[2] += ct * ((w0 + w1) - (u0 + u1));
        }
        const double x = rad[t] * st * ax * cp, y = rad[t] * st * ay * sp;
        double s0, c0, s1, c1;
        sincos(x + y, &s0, &c0);
        if (q) sincos(x - y, &s1, &c1);
        else s1 = s0, c1 = c0;
#pragma unroll
        for (int s = 0; s < 2; ++s) {
            if (s && jm == j) break;
            const double2 z = zph[(s ? jm : j) * TI3 + t];
            const double2 h0 = cmul3(cmul3(v[s][0], z), make_double2(c0, s0));
            const double2 h1 = cmul3(cmul3(v[s][1], z), make_double2(c1, s1));
            double2* o = g + (size_t)((s ? jm : j) * NM) * TI3 + t;
            if (grid_out) {
                grid_out[s ? atm : at] = h0;
                if (q) grid_out[(s ? atm : at) + neg] = h1;
            }
            if (q == 0) {
                o[0] = h0;
            } else {
                o[q * TI3] = make_double2(h0.x + h1.x, h0.y + h1.y);
                o[(NM - q) * TI3] = make_double2(h0.x - h1.x, h0.y - h1.y);
            }
        }
    }
    __syncthreads();
    // back over phi: G_m = sum_q exp(-i m phi_q) h_q, m and -m together
    for (int k = tid; k < L * TI3 * (M + 1); k += blockDim.x) {
        const int t = k % TI3, j = (k / TI3) % L, m = k / (TI3 * L);
        const double2* col = g + (size_t)j * NM * TI3 + t;
        double2 A = col[0], B = make_double2(0.0, 0.0);
        int e = 0;
        for (int q = 1; q <= M; ++q) {
            e += m;
            if (e >= NM) e -= NM;
            const double2 w = cs[e], p = col[q * TI3], d = col[(NM - q) * TI3];
            A.x = fma(w.x, p.x, A.x);
            A.y = fma(w.x, p.y, A.y);
            B.x = fma(w.y, d.x, B.x);
            B.y = fma(w.y, d.y, B.y);
        }
        G[((size_t)(M + m) * L + j) * TI3 + t] = make_double2(A.x + B.y, A.y - B.x);
        if (m) G[((size_t)(M - m) * L + j) * TI3 + t] = make_double2(A.x - B.y, A.y + B.x);
    }
    __syncthreads();
}

__device__ __forceinline__ void cos_table(double2* cs, int NM) {
    for (int k = threadIdx.x; k < NM; k += blockDim.x) {
        double sn, c;
        sincospi(2.0 * (double)k / NM, &sn, &c);
        cs[k] = make_double2(c, sn);
    }
}

// y = Y^H diag(exp(-i [w V + r (F_f1 + F_f2).n] ht)) Y x on TI3 radial points per block
// (w = 2, or w = 1 and no second sample for f2 < 0; x and y may alias; y may be null).
// grid_out: also stores the grid values [L][NM][N] after the phase, divided by NM.
// grid_in (values stored so): adds gscale * sum Im(conj(Y x) r n_c Y aux) into g1[c] and,
// unless null, g2[c], c = x, y, z.  The P^m products run on the tensor cores through
// exact digits, one m a warp.  What bounds it is the FP64 pipe: the phi sums and the sines.
__global__ void __launch_bounds__(128) k_tdse3d_potential(const double2* x, double2* y, const __grid_constant__ Angular3 a,
                                                          const double* __restrict__ V, const double* __restrict__ rr,
                                                          const double* __restrict__ F, int f1, int f2, double ht,
                                                          double2* grid_out, const double2* __restrict__ grid_in,
                                                          double gscale, double* g1, double* g2) {
    extern __shared__ __align__(16) unsigned char sm[];
    const int L = a.L, M = a.M, NM = 2 * M + 1, N = a.N, tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    double2* G = reinterpret_cast<double2*>(sm);
    double2* g = reinterpret_cast<double2*>(sm + grid3(L, NM));
    __half* dig = reinterpret_cast<__half*>(g) + (size_t)warp * DIG3;
    double2* cs = reinterpret_cast<double2*>(sm + grid3(L, NM) + second3(L, NM));
    double2* zph = cs + NM;
    __shared__ double red[3][4], rad[TI3];
    const int i0 = blockIdx.x * TI3, t = lane & 3, kq = lane >> 2;
    double f[3] = {0.0, 0.0, 0.0};
    if (F)
        for (int c = 0; c < 3; ++c) f[c] = F[3 * f1 + c] + (f2 >= 0 ? F[3 * f2 + c] : 0.0);
    cos_table(cs, NM);
    for (int k = tid; k < L * TI3; k += blockDim.x) {
        const int j = k / TI3, i = i0 + k % TI3;
        double sn, c;
        // (w V + r F_z eta) ht with the w at ht: 2 V may pass the largest number
        sincos(-(V[i] + (f2 >= 0 ? 0.5 : 1.0) * rr[i] * f[2] * a.eta[j]) * (f2 >= 0 ? 2.0 * ht : ht), &sn, &c);
        zph[k] = make_double2(c / NM, sn / NM);
    }
    if (tid < TI3) rad[tid] = rr[i0 + tid];
    for (int mi = warp; mi < NM; mi += 4) {   // G_m(eta_j) = sum_l P^m x_lm
        double2 v[4];
#pragma unroll
        for (int c = 0; c < 4; ++c)
            v[c] = 4 * kq + c < L ? x[(size_t)a.map[mi * L + 4 * kq + c] * N + i0 + t] : make_double2(0.0, 0.0);
        m_block(v, a.Pw + (size_t)abs(mi - M) * 2 * L3 * L3, dig, L, lane, [&](int r, int tp, double2 w) {
            const int j = pair_node(r, L);
            if (j >= 0) G[((size_t)mi * L + j) * TI3 + tp] = w;
        });
    }
    __syncthreads();
    double gs[3] = {0.0, 0.0, 0.0};
    phi_part(a, G, g, cs, zph, rad, -f[0] * ht, -f[1] * ht, i0, grid_out, grid_in, gs);
    if (grid_in) {   // block sums of the three components
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            for (int o = 16; o > 0; o >>= 1) gs[c] += __shfl_xor_sync(0xffffffffu, gs[c], o);
            if (lane == 0) red[c][warp] = gs[c];
        }
        __syncthreads();
        if (tid < 3) {
            const double s = gscale * (red[tid][0] + red[tid][1] + red[tid][2] + red[tid][3]);
            atomicAdd(g1 + tid, s);
            if (g2) atomicAdd(g2 + tid, s);
        }
    }
    if (!y) return;
    for (int mi = warp; mi < NM; mi += 4) {   // back over theta: psi_lm = sum_j P^m G_m
        double2 v[4];
#pragma unroll
        for (int c = 0; c < 4; ++c)
            v[c] = 4 * kq + c < L ? G[((size_t)mi * L + 4 * kq + c) * TI3 + t] : make_double2(0.0, 0.0);
        m_block(v, a.Pw + ((size_t)abs(mi - M) * 2 + 1) * L3 * L3, dig, L, lane, [&](int r, int tp, double2 w) {
            if (r < L) y[(size_t)a.map[mi * L + r] * N + i0 + tp] = w;
        });
    }
}

// The momentum-space middle of the velocity-gauge step (Eq. (81)) with all m,
// in place on the DSBT coefficients c[ch][s] at TI3 momentum slots
// n = 1..N per block (k~_n = n dk; storage s = n - 1 for even l, s = n for odd
// l with n = N at s = 0): the half kinetic phase exp(-i k^2 tau/4) with the
// plan's momentum of (l, s) (half_phase: the kinetic phase table of tau / 2);
// phi = Ytilde^H c with the factors (-i)^l s_l = 1 (even l) or i (odd l) of the
// modified harmonics (s_l: this library's sine/cosine signs); phi *= exp(i k~_n
// (A . n) tau) on the (theta, phi) grid; c = Ytilde phi with i^l s_l = 1 or -i; the
// half kinetic phase again.
__global__ void __launch_bounds__(128) k_tdse3d_velocity(double2* c, const __grid_constant__ Angular3 a,
                                                         const int* __restrict__ lch,
                                                         const double2* __restrict__ half_phase, int per_l, double dk,
                                                         const double* __restrict__ A, int aidx, double tau) {
    extern __shared__ __align__(16) unsigned char sm[];
    const int L = a.L, M = a.M, NM = 2 * M + 1, N = a.N, tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    double2* G = reinterpret_cast<double2*>(sm);
    double2* g = reinterpret_cast<double2*>(sm + grid3(L, NM));
    __half* dig = reinterpret_cast<__half*>(g) + (size_t)warp * DIG3;
    double2* cs = reinterpret_cast<double2*>(sm + grid3(L, NM) + second3(L, NM));
    double2* zph = cs + NM;
    __shared__ double rad[TI3];
    const int n0 = 1 + blockIdx.x * TI3, t = lane & 3, kq = lane >> 2;
    double f[3] = {0.0, 0.0, 0.0};
    if (A)
        for (int q = 0; q < 3; ++q) f[q] = A[3 * aidx + q];
    cos_table(cs, NM);
    for (int k = tid; k < L * TI3; k += blockDim.x) {
        double sn, cc;
        sincos(f[2] * a.eta[k / TI3] * ((n0 + k % TI3) * dk) * tau, &sn, &cc);
        zph[k] = make_double2(cc / NM, sn / NM);
    }
    if (tid < TI3) rad[tid] = (n0 + tid) * dk;
    auto slot = [&](int ch, int l, int n, double2& ph) {   // storage of momentum n, and its half kinetic phase
        const int sidx = (l & 1) ? (n % N) : n - 1;
        ph = per_l ? half_phase[(size_t)l * N + sidx] : half_phase[(size_t)(l & 1) * N + phase_entry(l, sidx, N)];
        return (size_t)ch * N + sidx;
    };
    for (int mi = warp; mi < NM; mi += 4) {   // gather, half kinetic phase, (-i)^l s_l
        double2 v[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            v[q] = make_double2(0.0, 0.0);
            if (4 * kq + q < L) {
                const int ch = a.map[mi * L + 4 * kq + q], l = lch[ch];
                double2 ph;
                const size_t at = slot(ch, l, n0 + t, ph);
                v[q] = cmul3(c[at], ph);
                if (l & 1) v[q] = make_double2(-v[q].y, v[q].x);   // times i
            }
        }
        m_block(v, a.Pw + (size_t)abs(mi - M) * 2 * L3 * L3, dig, L, lane, [&](int r, int tp, double2 w) {
            const int j = pair_node(r, L);
            if (j >= 0) G[((size_t)mi * L + j) * TI3 + tp] = w;
        });
    }
    __syncthreads();
    phi_part(a, G, g, cs, zph, rad, f[0] * tau, f[1] * tau, 0, nullptr, nullptr, nullptr);
    for (int mi = warp; mi < NM; mi += 4) {   // back to (l, m), i^l s_l, half phase, scatter
        double2 v[4];
#pragma unroll
        for (int q = 0; q < 4; ++q)
            v[q] = 4 * kq + q < L ? G[((size_t)mi * L + 4 * kq + q) * TI3 + t] : make_double2(0.0, 0.0);
        m_block(v, a.Pw + ((size_t)abs(mi - M) * 2 + 1) * L3 * L3, dig, L, lane, [&](int r, int tp, double2 w) {
            if (r >= L) return;
            const int ch = a.map[mi * L + r], l = lch[ch];
            if (l & 1) w = make_double2(w.y, -w.x);   // times -i
            double2 ph;
            const size_t at = slot(ch, l, n0 + tp, ph);
            c[at] = cmul3(w, ph);
        });
    }
}

Angular3 angular3(const dsbt_tdse3d* t) { return Angular3{t->Pw, t->map, t->eta, t->L, t->M, t->N}; }

// One angular pass with the samples f1 and (merged half steps) f2 >= 0; see k_tdse3d_potential.
int potential3d(const dsbt_tdse3d* t, const double2* x, double2* y, const double* F, int f1, int f2, double ht,
                cudaStream_t st, double2* grid_out = nullptr, const double2* grid_in = nullptr, double gscale = 0.0,
                double* g1 = nullptr, double* g2 = nullptr) {
    const size_t smem = smem3d(t->L, t->NM);
    if (smem > 48 * 1024)
        if (int rc0 = ensure_smem((const void*)k_tdse3d_potential, smem)) return rc0;
    ProfScope ps(kKTdsePot, st);
    k_tdse3d_potential<<<t->N / TI3, 128, smem, st>>>(x, y, angular3(t), t->V, t->rr, F, f1, f2, ht, grid_out, grid_in,
                                                      gscale, g1, g2);
    DSBT_CUDA_TRY(cudaGetLastError());
    return DSBT_OK;
}

// *out += sum over r_i > r_cut of |x|^2 (all channels); with mask != nullptr
// also mask = x on r_i > r_cut and 0 elsewhere (the adjoint start Pi psi_S).
__global__ void k_tdse3d_observable(const double2* __restrict__ x, double2* __restrict__ mask,
                                    const double* __restrict__ rr, int N, long long total, double r_cut,
                                    double* out) {
    double acc = 0.0;
    for (long long k = (long long)blockIdx.x * blockDim.x + threadIdx.x; k < total;
         k += (long long)gridDim.x * blockDim.x) {
        const bool in = rr[k % N] > r_cut;
        const double2 v = x[k];
        if (in) acc += v.x * v.x + v.y * v.y;
        if (mask) mask[k] = in ? v : make_double2(0.0, 0.0);
    }
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
    __shared__ double red[8];
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = acc;
    __syncthreads();
    if (threadIdx.x == 0) {
        double tsum = 0.0;
        for (int w = 0; w < (int)(blockDim.x >> 5); ++w) tsum += red[w];
        atomicAdd(out, tsum);
    }
}

int observable3d(const dsbt_tdse3d* t, const double2* x, double2* mask, double r_cut, double* out, cudaStream_t st) {
    const long long total = (long long)t->nchan * t->N;
    ProfScope ps(kKTdseReduce, st);
    k_tdse3d_observable<<<256, 256, 0, st>>>(x, mask, t->rr, t->N, total, r_cut, out);
    DSBT_CUDA_TRY(cudaGetLastError());
    return DSBT_OK;
}

// Half kinetic phases from the table of tau / 2 in the workspace.
int velocity3d(const dsbt_tdse3d* t, double2* c, const double* A, int aidx, void* kws, cudaStream_t st) {
    const size_t smem = smem3d(t->L, t->NM);
    if (smem > 48 * 1024)
        if (int rc0 = ensure_smem((const void*)k_tdse3d_velocity, smem)) return rc0;
    ProfScope ps(kKTdseAng, st);
    k_tdse3d_velocity<<<t->N / TI3, 128, smem, st>>>(c, angular3(t), t->lch, kinetic_phase_table(t->plan, kws, t->nchan),
                                                     t->plan->knl != nullptr, t->plan->dk, A, aidx, t->tau);
    DSBT_CUDA_TRY(cudaGetLastError());
    return DSBT_OK;
}

inline size_t a256(size_t x) { return (x + 255) & ~(size_t)255; }

}  // namespace
}  // namespace dsbt

using namespace dsbt;

extern "C" int dsbt_tdse3d_create(const dsbt_plan* plan, int L, int M, double tau, dsbt_tdse3d** out) {
    DSBT_CHECK_ARG(out != nullptr && plan != nullptr, "dsbt_tdse3d_create: NULL argument");
    *out = nullptr;
    DSBT_CHECK_ARG(plan->T64 != nullptr, "dsbt_tdse3d_create: the plan needs DSBT_PLAN_FP64");
    DSBT_CHECK_ARG(L >= 1 && L <= 32, "dsbt_tdse3d_create: L=%d not in 1..32", L);
    DSBT_CHECK_ARG(M >= 0 && M <= 12, "dsbt_tdse3d_create: M=%d not in 0..12", M);
    DSBT_CHECK_ARG(M + L - 1 <= plan->l_max, "dsbt_tdse3d_create: channels up to l=%d, plan l_max=%d", M + L - 1,
                   plan->l_max);
    DSBT_CHECK_ARG(isfinite(tau), "dsbt_tdse3d_create: tau must be finite");
    dsbt_tdse3d* t = new (std::nothrow) dsbt_tdse3d();
    if (!t) return DSBT_ERR_NOMEM;
    t->plan = plan;
    t->L = L;
    t->M = M;
    t->NM = 2 * M + 1;
    t->N = plan->N;
    t->tau = tau;
    // channels, l-major
    std::vector<int> map((size_t)t->NM * L, -1);
    t->counts.assign(plan->l_max + 1, 0);
    for (int l = 0; l <= M + L - 1; ++l)
        for (int mi = 0; mi < t->NM; ++mi) {
            const int m = mi - M, am = m < 0 ? -m : m;
            if (l < am || l > am + L - 1) continue;
            map[(size_t)mi * L + (l - am)] = (int)t->chan_l.size();
            t->chan_l.push_back(l);
            t->chan_m.push_back(m);
            ++t->counts[l];
        }
    t->nchan = (int)t->chan_l.size();
    std::vector<double> x, w, Pm, rr(t->N);
    tdse_gauss_legendre(L, x, w);
    std::vector<uint2> Pw((size_t)(M + 1) * 2 * L3 * L3, mm64::fixed_a_host(0.0));
    for (int m = 0; m <= M; ++m) {
        tdse_angular_rows(L, m, x, w, Pm);
        uint2* pt = Pw.data() + (size_t)m * 2 * L3 * L3;
        for (int r = 0; r < L3; ++r) {
            const int node = pair_node(r, L);
            for (int k = 0; k < L; ++k) {
                if (node >= 0) pt[r * L3 + k] = mm64::fixed_a_host(Pm[(size_t)k * L + node]);
                if (r < L) pt[(L3 + r) * L3 + k] = mm64::fixed_a_host(Pm[(size_t)r * L + k]);
            }
        }
    }
    const double dr = plan->r_max / plan->N;
    for (int i = 0; i < t->N; ++i) rr[i] = (i + 0.5) * dr;
    bool ok = cudaMalloc((void**)&t->Pw, Pw.size() * sizeof(uint2)) == cudaSuccess &&
              cudaMalloc((void**)&t->map, map.size() * sizeof(int)) == cudaSuccess &&
              cudaMalloc((void**)&t->lch, t->nchan * sizeof(int)) == cudaSuccess &&
              cudaMalloc((void**)&t->V, t->N * sizeof(double)) == cudaSuccess &&
              cudaMalloc((void**)&t->rr, t->N * sizeof(double)) == cudaSuccess &&
              cudaMalloc((void**)&t->eta, L * sizeof(double)) == cudaSuccess;
    ok = ok && cudaMemcpy(t->Pw, Pw.data(), Pw.size() * sizeof(uint2), cudaMemcpyHostToDevice) == cudaSuccess &&
         cudaMemcpy(t->map, map.data(), map.size() * sizeof(int), cudaMemcpyHostToDevice) == cudaSuccess &&
         cudaMemcpy(t->lch, t->chan_l.data(), t->nchan * sizeof(int), cudaMemcpyHostToDevice) == cudaSuccess &&
         cudaMemset(t->V, 0, t->N * sizeof(double)) == cudaSuccess &&
         cudaMemcpy(t->rr, rr.data(), t->N * sizeof(double), cudaMemcpyHostToDevice) == cudaSuccess &&
         cudaMemcpy(t->eta, x.data(), L * sizeof(double), cudaMemcpyHostToDevice) == cudaSuccess;
    if (!ok) {
        cudaGetLastError();
        cudaFree(t->Pw); cudaFree(t->map); cudaFree(t->lch); cudaFree(t->V); cudaFree(t->rr); cudaFree(t->eta);
        delete t;
        set_error("dsbt_tdse3d_create: device allocation or copy failed");
        return DSBT_ERR_NOMEM;
    }
    *out = t;
    return DSBT_OK;
}

extern "C" int dsbt_tdse3d_destroy(dsbt_tdse3d* t) {
    if (!t) return DSBT_OK;
    cudaDeviceSynchronize();
    cudaFree(t->Pw);
    cudaFree(t->map);
    cudaFree(t->lch);
    cudaFree(t->V);
    cudaFree(t->rr);
    cudaFree(t->eta);
    delete t;
    return DSBT_OK;
}

extern "C" int dsbt_tdse3d_channels(const dsbt_tdse3d* t, int* nchan, int* l_of, int* m_of) {
    DSBT_CHECK_ARG(t != nullptr, "dsbt_tdse3d_channels: NULL handle");
    if (nchan) *nchan = t->nchan;
    for (int c = 0; c < t->nchan; ++c) {
        if (l_of) l_of[c] = t->chan_l[c];
        if (m_of) m_of[c] = t->chan_m[c];
    }
    return DSBT_OK;
}

extern "C" int dsbt_tdse3d_set_potential(dsbt_tdse3d* t, const double* V, int n) {
    DSBT_CHECK_ARG(t != nullptr && V != nullptr, "dsbt_tdse3d_set_potential: NULL argument");
    DSBT_CHECK_ARG(n == t->N, "dsbt_tdse3d_set_potential: n=%d, grid has N=%d", n, t->N);
    DSBT_CUDA_TRY(cudaMemcpy(t->V, V, t->N * sizeof(double), cudaMemcpyHostToDevice));
    return DSBT_OK;
}

extern "C" size_t dsbt_tdse3d_workspace_size(const dsbt_tdse3d* t) {
    if (!t) return 0;
    return 2 * a256((size_t)t->nchan * t->N * sizeof(double2)) +
           dsbt_workspace_size(t->plan, t->nchan, DSBT_C128) + 512;
}

extern "C" int dsbt_tdse3d_propagate(const dsbt_tdse3d* t, void* psi, const double* F, int nsteps, int hold,
                                     void* workspace, size_t workspace_bytes, void* stream) {
    DSBT_CHECK_ARG(t != nullptr && psi != nullptr, "dsbt_tdse3d_propagate: NULL argument");
    DSBT_CHECK_ARG(nsteps >= 0 && hold >= 1, "dsbt_tdse3d_propagate: nsteps >= 0 and hold >= 1 required");
    const size_t need = dsbt_tdse3d_workspace_size(t);
    DSBT_CHECK_ARG(workspace != nullptr && workspace_bytes >= need,
                   "dsbt_tdse3d_propagate: workspace too small (need %zu bytes)", need);
    cudaStream_t st = (cudaStream_t)stream;
    unsigned char* base = (unsigned char*)(((uintptr_t)workspace + 255) & ~(uintptr_t)255);
    double2* tmp = (double2*)base;
    void* kws = base + 2 * a256((size_t)t->nchan * t->N * sizeof(double2));
    const size_t kws_b = dsbt_workspace_size(t->plan, t->nchan, DSBT_C128);
    double2* x = (double2*)psi;
    if (nsteps == 0) return DSBT_OK;
    int rc = kinetic_phase_fill(t->plan, kws, t->nchan, t->tau, st);
    if (!rc) rc = potential3d(t, x, tmp, F, 0, -1, 0.5 * t->tau, st);
    for (int s = 0; s < nsteps && !rc; ++s) {
        rc = grouped_device_call(kKineticReady, t->plan, t->counts.data(), DSBT_C128, 0.0, tmp, x, kws, kws_b, st);
        if (rc) break;
        if (s + 1 < nsteps) rc = potential3d(t, x, tmp, F, s / hold, (s + 1) / hold, 0.5 * t->tau, st);
        else rc = potential3d(t, x, x, F, s / hold, -1, 0.5 * t->tau, st);
    }
    return rc;
}

extern "C" int dsbt_tdse3d_propagate_velocity(const dsbt_tdse3d* t, void* psi, const double* F, const double* A,
                                              int nsteps, int hold, void* workspace, size_t workspace_bytes,
                                              void* stream) {
    DSBT_CHECK_ARG(t != nullptr && psi != nullptr, "dsbt_tdse3d_propagate_velocity: NULL argument");
    DSBT_CHECK_ARG(nsteps >= 0 && hold >= 1, "dsbt_tdse3d_propagate_velocity: nsteps >= 0 and hold >= 1 required");
    const size_t need = dsbt_tdse3d_workspace_size(t);
    DSBT_CHECK_ARG(workspace != nullptr && workspace_bytes >= need,
                   "dsbt_tdse3d_propagate_velocity: workspace too small (need %zu bytes)", need);
    cudaStream_t st = (cudaStream_t)stream;
    const size_t sb = a256((size_t)t->nchan * t->N * sizeof(double2));
    unsigned char* base = (unsigned char*)(((uintptr_t)workspace + 255) & ~(uintptr_t)255);
    double2* tmp = (double2*)base;
    double2* c = (double2*)(base + sb);
    void* kws = base + 2 * sb;
    const size_t kws_b = dsbt_workspace_size(t->plan, t->nchan, DSBT_C128);
    double2* x = (double2*)psi;
    if (nsteps == 0) return DSBT_OK;
    int rc = kinetic_phase_fill(t->plan, kws, t->nchan, 0.5 * t->tau, st);
    if (!rc) rc = potential3d(t, x, tmp, F, 0, -1, 0.5 * t->tau, st);
    for (int s = 0; s < nsteps && !rc; ++s) {
        rc = grouped_device_call(0, t->plan, t->counts.data(), DSBT_C128, 0.0, tmp, c, kws, kws_b, st);
        if (!rc) rc = velocity3d(t, c, A, s / hold, kws, st);
        if (!rc) rc = grouped_device_call(1, t->plan, t->counts.data(), DSBT_C128, 0.0, c, x, kws, kws_b, st);
        if (rc) break;
        if (s + 1 < nsteps) rc = potential3d(t, x, tmp, F, s / hold, (s + 1) / hold, 0.5 * t->tau, st);
        else rc = potential3d(t, x, x, F, s / hold, -1, 0.5 * t->tau, st);
    }
    return rc;
}

namespace dsbt {
namespace {

// Gradient workspace: nsteps / K + 1 checkpoints, a segment of K + 1 states,
// four more states (a, mu, nu, lambda), one DSBT workspace.
size_t grad3d_layout(const dsbt_tdse3d* t, int nsteps, int K, double2** ck, double2** seg, double2** a, double2** mu,
                     double2** nu, double2** lam, void** kws, void* base) {
    const size_t sb = a256((size_t)t->nchan * t->N * sizeof(double2));
    const size_t nck = (size_t)nsteps / K + 1;
    unsigned char* p = (unsigned char*)(((uintptr_t)base + 255) & ~(uintptr_t)255);
    size_t off = 0;
    auto take = [&](size_t b) { unsigned char* q = p + off; off += a256(b); return q; };
    unsigned char* c0 = take(sb * nck);
    unsigned char* s0 = take(sb * (K + 1));
    unsigned char* a0 = take(sb);
    unsigned char* m0 = take(sb);
    unsigned char* n0 = take(sb);
    unsigned char* l0 = take(sb);
    unsigned char* k0 = take(dsbt_workspace_size(t->plan, t->nchan, DSBT_C128));
    if (base) {
        *ck = (double2*)c0; *seg = (double2*)s0; *a = (double2*)a0; *mu = (double2*)m0; *nu = (double2*)n0;
        *lam = (double2*)l0; *kws = k0;
    }
    return off + 256;
}

}  // namespace
}  // namespace dsbt

extern "C" size_t dsbt_tdse3d_gradient_workspace_size(const dsbt_tdse3d* t, int nsteps, int checkpoint_every) {
    if (!t || nsteps < 0 || checkpoint_every < 1) return 0;
    return grad3d_layout(t, nsteps, checkpoint_every, nullptr, nullptr, nullptr, nullptr, nullptr, nullptr, nullptr,
                         nullptr);
}

extern "C" int dsbt_tdse3d_gradient(const dsbt_tdse3d* t, const void* psi0, const double* F, int nsamples, int nsteps,
                                    int hold, double r_cut, int checkpoint_every, double* O, double* dOdF,
                                    void* workspace, size_t workspace_bytes, void* stream) {
    DSBT_CHECK_ARG(t != nullptr && psi0 != nullptr && F != nullptr && O != nullptr && dOdF != nullptr,
                   "dsbt_tdse3d_gradient: NULL argument");
    const int K = checkpoint_every;
    DSBT_CHECK_ARG(K >= 1 && nsteps >= 0 && hold >= 1, "dsbt_tdse3d_gradient: K >= 1, nsteps >= 0, hold >= 1");
    DSBT_CHECK_ARG(nsamples >= (nsteps + hold - 1) / hold, "dsbt_tdse3d_gradient: nsamples < ceil(nsteps / hold)");
    const size_t need = dsbt_tdse3d_gradient_workspace_size(t, nsteps, K);
    DSBT_CHECK_ARG(workspace != nullptr && workspace_bytes >= need,
                   "dsbt_tdse3d_gradient: workspace too small (need %zu bytes)", need);
    cudaStream_t st = (cudaStream_t)stream;
    double2 *ck, *seg, *a, *mu, *nu, *lam;
    void* kws;
    grad3d_layout(t, nsteps, K, &ck, &seg, &a, &mu, &nu, &lam, &kws, workspace);
    const size_t kws_b = dsbt_workspace_size(t->plan, t->nchan, DSBT_C128);
    const size_t sb = (size_t)t->nchan * t->N * sizeof(double2);
    const size_t stride = a256(sb) / sizeof(double2);
    const double tau = t->tau, ht = 0.5 * tau;
    const int* counts = t->counts.data();
    DSBT_CUDA_TRY(cudaMemsetAsync(O, 0, sizeof(double), st));
    DSBT_CUDA_TRY(cudaMemsetAsync(dOdF, 0, (size_t)3 * nsamples * sizeof(double), st));
    if (nsteps == 0) return observable3d(t, (const double2*)psi0, nullptr, r_cut, O, st);
    auto smp = [&](int s) { return s / hold; };
    auto kin = [&](const double2* x, double2* y) {
        return grouped_device_call(kKineticReady, t->plan, counts, DSBT_C128, 0.0, x, y, kws, kws_b, st);
    };
    // forward sweep: a_s = Q_s psi_s, b_s = Kin a_s = psi_{s+1} before its half step;
    // checkpoint k holds b_{kK-1} (k = 0: psi_0)
    int rc = kinetic_phase_fill(t->plan, kws, t->nchan, tau, st);
    if (rc) return rc;
    DSBT_CUDA_TRY(cudaMemcpyAsync(ck, psi0, sb, cudaMemcpyDeviceToDevice, st));
    rc = potential3d(t, (const double2*)psi0, a, F, smp(0), -1, ht, st);
    const double2* b = nu;   // b_s of the latest step
    for (int s = 0; s < nsteps && !rc; ++s) {
        double2* to = (s + 1 < nsteps && (s + 1) % K == 0) ? ck + (size_t)((s + 1) / K) * stride : nu;
        rc = kin(a, to);
        b = to;
        if (!rc && s + 1 < nsteps) rc = potential3d(t, b, a, F, smp(s), smp(s + 1), ht, st);
    }
    // psi_S, the observable, lambda_S = Pi psi_S and mu = Q_{S-1}^H lambda_S
    if (!rc) rc = potential3d(t, b, lam, F, smp(nsteps - 1), -1, ht, st);
    if (!rc) rc = observable3d(t, lam, mu, r_cut, O, st);
    if (!rc) rc = potential3d(t, mu, mu, F, smp(nsteps - 1), -1, -ht, st);
    if (rc) return rc;
    // backward sweep, one checkpoint segment at a time
    const int nseg = (nsteps + K - 1) / K;
    for (int sg = nseg - 1; sg >= 0; --sg) {
        const int s0 = sg * K, s1 = (s0 + K < nsteps) ? s0 + K : nsteps;
        auto grid = [&](int s) { return seg + (size_t)(s - s0) * stride; };   // grid values of a_s
        const double2* c = ck + (size_t)sg * stride;
        if (sg < nseg - 1) rc = kinetic_phase_fill(t->plan, kws, t->nchan, tau, st);   // (the adjoint's table is in place)
        if (!rc)
            rc = s0 == 0 ? potential3d(t, c, a, F, smp(0), -1, ht, st, grid(0))
                         : potential3d(t, c, a, F, smp(s0 - 1), smp(s0), ht, st, grid(s0));
        for (int s = s0; s + 1 < s1 && !rc; ++s) {
            rc = kin(a, nu);
            if (!rc) rc = potential3d(t, nu, a, F, smp(s), smp(s + 1), ht, st, grid(s + 1));
        }
        if (!rc) rc = kinetic_phase_fill(t->plan, kws, t->nchan, -tau, st);
        for (int s = s1 - 1; s >= s0 && !rc; --s) {
            rc = kin(mu, nu);   // nu_s
            if (rc) break;
            // g_s into dO/dF_s and dO/dF_{s-1}; mu = Q_{s-1}^H Q_s^H nu_s
            double* g = dOdF + 3 * (size_t)smp(s);
            rc = s > 0 ? potential3d(t, nu, mu, F, smp(s), smp(s - 1), -ht, st, nullptr, grid(s), tau, g,
                                     dOdF + 3 * (size_t)smp(s - 1))
                       : potential3d(t, nu, nullptr, F, 0, -1, -ht, st, nullptr, grid(0), tau, g, nullptr);
        }
        if (rc) return rc;
    }
    return DSBT_OK;
}
