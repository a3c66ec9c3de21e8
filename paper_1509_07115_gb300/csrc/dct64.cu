// dct64.cu -- FP64 sine / cosine transforms on power-of-two grids, for calls of
// any number of channels (the transform itself as in dct_kernels.cuh).
//
// The FP64 units bound the transform: a quarter of an SM takes 76 clocks for one
// FP64 instruction of a warp (measured: 1.7 lanes per clock and SM), so a line of N
// points at 47 operations a point needs 15 us per 1024 points on a whole SM, and
// four times that on one warp.  A line therefore wants four full warps on each SM it
// uses, and a call with fewer lines than SMs wants several SMs a line:
//   EPT  elements per thread (16, 8 or 4: also the radix of the stages; fewer
//        elements make more warps of the same work)
//   CL   CTAs of a line, a thread-block cluster
// Elements are owned by columns: with T = N / EPT, thread lt holds the elements
// lt + r T, and every Stockham stage reads exactly a thread's own column (radix R:
// butterflies j = lt + u T, inputs j + r N / R, all lt modulo T).  A stage therefore
// only stores: each output goes to the shared memory of the CTA that owns its
// column, two buffers in turn, and one (cluster) barrier a stage is all that orders
// them.  The first stage takes its inputs straight from global memory, the last
// one leaves its outputs in the owner's registers: the inverse stores them to
// global memory, the forward exchanges columns lt and T - lt once for the
// post-processing.
//
// Measured on a GB300, forward / inverse (before: one 16-element-a-thread kernel per
// line, and its shared-memory passes): 32 channels of 1024 points 30 / 31 -> 17 / 16 us
// (two CTAs of 128 threads a line), 64 of 2048 points 33 / 34 -> 25 / 25 us (two of
// 256), 4 real lines of 1024 points 29 -> 16 us, 1024 channels of 2048 points 207 ->
// 200 / 195 us (the FP64 pipe's rate).  Spreading a line over 4 CTAs of half a warp
// each, or 16 elements a thread over 2 CTAs, gained nothing: the warps count.
#include "dct_kernels.cuh"

namespace dsbt {

namespace {

template <int CL>
__device__ __forceinline__ unsigned cluster_rank() {
    if (CL == 1) return 0;
    unsigned r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}

template <int CL>
__device__ __forceinline__ void line_sync() {
    if (CL == 1) {
        __syncthreads();
    } else {
        asm volatile("barrier.cluster.arrive.release.aligned;\nbarrier.cluster.wait.acquire.aligned;" ::: "memory");
    }
}

__device__ __forceinline__ uint32_t remote(const double2* p, unsigned rank) {
    uint32_t a = (uint32_t)__cvta_generic_to_shared(p), r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(rank));
    return r;
}

// Column owners: element i = row T + col belongs to CTA col / TC, at row TC + col % TC there.
template <int N, int CL, int EPT>
struct Columns {
    static constexpr int T = N / EPT, TC = T / CL;
    static constexpr int LEN = EPT * TC + EPT * TC / 16;   // padded elements of one buffer
    // radices: EPT as often as it goes, then REM
    static constexpr int log2(int n) { return n <= 1 ? 0 : 1 + log2(n / 2); }
    static constexpr int STAGES = log2(N) / log2(EPT), REM = 1 << (log2(N) % log2(EPT));
    static constexpr int EXCHANGES = STAGES - 1 + (REM > 1);

    static __device__ __forceinline__ void store(double2* buf, int i, double2 v) {
        const int col = i % T, at = padi((i / T) * TC + col % TC);
        if (CL == 1) {
            buf[at] = v;
        } else {
            asm volatile("st.shared::cluster.v2.f64 [%0], {%1, %2};" ::"r"(remote(buf + at, col / TC)), "d"(v.x), "d"(v.y)
                         : "memory");
        }
    }
    static __device__ __forceinline__ double2 load(const double2* buf, int i) {
        const int col = i % T, at = padi((i / T) * TC + col % TC);
        if (CL == 1) return buf[at];
        double2 v;
        asm volatile("ld.shared::cluster.v2.f64 {%0, %1}, [%2];"
                     : "=d"(v.x), "=d"(v.y)
                     : "r"(remote(buf + at, col / TC))
                     : "memory");
        return v;
    }
    // Row of x[e] after fft.
    static __device__ __forceinline__ constexpr int row_of(int e) {
        constexpr int RX = REM > 1 ? REM : EPT;
        return e / RX + (e % RX) * (EPT / RX);
    }

    // One stage of radix RX on the thread's column x (x[r] = element lt + r T).  Ls:
    // length of the finished sub-transforms.  x[u RX + q] becomes output q of butterfly u.
    template <int RX>
    static __device__ __forceinline__ void stage(double2* x, const double2* __restrict__ tw, int Ls, int lt) {
        constexpr int PER = EPT / RX;
        double2 y[EPT];
#pragma unroll
        for (int u = 0; u < PER; ++u) {
            const int k = (lt + u * T) & (Ls - 1), b = k * (N / (Ls * RX));
            double2* z = y + u * RX;
#pragma unroll
            for (int r = 0; r < RX; ++r) z[r] = x[u + r * PER];   // element j + r N / RX: row u + r PER
            if (Ls > 1) {
#pragma unroll
                for (int r = 1; r < RX; ++r) z[r] = cmul(z[r], tw[r * b]);
            }
            if (RX == 16) dft16(z);
            else if (RX == 8) dft8(z);
            else if (RX == 4) dft4(z[0], z[1], z[2], z[3]);
            else dft2(z[0], z[1]);
        }
#pragma unroll
        for (int r = 0; r < EPT; ++r) x[r] = y[r];
    }

    // Forward FFT of the column-owned line; x[e] ends as row row_of(e) of the column.
    static __device__ __forceinline__ void fft(double2* x, double2* bufs, const double2* __restrict__ tw, int lt) {
        const int col = lt % TC;
        int Ls = 1;
#pragma unroll
        for (int st = 0; st < STAGES; ++st) {
            stage<EPT>(x, tw, Ls, lt);
            if (st < EXCHANGES) {
                double2* buf = bufs + (st & 1) * LEN;
                const int k = lt & (Ls - 1), base = (lt - k) * EPT + k;
#pragma unroll
                for (int q = 0; q < EPT; ++q) store(buf, base + q * Ls, x[q]);
                line_sync<CL>();
#pragma unroll
                for (int r = 0; r < EPT; ++r) x[r] = buf[padi(r * TC + col)];
            }
            Ls *= EPT;
        }
        if constexpr (REM > 1) stage<REM>(x, tw, Ls, lt);
    }
};

struct LineAt {
    int l, line;
    size_t chan;
};

__device__ __forceinline__ LineAt line_at(const GroupTable& g, int chan, int cplx) {
    const int gi = find_group(g, chan), local = chan - g.chan0[gi];
    return {g.l[gi], g.line0[gi] + (cplx ? 2 * local : local), (size_t)chan};
}

template <int N, int CL, int EPT>
__global__ void __launch_bounds__(N / EPT / CL) k_dct64_fwd(const __grid_constant__ GroupTable g, int cplx,
                                                           const double* __restrict__ in, double* __restrict__ out,
                                                           const double2* __restrict__ tw,
                                                           const double2* __restrict__ post, DctScale<double> dsc) {
    using C = Columns<N, CL, EPT>;
    constexpr int T = N / EPT;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    double2* bufs = reinterpret_cast<double2*>(smem_raw);
    const unsigned rank = cluster_rank<CL>();
    const int lt = (int)rank * C::TC + threadIdx.x;
    const LineAt at = line_at(g, blockIdx.x / CL, cplx);
    const bool even = (at.l & 1) == 0;
    // v_i = x_{2i} for i < N / 2, x_{2(N-1-i)+1} (negated for even l) beyond
    double2 x[EPT];
#pragma unroll
    for (int r = 0; r < EPT; ++r) {
        const int i = lt + r * T, p = r < EPT / 2 ? 2 * i : 2 * (N - 1 - i) + 1;
        if (cplx) {
            const double* q = in + (at.chan * N + p) * 2;
            x[r] = make_double2(q[0], q[1]);
        } else {
            x[r] = make_double2(in[at.chan * N + p], 0.0);
        }
        if (r >= EPT / 2 && even) { x[r].x = -x[r].x; x[r].y = -x[r].y; }
    }
    if (CL > 1) line_sync<CL>();   // every CTA of the cluster runs before its memory is written
    C::fft(x, bufs, tw, lt);
    // columns lt and T - lt meet: V_k, V_{N-k} -> X_k, X_{N-k} (see k_dct_fwd)
    double2* buf = bufs + (C::EXCHANGES & 1) * C::LEN;
#pragma unroll
    for (int e = 0; e < EPT; ++e) buf[padi(C::row_of(e) * C::TC + (int)threadIdx.x)] = x[e];
    line_sync<CL>();
    double* o = out + (size_t)at.line * N;
    const double half = 0.5 * dsc.c1;
#pragma unroll
    for (int i = 0; i < EPT / 2; ++i) {   // k = lt + i T < N / 2
        const int k = lt + i * T;
        int k1 = N - k;
        const double2 a = buf[padi(i * C::TC + (int)threadIdx.x)];
        double2 X0, X1;
        if (k == 0) {   // its own partner; this thread also takes k = N / 2
            const double2 vh = buf[padi(EPT / 2 * C::TC)];
            const double h = 0.70710678118654752440 * dsc.c1;
            X0 = make_double2(a.x * dsc.c0, a.y * dsc.c0);
            X1 = make_double2(vh.x * h, vh.y * h);
            k1 = N / 2;
        } else {
            const double2 b = C::load(buf, N - k);
            double2 w = post[k];
            w.x *= half;
            w.y *= half;
            const double2 A = cmul(a, w), B = cmulc(b, w), D = csub(A, B);
            X0 = cadd(A, B);
            X1 = make_double2(-D.y, D.x);
        }
        const int i0 = even ? N - 1 - k : k, i1 = even ? N - 1 - k1 : k1;
        o[i0] = X0.x;
        o[i1] = X1.x;
        if (cplx) {
            o[N + i0] = X0.y;
            o[N + i1] = X1.y;
        }
    }
    if (CL > 1) line_sync<CL>();   // no CTA leaves while its columns are read
}

template <int N, int CL, int EPT>
__global__ void __launch_bounds__(N / EPT / CL) k_dct64_inv(const __grid_constant__ GroupTable g, int cplx,
                                                           const double* __restrict__ in, double* __restrict__ out,
                                                           const double2* __restrict__ tw,
                                                           const double2* __restrict__ post, DctScale<double> dsc) {
    using C = Columns<N, CL, EPT>;
    constexpr int T = N / EPT;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    double2* bufs = reinterpret_cast<double2*>(smem_raw);
    const unsigned rank = cluster_rank<CL>();
    const int lt = (int)rank * C::TC + threadIdx.x;
    const LineAt at = line_at(g, blockIdx.x / CL, cplx);
    const bool even = (at.l & 1) == 0;
    const double* li = in + (size_t)at.line * N;
    // conj(V_k), V_k = conj(w_k) (X_k - i X_{N-k}), k = lt + r T
    double2 x[EPT];
#pragma unroll
    for (int r = 0; r < EPT; ++r) {
        const int k = lt + r * T, s0 = even ? N - 1 - k : k, s1 = even ? k - 1 : N - k;
        double2 a = make_double2(li[s0], 0.0), b = make_double2(0.0, 0.0);
        if (k > 0) b.x = li[s1];
        if (cplx) {
            a.y = li[N + s0];
            if (k > 0) b.y = li[N + s1];
        }
        double2 w = post[k];
        const double sc = k == 0 ? dsc.c0 : dsc.c1;
        w.x *= sc;
        w.y *= sc;
        const double2 v = cmulc(make_double2(a.x + b.y, a.y - b.x), w);
        x[r] = make_double2(v.x, -v.y);
    }
    if (CL > 1) line_sync<CL>();
    C::fft(x, bufs, tw, lt);
#pragma unroll
    for (int e = 0; e < EPT; ++e) {
        const int i = lt + C::row_of(e) * T, p = i < N / 2 ? 2 * i : 2 * (N - 1 - i) + 1;
        const bool neg = even && i >= N / 2;
        const double re = neg ? -x[e].x : x[e].x, im = neg ? x[e].y : -x[e].y;
        if (cplx) {
            double* q = out + (at.chan * N + p) * 2;
            q[0] = re;
            q[1] = im;
        } else {
            out[at.chan * N + p] = re;
        }
    }
}

using Kernel64 = void (*)(GroupTable, int, const double*, double*, const double2*, const double2*, DctScale<double>);

template <int N, int CL, int EPT>
int launch64(bool fwd, const dsbt_plan* p, const GroupTable& g, bool cplx, const double* in, double* out,
             cudaStream_t st) {
    using C = Columns<N, CL, EPT>;
    const Kernel64 k = fwd ? (Kernel64)k_dct64_fwd<N, CL, EPT> : (Kernel64)k_dct64_inv<N, CL, EPT>;
    constexpr size_t smem = 2 * (size_t)C::LEN * sizeof(double2);
    static_assert(smem <= 227 * 1024, "the two buffers of a CTA's columns");
    if (smem > 48 * 1024)
        if (int rc = ensure_smem((const void*)k, smem)) return rc;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((unsigned)nchannels(g) * CL);
    cfg.blockDim = dim3(C::TC);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = CL;
    at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = CL > 1 ? 1 : 0;
    DSBT_CUDA_TRY(cudaLaunchKernelEx(&cfg, k, g, cplx ? 1 : 0, in, out, (const double2*)p->tw64,
                                     (const double2*)p->post64, fwd ? fwd_scale(N) : inv_scale(N)));
    return DSBT_OK;
}

// As many CTAs a line as still have an SM each and 128 threads, and at least as many
// as hold the line's two buffers: 278 KB at N = 8192, so two there for any number of
// channels (100: 134 / 142 us, 1000: 899 / 957 us).  EPT is fixed per grid, so a channel's bits do not depend on how many
// channels a call has.
template <int N>
int launch_n(bool fwd, const dsbt_plan* p, const GroupTable& g, bool cplx, const double* in, double* out,
             cudaStream_t st) {
    constexpr int EPT = N >= 8192 ? 8 : 4, T = N / EPT;
    const int n = nchannels(g);
    if constexpr (T >= 1024)
        if (8 * n <= kSMs) return launch64<N, 8, EPT>(fwd, p, g, cplx, in, out, st);
    if constexpr (T >= 512)
        if (4 * n <= kSMs) return launch64<N, 4, EPT>(fwd, p, g, cplx, in, out, st);
    if constexpr (T >= 256)
        if (2 * n <= kSMs) return launch64<N, 2, EPT>(fwd, p, g, cplx, in, out, st);
    return launch64<N, N >= 8192 ? 2 : 1, EPT>(fwd, p, g, cplx, in, out, st);
}

}  // namespace

bool dct64_supported(int N) { return N >= 256 && N <= 8192 && (N & (N - 1)) == 0; }

int dct64(bool fwd, const dsbt_plan* p, const GroupTable& g, bool cplx, const double* in, double* out,
          cudaStream_t st) {
    switch (p->N) {
        case 256: return launch_n<256>(fwd, p, g, cplx, in, out, st);
        case 512: return launch_n<512>(fwd, p, g, cplx, in, out, st);
        case 1024: return launch_n<1024>(fwd, p, g, cplx, in, out, st);
        case 2048: return launch_n<2048>(fwd, p, g, cplx, in, out, st);
        case 4096: return launch_n<4096>(fwd, p, g, cplx, in, out, st);
        case 8192: return launch_n<8192>(fwd, p, g, cplx, in, out, st);
    }
    set_error("dct64: N=%d not a power of two in 256..8192", p->N);
    return DSBT_ERR_INVALID;
}

}  // namespace dsbt
