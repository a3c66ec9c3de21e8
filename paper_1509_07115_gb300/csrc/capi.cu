// capi.cu -- C ABI entry points: argument checks, group tables, workspace
// layout, and the kernel sequence of each call.
//
//   forward  (Eqs. (18), (24)):  in -> F_l (sine/cosine kernel) -> T_l contraction -> out
//   inverse  (Eq. (25)):         in -> T_l^T contraction -> F_l^T kernel -> out
//   kinetic  (Eq. (81), A = 0):  in -> F_l -> T_l with exp(-i k~^2 tau/2) in the
//                                epilogue -> T_l^T -> F_l^T -> out
#include <math.h>

#include <algorithm>

#include "plan.cuh"

namespace dsbt {

namespace {

// TF32 split of caller data into planar lines (complex channel c -> lines 2c, 2c+1).
__global__ void k_split_lines(const float* __restrict__ in, float* __restrict__ hi, float* __restrict__ lo,
                              long long total) {
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= total) return;
    const float v = in[i];
    const float h = round_tf32(v);
    hi[i] = h;
    lo[i] = round_tf32(v - h);
}

__global__ void k_split_lines_c(const float2* __restrict__ in, float* __restrict__ hi,
                                float* __restrict__ lo, int N, long long total) {
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= total) return;
    const long long c = i / N, n = i % N;
    const float2 v = in[i];
    const float hr = round_tf32(v.x), hi_ = round_tf32(v.y);
    const size_t o = (size_t)(2 * c) * N + n;
    hi[o] = hr;
    lo[o] = round_tf32(v.x - hr);
    hi[o + N] = hi_;
    lo[o + N] = round_tf32(v.y - hi_);
}

// FP16 pair of caller data for the interval-scheme contraction: one CTA per
// channel (N values, or N complex values = two lines) computes ||psi||, picks
// 2^e with ||2^e psi|| in [2^12, 2^13) and writes hi = fp16(2^e x),
// lo = fp16(2^e x - hi) to the channel's planar lines and 2^-e to scale[line].
// HBM-bound when it streams: the channel is read once, 16 bytes a load where the
// caller's alignment allows (VEC), and held in registers between the norm and the
// stores (reading it twice in 4-byte loads took 30 us for 1271 real channels of 6400
// points; now 23 us).
constexpr int kSplitThreads = 256, kSplitChunks = 16;   // at most: chunks of 4 floats, 16384 floats (complex N = 8192)

template <bool CPLX, bool VEC>
__global__ void __launch_bounds__(kSplitThreads) k_split_f16(const float* __restrict__ in, int N, __half* __restrict__ hi,
                                                             __half* __restrict__ lo, float* __restrict__ scale) {
    const long long c = blockIdx.x;
    const int n4 = N * (CPLX ? 2 : 1) / 4;
    const float* x = in + c * (long long)n4 * 4;
    float4 v[kSplitChunks];
    float part = 0.f;
#pragma unroll
    for (int q = 0; q < kSplitChunks; ++q) {
        const int i = threadIdx.x + q * blockDim.x;
        if (i < n4) {
            if (VEC) v[q] = reinterpret_cast<const float4*>(x)[i];
            else v[q] = make_float4(x[4 * i], x[4 * i + 1], x[4 * i + 2], x[4 * i + 3]);
            part += (v[q].x * v[q].x + v[q].y * v[q].y) + (v[q].z * v[q].z + v[q].w * v[q].w);
        }
    }
    __shared__ float red[32];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) part += __shfl_xor_sync(0xffffffffu, part, o);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = part;
    __syncthreads();
    float sum = 0.f;
#pragma unroll
    for (int w = 0; w < kSplitThreads / 32; ++w)
        if (w < (int)(blockDim.x >> 5)) sum += red[w];
    const float nrm = sqrtf(sum);
    const int e = (nrm > 0.f && isfinite(nrm)) ? 12 - ilogbf(nrm) : 0;
    const float fs = ldexpf(1.f, e);
    const long long line = c * (CPLX ? 2 : 1);
    if (threadIdx.x < (CPLX ? 2 : 1)) scale[line + threadIdx.x] = ldexpf(1.f, -e);
    auto pair = [&](size_t at, float a, float b) {   // two consecutive points of a line
        const float2 f = make_float2(a * fs, b * fs);
        const __half2 h = __float22half2_rn(f);
        *reinterpret_cast<__half2*>(hi + at) = h;
        *reinterpret_cast<__half2*>(lo + at) = __float22half2_rn(make_float2(f.x - __low2float(h), f.y - __high2float(h)));
    };
#pragma unroll
    for (int q = 0; q < kSplitChunks; ++q) {
        const int i = threadIdx.x + q * blockDim.x;
        if (i >= n4) break;
        if (CPLX) {
            const size_t at = (size_t)line * N + 2 * i;
            pair(at, v[q].x, v[q].z);
            pair(at + N, v[q].y, v[q].w);
        } else {
            const size_t at = (size_t)line * N + 4 * i;
            pair(at, v[q].x, v[q].y);
            pair(at + 2, v[q].z, v[q].w);
        }
    }
}

// exp(-i k~_n^2 tau / 2) on the unified momentum grid (Eq. (65)): storage index
// k of parity class par (0: even l, n = k + 1; 1: odd l, n = k) maps to
// k~ = n dk, except the odd-l coefficient n = 0, which takes k~_N = N dk.
// Kinetic phase table exp(-i k^2 tau / 2): rows = 2 by parity of l with
// k = k~_n = n dk (n = 0 -> N dk) when knl is NULL, else rows = l_max + 1 with
// the plan's corrected momenta knl[l][s].
__global__ void k_phase(double2* ph64, float2* ph32, int N, double dk, double tau, const double* __restrict__ knl,
                        int rows) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= rows * N) return;
    double kt;
    if (knl) {
        kt = knl[i];
    } else {
        const int par = i / N, k = i % N;
        int n = (par == 0) ? k + 1 : k;
        if (n == 0) n = N;
        kt = n * dk;
    }
    double s, c;
    sincos(-0.5 * kt * kt * tau, &s, &c);
    if (ph64) ph64[i] = make_double2(c, s);
    if (ph32) ph32[i] = make_float2((float)c, (float)s);
}

// One warp per quarter of an SM: its sines are bound by the FP64 pipe.
constexpr int kPhaseThreads = 128;

// Rows of the phase table (see k_phase).
inline int phase_rows(const dsbt_plan* p) { return p->knl ? p->l_max + 1 : 2; }

inline size_t align256(size_t x) { return (x + 255) & ~(size_t)255; }

struct Workspace {
    // FP64 path
    double* f64a;
    double* f64b;
    double2* ph64;
    double* fast;    // scratch of the DSBT_PLAN_FAST64 contraction (or nullptr)
    // TF32 path
    float* hi_a;
    float* lo_a;
    float* hi_b;
    float* lo_b;
    float* planar;   // aliases hi_a
    float2* ph32;
    int* sched;      // tile-scheduler counter of the tensor-core contraction
    // interval-scheme path (plans with DSBT_PLAN_FAST_SPLIT): FP16 pairs of the
    // lines before (a) and between (b) the contractions, per-line unscale
    // factors, the augmented lines; planar aliases the a pair
    __half* h_hi_a;
    __half* h_lo_a;
    __half* h_hi_b;
    __half* h_lo_b;
    float* scale;
    void* ftc;
};

size_t lines_of(int total_channels, int dtype) {
    return (size_t)total_channels * (is_complex(dtype) ? 2 : 1);
}

size_t ws_bytes(const dsbt_plan* p, int total_channels, int dtype) {
    const size_t R = lines_of(total_channels, dtype);
    const int N = p->N;
    const size_t PR = (size_t)phase_rows(p) * N;
    if (is_fp64(dtype))
        return align256(R * N * sizeof(double)) * 2 + align256(PR * sizeof(double2)) +
               align256(fast_scratch_bytes(p, (int)R)) + 256;
    if (p->ftc)   // FP16 pairs a, b (4 B per value each), scale, phase, counter, augmented lines
        return align256(R * N * 4) * 2 + align256(R * sizeof(float)) + align256(PR * sizeof(float2)) + 256 +
               align256(ftc_scratch_bytes(p, R)) + 256;
    return align256(R * N * sizeof(float)) * 4 + align256(PR * sizeof(float2)) + 256 + 256;
}

Workspace carve(const dsbt_plan* pl, void* base, int total_channels, int dtype) {
    const int N = pl->N;
    const size_t PR = (size_t)phase_rows(pl) * N;
    Workspace w{};
    const size_t R = lines_of(total_channels, dtype);
    unsigned char* p = (unsigned char*)(((uintptr_t)base + 255) & ~(uintptr_t)255);
    if (is_fp64(dtype)) {
        const size_t b = align256(R * N * sizeof(double));
        w.f64a = (double*)p;
        w.f64b = (double*)(p + b);
        w.ph64 = (double2*)(p + 2 * b);
        w.fast = pl->fast ? (double*)(p + 2 * b + align256(PR * sizeof(double2))) : nullptr;
    } else if (pl->ftc) {
        const size_t b = align256(R * N * 4);   // one FP16 pair of every line
        w.h_hi_a = (__half*)p;
        w.h_lo_a = w.h_hi_a + R * N;
        w.planar = (float*)p;                   // FP32 lines after the last contraction
        w.h_hi_b = (__half*)(p + b);
        w.h_lo_b = w.h_hi_b + R * N;
        w.scale = (float*)(p + 2 * b);
        unsigned char* q = p + 2 * b + align256(R * sizeof(float));
        w.ph32 = (float2*)q;
        w.sched = (int*)(q + align256(PR * sizeof(float2)));
        w.ftc = q + align256(PR * sizeof(float2)) + 256;
    } else {
        const size_t b = align256(R * N * sizeof(float));
        w.hi_a = (float*)p;
        w.lo_a = (float*)(p + b);
        w.hi_b = (float*)(p + 2 * b);
        w.lo_b = (float*)(p + 3 * b);
        w.planar = w.hi_a;
        w.ph32 = (float2*)(p + 4 * b);
        w.sched = (int*)(p + 4 * b + align256(PR * sizeof(float2)));
    }
    return w;
}

int build_groups(const dsbt_plan* p, const int* counts, int ngroups_in, const int* ls, int dtype,
                 GroupTable& g) {
    g.ngroups = 0;
    int chan = 0, line = 0;
    const int per = is_complex(dtype) ? 2 : 1;
    for (int i = 0; i < ngroups_in; ++i) {
        const int c = counts[i];
        DSBT_CHECK_ARG(c >= 0, "negative channel count for l=%d", ls[i]);
        DSBT_CHECK_ARG(ls[i] >= 0 && ls[i] <= p->l_max, "l=%d outside the plan's 0..%d", ls[i], p->l_max);
        if (c == 0) continue;
        DSBT_CHECK_ARG(g.ngroups < kMaxGroups, "too many groups");
        DSBT_CHECK_ARG((long long)chan + c < (1LL << 30), "too many channels");
        g.l[g.ngroups] = ls[i];
        g.chan0[g.ngroups] = chan;
        g.line0[g.ngroups] = line;
        ++g.ngroups;
        chan += c;
        line += c * per;
    }
    g.chan0[g.ngroups] = chan;
    g.line0[g.ngroups] = line;
    g.total_lines = line;
    return DSBT_OK;
}

int check_common(const dsbt_plan* p, int dtype, const void* in, void* out, void* ws, size_t ws_b,
                 int total_channels) {
    DSBT_CHECK_ARG(p != nullptr, "plan is NULL");
    DSBT_CHECK_ARG(valid_dtype(dtype), "dtype=%d invalid", dtype);
    if (total_channels == 0) return DSBT_OK;
    DSBT_CHECK_ARG(in != nullptr && out != nullptr, "in/out is NULL");
    DSBT_CHECK_ARG(in != out, "in and out must not alias");
    DSBT_CHECK_ARG(ws != nullptr, "workspace is NULL");
    const size_t need = ws_bytes(p, total_channels, dtype);
    DSBT_CHECK_ARG(ws_b >= need, "workspace too small: %zu < %zu bytes", ws_b, need);
    if (is_fp64(dtype) && !p->T64) {
        set_error("FP64 dtype needs a plan built with DSBT_PLAN_FP64");
        return DSBT_ERR_UNSUPPORTED;
    }
    if (!is_fp64(dtype) && !p->has_tmaps && !p->ftc) {
        set_error("FP32 dtype needs a plan built with DSBT_PLAN_TF32X3 or DSBT_PLAN_FAST_SPLIT");
        return DSBT_ERR_UNSUPPORTED;
    }
    return DSBT_OK;
}

int run_forward(const dsbt_plan* p, const GroupTable& g, int dtype, const void* in, void* out,
                void* ws, cudaStream_t st) {
    if (g.total_lines == 0) return DSBT_OK;
    const bool cplx = is_complex(dtype);
    Workspace w = carve(p, ws, g.chan0[g.ngroups], dtype);
    int rc;
    if (is_fp64(dtype)) {
        rc = dct_forward_f64(p, g, cplx, (const double*)in, w.f64a, st);
        if (rc) return rc;
        return contract_f64(p, g, +1, w.f64a, 0, (double*)out, cplx ? 1 : 0, nullptr, st, w.fast);
    }
    if (p->ftc) {   // interval scheme on FP16 pairs
        rc = dct_forward_f16(p, g, cplx, (const float*)in, w.h_hi_a, w.h_lo_a, w.scale, st);
        if (rc) return rc;
        return contract_split_fast(p, g, +1, w.h_hi_a, w.h_lo_a, w.scale, cplx ? kOutUserC64 : kOutUserF32, out,
                                   nullptr, nullptr, w.ftc, st);
    }
    rc = dct_forward_f32(p, g, cplx, (const float*)in, w.hi_a, w.lo_a, st);
    if (rc) return rc;
    return contract_tf32x3(p, g, +1, w.hi_a, w.lo_a, cplx ? kOutUserC64 : kOutUserF32, (float*)out,
                           nullptr, nullptr, w.sched, st);
}

int run_inverse(const dsbt_plan* p, const GroupTable& g, int dtype, const void* in, void* out,
                void* ws, cudaStream_t st) {
    if (g.total_lines == 0) return DSBT_OK;
    const bool cplx = is_complex(dtype);
    Workspace w = carve(p, ws, g.chan0[g.ngroups], dtype);
    int rc;
    if (is_fp64(dtype)) {
        rc = contract_f64(p, g, -1, (const double*)in, cplx ? 1 : 0, w.f64a, 0, nullptr, st, w.fast);
        if (rc) return rc;
        return dct_inverse_f64(p, g, cplx, w.f64a, (double*)out, st);
    }
    if (p->ftc) {   // interval scheme on FP16 pairs
        {
            ProfScope ps(kKSplit, st);
            const bool vec = ((uintptr_t)in & 15) == 0;   // N is a multiple of 256: every channel starts alike
            const auto k = cplx ? (vec ? k_split_f16<true, true> : k_split_f16<true, false>)
                                : (vec ? k_split_f16<false, true> : k_split_f16<false, false>);
            // four chunks a thread where that leaves a warp, so that short channels fill theirs
            const int n4 = p->N * (cplx ? 2 : 1) / 4, th = std::min(kSplitThreads, std::max(32, n4 / 4 / 32 * 32));
            k<<<(unsigned)g.chan0[g.ngroups], th, 0, st>>>((const float*)in, p->N, w.h_hi_b, w.h_lo_b, w.scale);
        }
        DSBT_CUDA_TRY(cudaGetLastError());
        rc = contract_split_fast(p, g, -1, w.h_hi_b, w.h_lo_b, w.scale, kOutPlanarF32, w.planar, nullptr, nullptr,
                                 w.ftc, st);
        if (rc) return rc;
        return dct_inverse_f32(p, g, cplx, w.planar, (float*)out, st);
    }
    const long long total = (long long)g.chan0[g.ngroups] * p->N;
    const int bs = 256;
    {
    ProfScope ps(kKSplit, st);
    if (cplx)
        k_split_lines_c<<<(unsigned)((total + bs - 1) / bs), bs, 0, st>>>((const float2*)in, w.hi_b, w.lo_b,
                                                                          p->N, total);
    else
        k_split_lines<<<(unsigned)((total + bs - 1) / bs), bs, 0, st>>>((const float*)in, w.hi_b, w.lo_b,
                                                                        total);
    }
    DSBT_CUDA_TRY(cudaGetLastError());
    rc = contract_tf32x3(p, g, -1, w.hi_b, w.lo_b, kOutPlanarF32, w.planar, nullptr, nullptr, w.sched, st);
    if (rc) return rc;
    return dct_inverse_f32(p, g, cplx, w.planar, (float*)out, st);
}

int fill_phase64(const dsbt_plan* p, const Workspace& w, double tau, cudaStream_t st) {
    ProfScope ps(kKPhase, st);
    const int rows = phase_rows(p);
    k_phase<<<(rows * p->N + kPhaseThreads - 1) / kPhaseThreads, kPhaseThreads, 0, st>>>(w.ph64, nullptr, p->N, p->dk, tau, p->knl, rows);
    DSBT_CUDA_TRY(cudaGetLastError());
    return DSBT_OK;
}

// phase_ready (FP64): the workspace's table is already that of tau.
int run_kinetic(const dsbt_plan* p, const GroupTable& g, int dtype, double tau, const void* in, void* out,
                void* ws, cudaStream_t st, bool phase_ready = false) {
    if (g.total_lines == 0) return DSBT_OK;
    Workspace w = carve(p, ws, g.chan0[g.ngroups], dtype);
    const int N = p->N;
    int rc;
    if (is_fp64(dtype)) {
        rc = phase_ready ? DSBT_OK : fill_phase64(p, w, tau, st);
        if (!rc) rc = dct_forward_f64(p, g, true, (const double*)in, w.f64a, st);
        if (!rc) rc = contract_f64(p, g, +1, w.f64a, 0, w.f64b, 0, w.ph64, st, w.fast);
        if (!rc) rc = contract_f64(p, g, -1, w.f64b, 0, w.f64a, 0, nullptr, st, w.fast);
        if (!rc) rc = dct_inverse_f64(p, g, true, w.f64a, (double*)out, st);
        return rc;
    }
    {
        ProfScope ps(kKPhase, st);
        const int rows = phase_rows(p);
        k_phase<<<(rows * N + kPhaseThreads - 1) / kPhaseThreads, kPhaseThreads, 0, st>>>(nullptr, w.ph32, N, p->dk, tau, p->knl, rows);
    }
    DSBT_CUDA_TRY(cudaGetLastError());
    if (p->ftc) {   // interval scheme on FP16 pairs; the lines stay scaled until the last contraction
        rc = dct_forward_f16(p, g, true, (const float*)in, w.h_hi_a, w.h_lo_a, w.scale, st);
        if (!rc)
            rc = contract_split_fast(p, g, +1, w.h_hi_a, w.h_lo_a, w.scale, kOutPlanarSplit, w.h_hi_b, w.h_lo_b,
                                     w.ph32, w.ftc, st);
        if (!rc)
            rc = contract_split_fast(p, g, -1, w.h_hi_b, w.h_lo_b, w.scale, kOutPlanarF32, w.planar, nullptr,
                                     nullptr, w.ftc, st);
        if (!rc) rc = dct_inverse_f32(p, g, true, w.planar, (float*)out, st);
        return rc;
    }
    rc = dct_forward_f32(p, g, true, (const float*)in, w.hi_a, w.lo_a, st);
    if (!rc) rc = contract_tf32x3(p, g, +1, w.hi_a, w.lo_a, kOutPlanarSplit, w.hi_b, w.lo_b, w.ph32, w.sched, st);
    if (!rc) rc = contract_tf32x3(p, g, -1, w.hi_b, w.lo_b, kOutPlanarF32, w.planar, nullptr, nullptr, w.sched, st);
    if (!rc) rc = dct_inverse_f32(p, g, true, w.planar, (float*)out, st);
    return rc;
}

int grouped_call(int which, const dsbt_plan* p, const int* counts, int dtype, double tau, const void* in,
                 void* out, void* ws, size_t ws_b, void* stream, const long long* uoff = nullptr) {
    DSBT_CHECK_ARG(p != nullptr, "plan is NULL");
    DSBT_CHECK_ARG(counts != nullptr, "counts is NULL");
    int ls[kMaxGroups];
    long long total = 0;
    for (int l = 0; l <= p->l_max; ++l) {
        ls[l] = l;
        DSBT_CHECK_ARG(counts[l] >= 0, "counts[%d] negative", l);
        total += counts[l];
    }
    DSBT_CHECK_ARG(total < (1LL << 30), "too many channels");
    int rc = check_common(p, dtype, in, out, ws, ws_b, (int)total);
    if (rc || total == 0) return rc;
    GroupTable g;
    rc = build_groups(p, counts, p->l_max + 1, ls, dtype, g);
    if (rc) return rc;
    if (uoff) {   // channels gathered from the caller's arrays by offset: interval-scheme C64 paths only
        DSBT_CHECK_ARG(p->ftc != nullptr && dtype == DSBT_C64 && which != 1,
                       "channel offsets need a DSBT_PLAN_FAST_SPLIT plan, complex64, forward or kinetic");
        g.uoff = uoff;
    }
    cudaStream_t st = (cudaStream_t)stream;
    if (which == 0) return run_forward(p, g, dtype, in, out, ws, st);
    if (which == 1) return run_inverse(p, g, dtype, in, out, ws, st);
    DSBT_CHECK_ARG(is_complex(dtype), "kinetic step needs a complex dtype");
    DSBT_CHECK_ARG(isfinite(tau), "tau must be finite");
    return run_kinetic(p, g, dtype, tau, in, out, ws, st, which == kKineticReady && is_fp64(dtype));
}

int single_call(int which, const dsbt_plan* p, int l, int nchan, int dtype, const void* in, void* out,
                void* ws, size_t ws_b, void* stream) {
    DSBT_CHECK_ARG(p != nullptr, "plan is NULL");
    DSBT_CHECK_ARG(l >= 0 && l <= p->l_max, "l=%d outside the plan's 0..%d", l, p->l_max);
    DSBT_CHECK_ARG(nchan >= 0 && nchan < (1 << 30), "nchan=%d invalid", nchan);
    int rc = check_common(p, dtype, in, out, ws, ws_b, nchan);
    if (rc || nchan == 0) return rc;
    GroupTable g;
    rc = build_groups(p, &nchan, 1, &l, dtype, g);
    if (rc) return rc;
    cudaStream_t st = (cudaStream_t)stream;
    return which == 0 ? run_forward(p, g, dtype, in, out, ws, st) : run_inverse(p, g, dtype, in, out, ws, st);
}

}  // namespace

// Grouped forward with a scratch buffer supplied by the caller of this
// function (used by entry points that bring their own scratch memory).
int forward_grouped_with_scratch(const dsbt_plan* p, const int* counts, int dtype, const void* in,
                                 void* out, void* scratch, size_t scratch_bytes, cudaStream_t st) {
    return grouped_call(0, p, counts, dtype, 0.0, in, out, scratch, scratch_bytes, st);
}

// Grouped forward (which = 0), inverse (1) or kinetic step (2) on device
// buffers with a caller-supplied workspace (the host-streamed entry points).
int grouped_device_call(int which, const dsbt_plan* p, const int* counts, int dtype, double tau,
                        const void* in, void* out, void* ws, size_t ws_b, cudaStream_t st, const long long* uoff) {
    return grouped_call(which, p, counts, dtype, tau, in, out, ws, ws_b, st, uoff);
}

int real_step(const dsbt_plan* p, int l, int nchan, const double* in, double* b, double* out, const double* row_scale,
              void* ws, size_t ws_b, cudaStream_t st) {
    int rc = check_common(p, DSBT_F64, in, b, ws, ws_b, nchan);
    GroupTable g;
    if (!rc) rc = build_groups(p, &nchan, 1, &l, DSBT_F64, g);
    if (rc) return rc;
    Workspace w = carve(p, ws, nchan, DSBT_F64);
    rc = dct_forward_f64(p, g, false, in, w.f64a, st);
    if (!rc) rc = contract_f64(p, g, +1, w.f64a, 0, b, 0, nullptr, st, w.fast, row_scale);
    if (!rc) rc = contract_f64(p, g, -1, b, 0, w.f64a, 0, nullptr, st, w.fast);
    if (!rc) rc = dct_inverse_f64(p, g, false, w.f64a, out, st);
    return rc;
}

int kinetic_phase_fill(const dsbt_plan* p, void* ws, int total_channels, double tau, cudaStream_t st) {
    return fill_phase64(p, carve(p, ws, total_channels, DSBT_C128), tau, st);
}

const double2* kinetic_phase_table(const dsbt_plan* p, void* ws, int total_channels) {
    return carve(p, ws, total_channels, DSBT_C128).ph64;
}

}  // namespace dsbt

using namespace dsbt;

extern "C" size_t dsbt_workspace_size(const dsbt_plan* plan, int total_channels, int dtype) {
    if (!plan || total_channels < 0 || !valid_dtype(dtype)) return 0;
    return ws_bytes(plan, total_channels, dtype);
}

extern "C" int dsbt_forward(const dsbt_plan* plan, int l, int nchan, int dtype, const void* in, void* out,
                            void* workspace, size_t workspace_bytes, void* stream) {
    return single_call(0, plan, l, nchan, dtype, in, out, workspace, workspace_bytes, stream);
}

extern "C" int dsbt_inverse(const dsbt_plan* plan, int l, int nchan, int dtype, const void* in, void* out,
                            void* workspace, size_t workspace_bytes, void* stream) {
    return single_call(1, plan, l, nchan, dtype, in, out, workspace, workspace_bytes, stream);
}

extern "C" int dsbt_forward_grouped(const dsbt_plan* plan, const int* counts, int dtype, const void* in,
                                    void* out, void* workspace, size_t workspace_bytes, void* stream) {
    return grouped_call(0, plan, counts, dtype, 0.0, in, out, workspace, workspace_bytes, stream);
}

extern "C" int dsbt_inverse_grouped(const dsbt_plan* plan, const int* counts, int dtype, const void* in,
                                    void* out, void* workspace, size_t workspace_bytes, void* stream) {
    return grouped_call(1, plan, counts, dtype, 0.0, in, out, workspace, workspace_bytes, stream);
}

extern "C" int dsbt_kinetic_grouped(const dsbt_plan* plan, const int* counts, int dtype, double tau,
                                    const void* in, void* out, void* workspace, size_t workspace_bytes,
                                    void* stream) {
    return grouped_call(2, plan, counts, dtype, tau, in, out, workspace, workspace_bytes, stream);
}

extern "C" int dsbt_device_status(const dsbt_plan* plan, int reset, int* status_out) {
    DSBT_CHECK_ARG(plan != nullptr && status_out != nullptr, "NULL argument");
    unsigned s = 0;
    DSBT_CUDA_TRY(cudaMemcpy(&s, plan->status, sizeof(s), cudaMemcpyDeviceToHost));
    *status_out = (int)s;
    if (reset) DSBT_CUDA_TRY(cudaMemset(plan->status, 0, sizeof(unsigned)));
    return DSBT_OK;
}
