// Lane-vectorised mixed-radix FFT passes for the lattice grids.
//
// Sec. IV-B evaluates each Toeplitz block product with the FFT of its
// circulant embedding (Eqs. LJV3-LJV5) and generalises to 2-D lattices with
// 2-D FFTs.  Here every 2-D transform is two 1-D passes (grids that fit in
// shared memory take the fused transforms of fft2d.cu).  A pass transforms
// data[outer][P][inner] along P; the `inner` dimension holds independent
// sequences (local unknowns k, right-hand sides, or block entries (op,j,i))
// that sit next to each other in memory, so one CTA takes a P x W tile whose
// rows are W contiguous lanes (coalesced).  The first Stockham stage reads
// global memory into registers and the last one writes it (fft_core.cuh), so
// the tile crosses shared memory once per stage boundary.
//
// Pruning: only the first p_in points along P are read (the rest are the
// zero padding of the circulant embedding) and only the first p_out are
// written (the crop of the inverse transform).  The forward pass over the
// cell rows can read its input straight from the unique-unknown vector
// through U_o (x1 = U_o x, Eq. MVP), so no padded grid is ever written.
#include <algorithm>
#include <cmath>

#include "fft_core.cuh"

namespace emsurf {

namespace {

using namespace fftc;

constexpr int kFftThreads = 256;
constexpr int kFftMaxRad = 16;

// Gather source of the forward pass over cell rows: element (row iy, point
// ix, lane L = r*K + k) = sign * x[r][uo_index[(iy*nx + ix)*K + k]].
struct GatherSrc {
    const double2* x;
    const int32_t* idx;
    const int8_t* sgn;
    int nx, K, n_unique;
    const float2* xf;   // FP32 source instead of x when not null
};

// sign * x[r][u] of the gather, from the FP64 or the FP32 source; an FP32
// source into an FP32 grid needs no FP64 arithmetic
template <typename T2>
__device__ __forceinline__ T2 gather_value(const GatherSrc& gs, int r, size_t loc) {
    const size_t at = (size_t)r * gs.n_unique + gs.idx[loc];
    if (gs.xf) {
        const float2 xv = gs.xf[at];
        const float s = (float)gs.sgn[loc];
        if constexpr (sizeof(T2) == sizeof(float2)) return make_float2(s * xv.x, s * xv.y);
        else return mk<T2>((double)(s * xv.x), (double)(s * xv.y));
    }
    const double2 xv = gs.x[at];
    const double s = (double)gs.sgn[loc];
    return mk<T2>(s * xv.x, s * xv.y);
}

// Store epilogue of the inverse pass over the kept rows: point ix < nx of row
// iy, lane L = r*K + k, goes to y1[r][iy*nx + ix][k] = scale * value +
// sum_s mm[s][r][m][k] (the macromodel partials).
template <typename T2>
struct CropEpi {
    const T2* mm;
    T2* y1;
    int nsplit, R, M, nx, K;
    double scale;
};

template <typename T2>
__device__ __forceinline__ void crop_store(const CropEpi<T2>& ep, int iy, int p, long long L, T2 v) {
    const int r = (int)(L / ep.K), k = (int)(L % ep.K);
    const size_t m = (size_t)iy * ep.nx + p;
    // in the precision of the grid (no FP64 arithmetic on the FP32 path)
    using S = decltype(v.x);
    const S sc = (S)ep.scale;
    S ax = v.x * sc, ay = v.y * sc;
    for (int s = 0; s < ep.nsplit; ++s) {
        const T2 z = ep.mm[(((size_t)s * ep.R + r) * ep.M + m) * ep.K + k];
        ax += z.x;
        ay += z.y;
    }
    T2 o;
    o.x = ax;
    o.y = ay;
    ep.y1[((size_t)r * ep.M + m) * ep.K + k] = o;
}

// One pass over tiles of W lanes (a power of two up to 32).  In place: a tile's
// points are all read before any is written (one thread does both when there
// is a single stage).
template <typename T2, int SIGN, bool GATHER, bool EPI>
__global__ void __launch_bounds__(kFftThreads)
fft_pass_kernel(T2* __restrict__ data, FftStages f, FastDiv lanes, long long inner, long long outer_stride, int p_in,
                int p_out, const double2* __restrict__ twg, GatherSrc gs, CropEpi<T2> ep) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int P = f.P, W = (int)lanes.d;
    T2* tw = reinterpret_cast<T2*>(smem_raw);
    T2* cur = tw + P;
    T2* nxt = cur + P * W;
    for (int e = threadIdx.x; e < P; e += blockDim.x) {
        const double2 w = twg[e];
        tw[e] = mk<T2>(w.x, SIGN < 0 ? w.y : -w.y);
    }
    const long long lane0 = (long long)blockIdx.x * W;
    const int wl = (int)min((long long)W, inner - lane0);
    T2* base = data + (long long)blockIdx.y * outer_stride + lane0;
    // blockDim is a multiple of W: a thread stays on one lane
    const int myl = threadIdx.x & (W - 1);
    const bool live = myl < wl;
    int gr = 0, gk = 0;
    if constexpr (GATHER) {
        const long long L = lane0 + (live ? myl : 0);
        gr = (int)(L / gs.K);
        gk = (int)(L - (long long)gr * gs.K);
    }
    __syncthreads();
    auto ld0 = [&](int p, int l) {
        T2 v = mk<T2>(0.0, 0.0);
        if (live && p < p_in) {
            if constexpr (GATHER) v = gather_value<T2>(gs, gr, ((size_t)blockIdx.y * gs.nx + p) * gs.K + gk);
            else v = base[(long long)p * inner + l];
        }
        return v;
    };
    auto st1 = [&](int p, int l, T2 v) {
        if (live && p < p_out) {
            if constexpr (EPI) crop_store(ep, blockIdx.y, p, lane0 + l, v);
            else base[(long long)p * inner + l] = v;
        }
    };
    for (int s = 0; s < f.n; ++s) {
        const bool first = s == 0, last = s == f.n - 1;
        T2* out = cur;
        const T2* in = nxt;
        stage_any<SIGN, kFftMaxRad, T2>(
            f.rad[s], P, f.ns[s], lanes, tw, [&](int p, int l) { return first ? ld0(p, l) : in[p * W + l]; },
            [&](int p, int l, T2 v) {
                if (last) st1(p, l, v);
                else out[p * W + l] = v;
            });
        if (!last) __syncthreads();
        T2* t = cur;
        cur = nxt;
        nxt = t;
    }
}

template <typename T2, int SIGN, bool GATHER, bool EPI>
int launch_pass(T2* data, const FftPlan& plan, const FftStages& f, int W, size_t smem, long long inner,
                long long outer, long long outer_stride, int p_in, int p_out, const GatherSrc& gs,
                const CropEpi<T2>& ep, cudaStream_t st) {
    EMS_TRY(set_smem_once(fft_pass_kernel<T2, SIGN, GATHER, EPI>, smem));
    FastDiv lanes;
    lanes.set((uint32_t)W);
    const dim3 grid((unsigned)((inner + W - 1) / W), (unsigned)outer);
    fft_pass_kernel<T2, SIGN, GATHER, EPI><<<grid, kFftThreads, smem, st>>>(data, f, lanes, inner, outer_stride, p_in,
                                                                          p_out, plan.tw, gs, ep);
    EMS_CUDA(cudaGetLastError());
    return EMSURF_OK;
}

template <typename T2>
int pass_impl(T2* data, const FftPlan& plan, long long inner, long long outer, long long outer_stride,
              int sign, int p_in, int p_out, const GatherSrc& gs, bool gather, const CropEpi<T2>& ep,
              bool epi, cudaStream_t st) {
    if (outer <= 0 || inner <= 0) return EMSURF_OK;
    if (outer > 65535 || (inner + 7) / 8 > 2147483647LL) {
        set_error("fft_pass: grid too large (outer %lld, lanes %lld)", outer, inner);
        return EMSURF_EINVAL;
    }
    FftStages f;
    const size_t point = sizeof(T2);
    if (!fft_stages(plan.P, kFftMaxRad, f) || 2 * (size_t)plan.P * 8 * point > 200 * 1024) {
        set_error("FFT length %d too large for one shared-memory pass", plan.P);
        return EMSURF_EINVAL;
    }
    p_in = p_in < 0 ? plan.P : std::min(p_in, plan.P);
    p_out = p_out < 0 ? plan.P : std::min(p_out, plan.P);
    // 32 lanes while two blocks fit an SM, else 16 or 8
    const size_t bufs = f.n > 2 ? 2 : f.n > 1 ? 1 : 0;
    int W = 32;
    while (W > 8 && bufs * plan.P * W * point > 96 * 1024) W /= 2;
    const size_t smem = (bufs * W + 1) * plan.P * point;
    if (sign < 0 && gather)
        return launch_pass<T2, -1, true, false>(data, plan, f, W, smem, inner, outer, outer_stride, p_in, p_out, gs, ep, st);
    if (sign < 0)
        return launch_pass<T2, -1, false, false>(data, plan, f, W, smem, inner, outer, outer_stride, p_in, p_out, gs, ep, st);
    if (epi)
        return launch_pass<T2, +1, false, true>(data, plan, f, W, smem, inner, outer, outer_stride, p_in, p_out, gs, ep, st);
    return launch_pass<T2, +1, false, false>(data, plan, f, W, smem, inner, outer, outer_stride, p_in, p_out, gs, ep, st);
}

}  // namespace

int smallest_smooth_at_least(int n) {
    for (int m = (n < 1 ? 1 : n);; ++m) {
        int t = m;
        for (int p : {2, 3, 5})
            while (t % p == 0) t /= p;
        if (t == 1) return m;
    }
}

int fft_plan_create(FftPlan& plan, int P) {
    int t = P;
    for (int p : {2, 3, 5, 7})
        while (t > 1 && t % p == 0) t /= p;
    if (t != 1 || P < 1) {
        set_error("FFT length %d has a prime factor other than 2, 3, 5, 7", P);
        return EMSURF_EINVAL;
    }
    plan.P = P;
    std::vector<double2> h(P);
    const double two_pi = 6.283185307179586476925286766559;
    for (int k = 0; k < P; ++k) {
        // exact values on the axes; host libm elsewhere
        const double ang = two_pi * (double)k / (double)P;
        double c = std::cos(ang), s = std::sin(ang);
        if (4 * k == P) { c = 0.0; s = 1.0; }
        if (2 * k == P) { c = -1.0; s = 0.0; }
        if (4 * k == 3 * P) { c = 0.0; s = -1.0; }
        h[k] = make_double2(c, -s);
    }
    EMS_CUDA(cudaMalloc(&plan.tw, sizeof(double2) * P));
    EMS_CUDA(cudaMemcpy(plan.tw, h.data(), sizeof(double2) * P, cudaMemcpyHostToDevice));
    return EMSURF_OK;
}

void fft_plan_destroy(FftPlan& plan) {
    if (plan.tw) cudaFree(plan.tw);
    plan.tw = nullptr;
}

template <typename T2>
int fft_pass(T2* data, const FftPlan& plan, long long inner, long long outer,
             long long outer_stride, int sign, cudaStream_t st, int p_in, int p_out) {
    GatherSrc gs{nullptr, nullptr, nullptr, 0, 1, 0, nullptr};
    CropEpi<T2> ep{nullptr, nullptr, 0, 1, 1, 1, 1, 1.0};
    return pass_impl<T2>(data, plan, inner, outer, outer_stride, sign, p_in, p_out, gs, false, ep,
                         false, st);
}

template <typename T2>
int fft_pass_gather(T2* data, const FftPlan& plan, long long inner, long long outer,
                    long long outer_stride, int p_in, const double2* x, const int32_t* idx,
                    const int8_t* sgn, int nx, int K, int n_unique, cudaStream_t st, const float2* xf) {
    GatherSrc gs{x, idx, sgn, nx, K, n_unique, xf};
    CropEpi<T2> ep{nullptr, nullptr, 0, 1, 1, 1, 1, 1.0};
    return pass_impl<T2>(data, plan, inner, outer, outer_stride, -1, p_in, plan.P, gs, true, ep, false,
                         st);
}

template <typename T2>
int fft_pass_crop(T2* data, const FftPlan& plan, long long inner, long long outer,
                  long long outer_stride, int nx, const T2* mm, int nsplit, int R, int M, int K,
                  double scale, T2* y1, cudaStream_t st) {
    GatherSrc gs{nullptr, nullptr, nullptr, 0, 1, 0, nullptr};
    CropEpi<T2> ep{mm, y1, nsplit, R, M, nx, K, scale};
    return pass_impl<T2>(data, plan, inner, outer, outer_stride, +1, plan.P, nx, gs, false, ep, true,
                         st);
}

template int fft_pass<double2>(double2*, const FftPlan&, long long, long long, long long, int,
                               cudaStream_t, int, int);
template int fft_pass<float2>(float2*, const FftPlan&, long long, long long, long long, int,
                              cudaStream_t, int, int);
template int fft_pass_gather<double2>(double2*, const FftPlan&, long long, long long, long long, int,
                                      const double2*, const int32_t*, const int8_t*, int, int, int,
                                      cudaStream_t, const float2*);
template int fft_pass_gather<float2>(float2*, const FftPlan&, long long, long long, long long, int,
                                     const double2*, const int32_t*, const int8_t*, int, int, int,
                                     cudaStream_t, const float2*);
template int fft_pass_crop<double2>(double2*, const FftPlan&, long long, long long, long long, int,
                                    const double2*, int, int, int, int, double, double2*, cudaStream_t);
template int fft_pass_crop<float2>(float2*, const FftPlan&, long long, long long, long long, int,
                                   const float2*, int, int, int, int, double, float2*, cudaStream_t);

}  // namespace emsurf
