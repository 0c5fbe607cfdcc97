// Fused 2-D transforms of one product's grids (Sec. IV-B: the circulant
// embedding of the block-Toeplitz lattice operator, applied with 2-D FFTs).
//
// The pass-based transforms (fft.cu) run each 2-D FFT as two launches with
// the grid written to global memory in between.  While the px x py grid of W
// lanes (local unknowns k of one or more rhs) fits in shared memory, a CTA
// here does the gather of x1 = U_o x, both 1-D transforms and the store of
// X^ in one launch; the inverse does both inverse transforms, the crop to the
// lattice, the 1/P scale and the addition of the macromodel partials.
//
// The first stage of a transform reads global memory straight into registers
// and the last one writes it, so a lane's grid passes through shared memory
// once per stage boundary (three times for lengths of two stages).  Layouts
// there (W lanes contiguous, rows of odd length so that consecutive kx fall in
// different banks):
//   rows:    A[ix or kx][iy],   row stride (ny | 1) W
//   columns: B[kx][ky or iy],   row stride (py | 1) W
// Against the earlier kernels (every stage and both transposes through shared
// memory, run-time index divisions; grids other than the compiled squares up to
// 64 in four passes of a generic kernel): 24 x 24 boxes with 32 rhs 466 -> 278 us
// per direction, 20 x 13 boxes (40 x 25 grid) with 3 rhs 160 -> 22 us, 16 x 16
// with one rhs 11.2 -> 10.2 us.
#include <algorithm>

#include "fft_core.cuh"

namespace emsurf {
namespace {

using namespace fftc;

constexpr int kF2MaxRad = 10;
constexpr int kF2MaxLw = 5, kF2MaxW = 1 << kF2MaxLw;
constexpr int kF2MaxSplit = 8;   // macromodel partials (kMmSplit of the product)
constexpr size_t kF2MaxSmem = 220 * 1024;

struct F2Plan {
    FftStages x, y;
    FastDiv lx, ly;          // lanes of the x transforms (ny W) and of the y ones (px W)
    int lw = 0;              // log2 W
    int nx = 0, ny = 0;
    int buf0 = 0, buf1 = 0;  // elements of the two shared buffers
};

template <typename T2, int SIGN>
__device__ __forceinline__ void f2_twiddles(T2* tw, const double2* __restrict__ twg, int P) {
    for (int e = threadIdx.x; e < P; e += blockDim.x) {
        const double2 w = twg[e];
        tw[e] = mk<T2>(w.x, SIGN < 0 ? w.y : -w.y);
    }
}

// X^[ky * px + kx][lane] of x1 = U_o x (sign * x[r][uo_index[(iy nx + ix) K + k]],
// lane = r K + k), zero outside the lattice.  PC: px = py = PC at compile time,
// 0: any grid.
template <typename T2, int PC>
__global__ void __launch_bounds__(512)
fft2d_fwd_kernel(T2* __restrict__ Xg, long long lanes, F2Plan f, int K, int n_unique,
                 const double2* __restrict__ twx, const double2* __restrict__ twy, const double2* __restrict__ x,
                 const float2* __restrict__ xf, const int32_t* __restrict__ idx, const int8_t* __restrict__ sgn) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ int s_k[kF2MaxW], s_r[kF2MaxW];
    dep_trigger();
    T2* cur = reinterpret_cast<T2*>(smem_raw);
    T2* nxt = cur + f.buf0;
    T2* tx = nxt + f.buf1;
    const int px = PC > 0 ? PC : f.x.P, py = PC > 0 ? PC : f.y.P;
    T2* ty = PC > 0 ? tx : tx + px;
    f2_twiddles<T2, -1>(tx, twx, px);
    if (PC == 0) f2_twiddles<T2, -1>(ty, twy, py);
    const int lw = f.lw, W = 1 << lw, wm = W - 1, nx = f.nx, ny = f.ny;
    const long long lane0 = (long long)blockIdx.x * W;
    const int wl = (int)min((long long)W, lanes - lane0);
    if (threadIdx.x < W) {
        const long long L = lane0 + (threadIdx.x < wl ? threadIdx.x : 0);
        s_r[threadIdx.x] = (int)(L / K);
        s_k[threadIdx.x] = (int)(L % K);
    }
    __syncthreads();
    const int sx = (ny | 1) << lw, sy = (py | 1) << lw;     // row strides
    fft_stages_run<-1, PC, kF2MaxRad, T2>(f.x, f.lx, tx, [&](bool first, bool, auto&& go) {
        T2* out = cur;
        const T2* in = nxt;
        go(
            [&](int p, int l) {
                if (!first) return in[p * sx + l];
                T2 v = mk<T2>(0.0, 0.0);
                const int w = l & wm, iy = l >> lw;
                if (p < nx && w < wl) {
                    const int loc = (iy * nx + p) * K + s_k[w];
                    const size_t at = (size_t)s_r[w] * n_unique + idx[loc];
                    if (xf) {
                        const float sg = (float)sgn[loc];
                        const float2 xv = xf[at];
                        if constexpr (sizeof(T2) == sizeof(float2)) v = make_float2(sg * xv.x, sg * xv.y);
                        else v = mk<T2>((double)(sg * xv.x), (double)(sg * xv.y));
                    } else {
                        const double sg = (double)sgn[loc];
                        const double2 xv = x[at];
                        v = mk<T2>(sg * xv.x, sg * xv.y);
                    }
                }
                return v;
            },
            [&](int p, int l, T2 v) { out[p * sx + l] = v; });
        __syncthreads();
        T2* t = cur;
        cur = nxt;
        nxt = t;
    });
    // rows in `nxt`; rows iy >= ny are the zero padding
    T2* Xo = Xg + lane0;
    fft_stages_run<-1, PC, kF2MaxRad, T2>(f.y, f.ly, ty, [&](bool first, bool last, auto&& go) {
        T2* out = cur;
        const T2* in = nxt;
        go(
            [&](int p, int l) {
                const int w = l & wm, kx = l >> lw;
                if (first) return p < ny ? in[kx * sx + (p << lw) + w] : mk<T2>(0.0, 0.0);
                return in[kx * sy + (p << lw) + w];
            },
            [&](int p, int l, T2 v) {
                const int w = l & wm, kx = l >> lw;
                if (!last) out[kx * sy + (p << lw) + w] = v;
                else if (w < wl) Xo[(long long)(p * px + kx) * lanes + w] = v;
            });
        if (!last) __syncthreads();
        T2* t = cur;
        cur = nxt;
        nxt = t;
    });
}

// y1[r][iy nx + ix][k] = scale * IFFT2(Y^)[iy][ix] + sum_s mm[s][r][m][k] for
// the lattice points (the crop of the circulant embedding)
template <typename T2, int PC>
__global__ void __launch_bounds__(512)
fft2d_inv_kernel(const T2* __restrict__ Yg, long long lanes, F2Plan f, int K, int M, int R, int nsplit, double scale,
                 const double2* __restrict__ twx, const double2* __restrict__ twy, const T2* __restrict__ mm,
                 T2* __restrict__ y1) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ int s_k[kF2MaxW], s_r[kF2MaxW];
    dep_trigger();
    T2* cur = reinterpret_cast<T2*>(smem_raw);
    T2* nxt = cur + f.buf0;
    T2* tx = nxt + f.buf1;
    const int px = PC > 0 ? PC : f.x.P, py = PC > 0 ? PC : f.y.P;
    T2* ty = PC > 0 ? tx : tx + px;
    f2_twiddles<T2, +1>(tx, twx, px);
    if (PC == 0) f2_twiddles<T2, +1>(ty, twy, py);
    const int lw = f.lw, W = 1 << lw, wm = W - 1, nx = f.nx, ny = f.ny;
    const long long lane0 = (long long)blockIdx.x * W;
    const int wl = (int)min((long long)W, lanes - lane0);
    if (threadIdx.x < W) {
        const long long L = lane0 + (threadIdx.x < wl ? threadIdx.x : 0);
        s_r[threadIdx.x] = (int)(L / K);
        s_k[threadIdx.x] = (int)(L % K);
    }
    __syncthreads();
    const int sx = (ny | 1) << lw, sy = (py | 1) << lw;
    const T2* Yi = Yg + lane0;
    fft_stages_run<+1, PC, kF2MaxRad, T2>(f.y, f.ly, ty, [&](bool first, bool last, auto&& go) {
        T2* out = cur;
        const T2* in = nxt;
        go(
            [&](int p, int l) {
                const int w = l & wm, kx = l >> lw;
                if (!first) return in[kx * sy + (p << lw) + w];
                return w < wl ? Yi[(long long)(p * px + kx) * lanes + w] : mk<T2>(0.0, 0.0);
            },
            [&](int p, int l, T2 v) {
                const int w = l & wm, kx = l >> lw;
                if (!last) out[kx * sy + (p << lw) + w] = v;
                else if (p < ny) out[kx * sx + (p << lw) + w] = v;      // rows kept
            });
        __syncthreads();
        T2* t = cur;
        cur = nxt;
        nxt = t;
    });
    using S = typename Real<T2>::type;
    const S sc = (S)scale;
    const size_t split = (size_t)R * M * K;
    fft_stages_run<+1, PC, kF2MaxRad, T2>(f.x, f.lx, tx, [&](bool, bool last, auto&& go) {
        T2* out = cur;
        const T2* in = nxt;
        go([&](int p, int l) { return in[p * sx + l]; },
           [&](int p, int l, T2 v) {
               if (!last) {
                   out[p * sx + l] = v;
                   return;
               }
               const int w = l & wm, iy = l >> lw;
               if (p >= nx || w >= wl) return;
               const size_t at = ((size_t)s_r[w] * M + iy * nx + p) * K + s_k[w];
               T2 o;
               o.x = v.x * sc;
               o.y = v.y * sc;
               // all partials' loads in flight together
               T2 z[kF2MaxSplit];
#pragma unroll
               for (int q = 0; q < kF2MaxSplit; ++q)
                   if (q < nsplit) z[q] = mm[at + q * split];
#pragma unroll
               for (int q = 0; q < kF2MaxSplit; ++q)
                   if (q < nsplit) o = cadd(o, z[q]);
               y1[at] = o;
           });
        if (!last) __syncthreads();
        T2* t = cur;
        cur = nxt;
        nxt = t;
    });
}

int sm_count() {
    static int count[64] = {};      // per device, filled on first use
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return 152;
    if (!count[dev]) cudaDeviceGetAttribute(&count[dev], cudaDevAttrMultiProcessorCount, dev);
    return count[dev] > 0 ? count[dev] : 152;
}

// shared bytes of a plan of W = 2^lw lanes, and the buffers' sizes: the stages
// write the two buffers in turn (forward: x rows, then columns; inverse:
// columns, then rows), the last stage writes global memory
template <typename T2>
size_t f2_layout(F2Plan& f, int px, int py, bool inverse) {
    const int W = 1 << f.lw;
    const int sx = px * ((f.ny | 1) * W), sy = px * ((py | 1) * W);
    int size[2] = {0, 0}, at = 0;
    auto write = [&](int n) {
        size[at] = std::max(size[at], n);
        at ^= 1;
    };
    if (!inverse) {
        for (int s = 0; s < f.x.n; ++s) write(sx);
        for (int s = 0; s + 1 < f.y.n; ++s) write(sy);
    } else {
        for (int s = 0; s + 1 < f.y.n; ++s) write(sy);
        write(sx);
        for (int s = 0; s + 1 < f.x.n; ++s) write(sx);
    }
    f.buf0 = size[0];
    f.buf1 = size[1];
    f.lx.set((uint32_t)(f.ny * W));
    f.ly.set((uint32_t)(px * W));
    return (size_t)(f.buf0 + f.buf1 + px + py) * sizeof(T2);
}

// square grids with their own kernels
#define EMS_F2_SIZES(X) X(5) X(8) X(15) X(16) X(24) X(32) X(40) X(48) X(64)


// lanes per CTA: 32 bytes of them (a whole sector per bin), doubled while the grids
// of all stay below 4 KB (a stage of fewer lanes would leave most of a CTA's
// threads without a butterfly), halved while that leaves more than a tenth of the
// SMs without a CTA (16 x 16 boxes, one rhs: 144 CTAs of 4 lanes on 152 SMs, 10.2 us).
// One box with 33 rhs (K = 576): 47.6 -> 7.9 us per transform, 11 x 1 boxes with
// 33 (K = 324) 51.8 -> 14.9.
template <typename T2>
constexpr int f2_full_lw() { return sizeof(T2) == sizeof(float2) ? 2 : 1; }
template <typename T2>
int f2_pick_lanes(int points, long long lanes) {
    const int sms = sm_count();
    int lw = f2_full_lw<T2>();
    while (lw < kF2MaxLw && ((size_t)points << lw) * sizeof(T2) < 4096) ++lw;
    for (; lw > 0; --lw)
        if (((lanes - 1) >> lw) + 1 >= (long long)sms * 9 / 10) return lw;
    return 0;
}

template <typename T2>
int f2_plan(F2Plan& f, int px, int py, int nx, int ny, long long lanes, bool inverse, size_t& smem, int& threads) {
    if (!fft_stages(px, kF2MaxRad, f.x) || !fft_stages(py, kF2MaxRad, f.y)) {
        set_error("fused 2-D FFT: no plan for %d x %d", px, py);
        return EMSURF_EINVAL;
    }
    f.nx = nx;
    f.ny = ny;
    f.lw = f2_pick_lanes<T2>(px * py, lanes);
    smem = f2_layout<T2>(f, px, py, inverse);
    // measured (forward and inverse, average): float, 16 x 16 boxes, one rhs (144
    // CTAs of 4 lanes): 512 threads 10.2 us, 384 11.6, 256 12.4; 24 x 24 boxes, 32
    // rhs (4608 CTAs): 384 threads 278 us, 512 286, 256 304; double is bound by
    // the FP64 rate and small blocks even out its stages (12 x 9 boxes, 6 rhs:
    // 128 threads 100 us, 256 110, 384 144)
    const long long ctas = ((lanes - 1) >> f.lw) + 1;
    const int sms = sm_count();
    if (sizeof(T2) == sizeof(float2)) threads = ctas <= sms ? 512 : 384;
    else threads = ctas <= 2 * sms ? 256 : 128;
    // no more than the largest stage has butterflies (idle threads cost nothing in a
    // launch of one wave: there the same count as for larger grids)
    if (ctas <= sms) return EMSURF_OK;
    int work = 1 << f.lw;
    for (int s = 0; s < f.x.n; ++s) work = std::max(work, px / f.x.rad[s] * ny << f.lw);
    for (int s = 0; s < f.y.n; ++s) work = std::max(work, py / f.y.rad[s] * px << f.lw);
    threads = std::min(threads, (std::max(work, 64) + 31) / 32 * 32);
    return EMSURF_OK;
}

}  // namespace

template <typename T2>
bool fft2d_fused_ok(int px, int py, int nx, int ny) {
    F2Plan f;
    if (!fft_stages(px, kF2MaxRad, f.x) || !fft_stages(py, kF2MaxRad, f.y)) return false;
    if (f.x.n > 2 || f.y.n > 2) return false;
    f.nx = nx;
    f.ny = ny;
    f.lw = f2_full_lw<T2>();
    return std::max(f2_layout<T2>(f, px, py, false), f2_layout<T2>(f, px, py, true)) <= kF2MaxSmem;
}

template <typename T2>
int fft2d_forward(T2* Xg, int px, int py, long long lanes, int nx, int ny, int K, int n_unique, const double2* twx,
                  const double2* twy, const double2* x, const float2* xf, const int32_t* idx, const int8_t* sgn,
                  cudaStream_t st) {
    F2Plan f;
    size_t smem;
    int threads;
    EMS_TRY(f2_plan<T2>(f, px, py, nx, ny, lanes, false, smem, threads));
    auto go = [&](auto kern) -> int {
        EMS_TRY(set_smem_once(kern, smem));
        kern<<<(unsigned)(((lanes - 1) >> f.lw) + 1), threads, smem, st>>>(Xg, lanes, f, K, n_unique, twx, twy, x, xf,
                                                                          idx, sgn);
        EMS_CUDA(cudaGetLastError());
        return EMSURF_OK;
    };
    if (px == py) switch (px) {
#define EMS_F2_CASE(N) \
    case N: return go(fft2d_fwd_kernel<T2, N>);
        EMS_F2_SIZES(EMS_F2_CASE)
#undef EMS_F2_CASE
        default: break;
    }
    return go(fft2d_fwd_kernel<T2, 0>);
}

template <typename T2>
int fft2d_inverse(const T2* Yg, int px, int py, long long lanes, int nx, int ny, int K, int M, int R, int nsplit,
                  double scale, const double2* twx, const double2* twy, const T2* mm, T2* y1, cudaStream_t st) {
    F2Plan f;
    size_t smem;
    int threads;
    EMS_TRY(f2_plan<T2>(f, px, py, nx, ny, lanes, true, smem, threads));
    auto go = [&](auto kern) -> int {
        EMS_TRY(set_smem_once(kern, smem));
        kern<<<(unsigned)(((lanes - 1) >> f.lw) + 1), threads, smem, st>>>(Yg, lanes, f, K, M, R, nsplit, scale, twx,
                                                                          twy, mm, y1);
        EMS_CUDA(cudaGetLastError());
        return EMSURF_OK;
    };
    if (px == py) switch (px) {
#define EMS_F2_CASE(N) \
    case N: return go(fft2d_inv_kernel<T2, N>);
        EMS_F2_SIZES(EMS_F2_CASE)
#undef EMS_F2_CASE
        default: break;
    }
    return go(fft2d_inv_kernel<T2, 0>);
}

template bool fft2d_fused_ok<float2>(int, int, int, int);
template bool fft2d_fused_ok<double2>(int, int, int, int);
template int fft2d_forward<float2>(float2*, int, int, long long, int, int, int, int, const double2*, const double2*,
                                   const double2*, const float2*, const int32_t*, const int8_t*, cudaStream_t);
template int fft2d_forward<double2>(double2*, int, int, long long, int, int, int, int, const double2*, const double2*,
                                    const double2*, const float2*, const int32_t*, const int8_t*, cudaStream_t);
template int fft2d_inverse<float2>(const float2*, int, int, long long, int, int, int, int, int, int, double,
                                   const double2*, const double2*, const float2*, float2*, cudaStream_t);
template int fft2d_inverse<double2>(const double2*, int, int, long long, int, int, int, int, int, int, double,
                                    const double2*, const double2*, const double2*, double2*, cudaStream_t);

}  // namespace emsurf
