// Schur complement of the macromodels (Eq. Zmacromodel): LU elimination of the
// interior unknowns of every type at once, partial pivoting among the interior
// rows only, 32 columns at a time:
//   panel  LU of the interior rows of 32 columns, one CTA per type;
//   rows   L of the exterior rows (X U = A), digits of all L rows;
//   cols   the pivots' row exchanges and U = L^-1 A to the right, digits of U;
//   gemm   trailing block -= L U.
// FP64 runs at 2 FMA per clock and SM here, and 26 G of them (32 types of 928
// unknowns, 352 interior) take 41 ms; the trailing update, all but 3 % of them,
// runs on the tensor cores instead, on base-256 digits (digits.cuh) with levels
// 0 to 7 kept: the dropped products weigh 2^-57 of row maximum times column
// maximum, below FP64's own rounding.  352 rank-1 steps over the whole trailing
// block (one launch each): 122 ms; this: 12 ms.  Entries of L and U keep 55 bits
// below the maximum of their row (of L) or column (of U) of a panel instead of 53
// of their own.  Against a 113-bit Schur complement of the same tables (n = 2, 3; 56
// to 336 interior unknowns) the error in norm is 3.2e-16 to 7.4e-16 (in FP64
// arithmetic 4.8e-16 to 1.2e-15), that of the worst row 2.0e-15 (2.1e-15), that of
// the worst entry above 1e-6 of its row 4.0e-11 (4.5e-11).
#include <algorithm>

#include "digits.cuh"
#include "slab_lu.cuh"

namespace emsurf {
namespace {

constexpr int kLuNb = 32;                            // columns of a panel
constexpr int kLuLd = kLuNb + 1;                     // row stride of a panel in shared memory
constexpr int kLuPanelThreads = 512;
constexpr int kLuLevels = 8;
constexpr int kLuM = 128, kLuN = 64;                 // real rows and columns of a tile: 8 levels x 64 TMEM columns
constexpr int kLuADig = kLuM * 128, kLuBDig = kLuN * 128;   // bytes of one digit of a tile: 64 FP16 per row
constexpr int kLuATile = kSl * kLuADig, kLuBTile = kSl * kLuBDig;
constexpr int kLuGroup = 4;                          // column tiles of a CTA
constexpr int kLuGemmThreads = 288;                  // 8 epilogue warps, one for copies and MMAs
constexpr size_t kLuGemmSmem = 1024 + kLuATile + kLuBTile;

// Panel [c, c + kb) of a type: LU in place among the interior rows.
// src[j] = row (from c) that becomes row j < kb; mv[j] = (row, the original row
// below kb that moves there) for the row that row j was exchanged with, or -1.
template <bool SM>
__global__ void __launch_bounds__(kLuPanelThreads)
lu_panel_kernel(const SlabType* __restrict__ ty, int c, double2* __restrict__ B, int* __restrict__ src,
                int2* __restrict__ mv, int* __restrict__ perm_g, int max_nint, int* __restrict__ status) {
    const SlabType T = ty[blockIdx.x];
    const int n = T.nint - c, N = T.N;
    if (n <= 0) return;
    extern __shared__ __align__(16) unsigned char lu_smem[];
    const int kb = min(kLuNb, n);
    double2* G = B + T.offB + (size_t)c * N + c;
    double2* P = SM ? reinterpret_cast<double2*>(lu_smem) : G;
    const int ld = SM ? kLuLd : N;
    int* perm = perm_g + (size_t)blockIdx.x * max_nint;
    __shared__ double s_m[kLuPanelThreads / 32];
    __shared__ int s_i[kLuPanelThreads / 32];
    __shared__ int s_piv[kLuNb];
    __shared__ int s_p;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    for (int r = tid; r < n; r += kLuPanelThreads) perm[r] = r;
    if (SM)
        for (int e = tid; e < n * kLuNb; e += kLuPanelThreads) {
            const int r = e / kLuNb, j = e % kLuNb;
            if (j < kb) P[r * ld + j] = G[(size_t)r * N + j];
        }
    __syncthreads();
    bool singular = false;
    for (int j = 0; j < kb; ++j) {
        double best = -1.0;
        int at = j;
        for (int r = j + tid; r < n; r += kLuPanelThreads) {
            const double2 v = P[(size_t)r * ld + j];
            const double m = v.x * v.x + v.y * v.y;
            if (m > best) {
                best = m;
                at = r;
            }
        }
        auto take = [&](double m2, int i2) {
            if (m2 > best || (m2 == best && i2 < at)) {
                best = m2;
                at = i2;
            }
        };
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) take(__shfl_xor_sync(0xffffffffu, best, o), __shfl_xor_sync(0xffffffffu, at, o));
        if (lane == 0) {
            s_m[warp] = best;
            s_i[warp] = at;
        }
        __syncthreads();
        if (warp == 0) {
            best = lane < kLuPanelThreads / 32 ? s_m[lane] : -1.0;
            at = lane < kLuPanelThreads / 32 ? s_i[lane] : n;
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) take(__shfl_xor_sync(0xffffffffu, best, o), __shfl_xor_sync(0xffffffffu, at, o));
            if (lane == 0) {
                const bool ok = best > 0.0;
                s_p = ok ? at : -1;
                s_piv[j] = ok ? at : j;
                if (ok) {
                    const int t = perm[j];
                    perm[j] = perm[at];
                    perm[at] = t;
                }
            }
        }
        __syncthreads();
        const int p = s_p;
        if (p < 0) {                       // no pivot: the host reports it; what follows stays in bounds
            singular = true;
            for (int q = j + tid; q < kb; q += kLuPanelThreads) s_piv[q] = q;
            break;
        }
        if (p != j && tid < kb) {
            const double2 t = P[(size_t)j * ld + tid];
            P[(size_t)j * ld + tid] = P[(size_t)p * ld + tid];
            P[(size_t)p * ld + tid] = t;
        }
        __syncthreads();
        const double2 piv = P[(size_t)j * ld + j];
        const double dd = 1.0 / (piv.x * piv.x + piv.y * piv.y);
        const double2 inv = make_double2(piv.x * dd, -piv.y * dd);
        for (int r = j + 1 + tid; r < n; r += kLuPanelThreads) P[(size_t)r * ld + j] = cmul(P[(size_t)r * ld + j], inv);
        __syncthreads();
        const int w = kb - j - 1;
        for (int e = tid; e < (n - j - 1) * w; e += kLuPanelThreads) {
            const int r = j + 1 + e / w, x = j + 1 + e % w;
            const double2 l = P[(size_t)r * ld + j], u = P[(size_t)j * ld + x];
            double2 a = P[(size_t)r * ld + x];
            cfma(a, make_double2(-l.x, -l.y), u);
            P[(size_t)r * ld + x] = a;
        }
        __syncthreads();
    }
    __syncthreads();
    if (singular && tid == 0) atomicExch(status, 1);
    if (SM)
        for (int e = tid; e < n * kLuNb; e += kLuPanelThreads) {
            const int r = e / kLuNb, j = e % kLuNb;
            if (j < kb) G[(size_t)r * N + j] = P[r * ld + j];
        }
    for (int j = tid; j < kLuNb; j += kLuPanelThreads) {
        src[blockIdx.x * kLuNb + j] = j < kb ? perm[j] : -1;
        const int p = j < kb ? s_piv[j] : -1;
        mv[blockIdx.x * kLuNb + j] = p >= kb ? make_int2(p, perm[p]) : make_int2(-1, -1);
    }
}

// exponent of a row of L or a column of U (64 real sources) and 2^(ex - 8) (NaN
// where an entry was not finite): contributions below 2^-1000 may lose digits
__device__ __forceinline__ int lu_exp(unsigned long long mbits) {
    return max(sl_exp(mbits, 2 * kLuNb), -1000);
}
__device__ __forceinline__ double lu_pow(int ex) { return ex == kSlNan ? sl_nan() : sl_pow2(ex - 8); }

// L of the rows below the panel, one row per thread, and their digits: real rows
// 2 i = [Re, -Im] and 2 i + 1 = [Im, Re] of the 32 columns, 128-byte swizzled.
__global__ void __launch_bounds__(128)
lu_rows_kernel(const SlabType* __restrict__ ty, int c, const double2* __restrict__ B, unsigned char* __restrict__ A,
               double* __restrict__ rs, int tiles, int max_n) {
    const SlabType T = ty[blockIdx.y];
    if (T.nint <= c) return;
    const int kb = min(kLuNb, T.nint - c), N = T.N, rem = N - c - kb;
    __shared__ double2 s_u[kLuNb][kLuNb], s_inv[kLuNb];
    const double2* G = B + T.offB + (size_t)c * N + c;
    for (int e = threadIdx.x; e < kLuNb * kLuNb; e += blockDim.x) {
        const int i = e / kLuNb, j = e % kLuNb;
        const bool in = i < kb && j < kb && j >= i;
        const double2 u = in ? G[(size_t)i * N + j] : make_double2(0.0, 0.0);
        s_u[i][j] = u;
        if (i == j) {
            const double dd = in ? 1.0 / (u.x * u.x + u.y * u.y) : 0.0;
            s_inv[i] = make_double2(u.x * dd, -u.y * dd);
        }
    }
    __syncthreads();
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= rem) return;
    const int row = c + kb + i;
    const double2* g = B + T.offB + (size_t)row * N + c;
    double2 v[kLuNb];
#pragma unroll
    for (int j = 0; j < kLuNb; ++j) v[j] = j < kb ? g[j] : make_double2(0.0, 0.0);
    if (row >= T.nint) {
#pragma unroll
        for (int j = 0; j < kLuNb; ++j) {
            v[j] = cmul(v[j], s_inv[j]);
            const double2 m = make_double2(-v[j].x, -v[j].y);
#pragma unroll
            for (int x = j + 1; x < kLuNb; ++x) cfma(v[x], m, s_u[j][x]);
        }
    }
    unsigned long long mx = 0;
#pragma unroll
    for (int j = 0; j < kLuNb; ++j) mx = max(mx, max(sl_abs(v[j].x), sl_abs(v[j].y)));
    const int ex = lu_exp(mx);
    rs[(size_t)blockIdx.y * max_n + i] = lu_pow(ex);
    unsigned char* out = A + ((size_t)blockIdx.y * tiles + i / (kLuM / 2)) * kLuATile;
    const int r0 = 2 * (i % (kLuM / 2));
#pragma unroll
    for (int ch = 0; ch < kLuNb / 8; ++ch) {
        unsigned long long re[8], im[8], ni[8];
#pragma unroll
        for (int b = 0; b < 8; ++b) {
            re[b] = sl_digits(v[8 * ch + b].x, ex);
            im[b] = sl_digits(v[8 * ch + b].y, ex);
            ni[b] = sl_digits(-v[8 * ch + b].y, ex);
        }
#pragma unroll
        for (int t = 0; t < kSl; ++t) {
            auto put = [&](int r, int chunk, uint4 w) {
                *reinterpret_cast<uint4*>(out + t * kLuADig + r * 128 + ((chunk ^ (r & 7)) * 16)) = w;
            };
            const uint4 hr = sl_halves(re, t);
            put(r0, ch, hr);
            put(r0, 4 + ch, sl_halves(ni, t));
            put(r0 + 1, ch, sl_halves(im, t));
            put(r0 + 1, 4 + ch, hr);
        }
    }
}

// Row exchanges and U = L^-1 A of the columns right of the panel, one column per
// thread, and their digits ([Re; Im] of the 32 rows).  U itself is not needed
// again: only the exchanged rows are written back.
__global__ void __launch_bounds__(kLuN)
lu_cols_kernel(const SlabType* __restrict__ ty, int c, double2* __restrict__ B, const int* __restrict__ src,
               const int2* __restrict__ mv, unsigned char* __restrict__ D, double* __restrict__ cs, int tiles, int max_n) {
    const SlabType T = ty[blockIdx.y];
    if (T.nint <= c) return;
    const int kb = min(kLuNb, T.nint - c), N = T.N, rem = N - c - kb;
    __shared__ double2 s_l[kLuNb * (kLuNb - 1) / 2], s_o[kLuNb][kLuN];   // s_l: below the diagonal, row after row
    __shared__ int s_src[kLuNb];
    __shared__ int2 s_mv[kLuNb];
    const double2* G = B + T.offB + (size_t)c * N + c;
    for (int e = threadIdx.x; e < kLuNb * kLuNb; e += blockDim.x) {
        const int i = e / kLuNb, j = e % kLuNb;
        if (j < i) s_l[i * (i - 1) / 2 + j] = i < kb ? G[(size_t)i * N + j] : make_double2(0.0, 0.0);
    }
    if (threadIdx.x < kLuNb) {
        s_src[threadIdx.x] = src[blockIdx.y * kLuNb + threadIdx.x];
        s_mv[threadIdx.x] = mv[blockIdx.y * kLuNb + threadIdx.x];
    }
    __syncthreads();
    const int i = blockIdx.x * kLuN + threadIdx.x;
    if (i >= rem) return;
    double2* col = B + T.offB + (size_t)c * N + c + kb + i;
    double2 v[kLuNb];
#pragma unroll
    for (int j = 0; j < kLuNb; ++j) {
        v[j] = make_double2(0.0, 0.0);
        if (j < kb) s_o[j][threadIdx.x] = col[(size_t)j * N];
    }
#pragma unroll
    for (int j = 0; j < kLuNb; ++j)
        if (j < kb) v[j] = s_src[j] < kb ? s_o[s_src[j]][threadIdx.x] : col[(size_t)s_src[j] * N];
#pragma unroll 1
    for (int j = 0; j < kb; ++j)
        if (s_mv[j].x >= 0) col[(size_t)s_mv[j].x * N] = s_o[s_mv[j].y][threadIdx.x];
#pragma unroll
    for (int j = 0; j < kLuNb; ++j) {
        const double2 m = make_double2(-v[j].x, -v[j].y);
#pragma unroll
        for (int x = j + 1; x < kLuNb; ++x) cfma(v[x], m, s_l[x * (x - 1) / 2 + j]);
    }
    unsigned long long mx = 0;
#pragma unroll
    for (int j = 0; j < kLuNb; ++j) mx = max(mx, max(sl_abs(v[j].x), sl_abs(v[j].y)));
    const int ex = lu_exp(mx);
    cs[(size_t)blockIdx.y * max_n + i] = lu_pow(ex);
    unsigned char* out = D + ((size_t)blockIdx.y * tiles + blockIdx.x) * kLuBTile;
    const int r = threadIdx.x;
#pragma unroll
    for (int ch = 0; ch < kLuNb / 8; ++ch) {
        unsigned long long re[8], im[8];
#pragma unroll
        for (int b = 0; b < 8; ++b) {
            re[b] = sl_digits(v[8 * ch + b].x, ex);
            im[b] = sl_digits(v[8 * ch + b].y, ex);
        }
#pragma unroll
        for (int t = 0; t < kSl; ++t) {
            *reinterpret_cast<uint4*>(out + t * kLuBDig + r * 128 + ((ch ^ (r & 7)) * 16)) = sl_halves(re, t);
            *reinterpret_cast<uint4*>(out + t * kLuBDig + r * 128 + (((4 + ch) ^ (r & 7)) * 16)) = sl_halves(im, t);
        }
    }
}

// K-major descriptor, 128-byte swizzled rows, 8-row groups 1024 B apart
__device__ __forceinline__ uint64_t lu_desc(uint32_t addr) {
    return (uint64_t)((addr & 0x3FFFF) >> 4) | (1ull << 16) | (64ull << 32) | (1ull << 46) | (2ull << 61);
}
__device__ __forceinline__ void lu_mma(uint32_t d, uint64_t a, uint64_t b, uint32_t idesc, uint32_t acc) {
    asm volatile(
        "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
        " tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(d),
        "l"(a), "l"(b), "r"(idesc), "r"(acc));
}
// |x| < 2^51 to FP64 with one addition (conversions run at the FP64 rate)
__device__ __forceinline__ double lu_double(long long x) {
    return __longlong_as_double(0x4338000000000000ll + x) - 6755399441055744.0;
}

// Trailing block -= L U: 128 real rows x 64 columns per tile, the row tile stays
// in shared memory for kLuGroup column tiles.  34 digit pairs x 4 MMAs of 16
// sources per tile, then (levels as int64, two of them exact in FP64) 4 FP64
// operations per real number: the FP64 unit bounds it.
__global__ void __launch_bounds__(kLuGemmThreads, 1)
lu_gemm_kernel(const SlabType* __restrict__ ty, int c, double2* __restrict__ B, const unsigned char* __restrict__ A,
               const double* __restrict__ rs, int tiles_a, const unsigned char* __restrict__ D,
               const double* __restrict__ cs, int tiles_b, int max_n, int* __restrict__ status, int tries, int starve) {
    const SlabType T = ty[blockIdx.z];
    if (T.nint <= c) return;
    const int kb = min(kLuNb, T.nint - c), N = T.N, rem = N - c - kb;
    const int tile = blockIdx.x, ct0 = blockIdx.y * kLuGroup;
    if (tile * (kLuM / 2) >= rem || ct0 * kLuN >= rem) return;
    const int nct = min(kLuGroup, (rem + kLuN - 1) / kLuN - ct0);
    extern __shared__ __align__(16) unsigned char lu_smem[];
    unsigned char* sa = reinterpret_cast<unsigned char*>(((uintptr_t)lu_smem + 1023) & ~(uintptr_t)1023);
    unsigned char* sb = sa + kLuATile;
    __shared__ __align__(8) uint64_t full, done, tfree;
    __shared__ uint32_t tmem_slot;
    __shared__ int abort_flag;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (warp == 8) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(sl_addr(&tmem_slot)), "r"(512u));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    if (threadIdx.x == 0) {
        sl_init(&full, 1);
        sl_init(&done, 1);
        sl_init(&tfree, 8);
        abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    asm volatile("tcgen05.fence::before_thread_sync;");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;");
    const uint32_t tmem = tmem_slot;
    volatile int* abort_v = &abort_flag;
    if (warp == 8) {
        constexpr uint32_t idesc = (1u << 4) | ((uint32_t)(kLuN >> 3) << 17) | ((uint32_t)(kLuM >> 4) << 24);
        const uint64_t keep = l2_evict_last();
        const unsigned char* ga = A + ((size_t)blockIdx.z * tiles_a + tile) * kLuATile;
        const unsigned char* gb = D + ((size_t)blockIdx.z * tiles_b + ct0) * kLuBTile;
        const uint32_t tb = __shfl_sync(0xffffffffu, tmem, 0);
        bool copying = false, multiplying = false, ok = true;
        uint32_t fph = 0, dph = 0;
        for (int t = 0; t < nct; ++t) {
            if (lane == 0) {
                sl_expect(&full, kLuBTile + (t == 0 ? kLuATile : 0));
                if (t == 0 && !starve) sl_copy(sa, ga, kLuATile, &full, keep);
                if (!starve) sl_copy(sb, gb + (size_t)t * kLuBTile, kLuBTile, &full, keep);
            }
            __syncwarp();
            copying = true;
            // the operands are there and the last tile's sums have been read
            if (!sl_wait_warp(&full, fph, tries) || (t > 0 && !sl_wait_warp(&tfree, (uint32_t)(t - 1) & 1, tries))) {
                ok = false;
                break;
            }
            copying = false;
            fph ^= 1;
            asm volatile("tcgen05.fence::after_thread_sync;");
            const uint64_t da = lu_desc(sl_addr(sa)), db = lu_desc(sl_addr(sb));
            if (sl_elect()) {
#pragma unroll
                for (int l = 0; l < kLuLevels; ++l)
#pragma unroll
                    for (int s = (l < kSl ? 0 : l - kSl + 1); s <= (l < kSl ? l : kSl - 1); ++s)
#pragma unroll
                        for (int k = 0; k < 4; ++k)
                            lu_mma(tb + l * kLuN, da + s * (kLuADig / 16) + 2 * k, db + (l - s) * (kLuBDig / 16) + 2 * k, idesc,
                                   k > 0 || s > (l < kSl ? 0 : l - kSl + 1));
                sl_commit(&done);
            }
            __syncwarp();
            multiplying = true;
            if (!sl_wait_warp(&done, dph, tries)) {
                ok = false;
                break;
            }
            multiplying = false;
            dph ^= 1;
        }
        if (!ok) {
            if (lane == 0) atomicExch(status, 2);
            *abort_v = 1;
            // copies and MMAs in flight end before the CTA does
            if (copying) sl_wait_warp(&full, fph, tries);
            if (multiplying) sl_wait_warp(&done, dph, tries);
        }
    } else {
        const int qd = warp & 3, half = warp >> 2, rho = 32 * qd + lane;
        const uint32_t tl = tmem + ((uint32_t)(32 * qd) << 16) + half * (kLuN / 2);
        const int i = tile * (kLuM / 2) + (rho >> 1);
        const bool live = i < rem, im = lane & 1;
        // levels weigh 256^-l 2^-12 in units of 2^(ex_row + ex_col), the stored powers are 2^(ex - 8)
        const double rsc = live ? -rs[(size_t)blockIdx.z * max_n + i] * 0x1p-52 : 0.0;
        double2* row = B + T.offB + (size_t)(c + kb + (live ? i : 0)) * N + c + kb;
        for (int t = 0; t < nct; ++t) {
            if (sl_abort(abort_v) || !sl_wait_warp(&done, (uint32_t)t & 1, tries)) {
                if (lane == 0) atomicExch(status, 2);
                break;
            }
            asm volatile("tcgen05.fence::after_thread_sync;");
#pragma unroll 1
            for (int g = 0; g < kLuN / 2; g += 4) {
                uint32_t r[kLuLevels][4];
#pragma unroll
                for (int l = 0; l < kLuLevels; ++l) tmem_ld4(tl + l * kLuN + g, r[l]);
                asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
                double v[4];
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    long long hi = __float2int_rn(__uint_as_float(r[0][u])), lo = __float2int_rn(__uint_as_float(r[5][u]));
#pragma unroll
                    for (int l = 1; l < 5; ++l) hi = hi * 256 + __float2int_rn(__uint_as_float(r[l][u]));
#pragma unroll
                    for (int l = 6; l < 8; ++l) lo = lo * 256 + __float2int_rn(__uint_as_float(r[l][u]));
                    v[u] = fma(lu_double(hi), 0x1p24, lu_double(lo));
                }
                // the re lane takes columns 0 and 2 of four, the im lane 1 and 3
#pragma unroll
                for (int u = 0; u < 4; u += 2) {
                    const double o = __shfl_xor_sync(0xffffffffu, im ? v[u] : v[u + 1], 1);
                    const int x = (ct0 + t) * kLuN + half * (kLuN / 2) + g + u + im;
                    if (live && x < rem) {
                        const double sc = rsc * cs[(size_t)blockIdx.z * max_n + x];
                        double2 a = row[x];
                        a.x = fma(sc, im ? o : v[u], a.x);
                        a.y = fma(sc, im ? v[u + 1] : o, a.y);
                        row[x] = a;
                    }
                }
            }
            asm volatile("tcgen05.fence::before_thread_sync;");
            __syncwarp();
            if (lane == 0) sl_arrive(&tfree);
        }
    }
    asm volatile("tcgen05.fence::before_thread_sync;");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;");
    if (warp == 8) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512u));
}

struct LuSizes {
    int tiles_a, tiles_b;
    size_t a, d, rs, perm, src, mv;
    size_t total() const { return a + d + 2 * rs + perm + src + mv; }
};
LuSizes lu_sizes(int types, int max_n, int max_nint) {
    auto up = [](size_t b) { return (b + 255) & ~(size_t)255; };
    LuSizes s;
    s.tiles_a = (2 * max_n + kLuM - 1) / kLuM;
    s.tiles_b = (max_n + kLuN - 1) / kLuN;
    s.a = up((size_t)types * s.tiles_a * kLuATile);
    s.d = up((size_t)types * s.tiles_b * kLuBTile);
    s.rs = up((size_t)types * max_n * sizeof(double));
    s.perm = up((size_t)types * max_nint * sizeof(int));
    s.src = up((size_t)types * kLuNb * sizeof(int));
    s.mv = up((size_t)types * kLuNb * sizeof(int2));
    return s;
}

}  // namespace

size_t slab_lu_bytes(int types, int max_n, int max_nint) { return lu_sizes(types, max_n, max_nint).total(); }

// *status: 1 a singular interior block, 2 an expired wait
int slab_lu(const SlabType* ty, int types, int max_n, int max_nint, double2* B, void* work, int* status, cudaStream_t st) {
    const LuSizes z = lu_sizes(types, max_n, max_nint);
    unsigned char* w = static_cast<unsigned char*>(work);
    auto carve = [&](size_t b) {
        unsigned char* p = w;
        w += b;
        return p;
    };
    unsigned char *A = carve(z.a), *D = carve(z.d);
    double *rs = reinterpret_cast<double*>(carve(z.rs)), *cs = reinterpret_cast<double*>(carve(z.rs));
    int *perm = reinterpret_cast<int*>(carve(z.perm)), *src = reinterpret_cast<int*>(carve(z.src));
    int2* mv = reinterpret_cast<int2*>(carve(z.mv));
    const size_t panel = (size_t)max_nint * kLuLd * sizeof(double2);
    const bool sm = panel <= 220 * 1024;         // the panel of the largest type fits in shared memory
    // the limits only grow: another thread may be launching larger panels
    EMS_TRY(set_smem_once(lu_gemm_kernel, kLuGemmSmem));
    if (sm) EMS_TRY(set_smem_once(lu_panel_kernel<true>, panel));
    for (int c = 0; c < max_nint; c += kLuNb) {
        const int rem = max_n - c - 1;           // at most
        if (sm) lu_panel_kernel<true><<<types, kLuPanelThreads, panel, st>>>(ty, c, B, src, mv, perm, max_nint, status);
        else lu_panel_kernel<false><<<types, kLuPanelThreads, 0, st>>>(ty, c, B, src, mv, perm, max_nint, status);
        lu_rows_kernel<<<dim3((rem + 127) / 128, types), 128, 0, st>>>(ty, c, B, A, rs, z.tiles_a, max_n);
        lu_cols_kernel<<<dim3((rem + kLuN - 1) / kLuN, types), kLuN, 0, st>>>(ty, c, B, src, mv, D, cs, z.tiles_b, max_n);
        const int ta = (2 * rem + kLuM - 1) / kLuM, tc = (rem + kLuN - 1) / kLuN;
        lu_gemm_kernel<<<dim3(ta, (tc + kLuGroup - 1) / kLuGroup, types), kLuGemmThreads, kLuGemmSmem, st>>>(
            ty, c, B, A, rs, z.tiles_a, D, cs, z.tiles_b, max_n, status, kSlWait, 0);
        EMS_CUDA(cudaGetLastError());
    }
    return EMSURF_OK;
}

// One trailing update whose operands never arrive: every wait expires (no entry is
// touched).  Synchronises the stream.
int slab_lu_selftest(int tries, int* err, cudaStream_t st) {
    EMS_TRY(set_smem_once(lu_gemm_kernel, kLuGemmSmem));
    unsigned char* w = nullptr;
    EMS_CUDA(cudaMalloc(&w, 256 + 4 * sizeof(double2) + 4 * sizeof(double)));
    const SlabType ty{{0, 0}, {0, 0}, 2, 1, 0, 0};
    double2* B = reinterpret_cast<double2*>(w + 256);
    double* sc = reinterpret_cast<double*>(B + 4);
    cudaError_t e = cudaMemsetAsync(w, 0, 256 + 4 * sizeof(double2) + 4 * sizeof(double), st);
    if (e == cudaSuccess) e = cudaMemcpyAsync(w, &ty, sizeof(ty), cudaMemcpyHostToDevice, st);
    if (e == cudaSuccess) {
        lu_gemm_kernel<<<dim3(1, 1, 1), kLuGemmThreads, kLuGemmSmem, st>>>(reinterpret_cast<const SlabType*>(w), 0, B, w, sc, 1,
                                                                           w, sc + 2, 1, 2, err, tries, 1);
        e = cudaGetLastError();
    }
    const cudaError_t es = cudaStreamSynchronize(st);
    cudaFree(w);
    EMS_CUDA(e);
    EMS_CUDA(es);
    return EMSURF_OK;
}

}  // namespace emsurf
