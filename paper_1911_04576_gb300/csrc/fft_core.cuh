// Register DFTs and Stockham stages shared by the lattice transforms.
//
// A transform of length P runs as stages whose radices multiply to P
// (Stockham autosort; Govindaraju et al., SC 2008).  A thread holds one
// radix-R butterfly in registers, R up to 16 (primes by symmetric pairs,
// composites by one Cooley-Tukey step with compile-time twiddles), so lengths
// up to 100 take two stages and one pass through shared memory.  P, the radices
// and the lane counts are run-time values: index divisions use precomputed
// reciprocals.
#pragma once

#include <type_traits>
#include <utility>

#include "common.cuh"

namespace emsurf {
namespace fftc {

// cos and sin of 2 pi p / q, reduced to the first octant before the series
constexpr double oct_cos(double x) {
    double t = 1.0, s = 1.0;
    for (int i = 1; i < 12; ++i) {
        t *= -x * x / ((2 * i - 1) * (2 * i));
        s += t;
    }
    return s;
}
constexpr double oct_sin(double x) {
    double t = x, s = x;
    for (int i = 1; i < 12; ++i) {
        t *= -x * x / ((2 * i) * (2 * i + 1));
        s += t;
    }
    return s;
}
constexpr double kTwoPi = 6.283185307179586476925286766559;
constexpr double cos2pi(int p, int q) {
    p %= q;
    if (2 * p > q) p = q - p;
    if (4 * p > q) return -cos2pi(q - 2 * p, 2 * q);
    if (8 * p > q) return oct_sin(kTwoPi * (q - 4 * p) / (4 * q));
    return oct_cos(kTwoPi * p / q);
}
constexpr double sin2pi(int p, int q) {
    p %= q;
    if (2 * p > q) return -sin2pi(q - p, q);
    if (4 * p > q) return sin2pi(q - 2 * p, 2 * q);
    if (8 * p > q) return oct_cos(kTwoPi * (q - 4 * p) / (4 * q));
    return oct_sin(kTwoPi * p / q);
}

template <int I, int N, typename F>
__device__ __forceinline__ void static_for(F&& f) {
    if constexpr (I < N) {
        f(std::integral_constant<int, I>{});
        static_for<I + 1, N>(f);
    }
}

template <typename T2>
__device__ __forceinline__ T2 csub2(T2 a, T2 b) {
    T2 r;
    r.x = a.x - b.x;
    r.y = a.y - b.y;
    return r;
}

constexpr int first_factor(int R) {
    return R == 4 ? 2 : R == 6 ? 2 : R == 8 ? 2 : R == 9 ? 3 : R == 10 ? 2 : R == 12 ? 3 : R == 16 ? 4 : R;
}

// v <- DFT of v, e^{SIGN 2 pi i / R}
template <int SIGN, int R, typename T2>
__device__ __forceinline__ void dft(T2 (&v)[R]) {
    using S = typename Real<T2>::type;
    if constexpr (R == 1) {
    } else if constexpr (R == 2) {
        const T2 a = v[0], b = v[1];
        v[0] = cadd(a, b);
        v[1] = csub2(a, b);
    } else if constexpr (R == 3 || R == 5 || R == 7) {
        // sums and differences of the pairs (r, R - r)
        constexpr int Hn = (R - 1) / 2;
        T2 s[Hn], d[Hn];
        T2 sum = v[0];
        static_for<0, Hn>([&](auto r) {
            s[r] = cadd(v[r + 1], v[R - 1 - r]);
            d[r] = csub2(v[r + 1], v[R - 1 - r]);
            sum = cadd(sum, s[r]);
        });
        const T2 v0 = v[0];
        v[0] = sum;
        static_for<1, Hn + 1>([&](auto q) {
            T2 a = v0, b;
            b.x = b.y = (S)0;
            static_for<0, Hn>([&](auto r) {
                constexpr double c = cos2pi((q * (r + 1)) % R, R), sn = SIGN * sin2pi((q * (r + 1)) % R, R);
                a.x += (S)c * s[r].x;
                a.y += (S)c * s[r].y;
                b.x += (S)sn * d[r].x;
                b.y += (S)sn * d[r].y;
            });
            // a +- i b
            v[q].x = a.x - b.y;
            v[q].y = a.y + b.x;
            v[R - q].x = a.x + b.y;
            v[R - q].y = a.y - b.x;
        });
    } else if constexpr (R == 4) {
        const T2 s02 = cadd(v[0], v[2]), d02 = csub2(v[0], v[2]);
        const T2 s13 = cadd(v[1], v[3]), d13 = csub2(v[1], v[3]);
        v[0] = cadd(s02, s13);
        v[2] = csub2(s02, s13);
        v[1].x = d02.x - SIGN * d13.y;
        v[1].y = d02.y + SIGN * d13.x;
        v[3].x = d02.x + SIGN * d13.y;
        v[3].y = d02.y - SIGN * d13.x;
    } else {
        constexpr int A = first_factor(R), B = R / A;
        static_assert(A > 1 && A < R, "radix not supported");
        T2 t[R];
        static_for<0, B>([&](auto b) {
            T2 u[A];
            static_for<0, A>([&](auto a) { u[a] = v[B * a + b]; });
            dft<SIGN, A>(u);
            static_for<0, A>([&](auto ka) {
                if constexpr (b * ka == 0) {
                    t[ka * B + b] = u[ka];
                } else {
                    constexpr double c = cos2pi(b * ka, R), sn = SIGN * sin2pi(b * ka, R);
                    t[ka * B + b].x = (S)c * u[ka].x - (S)sn * u[ka].y;
                    t[ka * B + b].y = (S)c * u[ka].y + (S)sn * u[ka].x;
                }
            });
        });
        static_for<0, A>([&](auto ka) {
            T2 u[B];
            static_for<0, B>([&](auto b) { u[b] = t[ka * B + b]; });
            dft<SIGN, B>(u);
            static_for<0, B>([&](auto kb) { v[ka + A * kb] = u[kb]; });
        });
    }
}

// n / d for n d < 2^32
struct FastDiv {
    uint32_t d = 1, mul = 0;
    __host__ void set(uint32_t x) {
        d = x;
        mul = x > 1 ? (uint32_t)((0x100000000ull + x - 1) / x) : 0;
    }
    __device__ __forceinline__ int div(int n) const { return d == 1 ? n : (int)__umulhi((uint32_t)n, mul); }
};

constexpr int kMaxStages = 12;

// Radices of P: one stage up to 8 points, else two near-equal ones of at most
// max_rad (fewest passes through shared memory), else the largest factor
// first.  n = 0 if P has a prime factor above 7.
struct RadList {
    int n = 0;
    int r[kMaxStages] = {};
};
constexpr bool radix_ok(int r, int max_rad) {
    return r <= max_rad && ((r >= 2 && r <= 10) || r == 12 || r == 16);
}
constexpr RadList fft_radices(int P, int max_rad) {
    RadList f;
    if (P == 1 || (P <= 8 && radix_ok(P, max_rad))) {
        f.r[f.n++] = P;
        return f;
    }
    int left = P;
    while (left > 1) {
        if (f.n + 2 > kMaxStages) return RadList();
        int best = 0;
        for (int r = max_rad; r >= 2; --r)
            if (radix_ok(r, max_rad) && left % r == 0 && radix_ok(left / r, max_rad) && left / r <= r) best = r;
        if (best) {
            f.r[f.n++] = best;
            f.r[f.n++] = left / best;
            return f;
        }
        if (radix_ok(left, max_rad)) {
            f.r[f.n++] = left;
            return f;
        }
        int r0 = 0;
        for (int r = max_rad; r >= 2 && !r0; --r)
            if (radix_ok(r, max_rad) && left % r == 0) r0 = r;
        if (!r0) return RadList();
        f.r[f.n++] = r0;
        left /= r0;
    }
    return f;
}

struct FftStages {
    int P = 1, n = 1;
    int rad[kMaxStages] = {1};
    FastDiv ns[kMaxStages];      // product of the radices before stage s
};

inline bool fft_stages(int P, int max_rad, FftStages& f) {
    f = FftStages();
    f.P = P;
    const RadList l = P >= 1 ? fft_radices(P, max_rad) : RadList();
    f.n = l.n;
    int ns = 1;
    for (int s = 0; s < f.n; ++s) {
        f.rad[s] = l.r[s];
        f.ns[s].set((uint32_t)ns);
        ns *= f.rad[s];
    }
    return f.n > 0;
}

// One radix-R stage over `lanes` independent sequences: ld(p, l) reads point p
// of lane l, st(p, l, v) writes it; lanes run fastest over the threads.  PC,
// NSC > 0: compile-time length and radix product.
template <int SIGN, int R, int PC, int NSC, typename T2, typename Ld, typename St>
__device__ __forceinline__ void stage_run(int Pr, const FastDiv& ns, const FastDiv& lanes, const T2* __restrict__ tw,
                                          Ld&& ld, St&& st) {
    const int P = PC > 0 ? PC : Pr, NS = PC > 0 ? NSC : (int)ns.d;
    const int NR = P / R, L = (int)lanes.d;
    const int tstep = NR / NS;
    for (int e = threadIdx.x; e < NR * L; e += blockDim.x) {
        const int j = lanes.div(e), l = e - j * L;
        const int jn = PC > 0 ? j / NSC : ns.div(j), jm = j - jn * NS;
        T2 v[R];
#pragma unroll
        for (int r = 0; r < R; ++r) v[r] = ld(j + r * NR, l);
        if (NS > 1) {
#pragma unroll
            for (int r = 1; r < R; ++r) v[r] = cmul(v[r], tw[jm * r * tstep]);
        }
        dft<SIGN, R>(v);
        const int d = jn * NS * R + jm;
#pragma unroll
        for (int q = 0; q < R; ++q) st(d + q * NS, l, v[q]);
    }
}

template <int SIGN, int MAXR, typename T2, typename Ld, typename St>
__device__ __forceinline__ void stage_any(int R, int P, const FastDiv& ns, const FastDiv& lanes, const T2* tw, Ld&& ld,
                                          St&& st) {
    switch (R) {
#define EMS_FFT_RADIX(N) \
    case N:              \
        if constexpr (N <= MAXR) stage_run<SIGN, N, 0, 0, T2>(P, ns, lanes, tw, ld, st); \
        break;
        EMS_FFT_RADIX(1) EMS_FFT_RADIX(2) EMS_FFT_RADIX(3) EMS_FFT_RADIX(4) EMS_FFT_RADIX(5) EMS_FFT_RADIX(6)
        EMS_FFT_RADIX(7) EMS_FFT_RADIX(8) EMS_FFT_RADIX(9) EMS_FFT_RADIX(10) EMS_FFT_RADIX(12) EMS_FFT_RADIX(16)
#undef EMS_FFT_RADIX
        default: break;
    }
}

// All stages of one transform: body(first, last, go) for each, which calls go(ld, st)
// with the stage's source and destination.  PC > 0: a compile-time length,
// whose code holds its own radices only (small launches are bound by
// instruction fetch); 0: any length.
template <int SIGN, int PC, int MAXR, typename T2, typename F>
__device__ __forceinline__ void fft_stages_run(const FftStages& f, const FastDiv& lanes, const T2* tw, F&& body) {
    if constexpr (PC > 0) {
        constexpr RadList L = fft_radices(PC, MAXR);
        static_for<0, L.n>([&](auto s) {
            constexpr int ns = [](int k) {
                constexpr RadList l = fft_radices(PC, MAXR);
                int n = 1;
                for (int i = 0; i < k; ++i) n *= l.r[i];
                return n;
            }(s);
            constexpr RadList l = fft_radices(PC, MAXR);
            body(s == 0, s == L.n - 1, [&](auto&& ld, auto&& st) {
                stage_run<SIGN, l.r[s], PC, ns, T2>(PC, FastDiv(), lanes, tw, ld, st);
            });
        });
    } else {
        for (int s = 0; s < f.n; ++s)
            body(s == 0, s == f.n - 1, [&](auto&& ld, auto&& st) {
                stage_any<SIGN, MAXR, T2>(f.rad[s], f.P, f.ns[s], lanes, tw, ld, st);
            });
    }
}

}  // namespace fftc
}  // namespace emsurf
