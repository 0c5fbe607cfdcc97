// Tabulation of the Galerkin L and K blocks (Eqs. SIE_LOperator1,
// SIE_KOperator1 tested with RWG functions, Eq. blockZo) on the GPU.
//
//   L[m,n] = int int [Lam_m . Lam_n - (div Lam_m)(div' Lam_n)/k^2] G dS' dS
//   K[m,n] = int int Lam_m(r) . [grad_r G(r,r') x Lam_n(r')] dS' dS   (p.v.)
//   G = e^{-jkR} / (4 pi R)
//
// Quadrature (the paper names none): 7-point degree-5 Radon rule on both
// triangles; for blocks flagged singular (touching boxes, one cell) the 1/R
// and grad(1/R) parts are integrated over the source triangle in closed form
// (Wilton et al. 1984; Graglia 1993) and the remainder G - 1/(4 pi R) by the
// same rule.  Points within 1e-9 (relative) of the source plane take the
// principal value; point pairs within 1e-9 (relative) of each other are
// coincident (remainder at its R -> 0 limit, no gradient term).
//
// Stage 1: one thread per (block, test triangle, source triangle) computes
//          the 3x3 slot integrals of both operators into a scratch buffer
//          from the 3x3 barycentric moments of G and of its gradient factor.
// Stage 2: one thread per (block, test RWG, source RWG) sums the 2 x 2
//          triangle combinations of the two RWGs with their amplitudes.
// Blocks are processed in chunks so the scratch stays below 256 MB.
//
// Precision, against 113-bit quadrature of the same meshes (far blocks of 16 x 16
// lattices, n = 2, 3, 4): relative error of L 2.3e-15, 3.5e-15, 5.6e-15, of K 8.2e-16,
// 7.7e-16, 4.9e-16, with every point pair added to the slot integrals by itself 2.5e-15,
// 3.6e-15, 6.2e-15 and 8.5e-16, 6.4e-16, 4.8e-16.  The rounding of the distance times k
// R is what is left (a refined 1 / R changes nothing), so a 64-bit reference that
// rounds the same coordinates differs from tables by pair classes by a little more.
#include <algorithm>
#include <cmath>
#include <cstring>
#include <mutex>
#include <vector>

#include "common.cuh"

namespace emsurf {
namespace {

constexpr double kFourPi = 12.566370614359172953850573533118;
constexpr size_t kScratchBytes = 256ull << 20;

struct TriGeo {
    double v[9];     // vertices
    double q[21];    // quadrature points
    double area;
    double n[3];     // unit normal (v1-v0) x (v2-v0)
    double scale;    // max(|v1-v0|, |v2-v0|)
    double lh[9];    // unit vector of edge i, v_i -> v_{i+1}
    double u[9];     // its in-plane outward normal lh x n
};

struct RwgSlots {    // the two (triangle, slot) pairs of an RWG with amplitude sgn*len/(2A)
    int t[2];
    int s[2];
    double c[2];
};

__constant__ double c_wl[21];   // w_q lambda_u(q) of the rule at [3 q + u]

// the 7-point rule: the centroid, then two orbits of three points with one
// barycentric coordinate b and two a
constexpr double kS15 = 3.8729833462074168852;
constexpr double kRa1 = (6.0 - kS15) / 21.0, kRb1 = (9.0 + 2.0 * kS15) / 21.0;
constexpr double kRa2 = (6.0 + kS15) / 21.0, kRb2 = (9.0 - 2.0 * kS15) / 21.0;
constexpr double kRw0 = 9.0 / 40.0, kRw1 = (155.0 - kS15) / 1200.0, kRw2 = (155.0 + kS15) / 1200.0;

struct Vec3 {
    double x, y, z;
};
__device__ __forceinline__ Vec3 v3(const double* p) { return {p[0], p[1], p[2]}; }
__device__ __forceinline__ Vec3 operator+(Vec3 a, Vec3 b) { return {a.x + b.x, a.y + b.y, a.z + b.z}; }
__device__ __forceinline__ Vec3 operator-(Vec3 a, Vec3 b) { return {a.x - b.x, a.y - b.y, a.z - b.z}; }
__device__ __forceinline__ Vec3 operator*(double s, Vec3 a) { return {s * a.x, s * a.y, s * a.z}; }
__device__ __forceinline__ double dot(Vec3 a, Vec3 b) { return a.x * b.x + a.y * b.y + a.z * b.z; }
__device__ __forceinline__ Vec3 cross(Vec3 a, Vec3 b) {
    return {a.y * b.z - a.z * b.y, a.z * b.x - a.x * b.z, a.x * b.y - a.y * b.x};
}
__device__ __forceinline__ double norm3(Vec3 a) { return sqrt(dot(a, a)); }

// 4 pi G and 4 pi times the factor of grad_r G = (r - r') gfac, far form, from
// R2 = |r - r'|^2.  The phase is taken as kR / pi for sincospi, whose range
// reduction is exact.
__device__ __forceinline__ void green_far(double R2, double k, double kpi, double2& G, double2& gfac) {
    const double ri = rsqrt(R2), R1 = R2 * ri, R = fma(0.5 * ri, fma(-R1, R1, R2), R1);
    double s, c;
    sincospi(kpi * R, &s, &c);
    G = make_double2(c * ri, -s * ri);                           // e^{-jkR} / R
    const double kR = k * R, m = -ri * ri;
    // -(1 + jkR) e^{-jkR} / R^3
    gfac = make_double2(m * fma(-kR, G.y, G.x), m * fma(kR, G.x, G.y));
}

// 1/R (refined) and R of R2 = R^2 > 0
__device__ __forceinline__ double inv_dist(double R2, double& R) {
    const double ri = rsqrt(R2), R1 = R2 * ri;
    R = fma(0.5 * ri, fma(-R1, R1, R2), R1);
    return ri;
}

// Remainder after removing 1/R (times 4 pi), (e^{-jz} - 1) / R and
// (1 - (1 + jz) e^{-jz}) / R^3 for z = kR.  With the sine s and cosine c of z / 2
// no difference of near-equal terms is left (1 - cos z = 2 s^2,
// 1 - cos z - z sin z = 2 s (s - z c)) but one: sin z - z cos z takes its power
// series below 0.5.
__device__ __forceinline__ void green_smooth(double R2, double k, double kpi, double2& Gs, double2& gfac) {
    double R, s, c;
    const double ri = inv_dist(R2, R), z = k * R;
    sincospi(0.5 * kpi * R, &s, &c);
    const double s2 = 2.0 * s, sn = s2 * c, ri3 = ri * ri * ri;
    Gs = make_double2(-s2 * s * ri, -sn * ri);
    gfac.x = s2 * fma(-z, c, s) * ri3;
    if (z < 0.5) {
        // (sin z - z cos z) / z^3 = sum (-1)^(m+1) 2m / (2m + 1)! w^(m-1), w = z^2
        const double w = z * z;
        constexpr double f3 = 1.0 / 6, f5 = f3 / 20, f7 = f5 / 42, f9 = f7 / 72, f11 = f9 / 110, f13 = f11 / 156, f15 = f13 / 210;
        gfac.y = k * k * k * fma(w, fma(w, fma(w, fma(w, fma(w, fma(w, 14 * f15, -12 * f13), 10 * f11), -8 * f9), 6 * f7), -4 * f5), 2 * f3);
    } else {
        gfac.y = ri3 * fma(-z, fma(-s2, s, 1.0), sn);
    }
}

// Lossy region (Sec. II-B, k_v = w sqrt(mu0 eps_v) with complex eps_v): the
// same two functions for k = kr + j ki, e^{-jkR} = e^{ki R} e^{-j kr R}.
__device__ __forceinline__ double2 exp_mjkR(double R, double kpi, double ki) {
    double s, c;
    sincospi(kpi * R, &s, &c);
    const double m = exp(ki * R);
    return make_double2(m * c, -m * s);
}

__device__ __forceinline__ void green_far_cx(double R2, double kr, double kpi, double ki, double2& G, double2& gfac) {
    const double ri = rsqrt(R2), R1 = R2 * ri, R = fma(0.5 * ri, fma(-R1, R1, R2), R1);
    const double2 e = exp_mjkR(R, kpi, ki);
    G = make_double2(e.x * ri, e.y * ri);
    const double2 ae = cmul(make_double2(1.0 - ki * R, kr * R), G);     // (1 + jkR) e^{-jkR} / R
    const double d = -ri * ri;
    gfac = make_double2(ae.x * d, ae.y * d);
}

// e^a - 1: Taylor polynomial (relative error below 2^-57) for |a| < 1/64 (low loss)
__device__ __forceinline__ double expm1_small(double a) {
    if (fabs(a) < 0x1p-6) {
        constexpr double f2 = 1.0 / 2, f3 = f2 / 3, f4 = f3 / 4, f5 = f4 / 5, f6 = f5 / 6, f7 = f6 / 7;
        return a * fma(a, fma(a, fma(a, fma(a, fma(a, fma(a, f7, f6), f5), f4), f3), f2), 1.0);
    }
    return expm1(a);
}

__device__ __forceinline__ void green_smooth_cx(double R2, double kr, double kpi, double ki, double2& Gs,
                                                double2& gfac) {
    double R, s, c;
    const double ri = inv_dist(R2, R);
    const double2 z = make_double2(ki * R, -kr * R);                    // -jkR
    sincospi(0.5 * kpi * R, &s, &c);
    const double em = expm1_small(z.x), s2 = 2.0 * s;
    const double cs = fma(-s2, s, 1.0), sn = s2 * c, ez = 1.0 + em;
    Gs = make_double2(fma(em, cs, -s2 * s) * ri, -ez * sn * ri);        // (e^z - 1) / R
    const double r = 2.0 * z.x, q = fma(z.x, z.x, z.y * z.y);
    if (q < 0.25) {
        // (1 - (1 - z) e^z) / z^2 = sum z^m (m + 1) / (m + 2)!, the real polynomial at a
        // complex point by the recurrence of z^2 = 2 Re z z - |z|^2 (Knuth 4.6.4)
        double b1 = 0.0, b0 = 0.0;
#pragma unroll
        for (int m = 14; m >= 1; --m) {
            double f = 1.0;
#pragma unroll
            for (int i = 2; i <= m + 2; ++i) f /= i;                    // 1 / (m + 2)!
            const double t = fma(r, b0, fma(-q, b1, f * (m + 1)));
            b1 = b0;
            b0 = t;
        }
        // h = 1/2 - |z|^2 b1 + z b0
        const double hx = fma(z.x, b0, fma(-q, b1, 0.5)), hy = z.y * b0;
        const double2 jk = make_double2(ki, -kr), hh = cmul(cmul(jk, jk), make_double2(hx, hy));
        gfac = make_double2(hh.x * ri, hh.y * ri);
        return;
    }
    const double2 ae = cmul(make_double2(1.0 - z.x, -z.y), make_double2(ez * cs, -ez * sn));
    const double ri3 = ri * ri * ri;
    gfac = make_double2((1.0 - ae.x) * ri3, -ae.y * ri3);
}

__device__ __forceinline__ double edge_log(double lp, double lm, double Rp, double Rm, double R02) {
    // the operands are chosen first: one division and one logarithm for all lanes
    const bool ahead = lm >= 0.0, behind = lp <= 0.0;
    const double sp = Rp + lp, sm = Rm - lm;
    const double num = ahead ? sp : behind ? sm : sp * sm;
    const double den = ahead ? Rm + lm : behind ? Rp - lp : R02;
    return log(num / den);
}

// closed-form int 1/R, int (rho'-rho)/R, int grad_r(1/R) over source triangle;
// also returns rho (projection of r on the plane, after the in-plane snap)
__device__ __forceinline__ void potentials(Vec3 r, const TriGeo& T, double& I0, Vec3& I1, Vec3& Ig, Vec3& rho) {
    const Vec3 v0 = v3(T.v), n = v3(T.n);
    double d = dot(n, r - v0);
    if (fabs(d) <= 1e-9 * T.scale) d = 0.0;
    rho = r - d * n;
    const double ad = fabs(d), d2 = d * d;
    I0 = 0.0;
    I1 = {0.0, 0.0, 0.0};
    Vec3 fu = {0.0, 0.0, 0.0};
    // distances to the vertices, each the end of two edges
    Vec3 a[3];
    double Rv[3];
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        a[i] = v3(T.v + 3 * i) - rho;
        Rv[i] = sqrt(dot(a[i], a[i]) + d2);
    }
    // the edges' angles atan2(t l, R02 + |d| R), ends' difference, add up to the
    // solid angle: one atan2 of the product of the three complex numbers
    const double iu = 1.0 / fma(T.scale, T.scale, d2);
    double px = 1.0, py = 0.0;
    bool inside = true;
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        const Vec3 lh = v3(T.lh + 3 * i), u = v3(T.u + 3 * i);
        const double lp = dot(a[(i + 1) % 3], lh), lm = dot(a[i], lh);
        const double t = dot(a[i], u);
        const double R02 = t * t + d2;
        const double Rp = Rv[(i + 1) % 3], Rm = Rv[i];
        const double f = edge_log(lp, lm, Rp, Rm, R02);
        I0 += t * f;
        I1 = I1 + (0.5 * (R02 * f + lp * Rp - lm * Rm)) * u;
        fu = fu + f * u;
        if (ad > 0.0) {
            // in units of the triangle's size, so that the products stay in range
            const double xp = fma(ad, Rp, R02), xm = fma(ad, Rm, R02), yp = t * lp, ym = t * lm;
            const double X = (xp * iu) * (xm * iu) + (yp * iu) * (ym * iu), Y = (yp * iu) * (xm * iu) - (xp * iu) * (ym * iu);
            const double nx = px * X - py * Y;
            py = px * Y + py * X;
            px = nx;
            inside = inside && t > 0.0;
        }
    }
    double bsum = 0.0;
    if (ad > 0.0) {
        // in [0, pi] unless the projection is inside the triangle: there up to 2 pi
        bsum = atan2(py, px);
        if (inside && bsum < 0.0) bsum += 6.283185307179586476925286766559;
    }
    I0 -= ad * bsum;
    const double sg = (d > 0.0) - (d < 0.0);
    Ig = (-sg * bsum) * n - fu;
}

// Pairs of triangles that a lattice of boxes repeats: key of (block, test, source)
// = both shapes (triangles equal up to a shift along the box's grid) and the grid
// displacement between them.  tab[key] = row of the class in the table of slot
// integrals.
struct PairClasses {
    int* tab;                    // [shapes][shapes][nx][ny]
    const int* shape;            // [T]
    const int2* at;              // [T] grid position of each triangle
    const int2* off;             // [block] grid displacement of the test box
    int shapes, nx, ny, x0, y0;
    __device__ __forceinline__ size_t key(int b, int t, int s) const {
        const int2 d = off[b], p = at[t], q = at[s];
        return (((size_t)shape[t] * shapes + shape[s]) * nx + (p.x + d.x - q.x - x0)) * ny + (p.y + d.y - q.y - y0);
    }
};

// out[((b*Tt + t)*Ts + s)*18 + {0..8: L(i,j), 9..17: K(i,j)}]; CX: complex
// wavenumber k + j ki (lossy region), else ki is ignored; SING: closed-form
// 1/R parts.
//
// On a triangle r - v_i = sum_u lambda_u (v_u - v_i), so every slot integral
// is a combination of the 3 x 3 barycentric moments M[u][v] = sum_qp w_q w_p
// lambda_u(q) lambda_v(p) f(r_q, r'_p) of f = G and f = gfac:
//   L(i, j) = sum_{u != i, v != j} MG[u][v] (v_u - v_i).(s_v - s_j) - 4/k^2 sum MG
// and, with r - r' = a + c - b (a = r - v_i, b = r' - s_j, c = v_i - s_j),
// a.((r - r') x b) = c.(b x a):
//   K(i, j) = sum_{u != i, v != j} Mg[u][v] c.((s_v - s_j) x (v_u - v_i)),
// where the triple product depends, up to sign, on the two edges only (9
// values).  The kernel is bound by the FP64 rate (2 FMA per clock and SM):
// distance, rsqrt, sincospi and 7 operations for the moments are left per
// point pair, 0.135 ns on average over 25 blocks of 192 x 192 triangles
// (6.1 ms), against 0.37 ns (16.6 ms) when each point pair updated the 9 + 9
// slot integrals.  With closed-form parts (32 cells of 256 + 192 triangles in
// batches that fill the chip, pairs of the boxes' triangles once for all cells,
// 160 M point pairs if they were not): 48 ms (FP64 pipe 78 % busy at 7 warps per SM;
// 255 registers, spills of 0.5 % of the instructions), 59 ms without that, 100 ms with a full
// series beside the closed form of the remainder, three branches with a
// logarithm each per edge and three atan2 per point.
template <bool CX, bool SING>
__global__ void __launch_bounds__(128)
tri_pairs_kernel(const TriGeo* __restrict__ tg, int Tt, const TriGeo* __restrict__ sg, int Ts, int own,
                 int common, const double* __restrict__ shifts, int b0, double k, double ki, double2* __restrict__ out,
                 const int* __restrict__ reps, int n_reps) {
    int pair = blockIdx.x * blockDim.x + threadIdx.x, bl = blockIdx.y;
    size_t row = (size_t)bl * Tt * Ts + pair;
    if (reps) {
        // one member (b Tt + t) Ts + s of each class of pairs
        if (pair >= n_reps) return;
        row = pair;
        const int r = reps[pair];
        bl = r / (Tt * Ts);
        pair = r - bl * (Tt * Ts);
    } else if (pair >= Tt * Ts - common * common) {
        return;
    } else if (common) {
        // pairs of the first `common` triangles are left out: rows t < common start there
        const int w = Ts - common, first = common * w;
        pair = pair < first ? pair / w * Ts + common + pair % w : pair - first + common * Ts;
        row = (size_t)bl * Tt * Ts + pair;
    }
    const int t = pair / Ts, s = pair - t * Ts;
    // own: every block has its own mesh, test = source, not shifted; its first
    // `common` triangles are those of all blocks
    const TriGeo& A = tg[(own ? (b0 + bl) * Tt : 0) + t];
    const TriGeo& S = sg[(own ? (b0 + bl) * Ts : 0) + s];
    const Vec3 sh = own ? Vec3{0.0, 0.0, 0.0} : v3(shifts + 3 * (b0 + bl));
    const double kpi = k * 0.31830988618379067154;
    const double tiny2 = (1e-9 * S.scale) * (1e-9 * S.scale);
    // [G.x, G.y, g.x, g.y] of the moments
    double M[3][3][4];
#pragma unroll
    for (int u = 0; u < 3; ++u)
#pragma unroll
        for (int v = 0; v < 3; ++v)
#pragma unroll
            for (int c = 0; c < 4; ++c) M[u][v][c] = 0.0;
    // closed-form parts: sums over q of w_q lambda_u times I1 + I0 (rho - s_0), I0, Ig
    Vec3 PA[3], PC[3];
    double PB[3];
    if constexpr (SING) {
#pragma unroll
        for (int u = 0; u < 3; ++u) {
            PA[u] = PC[u] = {0.0, 0.0, 0.0};
            PB[u] = 0.0;
        }
    }
#pragma unroll 1
    for (int q = 0; q < 7; ++q) {
        const Vec3 r = v3(A.q + 3 * q) + sh;
        double N[3][4], base[4];
#pragma unroll
        for (int c = 0; c < 4; ++c) N[0][c] = N[1][c] = N[2][c] = base[c] = 0.0;
#pragma unroll
        for (int p = 0; p < 7; ++p) {
            const Vec3 diff = r - v3(S.q + 3 * p);
            const double R2 = dot(diff, diff);
            double2 G, g;
            if constexpr (SING) {
                // coincident points (up to rounding) take the R -> 0 limit of the
                // remainder: -jk/(4 pi) and no gradient term
                const bool same = R2 <= tiny2;
                const double Rs = same ? tiny2 : R2;
                if constexpr (CX) green_smooth_cx(Rs, k, kpi, ki, G, g);
                else green_smooth(Rs, k, kpi, G, g);
                if (same) {
                    G = make_double2(CX ? ki : 0.0, -k);
                    g = make_double2(0.0, 0.0);
                }
            } else {
                if constexpr (CX) green_far_cx(R2, k, kpi, ki, G, g);
                else green_far(R2, k, kpi, G, g);
            }
            const double f[4] = {G.x, G.y, g.x, g.y};
            const double wb = p == 0 ? kRw0 / 3.0 : p < 4 ? kRw1 * kRa1 : kRw2 * kRa2;
            const double wv = p < 4 ? kRw1 * (kRb1 - kRa1) : kRw2 * (kRb2 - kRa2);
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                base[c] = fma(wb, f[c], base[c]);
                if (p > 0) N[(p - 1) % 3][c] = fma(wv, f[c], N[(p - 1) % 3][c]);
            }
        }
        const double wl[3] = {c_wl[3 * q], c_wl[3 * q + 1], c_wl[3 * q + 2]};
#pragma unroll
        for (int v = 0; v < 3; ++v)
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                const double f = N[v][c] + base[c];
#pragma unroll
                for (int u = 0; u < 3; ++u) M[u][v][c] = fma(wl[u], f, M[u][v][c]);
            }
        if constexpr (SING) {
            double I0;
            Vec3 I1, Ig, rho;
            potentials(r, S, I0, I1, Ig, rho);
            const Vec3 PL = I1 + I0 * (rho - v3(S.v));
#pragma unroll
            for (int u = 0; u < 3; ++u) {
                PA[u] = PA[u] + wl[u] * PL;
                PB[u] = fma(wl[u], I0, PB[u]);
                PC[u] = PC[u] + wl[u] * Ig;
            }
        }
    }
    const Vec3 tv[3] = {v3(A.v) + sh, v3(A.v + 3) + sh, v3(A.v + 6) + sh};
    const Vec3 sv[3] = {v3(S.v), v3(S.v + 3), v3(S.v + 6)};
    // edge w of a triangle runs from vertex w + 1 to w + 2: dot products and
    // triple products of every edge pair
    double D[3][3], V[3][3];
#pragma unroll
    for (int w = 0; w < 3; ++w) {
        const Vec3 te = v3(A.v + 3 * ((w + 2) % 3)) - v3(A.v + 3 * ((w + 1) % 3));
#pragma unroll
        for (int x = 0; x < 3; ++x) {
            const Vec3 se = sv[(x + 2) % 3] - sv[(x + 1) % 3];
            D[w][x] = dot(te, se);
            V[w][x] = dot(tv[(w + 1) % 3] - sv[(x + 1) % 3], cross(se, te));
        }
    }
    double2 ik2;                                    // 4 / k^2
    if constexpr (CX) {
        const double2 k2 = make_double2(k * k - ki * ki, 2.0 * k * ki);
        const double d = 4.0 / (k2.x * k2.x + k2.y * k2.y);
        ik2 = make_double2(k2.x * d, -k2.y * d);
    } else {
        ik2 = make_double2(4.0 / (k * k), 0.0);
    }
    const double fr = A.area * S.area / kFourPi;    // regular part
    const double fs = A.area / kFourPi;             // closed-form part
    double2 sum = make_double2(0.0, 0.0);
#pragma unroll
    for (int u = 0; u < 3; ++u)
#pragma unroll
        for (int v = 0; v < 3; ++v) {
            sum.x += M[u][v][0];
            sum.y += M[u][v][1];
        }
    double2 div = make_double2(fr * sum.x, fr * sum.y);
    if constexpr (SING) div.x += fs * (PB[0] + PB[1] + PB[2]);
    if constexpr (CX) div = cmul(ik2, div);
    else div = make_double2(ik2.x * div.x, ik2.x * div.y);
    double2* o = out + row * 18;
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
        for (int j = 0; j < 3; ++j) {
            double l[2] = {0.0, 0.0}, kk[2] = {0.0, 0.0};
#pragma unroll
            for (int du = 1; du < 3; ++du)
#pragma unroll
                for (int dv = 1; dv < 3; ++dv) {
                    // vertex i + du and the edge between i and it: w = i + 2 (du = 1, i -> i + 1 runs
                    // along edge w) or w = i + 1 (du = 2, against it)
                    const int u = (i + du) % 3, v = (j + dv) % 3;
                    const int w = (i + 3 - du) % 3, x = (j + 3 - dv) % 3;
                    const double sgn = (du == dv) ? 1.0 : -1.0;
                    const double dd = sgn * D[w][x], vv = sgn * V[w][x];
                    l[0] = fma(dd, M[u][v][0], l[0]);
                    l[1] = fma(dd, M[u][v][1], l[1]);
                    kk[0] = fma(vv, M[u][v][2], kk[0]);
                    kk[1] = fma(vv, M[u][v][3], kk[1]);
                }
            double2 L = make_double2(fr * l[0] - div.x, fr * l[1] - div.y);
            double2 K = make_double2(fr * kk[0], fr * kk[1]);
            if constexpr (SING) {
                const Vec3 sj = sv[j] - sv[0], c = tv[i] - sv[j];
                double ls = 0.0, ks = 0.0;
#pragma unroll
                for (int du = 1; du < 3; ++du) {
                    const int u = (i + du) % 3;
                    const Vec3 te = v3(A.v + 3 * u) - v3(A.v + 3 * i);
                    ls += dot(te, PA[u] - PB[u] * sj);
                    ks += dot(PC[u], cross(c, te));
                }
                L.x += fs * ls;
                K.x += fs * ks;
            }
            o[3 * i + j] = L;
            o[9 + 3 * i + j] = K;
        }
}

// L[b][m][n], K[b][m][n] from the slot integrals of one chunk; own: every
// block's own RWGs, its K after its L, pairs of common triangles from Sc
__global__ void rwg_gather_kernel(const double2* __restrict__ S, const RwgSlots* __restrict__ tr,
                                  int Et, const RwgSlots* __restrict__ sr, int Es, int Tt, int Ts,
                                  int b0, int nb, int own, int common,
                                  const double2* __restrict__ Sc, double2* __restrict__ L,
                                  double2* __restrict__ K) {
    const size_t total = (size_t)nb * Et * Es;
    for (size_t e = blockIdx.x * (size_t)blockDim.x + threadIdx.x; e < total;
         e += (size_t)gridDim.x * blockDim.x) {
        const int n = (int)(e % Es);
        const size_t t2 = e / Es;
        const int m = (int)(t2 % Et);
        const int bl = (int)(t2 / Et);
        const RwgSlots A = tr[(own ? (b0 + bl) * Et : 0) + m], B = sr[(own ? (b0 + bl) * Es : 0) + n];
        double2 l = make_double2(0.0, 0.0), kk = make_double2(0.0, 0.0);
#pragma unroll
        for (int x = 0; x < 2; ++x)
#pragma unroll
            for (int y = 0; y < 2; ++y) {
                const double c = A.c[x] * B.c[y];
                const double2* p = A.t[x] < common && B.t[y] < common
                                       ? Sc + ((size_t)A.t[x] * common + B.t[y]) * 18
                                       : S + (((size_t)bl * Tt + A.t[x]) * Ts + B.t[y]) * 18;
                const int ij = 3 * A.s[x] + B.s[y];
                l.x += c * p[ij].x;
                l.y += c * p[ij].y;
                kk.x += c * p[9 + ij].x;
                kk.y += c * p[9 + ij].y;
            }
        const size_t o = ((size_t)(own ? 2 * (b0 + bl) : b0 + bl) * Et + m) * Es + n;
        L[o] = l;
        K[o] = kk;
    }
}

constexpr int kNoMember = 0x7f7f7f7f;        // memset pattern
// the lowest member (b T + t) T + s, b from b0, of every class of the blocks b0 ..
__global__ void mark_classes_kernel(PairClasses c, int T, int b0, int total) {
    for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < total; e += gridDim.x * blockDim.x) {
        const int b = e / (T * T), p = e - b * (T * T);
        atomicMin(c.tab + c.key(b0 + b, p / T, p % T), e);
    }
}
// rows for the marked classes (tab: member -> row) and their members; rows past
// cap are only counted
__global__ void number_classes_kernel(int* __restrict__ tab, size_t n, int* __restrict__ reps, int cap,
                                      int* __restrict__ count) {
    // whole warps: the vote and the shuffle are taken by all lanes
    for (size_t e0 = blockIdx.x * (size_t)blockDim.x; e0 < n; e0 += (size_t)gridDim.x * blockDim.x) {
        const size_t e = e0 + threadIdx.x;
        const int m = e < n ? tab[e] : kNoMember;
        const unsigned who = __ballot_sync(0xffffffffu, m != kNoMember);
        if (!who) continue;
        const int lane = threadIdx.x & 31, first = __ffs(who) - 1;
        int base = 0;
        if (lane == first) base = atomicAdd(count, __popc(who));
        base = __shfl_sync(0xffffffffu, base, first) + __popc(who & ((1u << lane) - 1));
        if (m == kNoMember) continue;
        tab[e] = base;
        if (base < cap) reps[base] = m;
    }
}
// L[slot][m][n], K[slot][m][n] from the classes' slot integrals, blocks b0 ..
__global__ void class_gather_kernel(const double2* __restrict__ S, PairClasses c, const RwgSlots* __restrict__ rw, int E,
                                    int b0, int nb, const int32_t* __restrict__ slot, double2* __restrict__ L,
                                    double2* __restrict__ K) {
    const size_t total = (size_t)nb * E * E;
    for (size_t e = blockIdx.x * (size_t)blockDim.x + threadIdx.x; e < total; e += (size_t)gridDim.x * blockDim.x) {
        const int n = (int)(e % E);
        const size_t t2 = e / E;
        const int m = (int)(t2 % E), b = b0 + (int)(t2 / E);
        const RwgSlots A = rw[m], B = rw[n];
        double2 l = make_double2(0.0, 0.0), kk = make_double2(0.0, 0.0);
#pragma unroll
        for (int x = 0; x < 2; ++x)
#pragma unroll
            for (int y = 0; y < 2; ++y) {
                const double f = A.c[x] * B.c[y];
                const double2* p = S + (size_t)c.tab[c.key(b, A.t[x], B.t[y])] * 18 + 3 * A.s[x] + B.s[y];
                const double2 pl = p[0], pk = p[9];
                l.x += f * pl.x;
                l.y += f * pl.y;
                kk.x += f * pk.x;
                kk.y += f * pk.y;
            }
        const size_t o = ((size_t)slot[b] * E + m) * E + n;
        L[o] = l;
        K[o] = kk;
    }
}

// ---------------------------------------------------------------- host side
void radon7(double bary[7][3], double w[7]) {
    const double s15 = std::sqrt(15.0);
    const double a1 = (6.0 - s15) / 21.0, b1 = (9.0 + 2.0 * s15) / 21.0;
    const double a2 = (6.0 + s15) / 21.0, b2 = (9.0 - 2.0 * s15) / 21.0;
    const double w1 = (155.0 - s15) / 1200.0, w2 = (155.0 + s15) / 1200.0;
    const double B[7][3] = {{1.0 / 3, 1.0 / 3, 1.0 / 3}, {b1, a1, a1}, {a1, b1, a1}, {a1, a1, b1},
                            {b2, a2, a2}, {a2, b2, a2}, {a2, a2, b2}};
    const double W[7] = {9.0 / 40.0, w1, w1, w1, w2, w2, w2};
    for (int q = 0; q < 7; ++q) {
        w[q] = W[q];
        for (int v = 0; v < 3; ++v) bary[q][v] = B[q][v];
    }
}

int prepare_mesh(const double* verts, const int32_t* tris, const int32_t* slot_rwg,
                 const int8_t* slot_sgn, int T, int E, std::vector<TriGeo>& geo,
                 std::vector<RwgSlots>& rw) {
    double bary[7][3], w[7];
    radon7(bary, w);
    geo.resize(T);
    rw.assign(E, RwgSlots{{-1, -1}, {0, 0}, {0.0, 0.0}});
    std::vector<int> seen(E, 0);
    for (int t = 0; t < T; ++t) {
        TriGeo& g = geo[t];
        double V[3][3];
        for (int v = 0; v < 3; ++v)
            for (int x = 0; x < 3; ++x) V[v][x] = g.v[3 * v + x] = verts[3 * tris[3 * t + v] + x];
        for (int q = 0; q < 7; ++q)
            for (int x = 0; x < 3; ++x)
                g.q[3 * q + x] = bary[q][0] * V[0][x] + bary[q][1] * V[1][x] + bary[q][2] * V[2][x];
        const double e1[3] = {V[1][0] - V[0][0], V[1][1] - V[0][1], V[1][2] - V[0][2]};
        const double e2[3] = {V[2][0] - V[0][0], V[2][1] - V[0][1], V[2][2] - V[0][2]};
        const double c[3] = {e1[1] * e2[2] - e1[2] * e2[1], e1[2] * e2[0] - e1[0] * e2[2],
                             e1[0] * e2[1] - e1[1] * e2[0]};
        const double cn = std::sqrt(c[0] * c[0] + c[1] * c[1] + c[2] * c[2]);
        if (!(cn > 0.0)) { set_error("degenerate triangle %d", t); return EMSURF_EINVAL; }
        g.area = 0.5 * cn;
        for (int x = 0; x < 3; ++x) g.n[x] = c[x] / cn;
        for (int i = 0; i < 3; ++i) {
            const double* p = V[i];
            const double* q = V[(i + 1) % 3];
            const double e[3] = {q[0] - p[0], q[1] - p[1], q[2] - p[2]};
            const double le = std::sqrt(e[0] * e[0] + e[1] * e[1] + e[2] * e[2]);
            double* lh = g.lh + 3 * i;
            for (int x = 0; x < 3; ++x) lh[x] = e[x] / le;
            for (int x = 0; x < 3; ++x) g.u[3 * i + x] = lh[(x + 1) % 3] * g.n[(x + 2) % 3] - lh[(x + 2) % 3] * g.n[(x + 1) % 3];
        }
        g.scale = std::max(std::sqrt(e1[0] * e1[0] + e1[1] * e1[1] + e1[2] * e1[2]),
                           std::sqrt(e2[0] * e2[0] + e2[1] * e2[1] + e2[2] * e2[2]));
        for (int i = 0; i < 3; ++i) {
            const int m = slot_rwg[3 * t + i];
            if (m < 0) continue;
            if (m >= E || seen[m] >= 2) { set_error("bad RWG slot map"); return EMSURF_EINVAL; }
            const double* p = V[(i + 1) % 3];
            const double* q = V[(i + 2) % 3];
            const double len = std::sqrt((p[0] - q[0]) * (p[0] - q[0]) + (p[1] - q[1]) * (p[1] - q[1]) +
                                         (p[2] - q[2]) * (p[2] - q[2]));
            RwgSlots& r = rw[m];
            const int x = seen[m]++;
            r.t[x] = t;
            r.s[x] = i;
            r.c[x] = (double)slot_sgn[3 * t + i] * len / (2.0 * g.area);
        }
    }
    for (int m = 0; m < E; ++m)
        if (seen[m] != 2) { set_error("RWG %d has %d triangles", m, seen[m]); return EMSURF_EINVAL; }
    return EMSURF_OK;
}

}  // namespace


namespace {
// w_q lambda_u(q) of the rule, the kernels' constant
void rule_moments(double wl[21]) {
    double bary[7][3], w[7];
    radon7(bary, w);
    for (int q = 0; q < 7; ++q)
        for (int u = 0; u < 3; ++u) wl[3 * q + u] = w[q] * bary[q][u];
}

// slot integrals of blocks b0 .. b0 + nc - 1 (singular: host flags), one
// launch per run of equal flags
cudaError_t launch_pairs(const TriGeo* tg, int Tt, const TriGeo* sg, int Ts, bool own, int common,
                         const double* shifts, const int8_t* singular, int b0, int nc, double k, double ki, double2* out, cudaStream_t st) {
    const unsigned gx = (unsigned)(((long long)Tt * Ts - (long long)common * common + 127) / 128);
    if (gx == 0) return cudaSuccess;
    for (int c = 0; c < nc;) {
        int e = c + 1;
        while (e < nc && (own || (singular[b0 + e] != 0) == (singular[b0 + c] != 0)) && e - c < 65535) ++e;
        const dim3 g(gx, (unsigned)(e - c));
        double2* o = out + (size_t)c * Tt * Ts * 18;
        const bool s = own || singular[b0 + c] != 0;
        if (ki != 0.0) {
            if (s) tri_pairs_kernel<true, true><<<g, 128, 0, st>>>(tg, Tt, sg, Ts, own, common, shifts, b0 + c, k, ki, o, nullptr, 0);
            else tri_pairs_kernel<true, false><<<g, 128, 0, st>>>(tg, Tt, sg, Ts, own, common, shifts, b0 + c, k, ki, o, nullptr, 0);
        } else {
            if (s) tri_pairs_kernel<false, true><<<g, 128, 0, st>>>(tg, Tt, sg, Ts, own, common, shifts, b0 + c, k, 0.0, o, nullptr, 0);
            else tri_pairs_kernel<false, false><<<g, 128, 0, st>>>(tg, Tt, sg, Ts, own, common, shifts, b0 + c, k, 0.0, o, nullptr, 0);
        }
        const cudaError_t err = cudaGetLastError();
        if (err != cudaSuccess) return err;
        c = e;
    }
    return cudaSuccess;
}
}  // namespace

// L, K: device [nb][Et][Es]; wavenumber k + j ki (ki = 0: lossless).  cells: nb meshes instead, each tested
// on itself (test = src = cells[b], singular), L = [nb][L, K][E][E].
static int tabulate_any(const MeshView* cells, const MeshView& test, const MeshView& src, const double* shifts,
                        const int8_t* singular, int nb, double k, double ki, double2* L, double2* K, cudaStream_t st) {
    if (!(k > 0.0) || !(ki <= 0.0) || nb < 1) {
        set_error("tabulate needs Re k > 0, Im k <= 0 and >= 1 block");
        return EMSURF_EINVAL;
    }
    const bool own = cells != nullptr;
    std::vector<TriGeo> tg, sgeo;
    std::vector<RwgSlots> tr, sr;
    for (int b = 0; b < (own ? nb : 0); ++b) {
        const MeshView& m = cells[b];
        EMS_TRY(prepare_mesh(m.verts, m.tris, m.slot_rwg, m.slot_sgn, m.T, m.E, sgeo, sr));
        tg.insert(tg.end(), sgeo.begin(), sgeo.end());
        tr.insert(tr.end(), sr.begin(), sr.end());
    }
    if (!own) {
        EMS_TRY(prepare_mesh(test.verts, test.tris, test.slot_rwg, test.slot_sgn, test.T, test.E, tg, tr));
        EMS_TRY(prepare_mesh(src.verts, src.tris, src.slot_rwg, src.slot_sgn, src.T, src.E, sgeo, sr));
    }
    double wl[21];
    rule_moments(wl);
    EMS_CUDA(cudaMemcpyToSymbolAsync(c_wl, wl, sizeof(wl), 0, cudaMemcpyHostToDevice, st));
    const size_t per_block = (size_t)test.T * src.T * 18 * sizeof(double2);
    const int chunk = (int)std::max<size_t>(1, std::min<size_t>(nb, kScratchBytes / per_block));
    // leading triangles that all cells share (a library's boxes), bit for bit: their
    // pairs are integrated once
    int common = own && nb > 1 ? test.T : 0;
    for (int b = 1; b < (own ? nb : 0); ++b) {
        int c = 0;
        while (c < common && !std::memcmp(&tg[c], &tg[(size_t)b * test.T + c], sizeof(TriGeo))) ++c;
        common = c;
    }
    TriGeo *dtg = nullptr, *dsg = nullptr;
    RwgSlots *dtr = nullptr, *dsr = nullptr;
    double* dsh = nullptr;
    double2 *scratch = nullptr, *shared = nullptr;
    int status = EMSURF_OK;
    auto fail = [&](cudaError_t e, const char* what) {
        set_error("tabulate: %s: %s", what, cudaGetErrorString(e));
        status = EMSURF_ECUDA;
    };
    cudaError_t e;
    if ((e = cudaMalloc(&dtg, sizeof(TriGeo) * tg.size())) != cudaSuccess) fail(e, "alloc");
    if (!status && !own && (e = cudaMalloc(&dsg, sizeof(TriGeo) * sgeo.size())) != cudaSuccess) fail(e, "alloc");
    if (!status && (e = cudaMalloc(&dtr, sizeof(RwgSlots) * tr.size())) != cudaSuccess) fail(e, "alloc");
    if (!status && !own && (e = cudaMalloc(&dsr, sizeof(RwgSlots) * sr.size())) != cudaSuccess) fail(e, "alloc");
    if (!status && !own && (e = cudaMalloc(&dsh, sizeof(double) * 3 * nb)) != cudaSuccess) fail(e, "alloc");
    if (!status && (e = cudaMalloc(&scratch, per_block * chunk)) != cudaSuccess) fail(e, "scratch alloc");
    if (!status && common && (e = cudaMalloc(&shared, (size_t)common * common * 18 * sizeof(double2))) != cudaSuccess)
        fail(e, "scratch alloc");
    if (!status) {
        cudaMemcpyAsync(dtg, tg.data(), sizeof(TriGeo) * tg.size(), cudaMemcpyHostToDevice, st);
        cudaMemcpyAsync(dtr, tr.data(), sizeof(RwgSlots) * tr.size(), cudaMemcpyHostToDevice, st);
        if (!own) {
            cudaMemcpyAsync(dsg, sgeo.data(), sizeof(TriGeo) * sgeo.size(), cudaMemcpyHostToDevice, st);
            cudaMemcpyAsync(dsr, sr.data(), sizeof(RwgSlots) * sr.size(), cudaMemcpyHostToDevice, st);
            cudaMemcpyAsync(dsh, shifts, sizeof(double) * 3 * nb, cudaMemcpyHostToDevice, st);
        }
        const TriGeo* ds = own ? dtg : dsg;
        const RwgSlots* drs = own ? dtr : dsr;
        if (common && (e = launch_pairs(dtg, common, dtg, common, true, 0, dsh, singular, 0, 1, k, ki, shared, st)) != cudaSuccess)
            fail(e, "tri_pairs_kernel");
        for (int b0 = 0; b0 < nb && !status; b0 += chunk) {
            const int nc = std::min(chunk, nb - b0);
            e = launch_pairs(dtg, test.T, ds, src.T, own, common, dsh, singular, b0, nc, k, ki, scratch, st);
            if (e != cudaSuccess) { fail(e, "tri_pairs_kernel"); break; }
            const size_t tot = (size_t)nc * test.E * src.E;
            const int g2 = (int)std::min<size_t>((tot + 255) / 256, 152 * 64);
            rwg_gather_kernel<<<g2, 256, 0, st>>>(scratch, dtr, test.E, drs, src.E, test.T, src.T, b0, nc, own, common, shared, L,
                                                  own ? L + (size_t)test.E * src.E : K);
            if ((e = cudaGetLastError()) != cudaSuccess) { fail(e, "rwg_gather_kernel"); break; }
        }
        if (!status && (e = cudaStreamSynchronize(st)) != cudaSuccess) fail(e, "synchronize");
    }
    cudaFree(dtg);
    cudaFree(dsg);
    cudaFree(dtr);
    cudaFree(dsr);
    cudaFree(dsh);
    cudaFree(scratch);
    cudaFree(shared);
    return status;
}

int tabulate_blocks_cx(const MeshView& test, const MeshView& src, const double* shifts,
                       const int8_t* singular, int nb, double k, double ki, double2* L, double2* K,
                       cudaStream_t st) {
    return tabulate_any(nullptr, test, src, shifts, singular, nb, k, ki, L, K, st);
}

// LK[b] = L, K of cell b on itself; all meshes have the same number of triangles and RWGs
int tabulate_cells_cx(const std::vector<MeshView>& cells, double k, double ki, double2* LK, cudaStream_t st) {
    return tabulate_any(cells.data(), cells[0], cells[0], nullptr, nullptr, (int)cells.size(), k, ki, LK, nullptr, st);
}

// L, K of one box against its copies at the grid displacements off (box sides of
// nq grid steps; the first n_touch blocks touch), block b at slot[b].  The mesh
// repeats itself along its faces and from box to box, so most pairs of triangles
// are shifted copies of others: one of each class is integrated (16 x 16 boxes
// of 192 triangles: 1.6 of 4.9 million pairs), and the blocks are gathered from
// the classes' table.  Chunks of blocks keep the table below kScratchBytes.
static int tabulate_lattice(const MeshView& m, const std::vector<int2>& off, int nq, double a, double b_, int n_touch,
                            double k, double2* L, double2* K, const std::vector<int32_t>& slot, cudaStream_t st) {
    if (!(k > 0.0)) {
        set_error("tabulate needs k > 0");
        return EMSURF_EINVAL;
    }
    std::vector<TriGeo> geo;
    std::vector<RwgSlots> rw;
    EMS_TRY(prepare_mesh(m.verts, m.tris, m.slot_rwg, m.slot_sgn, m.T, m.E, geo, rw));
    const int nb = (int)off.size(), T = m.T;
    const double hx = a / nq, hy = b_ / nq;
    // grid position of each triangle's lowest corner and its shape: equal vertices
    // relative to it, in any order of triangles; one off the grid is a shape of its own
    std::vector<int> shape(T, -1);
    std::vector<int2> at(T);
    std::vector<int> first;                       // a triangle of each shape
    double mx = geo[0].v[0], my = geo[0].v[1];
    for (const TriGeo& g : geo)
        for (int v = 0; v < 3; ++v) {
            mx = std::min(mx, g.v[3 * v]);
            my = std::min(my, g.v[3 * v + 1]);
        }
    auto corner = [&](const TriGeo& g, int x) { return std::min(g.v[x], std::min(g.v[3 + x], g.v[6 + x])); };
    for (int t = 0; t < T; ++t) {
        const double px = (corner(geo[t], 0) - mx) / hx, py = (corner(geo[t], 1) - my) / hy;
        at[t] = make_int2((int)std::lround(px), (int)std::lround(py));
        const bool on = std::fabs(px - at[t].x) <= 1e-9 && std::fabs(py - at[t].y) <= 1e-9;
        for (int f = 0; on && f < (int)first.size() && shape[t] < 0; ++f) {
            bool same = true;
            for (int v = 0; v < 9 && same; ++v) {
                const int x = v % 3;
                const double u = geo[t].v[v] - (x < 2 ? corner(geo[t], x) : 0.0);
                const double w = geo[first[f]].v[v] - (x < 2 ? corner(geo[first[f]], x) : 0.0);
                same = std::fabs(u - w) <= 1e-9 * std::min(hx, hy);
            }
            if (same) shape[t] = f;
        }
        if (shape[t] < 0) {
            shape[t] = (int)first.size();
            first.push_back(t);
        }
    }
    const int S = (int)first.size();
    std::vector<double> shifts(3 * (size_t)nb);
    for (int b = 0; b < nb; ++b) {
        shifts[3 * b] = off[b].x / nq * a;
        shifts[3 * b + 1] = off[b].y / nq * b_;
        shifts[3 * b + 2] = 0.0;
    }
    // classes of blocks b0 .. b0 + nc: extent of the displacements
    auto extent = [&](int b0, int nc, PairClasses& c) {
        int lx = off[b0].x, hx_ = lx, ly = off[b0].y, hy_ = ly;
        for (int b = b0; b < b0 + nc; ++b) {
            lx = std::min(lx, off[b].x);
            hx_ = std::max(hx_, off[b].x);
            ly = std::min(ly, off[b].y);
            hy_ = std::max(hy_, off[b].y);
        }
        c.x0 = lx - nq;
        c.y0 = ly - nq;
        c.nx = hx_ - lx + 2 * nq + 1;
        c.ny = hy_ - ly + 2 * nq + 1;
        return (size_t)S * S * c.nx * c.ny;
    };
    constexpr size_t kTabBytes = 64ull << 20;
    const int cap = (int)std::max<size_t>(kScratchBytes / (18 * sizeof(double2)), (size_t)T * T);
    // the most blocks a chunk may have, then less until its classes fit
    auto chunk_of = [&](int b0, int end) {
        PairClasses c;
        int nc = (int)std::min<long long>(end - b0, kNoMember / ((long long)T * T));
        while (nc > 1 && extent(b0, nc, c) * sizeof(int) > kTabBytes) nc = (nc + 1) / 2;
        return std::max(nc, 1);
    };
    // a chunk's extent is that of one block, below the limit, or that of all blocks
    PairClasses whole;
    const size_t one = (size_t)S * S * (2 * nq + 1) * (2 * nq + 1);
    const size_t tab_n = std::min(std::max(kTabBytes / sizeof(int), one), extent(0, nb, whole));
    double wl[21];
    rule_moments(wl);
    EMS_CUDA(cudaMemcpyToSymbolAsync(c_wl, wl, sizeof(wl), 0, cudaMemcpyHostToDevice, st));
    // one buffer: class table, members, slot integrals, then the mesh and the blocks
    size_t bytes = 0;
    auto part = [&](size_t n) {
        const size_t o = bytes;
        bytes += (n + 255) & ~(size_t)255;
        return o;
    };
    const long long all = (long long)nb * T * T;
    const int rows = (int)std::min<long long>(cap, all);
    const size_t o_tab = part(tab_n * sizeof(int)), o_rep = part((size_t)rows * sizeof(int)), o_cnt = part(sizeof(int)),
                 o_S = part((size_t)rows * 18 * sizeof(double2)), o_geo = part(T * sizeof(TriGeo)),
                 o_rw = part(m.E * sizeof(RwgSlots)), o_sh = part(T * sizeof(int)), o_at = part(T * sizeof(int2)),
                 o_off = part(nb * sizeof(int2)), o_slot = part(nb * sizeof(int32_t)), o_shift = part(3 * nb * sizeof(double));
    unsigned char* w = nullptr;
    cudaError_t e = cudaMalloc(&w, bytes);
    if (e != cudaSuccess) {
        cudaGetLastError();
        set_error("tabulate: device allocation of %zu bytes: %s", bytes, cudaGetErrorString(e));
        return EMSURF_ECUDA;
    }
    auto put = [&](size_t o, const void* src, size_t n) {
        if (e == cudaSuccess) e = cudaMemcpyAsync(w + o, src, n, cudaMemcpyHostToDevice, st);
    };
    put(o_geo, geo.data(), T * sizeof(TriGeo));
    put(o_rw, rw.data(), m.E * sizeof(RwgSlots));
    put(o_sh, shape.data(), T * sizeof(int));
    put(o_at, at.data(), T * sizeof(int2));
    put(o_off, off.data(), nb * sizeof(int2));
    put(o_slot, slot.data(), nb * sizeof(int32_t));
    put(o_shift, shifts.data(), 3 * nb * sizeof(double));
    int *tab = reinterpret_cast<int*>(w + o_tab), *reps = reinterpret_cast<int*>(w + o_rep), *cnt = reinterpret_cast<int*>(w + o_cnt);
    double2* U = reinterpret_cast<double2*>(w + o_S);
    const TriGeo* dg = reinterpret_cast<const TriGeo*>(w + o_geo);
    const RwgSlots* dr = reinterpret_cast<const RwgSlots*>(w + o_rw);
    const double* dsh = reinterpret_cast<const double*>(w + o_shift);
    for (int b0 = 0; b0 < nb && e == cudaSuccess;) {
        const bool touch = b0 < n_touch;
        int nc = chunk_of(b0, touch ? n_touch : nb), n_cls = 0;
        PairClasses c{tab, reinterpret_cast<const int*>(w + o_sh), reinterpret_cast<const int2*>(w + o_at),
                      reinterpret_cast<const int2*>(w + o_off), S, 0, 0, 0, 0};
        for (;;) {
            const size_t n = extent(b0, nc, c);
            const int total = nc * T * T;
            e = cudaMemsetAsync(tab, 0x7f, n * sizeof(int), st);          // 0x7f7f7f7f: no member
            if (e == cudaSuccess) e = cudaMemsetAsync(cnt, 0, sizeof(int), st);
            if (e != cudaSuccess) break;
            mark_classes_kernel<<<std::min((total + 255) / 256, 152 * 32), 256, 0, st>>>(c, T, b0, total);
            number_classes_kernel<<<(int)std::min<size_t>((n + 255) / 256, 152 * 16), 256, 0, st>>>(tab, n, reps, rows, cnt);
            e = cudaGetLastError();
            if (e == cudaSuccess) e = cudaMemcpyAsync(&n_cls, cnt, sizeof(int), cudaMemcpyDeviceToHost, st);
            if (e == cudaSuccess) e = cudaStreamSynchronize(st);
            if (e != cudaSuccess || n_cls <= rows) break;
            nc = std::max(1, std::min(nc - 1, (int)((double)nc * rows / n_cls * 0.95)));
        }
        if (e != cudaSuccess) break;
        const dim3 g((unsigned)((n_cls + 127) / 128));
        if (touch) tri_pairs_kernel<false, true><<<g, 128, 0, st>>>(dg, T, dg, T, 0, 0, dsh, b0, k, 0.0, U, reps, n_cls);
        else tri_pairs_kernel<false, false><<<g, 128, 0, st>>>(dg, T, dg, T, 0, 0, dsh, b0, k, 0.0, U, reps, n_cls);
        const size_t tot = (size_t)nc * m.E * m.E;
        class_gather_kernel<<<(int)std::min<size_t>((tot + 255) / 256, 152 * 64), 256, 0, st>>>(
            U, c, dr, m.E, b0, nc, reinterpret_cast<const int32_t*>(w + o_slot), L, K);
        e = cudaGetLastError();
        b0 += nc;
    }
    const cudaError_t es = cudaStreamSynchronize(st);
    if (e == cudaSuccess) e = es;
    cudaFree(w);
    if (e != cudaSuccess) {
        set_error("tabulate: %s", cudaGetErrorString(e));
        return EMSURF_ECUDA;
    }
    return EMSURF_OK;
}

int tabulate_blocks(const MeshView& test, const MeshView& src, const double* shifts,
                    const int8_t* singular, int nb, double k, double2* L, double2* K,
                    cudaStream_t st) {
    return tabulate_blocks_cx(test, src, shifts, singular, nb, k, 0.0, L, K, st);
}

// ---------------------------------------------------------------------------
// Allocation-free tabulation.  Scratch lives in one file-scope device array
// that every GPU loading this library holds until the process exits.  Host
// code must not use the array's name as a device address (it is a host-side
// stand-in); the device address comes from cudaGetSymbolAddress, taken once
// per device with that device current and cached.
namespace {

constexpr size_t kNoAllocBytes = 64ull << 20;   // 64 MiB per device
static __device__ __align__(256) unsigned char g_tab_scratch[kNoAllocBytes];

std::mutex g_tab_scratch_mu;
constexpr int kMaxDevices = 64;
struct ScratchAddr {
    void* ctx = nullptr;     // context the address was taken in
    void* addr = nullptr;
};
ScratchAddr g_tab_scratch_addr[kMaxDevices];

// cuCtxGetCurrent through the runtime's driver entry point (no link to the
// driver library); a context created after a device reset gets a new handle,
// so the cached address is taken again in it
using CtxGetCurrentFn = int (*)(void**);
CtxGetCurrentFn ctx_get_current() {
    static CtxGetCurrentFn fn = [] {
        void* f = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuCtxGetCurrent", &f, 12000, cudaEnableDefault, &q) !=
                cudaSuccess || q != cudaDriverEntryPointSuccess)
            f = nullptr;
        return reinterpret_cast<CtxGetCurrentFn>(f);
    }();
    return fn;
}

int scratch_address(void** out) {
    int dev = -1;
    EMS_CUDA(cudaGetDevice(&dev));
    if (dev < 0 || dev >= kMaxDevices) {
        set_error("device ordinal %d outside [0, %d)", dev, kMaxDevices);
        return EMSURF_EINVAL;
    }
    const CtxGetCurrentFn fn = ctx_get_current();
    void* ctx = nullptr;
    if (fn) fn(&ctx);
    std::lock_guard<std::mutex> lock(g_tab_scratch_mu);
    ScratchAddr& c = g_tab_scratch_addr[dev];
    if (!c.addr || !ctx || c.ctx != ctx) {
        void* p = nullptr;
        // binds the device's primary context if none is current yet
        const cudaError_t e = cudaGetSymbolAddress(&p, g_tab_scratch);
        if (e != cudaSuccess || !p) {
            set_error("cudaGetSymbolAddress of the static scratch failed on device %d: %s", dev,
                      cudaGetErrorString(e));
            return EMSURF_ECUDA;
        }
        if (fn && !ctx) fn(&ctx);
        c.ctx = ctx;
        c.addr = p;
    }
    *out = c.addr;
    return EMSURF_OK;
}

size_t align256(size_t b) { return (b + 255) & ~size_t(255); }

int tabulate_blocks_noalloc(const MeshView& test, const MeshView& src, const double* shifts,
                            const int8_t* singular, int nb, double k, double2* L, double2* K,
                            cudaStream_t st) {
    if (!(k > 0.0) || nb < 1) { set_error("tabulate needs k > 0 and >= 1 block"); return EMSURF_EINVAL; }
    std::vector<TriGeo> tg, sgeo;
    std::vector<RwgSlots> tr, sr;
    EMS_TRY(prepare_mesh(test.verts, test.tris, test.slot_rwg, test.slot_sgn, test.T, test.E, tg, tr));
    EMS_TRY(prepare_mesh(src.verts, src.tris, src.slot_rwg, src.slot_sgn, src.T, src.E, sgeo, sr));
    // carve the static array: geometry, then the per-chunk pair integrals
    const size_t o_tg = 0;
    const size_t o_sg = o_tg + align256(sizeof(TriGeo) * tg.size());
    const size_t o_tr = o_sg + align256(sizeof(TriGeo) * sgeo.size());
    const size_t o_sr = o_tr + align256(sizeof(RwgSlots) * tr.size());
    const size_t o_sh = o_sr + align256(sizeof(RwgSlots) * sr.size());
    const size_t o_pairs = o_sh + align256(sizeof(double) * 3 * (size_t)nb);
    const size_t per_block = (size_t)test.T * src.T * 18 * sizeof(double2);
    if (o_pairs + per_block > kNoAllocBytes) {
        set_error("emsurf_tabulate_noalloc needs %zu bytes of scratch for these meshes and %d "
                  "blocks; its static scratch holds %zu bytes",
                  o_pairs + per_block, nb, kNoAllocBytes);
        return EMSURF_EINVAL;
    }
    void* base = nullptr;
    EMS_TRY(scratch_address(&base));
    unsigned char* b = static_cast<unsigned char*>(base);
    TriGeo* dtg = reinterpret_cast<TriGeo*>(b + o_tg);
    TriGeo* dsg = reinterpret_cast<TriGeo*>(b + o_sg);
    RwgSlots* dtr = reinterpret_cast<RwgSlots*>(b + o_tr);
    RwgSlots* dsr = reinterpret_cast<RwgSlots*>(b + o_sr);
    double* dsh = reinterpret_cast<double*>(b + o_sh);
    double2* pairs = reinterpret_cast<double2*>(b + o_pairs);
    const int chunk = (int)std::min<size_t>(nb, (kNoAllocBytes - o_pairs) / per_block);
    double wl[21];
    rule_moments(wl);
    // from the first queued copy on, every return goes through the stream
    // synchronisation below, so no queued work outlives the call
    int status = EMSURF_OK;
    auto step = [&](cudaError_t e, const char* what) {
        if (status == EMSURF_OK && e != cudaSuccess) {
            set_error("emsurf_tabulate_noalloc: %s: %s", what, cudaGetErrorString(e));
            status = EMSURF_ECUDA;
        }
    };
    step(cudaMemcpyToSymbolAsync(c_wl, wl, sizeof(wl), 0, cudaMemcpyHostToDevice, st), "copy weights");
    if (!status) step(cudaMemcpyAsync(dtg, tg.data(), sizeof(TriGeo) * tg.size(), cudaMemcpyHostToDevice, st), "copy");
    if (!status) step(cudaMemcpyAsync(dsg, sgeo.data(), sizeof(TriGeo) * sgeo.size(), cudaMemcpyHostToDevice, st), "copy");
    if (!status) step(cudaMemcpyAsync(dtr, tr.data(), sizeof(RwgSlots) * tr.size(), cudaMemcpyHostToDevice, st), "copy");
    if (!status) step(cudaMemcpyAsync(dsr, sr.data(), sizeof(RwgSlots) * sr.size(), cudaMemcpyHostToDevice, st), "copy");
    if (!status) step(cudaMemcpyAsync(dsh, shifts, sizeof(double) * 3 * nb, cudaMemcpyHostToDevice, st), "copy");
    // every pair integral is written before it is read, so nothing needs clearing
    for (int b0 = 0; b0 < nb && !status; b0 += chunk) {
        const int nc = std::min(chunk, nb - b0);
        step(launch_pairs(dtg, test.T, dsg, src.T, false, 0, dsh, singular, b0, nc, k, 0.0, pairs, st), "tri_pairs_kernel");
        if (status) break;
        const size_t tot = (size_t)nc * test.E * src.E;
        const int g2 = (int)std::min<size_t>((tot + 255) / 256, 152 * 64);
        rwg_gather_kernel<<<g2, 256, 0, st>>>(pairs, dtr, test.E, dsr, src.E, test.T, src.T, b0, nc, 0, 0,
                                              nullptr, L, K);
        step(cudaGetLastError(), "rwg_gather_kernel");
    }
    step(cudaStreamSynchronize(st), "synchronize");
    return status;
}

}  // namespace

}  // namespace emsurf

using namespace emsurf;

extern "C" {

EMSURF_API int emsurf_tabulate_noalloc(const double* test_verts, const int32_t* test_tris,
                                       const int32_t* test_slot_rwg, const int8_t* test_slot_sgn,
                                       int32_t test_T, int32_t test_E, const double* src_verts,
                                       const int32_t* src_tris, const int32_t* src_slot_rwg,
                                       const int8_t* src_slot_sgn, int32_t src_T, int32_t src_E,
                                       const double* shifts, const int8_t* singular,
                                       int32_t n_blocks, double k, emsurf_c128* L, emsurf_c128* K,
                                       void* stream) {
    if (!test_verts || !test_tris || !test_slot_rwg || !test_slot_sgn || !src_verts || !src_tris ||
        !src_slot_rwg || !src_slot_sgn || !shifts || !singular || !L || !K || test_T < 1 ||
        src_T < 1 || test_E < 1 || src_E < 1) {
        set_error("emsurf_tabulate_noalloc: NULL pointer or empty mesh");
        return EMSURF_EINVAL;
    }
    MeshView t{test_verts, test_tris, test_slot_rwg, test_slot_sgn, test_T, test_E};
    MeshView s{src_verts, src_tris, src_slot_rwg, src_slot_sgn, src_T, src_E};
    return tabulate_blocks_noalloc(t, s, shifts, singular, n_blocks, k, reinterpret_cast<double2*>(L),
                                   reinterpret_cast<double2*>(K), reinterpret_cast<cudaStream_t>(stream));
}

EMSURF_API int emsurf_tabulate(const double* test_verts, const int32_t* test_tris,
                               const int32_t* test_slot_rwg, const int8_t* test_slot_sgn,
                               int32_t test_T, int32_t test_E, const double* src_verts,
                               const int32_t* src_tris, const int32_t* src_slot_rwg,
                               const int8_t* src_slot_sgn, int32_t src_T, int32_t src_E,
                               const double* shifts, const int8_t* singular, int32_t n_blocks,
                               double k, emsurf_c128* L, emsurf_c128* K, void* stream) {
    if (!test_verts || !test_tris || !test_slot_rwg || !test_slot_sgn || !src_verts || !src_tris ||
        !src_slot_rwg || !src_slot_sgn || !shifts || !singular || !L || !K || test_T < 1 ||
        src_T < 1 || test_E < 1 || src_E < 1) {
        set_error("emsurf_tabulate: NULL pointer or empty mesh");
        return EMSURF_EINVAL;
    }
    MeshView t{test_verts, test_tris, test_slot_rwg, test_slot_sgn, test_T, test_E};
    MeshView s{src_verts, src_tris, src_slot_rwg, src_slot_sgn, src_T, src_E};
    return tabulate_blocks(t, s, shifts, singular, n_blocks, k, reinterpret_cast<double2*>(L),
                           reinterpret_cast<double2*>(K), reinterpret_cast<cudaStream_t>(stream));
}

}  // extern "C"

namespace emsurf {
namespace {
// T(d) <- (T(d) + T(-d)^T) / 2 for both tables in place, for the listed pairs
// (o, om) of the offsets d and -d (o == om: d = 0), blockIdx.y = pair, one
// thread per entry pair.
__global__ void reciprocal_part_kernel(double2* __restrict__ L, double2* __restrict__ K,
                                       const int2* __restrict__ pairs, int E) {
    const size_t EE = (size_t)E * E;
    const int o = pairs[blockIdx.y].x, om = pairs[blockIdx.y].y;
    for (size_t e = blockIdx.x * (size_t)blockDim.x + threadIdx.x; e < EE; e += (size_t)gridDim.x * blockDim.x) {
        const int i = (int)(e / E), j = (int)(e % E);
        if (o == om && i >= j) continue;
        const size_t p = (size_t)o * EE + e, q = (size_t)om * EE + (size_t)j * E + i;
        double2 t[2] = {L[p], K[p]};
        double2 u[2] = {L[q], K[q]};
        const double2 sl = make_double2((t[0].x + u[0].x) * 0.5, (t[0].y + u[0].y) * 0.5);
        const double2 sk = make_double2((t[1].x + u[1].x) * 0.5, (t[1].y + u[1].y) * 0.5);
        L[p] = sl;
        L[q] = sl;
        K[p] = sk;
        K[q] = sk;
    }
}

// One offset that takes its block from offset `rep` through group element
// `elem` (bits 0..2: the box's x, y and x <-> y mirrors) and, with bit 3, the
// transpose of reciprocity.
struct OffsetImage {
    int32_t slot, rep, elem;
};

// T(d')[pi(i)][pi(j)] = s sign(i) sign(j) T(d)[i][j] (transposed with bit 3),
// s = 1 for L and det(g) for K.  inv[g][n] = pi^-1(n) | (sign < 0) << 31.
// One CTA per 32 x 32 tile of an output block: its source entries lie in 32
// rows (columns) of the L2-resident source block.
__global__ void __launch_bounds__(256)
expand_offsets_kernel(double2* __restrict__ L, double2* __restrict__ K, const OffsetImage* __restrict__ img,
                      const uint32_t* __restrict__ inv, int E) {
    const OffsetImage m = img[blockIdx.z];
    const uint32_t* pi = inv + (size_t)(m.elem & 7) * E;
    const bool tr = m.elem & 8;
    const double det = (__popc(m.elem & 7) & 1) ? -1.0 : 1.0;
    const size_t EE = (size_t)E * E, src = (size_t)m.rep * EE, dst = (size_t)m.slot * EE;
    const int j = blockIdx.x * 32 + threadIdx.x;
    if (j >= E) return;
    const uint32_t pj = pi[j];
#pragma unroll
    for (int r = 0; r < 32; r += 8) {
        const int i = blockIdx.y * 32 + r + threadIdx.y;
        if (i >= E) break;
        const uint32_t pr = pi[i];
        const size_t a = pr & 0x7fffffffu, b = pj & 0x7fffffffu;
        const size_t at = src + (tr ? b * E + a : a * E + b);
        const double s = ((pr ^ pj) >> 31) ? -1.0 : 1.0;
        const double2 l = L[at], k = K[at];
        L[dst + (size_t)i * E + j] = make_double2(s * l.x, s * l.y);
        K[dst + (size_t)i * E + j] = make_double2(s * det * k.x, s * det * k.y);
    }
}
}  // namespace
}  // namespace emsurf

extern "C" {

// The tables' symmetries leave few offsets to integrate: with the box's
// mirrors g (emsurf_setup_box_mirrors) L(g d) = P_g L(d) P_g^T and K(g d) =
// det(g) P_g K(d) P_g^T, and the reciprocal part obeys T(-d) = T(d)^T (exact
// for the two-sided quadrature of offsets that do not touch).  One offset of
// each orbit is integrated (136 of 961 on a 16 x 16 lattice of square cells
// with even n), touching ones together with their -d; the others are signed
// permutations of it.  Tabulation is bound by the FP64 rate, so its time
// follows the integrated pairs: 15.4 ms for 16 x 16 boxes of 288 RWGs, 38 ms
// without the classes of shifted pairs, 650 ms with every offset integrated
// point pair by point pair.
EMSURF_API int emsurf_tabulate_offsets(double a, double b, double h, int32_t n,
                                       const double* zlevels, int32_t nx, int32_t ny, double k,
                                       emsurf_c128* L, emsurf_c128* K, void* stream) {
    if (n < 1 || nx < 1 || ny < 1 || !L || !K) {
        set_error("emsurf_tabulate_offsets: bad sizes or NULL output");
        return EMSURF_EINVAL;
    }
    int32_t V, T, E;
    EMS_TRY(emsurf_setup_box_counts(n, &V, &T, &E));
    std::vector<double> verts(3 * V);
    std::vector<int32_t> tris(3 * T), edges(2 * E), tp(E), tm(E), srw(3 * T);
    std::vector<int8_t> ssg(3 * T);
    EMS_TRY(emsurf_setup_box_mesh(a, b, h, n, zlevels, verts.data(), tris.data(), edges.data(),
                                  tp.data(), tm.data(), srw.data(), ssg.data()));
    // inverse signed permutations of the 8 products of mirrors (P_g = Px^a Py^b Pd^c)
    std::vector<int32_t> perm(3 * (size_t)E);
    std::vector<int8_t> sign(3 * (size_t)E);
    int32_t mask = 0;
    EMS_TRY(emsurf_setup_box_mirrors(a, b, n, perm.data(), sign.data(), &mask));
    std::vector<uint32_t> inv(8 * (size_t)E);
    for (int g = 0; g < 8; ++g) {
        if (g & ~mask) continue;
        for (int e = 0; e < E; ++e) {
            int at = e, sg = 1;
            for (int bit : {2, 1, 0})           // the x <-> y mirror first
                if (g & (1 << bit)) {
                    sg *= sign[(size_t)bit * E + at];
                    at = perm[(size_t)bit * E + at];
                }
            inv[(size_t)g * E + at] = (uint32_t)e | (sg < 0 ? 0x80000000u : 0u);
        }
    }
    const int nox = 2 * nx - 1, noy = 2 * ny - 1, nof = nox * noy;
    std::vector<int32_t> rep_of(nof, -1);
    std::vector<int32_t> slot;                  // integrated offsets: touching ones first
    std::vector<int2> touch;                    // (d, -d) of the touching representatives
    std::vector<OffsetImage> image;
    std::vector<int32_t> far;
    auto touching = [](int dx, int dy) { return std::abs(dx) <= 1 && std::abs(dy) <= 1; };
    for (int o = 0; o < nof; ++o) {
        if (rep_of[o] >= 0) continue;
        const int dx = o % nox - (nx - 1), dy = o / nox - (ny - 1);
        rep_of[o] = o;
        if (touching(dx, dy)) {
            slot.push_back(o);
            const int om = nof - 1 - o;
            if (om != o) {
                slot.push_back(om);
                rep_of[om] = o;                 // its reciprocal part is written with d's
            }
            touch.push_back(make_int2(o, om));
        } else {
            far.push_back(o);
        }
        // d' and -d' together, so that T(-d') = T(d')^T entry by entry
        for (int g = 0; g < 8; ++g) {
            if (g & ~mask) continue;
            int x = dx, y = dy;
            if (g & 4) std::swap(x, y);
            if (g & 1) x = -x;
            if (g & 2) y = -y;
            if (std::abs(x) >= nx || std::abs(y) >= ny) continue;
            const int q = (y + ny - 1) * nox + x + nx - 1, qm = nof - 1 - q;
            for (const OffsetImage& m : {OffsetImage{q, o, g}, OffsetImage{qm, o, g | 8}})
                if (rep_of[m.slot] < 0) {
                    rep_of[m.slot] = o;
                    image.push_back(m);
                }
        }
    }
    const int n_touch = (int)slot.size();
    slot.insert(slot.end(), far.begin(), far.end());
    std::vector<int2> off(slot.size());
    for (size_t i = 0; i < slot.size(); ++i)
        off[i] = make_int2((slot[i] % nox - (nx - 1)) * n, (slot[i] / nox - (ny - 1)) * n);
    MeshView mv{verts.data(), tris.data(), srw.data(), ssg.data(), T, E};
    cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
    double2* Ld = reinterpret_cast<double2*>(L);
    double2* Kd = reinterpret_cast<double2*>(K);
    EMS_TRY(tabulate_lattice(mv, off, n, a, b, n_touch, k, Ld, Kd, slot, st));
    // reciprocal part of the touching blocks, then the images
    unsigned char* dbuf = nullptr;
    const size_t b_touch = touch.size() * sizeof(int2), b_inv = inv.size() * sizeof(uint32_t);
    const size_t b_img = std::max<size_t>(1, image.size()) * sizeof(OffsetImage);
    if (cudaMalloc(&dbuf, b_touch + b_inv + b_img) != cudaSuccess) {
        cudaGetLastError();
        set_error("emsurf_tabulate_offsets: device allocation failed");
        return EMSURF_ENOMEM;
    }
    int2* dtouch = reinterpret_cast<int2*>(dbuf);
    uint32_t* dinv = reinterpret_cast<uint32_t*>(dbuf + b_touch);
    OffsetImage* dimg = reinterpret_cast<OffsetImage*>(dbuf + b_touch + b_inv);
    cudaError_t e = cudaMemcpyAsync(dtouch, touch.data(), b_touch, cudaMemcpyHostToDevice, st);
    if (e == cudaSuccess) e = cudaMemcpyAsync(dinv, inv.data(), b_inv, cudaMemcpyHostToDevice, st);
    if (e == cudaSuccess && !image.empty())
        e = cudaMemcpyAsync(dimg, image.data(), image.size() * sizeof(OffsetImage), cudaMemcpyHostToDevice, st);
    if (e == cudaSuccess) {
        const size_t EE = (size_t)E * E;
        reciprocal_part_kernel<<<dim3((unsigned)std::min<size_t>((EE + 255) / 256, 1024), (unsigned)touch.size()), 256,
                                 0, st>>>(Ld, Kd, dtouch, E);
        e = cudaGetLastError();
    }
    for (size_t i0 = 0; i0 < image.size() && e == cudaSuccess; i0 += 65535) {
        const dim3 grid((E + 31) / 32, (E + 31) / 32, (unsigned)std::min<size_t>(65535, image.size() - i0));
        expand_offsets_kernel<<<grid, dim3(32, 8), 0, st>>>(Ld, Kd, dimg + i0, dinv, E);
        e = cudaGetLastError();
    }
    const cudaError_t es = cudaStreamSynchronize(st);
    cudaFree(dbuf);
    if (e == cudaSuccess) e = es;
    if (e != cudaSuccess) {
        set_error("emsurf_tabulate_offsets: %s", cudaGetErrorString(e));
        return EMSURF_ECUDA;
    }
    return EMSURF_OK;
}

}  // extern "C"
