// Excitation vector (Eq. out) and far field / RCS (Sec. III-D: fields
// radiated by the solved box currents through the free-space operators).
//
// Plane wave E_inc = e^{-jk khat.r} ehat, |E_inc| = 1 V/m, eta0 H_inc =
// (khat x ehat) e^{-jk khat.r}.  V^(m) tests E_inc (rows J) and eta0 H_inc
// (rows M) with the RWGs of box m; since box m is box 0 translated by c_m,
// V^(m) = e^{-jk khat.c_m} V^(0) exactly.  V~ = U_o^T V (Eq. final).
//
// Far field, E ~ F e^{-jkr}/r:  F = -(jk/4pi) [N_perp - rhat x L_M] with
// N = sum_m e^{jk rhat.c_m} sum_e x_J[m,e] R_e(rhat),
// L_M = same with x_M, R_e(rhat) = int Lam_e e^{jk rhat.r'} dS' on box 0,
// x = U_o Y~.  Bistatic RCS sigma = 4 pi |F|^2 / |E_inc|^2.
#include <algorithm>
#include <cmath>
#include <cstring>
#include <vector>

#include "common.cuh"

namespace emsurf {
namespace {

constexpr double kFourPi = 12.566370614359172953850573533118;

// per RWG: 14 quadrature points (7 on T+, 7 on T-), weight w*A*sgn*len/(2A),
// free vertex of the point's triangle
struct RwgQuad {
    double r[14][3];
    double w[14];
    double p[14][3];
};

__device__ __forceinline__ double2 cexpj(double phase) {   // e^{j phase}
    double s, c;
    sincos(phase, &s, &c);
    return make_double2(c, s);
}

__device__ __forceinline__ double2 cexpjpi(double phase) {   // e^{j pi phase}
    double s, c;
    sincospi(phase, &s, &c);
    return make_double2(c, s);
}

// V0[r][e] = <Lam_e, ehat e^{-jk khat.r}>, V0[r][E+e] = <Lam_e, (khat x ehat) e^{..}>
__global__ void excitation_box_kernel(const RwgQuad* __restrict__ q, int E, int R,
                                      const double* __restrict__ khat, const double* __restrict__ ehat,
                                      double k, double2* __restrict__ V0) {
    const int e = blockIdx.x * blockDim.x + threadIdx.x;
    const int r = blockIdx.y;
    if (e >= E) return;
    const double* kh = khat + 3 * r;
    const double* eh = ehat + 3 * r;
    const double hv[3] = {kh[1] * eh[2] - kh[2] * eh[1], kh[2] * eh[0] - kh[0] * eh[2],
                          kh[0] * eh[1] - kh[1] * eh[0]};
    double2 vE = make_double2(0.0, 0.0), vH = make_double2(0.0, 0.0);
    const RwgQuad& Q = q[e];
    for (int i = 0; i < 14; ++i) {
        const double a[3] = {Q.r[i][0] - Q.p[i][0], Q.r[i][1] - Q.p[i][1], Q.r[i][2] - Q.p[i][2]};
        const double2 ph = cexpj(-k * (kh[0] * Q.r[i][0] + kh[1] * Q.r[i][1] + kh[2] * Q.r[i][2]));
        const double pe = Q.w[i] * (a[0] * eh[0] + a[1] * eh[1] + a[2] * eh[2]);
        const double phh = Q.w[i] * (a[0] * hv[0] + a[1] * hv[1] + a[2] * hv[2]);
        vE.x += pe * ph.x;
        vE.y += pe * ph.y;
        vH.x += phh * ph.x;
        vH.y += phh * ph.y;
    }
    V0[(size_t)r * 2 * E + e] = vE;
    V0[(size_t)r * 2 * E + E + e] = vH;
}

// V~[r][u] = sum over (m,k) of u: sign * e^{-jk khat.c_m} V0[r][k]
__global__ void excitation_scatter_kernel(const double2* __restrict__ V0, const int32_t* __restrict__ ptr,
                                          const int32_t* __restrict__ ent, const int8_t* __restrict__ esg,
                                          int nx, double a, double b, const double* __restrict__ khat,
                                          double k, int K, int n_unique, int R,
                                          double2* __restrict__ V) {
    const size_t total = (size_t)R * n_unique;
    for (size_t e = blockIdx.x * (size_t)blockDim.x + threadIdx.x; e < total;
         e += (size_t)gridDim.x * blockDim.x) {
        const int u = (int)(e % n_unique), r = (int)(e / n_unique);
        const double* kh = khat + 3 * r;
        double2 acc = make_double2(0.0, 0.0);
        for (int q = ptr[u]; q < ptr[u + 1]; ++q) {
            const int loc = ent[q];
            const int m = loc / K, kk = loc % K;
            const double cx = (m % nx) * a, cy = (m / nx) * b;
            const double2 ph = cexpj(-k * (kh[0] * cx + kh[1] * cy));
            const double2 v = cmul(ph, V0[(size_t)r * K + kk]);
            const double s = (double)esg[q];
            acc.x += s * v.x;
            acc.y += s * v.y;
        }
        V[e] = acc;
    }
}

// X1[m][r K + k] = sign * Y[r][idx[m K + k]]: every cell's box currents
template <typename C>
__global__ void gather_cells_kernel(const double2* __restrict__ Y, const int32_t* __restrict__ idx,
                                    const int8_t* __restrict__ sgn, int M, int K, int R, int n_unique,
                                    C* __restrict__ X1) {
    const size_t N = (size_t)R * K, total = (size_t)M * N;
    for (size_t e = blockIdx.x * (size_t)blockDim.x + threadIdx.x; e < total; e += (size_t)gridDim.x * blockDim.x) {
        const size_t m = e / N, rem = e - m * N;
        const int r = (int)(rem / K), kk = (int)(rem - (size_t)r * K);
        const size_t loc = m * K + kk;
        const double s = (double)sgn[loc];
        const double2 y = Y[(size_t)r * n_unique + idx[loc]];
        C v;
        v.x = s * y.x;
        v.y = s * y.y;
        X1[e] = v;
    }
}

// The array factor of every column: S[d][n] = sum_m e^{jk rhat_d . c_m}
// X1[m][n], c_m = (ix a, iy b, 0).  A block computes 32 directions x 96
// columns, 16 cells at a time (8 where the tables leave no room for more): X1
// and the cells' phases are staged in shared memory, the phases as products of
// the direction's e^{jk rx a ix} and e^{jk ry b iy} (from phase_table_kernel).
// A warp holds 4 directions, each lane 3 columns, so a phase is one broadcast
// read for the warp.  T: arithmetic type (double for FP64 handles; float, with float
// accumulation over the cells, for FP32 / MIXED handles).  Bound by the FMA
// rate.  16 x 16 cells, 576 columns, 65,160 directions (1.1 ms at the FP32 FMA
// rate): 1.9 ms and 0.14 ms for the tables; 3.5 ms with 2 x 4 sums per thread, the tables formed by
// every block, and the phase product and the cell's index division redone by
// every thread.  64 directions per block (8 per warp) left one block per SM
// and took a quarter longer.
constexpr int kLsM = 16, kLsThreads = 256, kLsCpt = 3, kLsDpt = 4;

// tab[d][i] = e^{jk rx a i} for i < nx, e^{jk ry b (i - nx)} for the ny above
template <typename T, typename C>
__global__ void phase_table_kernel(const double* __restrict__ rhat, int nd, int nx, int ny, double a, double b,
                                   double k, C* __restrict__ tab) {
    const int n = nx + ny;
    const long long total = (long long)nd * n;
    for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < total; e += (long long)gridDim.x * blockDim.x) {
        const int d = (int)(e / n), i = (int)(e - (long long)d * n);
        double sn, cs;
        sincos(i < nx ? k * a * rhat[3 * d] * i : k * b * rhat[3 * d + 1] * (i - nx), &sn, &cs);
        tab[e].x = (T)cs;
        tab[e].y = (T)sn;
    }
}

// shared bytes of a block with ms cells per stage
template <typename C>
size_t lattice_sum_smem(int ms, int nx, int ny) {
    return ((size_t)ms * (32 * kLsCpt + 8 * kLsDpt) + (size_t)8 * kLsDpt * (nx + ny)) * sizeof(C);
}

template <typename T, typename C, int MS>
__global__ void __launch_bounds__(kLsThreads)
lattice_sum_kernel(const C* __restrict__ X1, int M, int N, int nx, int ny, const C* __restrict__ tab, int nd,
                   C* __restrict__ S) {
    constexpr int DPT = kLsDpt, ND = 8 * DPT, NC = 32 * kLsCpt;
    constexpr int kXPer = MS * NC / kLsThreads;        // X1 entries of a thread and stage
    extern __shared__ __align__(16) unsigned char smem_raw[];
    C* xs = reinterpret_cast<C*>(smem_raw);            // [MS][NC]
    C* ps = xs + MS * NC;                              // [MS][ND]
    C* px = ps + MS * ND;                              // [nx][ND]
    C* py = px + nx * ND;                              // [ny][ND]
    const int d0 = blockIdx.y * ND, n0 = blockIdx.x * NC;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (int e = threadIdx.x; e < ND * (nx + ny); e += blockDim.x) {
        const int i = e / ND, dd = e - i * ND, d = d0 + dd;
        C v;
        v.x = (T)1;
        v.y = (T)0;
        if (d < nd) v = tab[(size_t)d * (nx + ny) + i];
        px[e] = v;
    }
    C acc[DPT][kLsCpt];
#pragma unroll
    for (int i = 0; i < DPT; ++i)
#pragma unroll
        for (int c = 0; c < kLsCpt; ++c) acc[i][c].x = acc[i][c].y = (T)0;
    // one stage's cells are summed on their own and then added: fewer roundings
    // at the size of the whole sum
    C part[DPT][kLsCpt];
    C xr[kXPer];
    auto load = [&](int m0) {
#pragma unroll
        for (int q = 0; q < kXPer; ++q) {
            const int e = threadIdx.x + q * kLsThreads, mm = e / NC, c = e - mm * NC;
            xr[q].x = xr[q].y = (T)0;
            if (m0 + mm < M && n0 + c < N) xr[q] = X1[(size_t)(m0 + mm) * N + n0 + c];
        }
    };
    load(0);
    for (int m0 = 0; m0 < M; m0 += MS) {
        __syncthreads();
#pragma unroll
        for (int q = 0; q < kXPer; ++q) xs[threadIdx.x + q * kLsThreads] = xr[q];
        for (int e = threadIdx.x; e < MS * ND; e += kLsThreads) {
            const int mm = e / ND, dd = e - mm * ND, m = min(m0 + mm, M - 1), iy = m / nx, ix = m - iy * nx;
            const C u = px[ix * ND + dd], w = py[iy * ND + dd];
            C v;
            v.x = u.x * w.x - u.y * w.y;
            v.y = u.x * w.y + u.y * w.x;
            ps[e] = v;
        }
        if (m0 + MS < M) load(m0 + MS);
        __syncthreads();
#pragma unroll
        for (int i = 0; i < DPT; ++i)
#pragma unroll
            for (int c = 0; c < kLsCpt; ++c) part[i][c].x = part[i][c].y = (T)0;
        // cells past M: X1 is zero there
#pragma unroll 4
        for (int mm = 0; mm < MS; ++mm) {
            C x[kLsCpt];
#pragma unroll
            for (int c = 0; c < kLsCpt; ++c) x[c] = xs[mm * NC + lane + 32 * c];
            const C* pw = ps + mm * ND + warp * DPT;
#pragma unroll
            for (int i = 0; i < DPT; i += 2) {
                // two directions' phases (16 or 32 bytes, the same for the whole warp)
                const C pa = pw[i], pb = pw[i + 1];
#pragma unroll
                for (int c = 0; c < kLsCpt; ++c) {
                    part[i][c].x += pa.x * x[c].x;
                    part[i][c].x -= pa.y * x[c].y;
                    part[i][c].y += pa.x * x[c].y;
                    part[i][c].y += pa.y * x[c].x;
                    part[i + 1][c].x += pb.x * x[c].x;
                    part[i + 1][c].x -= pb.y * x[c].y;
                    part[i + 1][c].y += pb.x * x[c].y;
                    part[i + 1][c].y += pb.y * x[c].x;
                }
            }
        }
#pragma unroll
        for (int i = 0; i < DPT; ++i)
#pragma unroll
            for (int c = 0; c < kLsCpt; ++c) {
                acc[i][c].x += part[i][c].x;
                acc[i][c].y += part[i][c].y;
            }
    }
#pragma unroll
    for (int i = 0; i < DPT; ++i) {
        const int d = d0 + warp * DPT + i;
        if (d >= nd) continue;
#pragma unroll
        for (int c = 0; c < kLsCpt; ++c) {
            const int n = n0 + lane + 32 * c;
            if (n < N) S[(size_t)d * N + n] = acc[i][c];
        }
    }
}

// The box as translates of a few triangle shapes: with t = shape c moved by
// its first vertex (X[ix], Y[iy], Z[iz]) the radiation integral of slot i of t
// is  sgn e^{jk rhat . v0_t} U_{c,i}(rhat),
// U_{c,i} = len_i / (2A) int_c (r' - v_i) e^{jk rhat . r'}.  A shape's slot i has
// the same len_i / (2A) on every member, so
//   N = sum_{c,i} U_{c,i} sum_{t in c} sgn e^{jk rhat . v0_t} S[rwg(t, i)]:
// the phases need one sincos per distinct coordinate and the U ones 7 per
// shape (about 155 per direction for 288 RWGs, 20 shapes) instead of 14 per
// RWG (4032).
struct BoxShape {
    double r[21];       // quadrature points relative to v_0
    double f[63];       // [i][q][x] w_q A len_i / (2A) (r_q - v_i)
    double v[9];        // vertices relative to v_0
};
struct BoxTri {
    int16_t ix, iy, iz, shape;
};
struct BoxMember {
    int32_t tri, rwg;   // rwg | (sgn < 0) << 31
};
struct BoxShapes {
    std::vector<BoxShape> shape;
    std::vector<BoxTri> tri;
    std::vector<double> coord;          // X, Y, Z one after the other
    int nc[3] = {0, 0, 0};
    std::vector<int32_t> slot;          // 3 shape + i, most members first
    std::vector<int32_t> ptr;           // members of slot[s]: ptr[s] .. ptr[s + 1]
    std::vector<BoxMember> mem;
};
struct BoxDev {
    const BoxShape* shape;
    const BoxTri* tri;
    const double* coord;
    const int32_t *slot, *ptr;
    const BoxMember* mem;
    int nshape, ntri, nx, ny, nz, nslot;
};

// F[r][d] = -(jk/4pi) [N_perp - rhat x L_M] of the column sums S[d][r K + e]
// (S_J in e < E, S_M in e >= E), one warp per direction; lanes share the
// coordinate phases, the shapes' points and the (shape, slot) sums through the
// warp's shared memory; the last step, from the six sums to F, is done for up to 32
// rhs at once.  by_rhs: 32 rhs at a time, one per lane, each lane all members (boxes
// with few of them leave lanes idle otherwise).  tri_ph: the triangles' phases are kept there too (else
// they are formed per member).  blockIdx.y takes rp of the R rhs: few directions
// with many rhs would leave SMs without a warp.  All FP64, and bound by its rate.
// 16 x 16 boxes of 288 RWGs, 65,160 directions: 2.9 ms;
// with the radiation vectors of every (direction, RWG) written out first this
// and the kernel before it took 20.6 ms.
constexpr int kFfWarps = 4;     // directions per block (fewer where their shared memory does not fit)

template <typename C>
__global__ void __launch_bounds__(32 * kFfWarps)
far_field_kernel(const C* __restrict__ S, BoxDev g, const double* __restrict__ rhat, int nd, int E, int R, int rp, double k,
                 bool tri_ph, bool by_rhs, double2* __restrict__ F, double* __restrict__ rcs, int ndir_all) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int ncoord = g.nx + g.ny + g.nz;
    const int per = ncoord + 7 * g.nshape + 3 * g.nslot + (tri_ph ? g.ntri : 0);
    double2* cp = reinterpret_cast<double2*>(smem_raw) + (size_t)warp * per;   // coordinate phases
    double2* eq = cp + ncoord;                                                 // point phases [shape][7]
    double2* U = eq + 7 * g.nshape;                                            // [slot][3]
    double2* tp = U + 3 * g.nslot;                                             // triangle phases
    const int K = 2 * E;
    const int nw = blockDim.x >> 5, r_lo = blockIdx.y * rp, r_hi = min(R, r_lo + rp);
    const double kpi = k * 0.31830988618379067154, k4 = k / kFourPi;
    for (int d = blockIdx.x * nw + warp; d < nd; d += gridDim.x * nw) {
        const double rh[3] = {rhat[3 * d], rhat[3 * d + 1], rhat[3 * d + 2]};
        __syncwarp();
        for (int e = lane; e < ncoord; e += 32)
            cp[e] = cexpjpi(kpi * (e < g.nx ? rh[0] : e < g.nx + g.ny ? rh[1] : rh[2]) * g.coord[e]);
        for (int e = lane; e < 7 * g.nshape; e += 32) {
            const int c = e / 7, q = e - 7 * c;
            const double* r = g.shape[c].r + 3 * q;
            eq[e] = cexpjpi(kpi * (rh[0] * r[0] + rh[1] * r[1] + rh[2] * r[2]));
        }
        __syncwarp();
        auto tri_phase = [&](const BoxTri t) {
            return cmul(cmul(cp[t.ix], cp[g.nx + t.iy]), cp[g.nx + g.ny + t.iz]);
        };
        if (tri_ph)
            for (int t = lane; t < g.ntri; t += 32) tp[t] = tri_phase(g.tri[t]);
        for (int s = lane; s < g.nslot; s += 32) {
            const int c = g.slot[s] / 3, i = g.slot[s] - 3 * c;
            const double* H = g.shape[c].f + 21 * i;
            double2 u[3] = {make_double2(0, 0), make_double2(0, 0), make_double2(0, 0)};
            for (int q = 0; q < 7; ++q) {
                const double2 p = eq[7 * c + q];
#pragma unroll
                for (int x = 0; x < 3; ++x) {
                    const double f = H[3 * q + x];
                    u[x].x = fma(f, p.x, u[x].x);
                    u[x].y = fma(f, p.y, u[x].y);
                }
            }
#pragma unroll
            for (int x = 0; x < 3; ++x) U[3 * s + x] = u[x];
        }
        __syncwarp();
        // F and RCS of one rhs from its sums N, L (NL)
        auto finish = [&](const double2 (&NL)[6], int rl) {
            const double2 *N = NL, *L = NL + 3;
            double2 rn = make_double2(0, 0);
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                rn.x += rh[c] * N[c].x;
                rn.y += rh[c] * N[c].y;
            }
            double mag = 0.0;
            double2* f = F + ((size_t)rl * ndir_all + d) * 3;
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                const int c1 = (c + 1) % 3, c2 = (c + 2) % 3;
                // N_perp - rhat x L, times -(jk / 4pi)
                const double2 rxl = make_double2(rh[c1] * L[c2].x - rh[c2] * L[c1].x,
                                                 rh[c1] * L[c2].y - rh[c2] * L[c1].y);
                const double2 w = make_double2(N[c].x - rn.x * rh[c] - rxl.x, N[c].y - rn.y * rh[c] - rxl.y);
                const double2 fc = make_double2(k4 * w.y, -k4 * w.x);
                f[c] = fc;
                mag += fc.x * fc.x + fc.y * fc.y;
            }
            if (rcs) rcs[(size_t)rl * ndir_all + d] = kFourPi * mag;
        };
        // sums of a rhs from its column sums sr over slots s0, s0 + step, ..
        auto slots = [&](const C* sr, int s0, int step, double2 (&NL)[6]) {
#pragma unroll
            for (int x = 0; x < 6; ++x) NL[x] = make_double2(0, 0);
            for (int s = s0; s < g.nslot; s += step) {
                double2 aj = make_double2(0, 0), am = make_double2(0, 0);
                for (int q = g.ptr[s]; q < g.ptr[s + 1]; ++q) {
                    const BoxMember b = g.mem[q];
                    const int e = b.rwg & 0x7fffffff;
                    C sj = sr[e], sm = sr[E + e];
                    if (b.rwg < 0) {
                        sj.x = -sj.x;
                        sj.y = -sj.y;
                        sm.x = -sm.x;
                        sm.y = -sm.y;
                    }
                    const double2 ph = tri_ph ? tp[b.tri] : tri_phase(g.tri[b.tri]);
                    cfma(aj, ph, make_double2((double)sj.x, (double)sj.y));
                    cfma(am, ph, make_double2((double)sm.x, (double)sm.y));
                }
#pragma unroll
                for (int x = 0; x < 3; ++x) {
                    const double2 u = U[3 * s + x];
                    cfma(NL[x], aj, u);
                    cfma(NL[3 + x], am, u);
                }
            }
        };
        const C* sd = S + (size_t)d * R * K;
        double2 NL[6];
        int r_at = r_lo;
        for (; by_rhs && r_hi - r_at >= 32; r_at += 32) {
            slots(sd + (size_t)(r_at + lane) * K, 0, 1, NL);
            finish(NL, r_at + lane);
        }
        // the sums of up to 32 rhs, one rhs per lane
        for (int r = r_at; r < r_hi; ++r) {
            double2 part[6];
            slots(sd + (size_t)r * K, lane, 32, part);
            // reduce-scatter of the 12 sums (padded to 16) over the warp: lanes 2 v
            // and 2 v + 1 end with value v, which the lane of this rhs takes
            double v[16];
#pragma unroll
            for (int x = 0; x < 6; ++x) {
                v[2 * x] = part[x].x;
                v[2 * x + 1] = part[x].y;
            }
            v[12] = v[13] = v[14] = v[15] = 0.0;
#pragma unroll
            for (int n = 16, D = 16; n > 1; n >>= 1, D >>= 1) {
                const bool up = lane & D;
#pragma unroll
                for (int c = 0; c < n / 2; ++c) {
                    const double send = up ? v[c] : v[c + n / 2];
                    const double keep = up ? v[c + n / 2] : v[c];
                    v[c] = keep + __shfl_xor_sync(0xffffffffu, send, D);
                }
            }
            v[0] += __shfl_xor_sync(0xffffffffu, v[0], 1);
#pragma unroll
            for (int x = 0; x < 6; ++x) {
                const double re = __shfl_sync(0xffffffffu, v[0], 4 * x), im = __shfl_sync(0xffffffffu, v[0], 4 * x + 2);
                if (lane == ((r - r_at) & 31)) NL[x] = make_double2(re, im);
            }
            if (((r - r_at) & 31) != 31 && r + 1 < r_hi) continue;
            const int rl = r - ((r - r_at) & 31) + lane;            // this lane's rhs
            if (rl > r) continue;
            finish(NL, rl);
        }
    }
}

int box_quadrature(double a, double b, double h, int n, const double* zlevels, int E_expected,
                   std::vector<RwgQuad>& out) {
    int32_t V, T, E;
    EMS_TRY(emsurf_setup_box_counts(n, &V, &T, &E));
    if (E != E_expected) {
        set_error("box mesh n=%d has %d RWGs, the handle has %d", n, E, E_expected);
        return EMSURF_EINVAL;
    }
    std::vector<double> verts(3 * V);
    std::vector<int32_t> tris(3 * T), edges(2 * E), tp(E), tm(E), srw(3 * T);
    std::vector<int8_t> ssg(3 * T);
    EMS_TRY(emsurf_setup_box_mesh(a, b, h, n, zlevels, verts.data(), tris.data(), edges.data(),
                                  tp.data(), tm.data(), srw.data(), ssg.data()));
    const double s15 = std::sqrt(15.0);
    const double a1 = (6.0 - s15) / 21.0, b1 = (9.0 + 2.0 * s15) / 21.0;
    const double a2 = (6.0 + s15) / 21.0, b2 = (9.0 - 2.0 * s15) / 21.0;
    const double w1 = (155.0 - s15) / 1200.0, w2 = (155.0 + s15) / 1200.0;
    const double B[7][3] = {{1.0 / 3, 1.0 / 3, 1.0 / 3}, {b1, a1, a1}, {a1, b1, a1}, {a1, a1, b1},
                            {b2, a2, a2}, {a2, b2, a2}, {a2, a2, b2}};
    const double W[7] = {9.0 / 40.0, w1, w1, w1, w2, w2, w2};
    out.assign(E, RwgQuad{});
    std::vector<int> seen(E, 0);
    for (int t = 0; t < T; ++t) {
        double P[3][3];
        for (int v = 0; v < 3; ++v)
            for (int x = 0; x < 3; ++x) P[v][x] = verts[3 * tris[3 * t + v] + x];
        const double e1[3] = {P[1][0] - P[0][0], P[1][1] - P[0][1], P[1][2] - P[0][2]};
        const double e2[3] = {P[2][0] - P[0][0], P[2][1] - P[0][1], P[2][2] - P[0][2]};
        const double c[3] = {e1[1] * e2[2] - e1[2] * e2[1], e1[2] * e2[0] - e1[0] * e2[2],
                             e1[0] * e2[1] - e1[1] * e2[0]};
        const double A = 0.5 * std::sqrt(c[0] * c[0] + c[1] * c[1] + c[2] * c[2]);
        for (int i = 0; i < 3; ++i) {
            const int m = srw[3 * t + i];
            const double* p = P[(i + 1) % 3];
            const double* qv = P[(i + 2) % 3];
            const double len = std::sqrt((p[0] - qv[0]) * (p[0] - qv[0]) + (p[1] - qv[1]) * (p[1] - qv[1]) +
                                         (p[2] - qv[2]) * (p[2] - qv[2]));
            const double amp = ssg[3 * t + i] * len / (2.0 * A);
            const int base = 7 * seen[m]++;
            for (int q = 0; q < 7; ++q) {
                for (int x = 0; x < 3; ++x) {
                    out[m].r[base + q][x] = B[q][0] * P[0][x] + B[q][1] * P[1][x] + B[q][2] * P[2][x];
                    out[m].p[base + q][x] = P[i][x];
                }
                out[m].w[base + q] = W[q] * A * amp;
            }
        }
    }
    return EMSURF_OK;
}

// index of x in v (appended when no entry lies within tol)
int coord_index(std::vector<double>& v, double x, double tol) {
    for (size_t i = 0; i < v.size(); ++i)
        if (std::fabs(v[i] - x) <= tol) return (int)i;
    v.push_back(x);
    return (int)v.size() - 1;
}

int box_shapes(double a, double b, double h, int n, const double* zlevels, int E_expected, BoxShapes& out) {
    int32_t V, T, E;
    EMS_TRY(emsurf_setup_box_counts(n, &V, &T, &E));
    if (E != E_expected) {
        set_error("box mesh n=%d has %d RWGs, the handle has %d", n, E, E_expected);
        return EMSURF_EINVAL;
    }
    std::vector<double> verts(3 * V);
    std::vector<int32_t> tris(3 * T), edges(2 * E), tp(E), tm(E), srw(3 * T);
    std::vector<int8_t> ssg(3 * T);
    EMS_TRY(emsurf_setup_box_mesh(a, b, h, n, zlevels, verts.data(), tris.data(), edges.data(),
                                  tp.data(), tm.data(), srw.data(), ssg.data()));
    const double s15 = std::sqrt(15.0);
    const double a1 = (6.0 - s15) / 21.0, b1 = (9.0 + 2.0 * s15) / 21.0;
    const double a2 = (6.0 + s15) / 21.0, b2 = (9.0 - 2.0 * s15) / 21.0;
    const double w1 = (155.0 - s15) / 1200.0, w2 = (155.0 + s15) / 1200.0;
    const double B[7][3] = {{1.0 / 3, 1.0 / 3, 1.0 / 3}, {b1, a1, a1}, {a1, b1, a1}, {a1, a1, b1},
                            {b2, a2, a2}, {a2, b2, a2}, {a2, a2, b2}};
    const double W[7] = {9.0 / 40.0, w1, w1, w1, w2, w2, w2};
    // translates agree to rounding; distinct ones differ by parts of an edge
    const double tol = 1e-12 * std::max(std::max(std::fabs(a), std::fabs(b)), std::fabs(h));
    std::vector<double> coord[3];
    out.tri.resize(T);
    for (int t = 0; t < T; ++t) {
        double P[3][3], e[9];
        for (int v = 0; v < 3; ++v)
            for (int x = 0; x < 3; ++x) P[v][x] = verts[3 * tris[3 * t + v] + x];
        for (int v = 0; v < 3; ++v)
            for (int x = 0; x < 3; ++x) e[3 * v + x] = P[v][x] - P[0][x];
        size_t c = 0;
        for (; c < out.shape.size(); ++c) {
            double dmax = 0.0;
            for (int q = 0; q < 9; ++q) dmax = std::max(dmax, std::fabs(out.shape[c].v[q] - e[q]));
            if (dmax <= tol) break;
        }
        if (c == out.shape.size()) {
            BoxShape s;
            for (int q = 0; q < 9; ++q) s.v[q] = e[q];
            const double cr[3] = {e[4] * e[8] - e[5] * e[7], e[5] * e[6] - e[3] * e[8], e[3] * e[7] - e[4] * e[6]};
            const double A = 0.5 * std::sqrt(cr[0] * cr[0] + cr[1] * cr[1] + cr[2] * cr[2]);
            for (int q = 0; q < 7; ++q)
                for (int x = 0; x < 3; ++x) s.r[3 * q + x] = B[q][1] * e[3 + x] + B[q][2] * e[6 + x];
            for (int i = 0; i < 3; ++i) {
                const double *p = e + 3 * ((i + 1) % 3), *q = e + 3 * ((i + 2) % 3);
                const double len = std::sqrt((p[0] - q[0]) * (p[0] - q[0]) + (p[1] - q[1]) * (p[1] - q[1]) +
                                             (p[2] - q[2]) * (p[2] - q[2]));
                for (int g = 0; g < 7; ++g)
                    for (int x = 0; x < 3; ++x)
                        s.f[21 * i + 3 * g + x] = W[g] * A * (len / (2.0 * A)) * (s.r[3 * g + x] - e[3 * i + x]);
            }
            out.shape.push_back(s);
        }
        BoxTri& bt = out.tri[t];
        bt.shape = (int16_t)c;
        bt.ix = (int16_t)coord_index(coord[0], P[0][0], tol);
        bt.iy = (int16_t)coord_index(coord[1], P[0][1], tol);
        bt.iz = (int16_t)coord_index(coord[2], P[0][2], tol);
    }
    for (int x = 0; x < 3; ++x) {
        out.nc[x] = (int)coord[x].size();
        out.coord.insert(out.coord.end(), coord[x].begin(), coord[x].end());
    }
    std::vector<std::vector<BoxMember>> mem(3 * out.shape.size());
    for (int t = 0; t < T; ++t)
        for (int i = 0; i < 3; ++i) {
            const int m = srw[3 * t + i];
            if (m < 0) continue;
            mem[3 * (size_t)out.tri[t].shape + i].push_back(
                BoxMember{t, ssg[3 * t + i] < 0 ? (int32_t)((uint32_t)m | 0x80000000u) : m});
        }
    out.slot.resize(mem.size());
    for (size_t s = 0; s < mem.size(); ++s) out.slot[s] = (int32_t)s;
    std::stable_sort(out.slot.begin(), out.slot.end(),
                     [&](int x, int y) { return mem[x].size() > mem[y].size(); });
    out.ptr.assign(1, 0);
    for (int s : out.slot) {
        out.mem.insert(out.mem.end(), mem[s].begin(), mem[s].end());
        out.ptr.push_back((int32_t)out.mem.size());
    }
    return EMSURF_OK;
}

template <typename T>
int to_device(T** d, const T* h, size_t n, cudaStream_t st) {
    EMS_CUDA(cudaMalloc(d, sizeof(T) * std::max<size_t>(n, 1)));
    EMS_CUDA(cudaMemcpyAsync(*d, h, sizeof(T) * n, cudaMemcpyHostToDevice, st));
    return EMSURF_OK;
}

struct Scoped {
    std::vector<void*> p;
    cudaStream_t st = nullptr;
    bool wait = false;
    ~Scoped() {
        if (wait) cudaStreamSynchronize(st);
        for (void* x : p) cudaFree(x);
    }
};
constexpr size_t kFfKeep = 8 << 20;

template <typename T, typename C, int MS>
int launch_lattice_sum(emsurf_handle* h, const C* X1, int N, const C* tab, int nd, C* S, cudaStream_t st) {
    constexpr int ND = 8 * kLsDpt, kMaxDirs = 65535 * ND;      // directions in grid rows
    const size_t smem = lattice_sum_smem<C>(MS, h->nx, h->ny);
    EMS_TRY(set_smem_once(lattice_sum_kernel<T, C, MS>, smem));
    for (int d0 = 0; d0 < nd; d0 += kMaxDirs) {
        const int n = std::min(nd - d0, kMaxDirs);
        const dim3 g((unsigned)((N + 32 * kLsCpt - 1) / (32 * kLsCpt)), (unsigned)((n + ND - 1) / ND));
        lattice_sum_kernel<T, C, MS><<<g, kLsThreads, smem, st>>>(X1, h->M, N, h->nx, h->ny,
                                                                   tab + (size_t)d0 * (h->nx + h->ny), n, S + (size_t)d0 * N);
        EMS_CUDA(cudaGetLastError());
    }
    return EMSURF_OK;
}

template <typename T, typename C>
int far_field_run(emsurf_handle* h, const BoxShapes& box, double a, double b, double k, const emsurf_c128* Y,
                  int nrhs, int ndir, const double* rhat, emsurf_c128* F, double* rcs, cudaStream_t st) {
    const int E = h->E, K = h->K, M = h->M, N = nrhs * K;
    // cells per stage of the lattice sum: the phase tables take what room they need
    constexpr size_t kMaxSmem = 227 * 1024;
    const int ms = lattice_sum_smem<C>(kLsM, h->nx, h->ny) <= kMaxSmem ? kLsM : kLsM / 2;
    if (lattice_sum_smem<C>(ms, h->nx, h->ny) > kMaxSmem) {
        set_error("emsurf_far_field: lattice %d x %d too large for the phase tables", h->nx, h->ny);
        return EMSURF_EINVAL;
    }
    // directions in chunks whose column sums stay in L2 between the two kernels
    // (at least enough directions to fill the device), sums and phase tables below
    // 512 MB
    const size_t per_dir = (size_t)(N + h->nx + h->ny) * sizeof(C);
    const int chunk = (int)std::min<size_t>(
        ndir, std::max<size_t>(1, std::min<size_t>(std::max<size_t>(4096, (48ull << 20) / ((size_t)N * sizeof(C))),
                                                   (512ull << 20) / per_dir)));
    // one device buffer: currents, column sums, directions and the box tables
    size_t bytes = 0;
    auto part = [&](size_t n) {
        const size_t at = bytes;
        bytes += (n + 255) & ~(size_t)255;
        return at;
    };
    const size_t o_x = part(sizeof(C) * (size_t)M * N), o_s = part(sizeof(C) * (size_t)chunk * N);
    const size_t o_p = part(sizeof(C) * (size_t)chunk * (h->nx + h->ny));
    const size_t o_r = part(sizeof(double) * 3 * (size_t)ndir);
    const size_t o_tab = bytes;
    const size_t o_shape = part(box.shape.size() * sizeof(BoxShape)), o_tri = part(box.tri.size() * sizeof(BoxTri));
    const size_t o_coord = part(box.coord.size() * sizeof(double)), o_slot = part(box.slot.size() * sizeof(int32_t));
    const size_t o_ptr = part(box.ptr.size() * sizeof(int32_t)), o_mem = part(box.mem.size() * sizeof(BoxMember));
    // up to kFfKeep bytes stay with the handle (an allocation that CUDA has to map
    // costs as much as a small far field), more are allocated for the call
    Scoped sc;
    unsigned char* buf = nullptr;
    if (bytes <= kFfKeep && h->ff_bytes < bytes) {
        dev_free(h, h->ff_buf, h->ff_bytes);
        h->ff_buf = nullptr;
        h->ff_bytes = 0;
        size_t keep = 256 << 10;
        while (keep < bytes) keep *= 2;
        if (dev_alloc(h, &h->ff_buf, keep) == EMSURF_OK) h->ff_bytes = keep;
    }
    if (bytes <= h->ff_bytes) {
        buf = static_cast<unsigned char*>(h->ff_buf);
        sc.st = st;                      // nothing of this call is in flight after it
        sc.wait = true;
    } else {
        EMS_CUDA(cudaMalloc(&buf, bytes));
        sc.p.push_back(buf);
    }
    std::vector<unsigned char> tab(bytes - o_tab);
    auto fill = [&](size_t at, const auto& v) { std::memcpy(tab.data() + at - o_tab, v.data(), v.size() * sizeof(v[0])); };
    fill(o_shape, box.shape);
    fill(o_tri, box.tri);
    fill(o_coord, box.coord);
    fill(o_slot, box.slot);
    fill(o_ptr, box.ptr);
    fill(o_mem, box.mem);
    EMS_CUDA(cudaMemcpyAsync(buf + o_tab, tab.data(), tab.size(), cudaMemcpyHostToDevice, st));
    EMS_CUDA(cudaMemcpyAsync(buf + o_r, rhat, sizeof(double) * 3 * (size_t)ndir, cudaMemcpyHostToDevice, st));
    C *X1 = reinterpret_cast<C*>(buf + o_x), *S = reinterpret_cast<C*>(buf + o_s);
    const double* dr = reinterpret_cast<const double*>(buf + o_r);
    const BoxDev g{reinterpret_cast<const BoxShape*>(buf + o_shape), reinterpret_cast<const BoxTri*>(buf + o_tri),
                   reinterpret_cast<const double*>(buf + o_coord), reinterpret_cast<const int32_t*>(buf + o_slot),
                   reinterpret_cast<const int32_t*>(buf + o_ptr), reinterpret_cast<const BoxMember*>(buf + o_mem),
                   (int)box.shape.size(), (int)box.tri.size(), box.nc[0], box.nc[1], box.nc[2], (int)box.slot.size()};
    gather_cells_kernel<C><<<(int)std::min<size_t>(((size_t)M * N + 255) / 256, 152 * 32), 256, 0, st>>>(
        reinterpret_cast<const double2*>(Y), h->d_uo_index, h->d_uo_sign, M, K, nrhs, h->n_unique, X1);
    EMS_CUDA(cudaGetLastError());
    // far field: triangle phases in shared memory while those of four warps fit an SM
    // (20,000 directions, 16 x 16 per face: 13.4 ms, formed per member 14.2; 18 x 18,
    // where two warps would fit: 30.3 and 17.9)
    const size_t per = (box.coord.size() + 7 * box.shape.size() + 3 * box.slot.size()) * sizeof(double2);
    const size_t per_ph = per + box.tri.size() * sizeof(double2);
    const bool ph = 4 * per_ph <= 224 * 1024;
    int warps = kFfWarps;
    while (warps > 1 && (ph ? per_ph : per) * warps > 200 * 1024) warps /= 2;
    const size_t fsm = (ph ? per_ph : per) * warps;
    EMS_TRY(set_smem_once(far_field_kernel<C>, fsm));
    // 32 rhs at a time by lanes: FP64 operations of a warp for them against 32 times
    // those of a rhs by slots
    long long by_lane = 8 * (long long)box.mem.size() + 24 * (long long)box.slot.size() + 42, by_slot = 17;
    for (size_t s = 0; s < box.slot.size(); s += 32) by_slot += 8 * (box.ptr[s + 1] - box.ptr[s]) + 24;
    const bool by_rhs = by_lane < 32 * by_slot;
    double2* Fo = reinterpret_cast<double2*>(F);
    for (int d0 = 0; d0 < ndir; d0 += chunk) {
        const int nd = std::min(chunk, ndir - d0);
        const double* drc = dr + 3 * (size_t)d0;
        C* tab = reinterpret_cast<C*>(buf + o_p);
        const size_t tn = (size_t)nd * (h->nx + h->ny);
        phase_table_kernel<T, C><<<(int)std::min<size_t>((tn + 127) / 128, 152 * 32), 128, 0, st>>>(drc, nd, h->nx, h->ny, a,
                                                                                               b, k, tab);
        EMS_CUDA(cudaGetLastError());
        if (ms == kLsM) EMS_TRY((launch_lattice_sum<T, C, kLsM>(h, X1, N, tab, nd, S, st)));
        else EMS_TRY((launch_lattice_sum<T, C, kLsM / 2>(h, X1, N, tab, nd, S, st)));
        // rhs in groups while the device has room for all of them at once (8 warps per SM
        // keep its FP64 unit busy): each forms its directions' phases again
        const int blocks = std::min((nd + warps - 1) / warps, h->num_sms * 32);
        const int groups = std::max(1, std::min(std::min(nrhs, 65535), 8 * h->num_sms / (blocks * warps)));
        int rn = (nrhs + groups - 1) / groups;
        if (by_rhs && rn < 32 && (long long)blocks * (nrhs / 32) >= h->num_sms) rn = 32;
        far_field_kernel<C><<<dim3(blocks, (nrhs + rn - 1) / rn), 32 * warps, fsm, st>>>(
            S, g, drc, nd, E, nrhs, rn, k, ph, by_rhs, Fo + (size_t)d0 * 3, rcs ? rcs + d0 : nullptr, ndir);
        EMS_CUDA(cudaGetLastError());
    }
    sc.wait = false;
    EMS_CUDA(cudaStreamSynchronize(st));
    return EMSURF_OK;
}

}  // namespace
}  // namespace emsurf

using namespace emsurf;

extern "C" {

EMSURF_API int emsurf_excitation(emsurf_handle* h, double a, double b, double hgt, int32_t n,
                                 const double* zlevels, double k, int32_t nrhs, const double* khat, const double* ehat,
                                 emsurf_c128* V, void* stream) {
    if (!h || !khat || !ehat || !V || nrhs < 1 || !(k > 0.0)) {
        set_error("emsurf_excitation: bad arguments");
        return EMSURF_EINVAL;
    }
    cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
    std::vector<RwgQuad> q;
    EMS_TRY(box_quadrature(a, b, hgt, n, zlevels, h->E, q));
    Scoped sc;
    RwgQuad* dq;
    double *dk, *de;
    double2* V0;
    EMS_TRY(to_device(&dq, q.data(), q.size(), st));
    sc.p.push_back(dq);
    EMS_TRY(to_device(&dk, khat, 3 * (size_t)nrhs, st));
    sc.p.push_back(dk);
    EMS_TRY(to_device(&de, ehat, 3 * (size_t)nrhs, st));
    sc.p.push_back(de);
    EMS_CUDA(cudaMalloc(&V0, sizeof(double2) * nrhs * h->K));
    sc.p.push_back(V0);
    excitation_box_kernel<<<dim3((h->E + 127) / 128, nrhs), 128, 0, st>>>(dq, h->E, nrhs, dk, de, k, V0);
    EMS_CUDA(cudaGetLastError());
    const size_t tot = (size_t)nrhs * h->n_unique;
    excitation_scatter_kernel<<<(int)std::min<size_t>((tot + 255) / 256, 152 * 32), 256, 0, st>>>(
        V0, h->d_inv_ptr, h->d_inv_ent, h->d_inv_sgn, h->nx, a, b, dk, k, h->K, h->n_unique, nrhs,
        reinterpret_cast<double2*>(V));
    EMS_CUDA(cudaGetLastError());
    EMS_CUDA(cudaStreamSynchronize(st));
    return EMSURF_OK;
}

EMSURF_API int emsurf_far_field(emsurf_handle* h, double a, double b, double hgt, int32_t n,
                                const double* zlevels, double k,
                                const emsurf_c128* Y, int32_t nrhs, int32_t ndir, const double* rhat,
                                emsurf_c128* F, double* rcs, void* stream) {
    if (!h || !Y || !rhat || !F || nrhs < 1 || ndir < 1 || !(k > 0.0)) {
        set_error("emsurf_far_field: bad arguments");
        return EMSURF_EINVAL;
    }
    cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
    BoxShapes box;
    EMS_TRY(box_shapes(a, b, hgt, n, zlevels, h->E, box));
    if (h->precision == EMSURF_FP64) return far_field_run<double, double2>(h, box, a, b, k, Y, nrhs, ndir, rhat, F, rcs, st);
    return far_field_run<float, float2>(h, box, a, b, k, Y, nrhs, ndir, rhat, F, rcs, st);
}

}  // extern "C"
