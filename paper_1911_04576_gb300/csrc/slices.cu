// FP64-accuracy products on the tensor cores: exact integer slices.
//
// FP64 runs at ~1/60 of the FP32 rate on this part, and double-single FP32
// arithmetic needs 12 FP32 operations per real multiply-add.  Here every
// operand is cut into 7 balanced base-256 digits of a 55-bit integer,
//   v = 2^(ex - 54) sum_t d_t 256^(6 - t),  d_t in [-128, 127],
// with one power of two 2^ex above the largest component of each matrix row
// and of each vector (Ozaki, Ogita, Oishi, Rump 2012: error-free splitting).
// Digits are exact in FP16, their products exact in FP32, and a sum of up to
// 7 x 128 products stays below 2^24, so kind::f16 MMAs with FP32 accumulation
// in TMEM add them without rounding.  Digit pairs s + t = l share an
// accumulator column (level l); levels 0..6 are kept (the dropped pairs weigh
// 2^-50 of row maximum times vector maximum), read back as integers, summed in
// int64 over the 128-wide K chunks, combined into complex products there and
// turned into FP64 once per output.
//
// Two problems share one launch:
//   bins        y^(k) = B^(k) x^(k): per bin 4E real rows (4 i + 2 op + c, op in
//               {L, K}, c = re, im) over the E sources; columns (rhs, x_J/x_M,
//               re/im);
//   macromodels y = Z~^t x1 of the cells of a type: 2K real rows (2 k + c) over
//               K; columns (cell and rhs, re/im).
//
// The matrix digits are stored as bytes (d + 128), 7 per real number: planes
// [matrix][row tile of 128][16-source block][digit][row][16 bytes], streamed
// through a ring of their own whose slots are free as soon as a warp set has
// read them.  The warp set turns them into FP16 (byte into the mantissa of 1024 + b, minus 1152)
// and writes them into TMEM, so the A operand never passes through shared
// memory as FP16.  The vectors' digits are FP16 in 64-byte swizzled rows
// (t, v), preceded by 6 V rows of zeros that stay in shared memory: digit s of
// the matrix multiplies the rows from -s V on, so that digit t lands in the
// columns of level s + t and every MMA of a tile has the same shape and the
// same accumulator (which keeps them in order).
//
// Warps: 0-7 epilogue (half of the columns each), 8-15 byte to FP16 in two sets
// that take 16-source blocks in turn, 16 and 18 bulk copies of matrix and
// vector digits, 17 MMA.  A 128 x N x 16 MMA with A in TMEM takes 68-86 cycles
// for N up to 176 (measured), and each wait about as long as two of them, so the
// MMA warp bounds the kernel: it waits once per two blocks on all it needs (the
// byte-to-FP16 warps see to the vector digits and give their slots back).  Every
// wait is bounded: on expiry the kernel sets the error flag, waits (bounded) for
// its copies and MMAs in flight, frees TMEM and returns.
//
// Measured, product of a 16 x 16 lattice with K = 576 (2.38 GB of digits, 350 us
// at the copy rate): 1161 us in double-single FP32, 568 us here (600 us with waits
// that every lane left by itself); 12 x 9, K = 576 and 6 rhs: 6575 us, 556 us (27 us
// more with 8 instead of 12 macromodel columns per entry).
//
// Precision.  An entry of a matrix row or of a vector keeps the 55 bits below the
// row's or vector's maximum, where double-single kept 48 of its own: an entry 2^-8
// below the maximum has fewer.  The bound is on row maximum times vector maximum
// instead of on each term.  Measured against 113-bit arithmetic (3 x 2 slab cells, K
// = 324, entries of x spread over 0, 4, 8, 12 decades): error in norm 2.8e-15, 6.8e-15,
// 8.2e-15, 7.7e-15, double-single 4.5e-14 at each; largest error over (|A| |x|)_i
// 3.5e-15, 2.1e-14, 4.0e-14, 5.2e-14, double-single 7.1e-14, 1.7e-13, 4.0e-13, 4.6e-13.
// The term of a row's entry 2^-p below its maximum with the vector's largest entry
// has 55 - p bits, fewer than double-single's 48 for p above 7: the fixed point
// loses where only such terms make up a sum.
#include <algorithm>
#include <vector>

#include "digits.cuh"

namespace emsurf {
namespace {

constexpr int kSlRows = 128;                 // rows per tile (TMEM lanes)
constexpr int kSlK = 32;                     // sources per stage
constexpr int kSlChunk = 4;                  // stages per exact accumulation (128 sources)
constexpr int kSlKbBytes = kSl * 16;         // bytes per row and 16-source block
constexpr int kSlABytes = kSlKbBytes * kSlRows;         // one 16-source block of a tile
constexpr int kSlMaxStages = 14, kSlXStages = 4;
constexpr int kSlEpi = 8, kSlWarps = kSlEpi + 8 + 3, kSlThreads = 32 * kSlWarps;
constexpr int kSlWarpA = kSlWarps - 3, kSlWarpM = kSlWarps - 2, kSlWarpX = kSlWarps - 1;
constexpr uint32_t kSlTmemCols = 512, kSlAStep = kSl * 8;   // TMEM columns; of one 16-source block of A
constexpr int kSlMaxSlots = 4;               // A blocks in TMEM, at the end of its columns
constexpr size_t kSlSmemMax = 224 * 1024;
constexpr int kSlMaxV = 24;                  // vector columns of one launch (a multiple of 8: swizzle groups):
                                             // two accumulators and two A blocks fit in TMEM
constexpr int kSlRhs = kSlMaxV / 4;          // rhs per launch
constexpr int kSlSplit = 256;                // threads of a splitting block
// sl_wait_warp for two or three barriers at once (their latencies overlap)
__device__ __forceinline__ bool sl_wait3(uint64_t* b0, uint32_t p0, uint64_t* b1, uint32_t p1, uint64_t* b2, uint32_t p2,
                                         bool third, int tries) {
    for (int it = 0; it < tries; ++it) {
        uint32_t ok;
        asm volatile(
            "{\n .reg .pred p, q, r, t;\n setp.ne.b32 t, %8, 0;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, %7;\n"
            " mbarrier.try_wait.parity.shared::cta.b64 q, [%3], %4, %7;\n setp.eq.b32 r, %8, 0;\n"
            " @t mbarrier.try_wait.parity.shared::cta.b64 r, [%5], %6, %7;\n"
            " and.pred p, p, q;\n and.pred p, p, r;\n selp.u32 %0, 1, 0, p;\n}\n"
            : "=r"(ok)
            : "r"(sl_addr(b0)), "r"(p0), "r"(sl_addr(b1)), "r"(p1), "r"(sl_addr(b2)), "r"(p2), "r"(20000u),
              "r"((uint32_t)third)
            : "memory");
        if (__all_sync(0xffffffffu, ok)) return true;
    }
    return false;
}
// K-major descriptor, 64-byte swizzled rows, 8-row groups 512 B apart
__device__ __forceinline__ uint64_t sl_desc(uint32_t addr) {
    return (uint64_t)((addr & 0x3FFFF) >> 4) | (1ull << 16) | (32ull << 32) | (1ull << 46) | (4ull << 61);
}
__device__ __forceinline__ void tmem_st8(uint32_t t, const uint32_t (&r)[8]) {
    asm volatile("tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8};" ::"r"(t), "r"(r[0]),
                 "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7])
                 : "memory");
}
__host__ __device__ constexpr int sl_up16(int n) { return (n + 15) & ~15; }

struct SlProb {
    const unsigned char* A;      // digit planes
    const int* rs;               // [matrix][row / 2] exponent of each complex row (sl_exp)
    const unsigned char* X;      // vector digits [x matrix][stage][Np][64 bytes]
    const int* xs;               // [x matrix][V / 2] exponent of each complex vector
    int nk16, nst, rows, tiles, V, Np, items, xmats;
    int live;                    // bins: rhs of this launch
};

struct SlArgs {
    SlProb p[2];                 // bins, macromodels
    int stages, z_bytes, x_bytes;   // matrix ring depth, bytes of a vector slot's zero rows and vector rows
    int slots, d_step;           // A blocks in TMEM, spacing of the two accumulators
    // bins
    double2* Y;                  // [bins][R][2E]
    int E, R, r0;
    double2 co[4];
    // macromodels
    double2* Ymm;                // [R][M][K]
    const int2* ent;             // (type, first column)
    const int32_t *type_ptr, *type_cells;
    int K, M;
    int* err;
    int tries;                   // of a wait
    int starve;                  // self-test: the vectors' digits never arrive
};

// Range of items of CTA b: items whose first stage lies in its share of all stages.
__device__ __forceinline__ int sl_item_at(const SlArgs& g, long long q) {
    const long long s0 = (long long)g.p[0].items * g.p[0].nst;
    if (q <= s0) return g.p[0].nst ? (int)((q + g.p[0].nst - 1) / g.p[0].nst) : 0;
    return g.p[0].items + (int)((q - s0 + g.p[1].nst - 1) / g.p[1].nst);
}

__global__ void __launch_bounds__(kSlThreads, 1) slices_kernel(SlArgs g) {
    constexpr int V4 = kSlMaxV / 8;          // groups of four columns per epilogue half
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    unsigned char* smem = reinterpret_cast<unsigned char*>(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    __shared__ __align__(8) uint64_t full[kSlMaxStages], empty[kSlMaxStages], xfull[kSlXStages], xempty[kSlXStages],
        afull[kSlMaxSlots], aempty[kSlMaxSlots], dfull[2], dempty[2], mma_done;
    __shared__ uint32_t tmem_slot;
    __shared__ int abort_flag;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (warp == kSlWarpM) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(sl_addr(&tmem_slot)),
                     "r"(kSlTmemCols));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    const int xslot = g.z_bytes + g.x_bytes;
    unsigned char* xring = smem + g.stages * kSlABytes;
    for (int s = 0; s < kSlXStages; ++s)
        for (int e = threadIdx.x; e < g.z_bytes / 16; e += blockDim.x)
            reinterpret_cast<uint4*>(xring + s * xslot)[e] = make_uint4(0u, 0u, 0u, 0u);
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    if (threadIdx.x == 0) {
        for (int s = 0; s < g.stages; ++s) {
            sl_init(&full[s], 1);
            sl_init(&empty[s], 4);
        }
        for (int s = 0; s < kSlXStages; ++s) {
            sl_init(&xfull[s], 1);
            sl_init(&xempty[s], 1);
        }
        for (int a = 0; a < kSlMaxSlots; ++a) {
            sl_init(&afull[a], 4);
            sl_init(&aempty[a], 1);
        }
        for (int a = 0; a < 2; ++a) {
            sl_init(&dfull[a], 1);
            sl_init(&dempty[a], kSlEpi);
        }
        sl_init(&mma_done, 1);
        abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    asm volatile("tcgen05.fence::before_thread_sync;");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;");
    const uint32_t tmem = tmem_slot;
    volatile int* abort_v = &abort_flag;
    const uint32_t a_col = kSlTmemCols - g.slots * kSlAStep;
    const int slots = g.slots;
    const long long total = (long long)g.p[0].items * g.p[0].nst + (long long)g.p[1].items * g.p[1].nst;
    const int i_lo = sl_item_at(g, (long long)blockIdx.x * total / gridDim.x);
    const int i_hi = sl_item_at(g, (long long)(blockIdx.x + 1) * total / gridDim.x);

    if (warp == kSlWarpA || warp == kSlWarpX) {
        // ------------------------------------------------ copies: matrix digits, vector digits
        if (lane == 0) {
            const bool mat_side = warp == kSlWarpA;
            const uint64_t once = l2_evict_first(), keep = l2_evict_last();
            const int depth = mat_side ? g.stages : kSlXStages;
            uint64_t *fb = mat_side ? full : xfull, *eb = mat_side ? empty : xempty;
            int st = 0;
            long long issued = 0;
            uint32_t ph = 0;
            bool ok = true;
            if (!mat_side) dep_wait();           // the matrix digits do not depend on the splitting kernel
            const int i_end = g.starve && !mat_side ? i_lo : i_hi;
            for (int it = i_lo; it < i_end && ok && !*abort_v; ++it) {
                const int w = it >= g.p[0].items;
                const SlProb& p = g.p[w];
                const int loc = w ? it - g.p[0].items : it, xm = loc / p.tiles, tile = loc - xm * p.tiles;
                const int mat = w ? g.ent[xm].x : xm;
                const int rows = min(kSlRows, p.rows - tile * kSlRows);
                const unsigned char* a = p.A + ((size_t)mat * p.rows + (size_t)tile * kSlRows) * p.nk16 * kSlKbBytes;
                const unsigned char* x = p.X + (size_t)xm * p.nst * p.Np * 64;
                const int steps = mat_side ? p.nk16 : p.nst;
                for (int s = 0; s < steps; ++s) {
                    if (!sl_wait(&eb[st], ph ^ 1, g.tries)) {
                        atomicExch(g.err, 20);
                        ok = false;
                        break;
                    }
                    if (mat_side) {
                        const uint32_t n = (uint32_t)(kSlKbBytes * rows);
                        sl_expect(&fb[st], n);
                        // the macromodels are read by several items and products
                        sl_copy(smem + st * kSlABytes, a + (size_t)s * n, n, &fb[st], w ? keep : once);
                    } else {
                        const uint32_t n = (uint32_t)(p.Np * 64);
                        sl_expect(&fb[st], n);
                        sl_copy(xring + st * xslot + g.z_bytes, x + (size_t)s * n, n, &fb[st], keep);
                    }
                    ++issued;
                    if (++st == depth) {
                        st = 0;
                        ph ^= 1;
                    }
                }
            }
            if (!ok) *abort_v = 1;
            // every copy has landed before the CTA can exit
            for (long long u = issued > depth ? issued - depth : 0; u < issued; ++u)
                if (!sl_wait(&fb[u % depth], (uint32_t)((u / depth) & 1), kSlWait)) atomicExch(g.err, 20);
        }
    } else if (warp == kSlWarpM) {
        // ------------------------------------------------ MMA
        const uint32_t go = lane == 0;
        const uint32_t tb = __shfl_sync(0xffffffffu, tmem, 0);
        int xst = 0, db = 0, slot = 0;
        uint32_t dph = 0, sph = 0;
        bool any = false, ok = true;
        for (int it = i_lo; it < i_hi && ok && !sl_abort(abort_v); ++it) {
            const SlProb& p = g.p[it >= g.p[0].items];
            const uint32_t idesc = (1u << 4) | ((uint32_t)(p.Np >> 3) << 17) | ((uint32_t)(kSlRows >> 4) << 24);
            const uint32_t back = (uint32_t)p.V * 4;        // one digit's rows in descriptor units of 16 bytes
            const int nk16 = p.nk16;
            // Two blocks of A (one vector stage) at a time where TMEM has four slots,
            // else one: the waits cost more than the issue.
            int kc = 0;
            for (int k = 0; k < nk16;) {
                const bool odd = k & 1, two = slots == kSlMaxSlots && k + 1 < nk16;
                const int slot2 = slot + 1 == slots ? 0 : slot + 1;
                const uint32_t sph2 = slot2 ? sph : sph ^ 1;
                const bool first = kc == 0;
                if (!sl_wait3(&afull[slot], sph, &afull[two ? slot2 : slot], two ? sph2 : sph, &dempty[db],
                              dph ^ 1, first, g.tries)) {
                    if (go) atomicExch(g.err, 21);
                    ok = false;
                    break;
                }
                asm volatile("tcgen05.fence::after_thread_sync;");
                const uint32_t d = tb + (uint32_t)(db * g.d_step), ta = tb + a_col + slot * kSlAStep,
                               ta2 = tb + a_col + slot2 * kSlAStep;
                const uint64_t bd = sl_desc(sl_addr(xring + xst * xslot + g.z_bytes)) + (odd ? 2 : 0);
                k += two ? 2 : 1;
                kc += two ? 2 : 1;
                const bool flush = kc == 2 * kSlChunk || k >= nk16;
                if (sl_elect()) {
                    if (first) sl_mma<false>(d, ta, bd, idesc);
                    else sl_mma<true>(d, ta, bd, idesc);
#pragma unroll
                    for (int sl = 1; sl < kSl; ++sl) sl_mma<true>(d, ta + sl * 8, bd - sl * back, idesc);
                    sl_commit(&aempty[slot]);
                    if (two) {
#pragma unroll
                        for (int sl = 0; sl < kSl; ++sl) sl_mma<true>(d, ta2 + sl * 8, bd + 2 - sl * back, idesc);
                        sl_commit(&aempty[slot2]);
                    }
                    if (flush) sl_commit(&dfull[db]);
                }
                __syncwarp();
                any = true;
                if (flush) {
                    kc = 0;
                    dph ^= (uint32_t)db;
                    db ^= 1;
                }
                slot = two ? slot2 : slot;
                sph = two ? sph2 : sph;
                if (++slot == slots) {
                    slot = 0;
                    sph ^= 1;
                }
                if ((odd || two || k >= nk16) && ++xst == kSlXStages) xst = 0;
            }
        }
        if (!ok) *abort_v = 1;
        if (any) {
            if (sl_elect()) sl_commit(&mma_done);
            __syncwarp();
            if (!sl_wait_warp(&mma_done, 0, kSlWait) && go) atomicExch(g.err, 23);
        }
    } else if (warp >= kSlEpi) {
        // ------------------------------------------------ bytes to FP16 in TMEM
        const int set = (warp - kSlEpi) >> 2, qd = warp & 3, row = 32 * qd + lane;
        const uint32_t ta = tmem + ((uint32_t)(32 * qd) << 16) + a_col;
        const __half2 off = __floats2half2_rn(1152.f, 1152.f);
        int st = 0, q = 0, slot = 0, xst = 0;
        uint32_t ph = 0, sph = 0, xph = 0;
        // vector slot + 1 of the last kSlMaxSlots blocks that end a vector stage (else 0)
        int ends[kSlMaxSlots] = {};
        bool ok = true;
        for (int it = i_lo; it < i_hi && ok && !sl_abort(abort_v); ++it) {
            const int w = it >= g.p[0].items;
            const SlProb& p = g.p[w];
            const int loc = w ? it - g.p[0].items : it, tile = loc % p.tiles;
            const int rows = min(kSlRows, p.rows - tile * kSlRows), rr = min(row, rows - 1);
            const int nk16 = p.nk16;
            for (int k = 0; k < nk16; ++k, ++q) {
                const bool end = (k & 1) || k == nk16 - 1;
                const int done = slots == kSlMaxSlots ? ends[kSlMaxSlots - 1] : ends[1];
                if ((q & 1) == set) {
                    if (!sl_wait_warp(&full[st], ph, g.tries)) {
                        if (lane == 0) atomicExch(g.err, 24);
                        ok = false;
                        break;
                    }
                    const uint4* a = reinterpret_cast<const uint4*>(smem + st * kSlABytes);
                    uint4 v[kSl];
#pragma unroll
                    for (int sl = 0; sl < kSl; ++sl) v[sl] = a[sl * rows + rr];
                    __syncwarp();
                    if (lane == 0) sl_arrive(&empty[st]);
                    // the block `slots` before this one has been multiplied: its TMEM slot
                    // is free, and its vector slot if it was the stage's last
                    if (!sl_wait_warp(&aempty[slot], sph ^ 1, g.tries)) {
                        if (lane == 0) atomicExch(g.err, 25);
                        ok = false;
                        break;
                    }
                    if (done && qd == 0 && lane == 0) sl_arrive(&xempty[done - 1]);
                    if (!sl_wait_warp(&xfull[xst], xph, g.tries)) {
                        if (lane == 0) atomicExch(g.err, 26);
                        ok = false;
                        break;
                    }
                    asm volatile("tcgen05.fence::after_thread_sync;");
#pragma unroll
                    for (int sl = 0; sl < kSl; ++sl) {
                        const uint32_t b[4] = {v[sl].x, v[sl].y, v[sl].z, v[sl].w};
                        uint32_t h[8];
#pragma unroll
                        for (int c = 0; c < 4; ++c) {
                            // FP16 0x6400 | byte = 1024 + byte; minus 1152 gives byte - 128
                            const uint32_t lo = __byte_perm(b[c], 0x64646464u, 0x4140), hi = __byte_perm(b[c], 0x64646464u, 0x4342);
                            const __half2 l2 = __hsub2(*reinterpret_cast<const __half2*>(&lo), off);
                            const __half2 h2 = __hsub2(*reinterpret_cast<const __half2*>(&hi), off);
                            h[2 * c] = *reinterpret_cast<const uint32_t*>(&l2);
                            h[2 * c + 1] = *reinterpret_cast<const uint32_t*>(&h2);
                        }
                        tmem_st8(ta + slot * kSlAStep + sl * 8, h);
                    }
                    asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
                    asm volatile("tcgen05.fence::before_thread_sync;");
                    __syncwarp();
                    if (lane == 0) sl_arrive(&afull[slot]);
                }
#pragma unroll
                for (int i = kSlMaxSlots - 1; i > 0; --i) ends[i] = ends[i - 1];
                ends[0] = end ? xst + 1 : 0;
                if (++st == g.stages) {
                    st = 0;
                    ph ^= 1;
                }
                if (++slot == slots) {
                    slot = 0;
                    sph ^= 1;
                }
                if (end && ++xst == kSlXStages) {
                    xst = 0;
                    xph ^= 1;
                }
            }
        }
        if (!ok) *abort_v = 1;
    } else {
        // ------------------------------------------------ epilogue
        dep_wait();
        const int qd = warp & 3, half = warp >> 2, rho = 32 * qd + lane;
        const uint32_t tl = tmem + ((uint32_t)(32 * qd) << 16);
        int db = 0;
        uint32_t dph = 0;
        bool ok = true;
        for (int it = i_lo; it < i_hi && ok && !sl_abort(abort_v); ++it) {
            const int w = it >= g.p[0].items;
            const SlProb& p = g.p[w];
            const int loc = w ? it - g.p[0].items : it, xm = loc / p.tiles, tile = loc - xm * p.tiles;
            const int V = p.V, row = tile * kSlRows + rho;
            const int g0 = half * (V / 8);           // first group of four columns, V / 8 groups each
            // sums in units of level 5 (level 6 rounded to it)
            long long acc[4 * V4];
#pragma unroll
            for (int v = 0; v < 4 * V4; ++v) acc[v] = 0;
            for (int s = 0; s < p.nst; s += kSlChunk) {
                if (!sl_wait_warp(&dfull[db], dph, g.tries)) {
                    if (lane == 0) atomicExch(g.err, 27);
                    ok = false;
                    break;
                }
                asm volatile("tcgen05.fence::after_thread_sync;");
                const uint32_t d = tl + (uint32_t)(db * g.d_step);
#pragma unroll
                for (int c = 0; c < V4; ++c) {
                    if (8 * c < V) {
                        uint32_t r[kSl][4];
#pragma unroll
                        for (int l = 0; l < kSl; ++l) tmem_ld4(d + l * V + 4 * (g0 + c), r[l]);
                        asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
                        for (int u = 0; u < 4; ++u) {
                            long long a = __float2int_rn(__uint_as_float(r[0][u]));
#pragma unroll
                            for (int l = 1; l < 6; ++l) a = a * 256 + __float2int_rn(__uint_as_float(r[l][u]));
                            acc[4 * c + u] += a + ((__float2int_rn(__uint_as_float(r[6][u])) + 128) >> 8);
                        }
                    }
                }
                asm volatile("tcgen05.fence::before_thread_sync;");
                __syncwarp();
                if (lane == 0) sl_arrive(&dempty[db]);
                dph ^= (uint32_t)db;
                db ^= 1;
            }
            if (!ok) break;
            const int mat = w ? g.ent[xm].x : xm;
            // digits: v = 2^(ex - 6) sum d_t 256^-t; level l weighs 256^-l 2^-12, so
            // level 5 is 2^-52
            const int rex = row < p.rows ? p.rs[(size_t)mat * (p.rows / 2) + (row >> 1)] : 0;
            const int* xs = p.xs + (size_t)xm * (V / 2);
            const bool im = rho & 1;
            int c0 = 0, nt = 0;
            if (w) {
                c0 = g.type_ptr[mat];
                nt = (g.type_ptr[mat + 1] - c0) * g.R;
            }
#pragma unroll
            for (int c = 0; c < V4; ++c) {
                const int cc = g0 + c;
                if (8 * c >= V || (!w && cc >= p.live)) continue;
                // rows re and im of one complex row on neighbouring lanes (same scale):
                // the re lane forms the product with the first complex vector of the
                // group of two, the im lane with the second
                const long long* q = acc + 4 * c;
                const long long t0 = __shfl_xor_sync(0xffffffffu, im ? q[0] : q[2], 1);
                const long long t1 = __shfl_xor_sync(0xffffffffu, im ? q[1] : q[3], 1);
                const long long pr = im ? t0 - q[3] : q[0] - t1, pi = im ? t1 + q[2] : q[1] + t0;
                // the sums scaled by 2^e, in two steps where that power or a product with it
                // (below 2^63) could leave FP64's range; a component that was not finite
                // (kSlNan) marks every output
                const int e = rex + xs[2 * cc + (im ? 1 : 0)] - 52;
                double2 u = make_double2((double)pr, (double)pi);
                if (e >= -1000 && e <= 900) {
                    const double sc = sl_pow2(e);
                    u = make_double2(u.x * sc, u.y * sc);
                } else {
                    const int e1 = max(min(e, 2000), -2000), e0 = e1 / 2;
                    const double sc = sl_pow2(e0), s2 = e > 4000 ? sl_nan() : sl_pow2(e1 - e0);
                    u = make_double2(u.x * sc * s2, u.y * sc * s2);
                }
                if (!w) {
                    // y_J = a L x_J + b K x_M, y_M = g K x_J + d L x_M
                    const int role = rho & 3;                  // L x_J, L x_M, K x_J, K x_M
                    const double2 cf = role == 0 ? g.co[0] : role == 1 ? g.co[3] : role == 2 ? g.co[2] : g.co[1];
                    u = cmul(cf, u);
                    const double px = __shfl_xor_sync(0xffffffffu, u.x, 3), py = __shfl_xor_sync(0xffffffffu, u.y, 3);
                    const int i = row >> 2;
                    if (!im && i < g.E)
                        g.Y[((size_t)xm * g.R + g.r0 + cc) * 2 * g.E + (role == 2 ? g.E : 0) + i] =
                            make_double2(u.x + px, u.y + py);
                } else {
                    const int col = g.ent[xm].y + 2 * cc + (im ? 1 : 0);
                    if (row < p.rows && col < nt) {
                        const int cell = g.type_cells[c0 + col / g.R];
                        g.Ymm[((size_t)(col % g.R) * g.M + cell) * g.K + (row >> 1)] = u;
                    }
                }
            }
        }
        if (!ok) *abort_v = 1;
    }
    asm volatile("tcgen05.fence::before_thread_sync;");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;");
    if (warp == kSlWarpM)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kSlTmemCols));
}

// ---------------------------------------------------------------- splitting
// Planes of one row per threadIdx.x, its sources shared by the kSlRowParts values of
// threadIdx.y: rows of bins (MM false) from B^[bin][op][j][i], of macromodels from
// Zt[t][k'][k]; blockIdx.x = tile, blockIdx.y = matrix.  With one thread per row a
// few matrices left the threads waiting for one load after another (create of one
// box with K = 576: 1.24 ms, 1.00 with the parts and one upload of the entries).
constexpr int kSlRowParts = 4;
template <bool MM>
__global__ void __launch_bounds__(kSlRows * kSlRowParts)
slice_rows_kernel(const double2* __restrict__ src, int n, int rows, int nk16, size_t m0, unsigned char* __restrict__ A,
                  int* __restrict__ rs) {
    const size_t mat = m0 + blockIdx.y;
    const int tile = blockIdx.x, rho = threadIdx.x, row = tile * kSlRows + rho;
    const int rt = min(kSlRows, rows - tile * kSlRows), part = threadIdx.y;
    __shared__ unsigned long long s_mx[kSlRowParts][kSlRows];
    const int c = row & 1;
    const double2* s = MM ? src + (mat * n) * n + (row >> 1) : src + ((mat * 2 + ((row >> 1) & 1)) * n) * n + (row >> 2);
    unsigned long long mx = 0;
    for (int j = part; j < n && rho < rt; j += kSlRowParts) {
        const double2 v = s[(size_t)j * n];
        mx = max(mx, max(sl_abs(v.x), sl_abs(v.y)));
    }
    s_mx[part][rho] = mx;
    __syncthreads();
    if (rho >= rt) return;
#pragma unroll
    for (int q = 0; q < kSlRowParts; ++q) mx = max(mx, s_mx[q][rho]);
    const int ex = sl_exp(mx, n);
    if (c == 0 && part == 0) rs[(mat * rows + row) >> 1] = ex;
    unsigned char* out = A + (mat * rows + (size_t)tile * kSlRows) * nk16 * kSlKbBytes;
    for (int kb = part; kb < nk16; kb += kSlRowParts) {
        uint32_t w[kSl][4];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
#pragma unroll
            for (int t = 0; t < kSl; ++t) w[t][q] = 0;
#pragma unroll
            for (int b = 0; b < 4; ++b) {
                const int j = kb * 16 + 4 * q + b;
                unsigned long long d = 0x80808080808080ull;
                if (j < n) {
                    const double2 v = s[(size_t)j * n];
                    d = sl_digits(c ? v.y : v.x, ex);
                }
#pragma unroll
                for (int t = 0; t < kSl; ++t) w[t][q] |= (uint32_t)(d >> 8 * (kSl - 1 - t) & 0xff) << (8 * b);
            }
        }
#pragma unroll
        for (int t = 0; t < kSl; ++t)
            reinterpret_cast<uint4*>(out)[(kb * kSl + t) * rt + rho] = make_uint4(w[t][0], w[t][1], w[t][2], w[t][3]);
    }
}

// Digits of complex vectors v0, v0 + 1 of an x matrix (V / 2 of n entries each),
// one pair per block: load(v, j) = entry j of vector v (zero past the live
// ones).  The block of the last pair also clears the padding rows.
template <typename Load>
__device__ __forceinline__ void slice_vectors(int n, int nst, int V, int Np, int v0, Load&& load,
                                              unsigned char* __restrict__ X, int* __restrict__ xs) {
    dep_trigger();
    extern __shared__ double2 s_v[];         // [2][n]
    __shared__ unsigned long long s_mx[2];
    __shared__ int s_ex[2];
    const int lane = threadIdx.x & 31;
    if (threadIdx.x < 2) s_mx[threadIdx.x] = 0;
    __syncthreads();
    {
        // half of the threads per vector
        const int h = threadIdx.x >= blockDim.x / 2, v = v0 + h;
        unsigned long long mx = 0;
#pragma unroll 4
        for (int j = threadIdx.x - h * (blockDim.x / 2); j < n; j += blockDim.x / 2) {
            const double2 a = load(v, j);
            s_v[h * n + j] = a;
            mx = max(mx, max(sl_abs(a.x), sl_abs(a.y)));
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, o));
        if (lane == 0) atomicMax(&s_mx[h], mx);
    }
    __syncthreads();
    if (threadIdx.x < 2) {
        const int ex = sl_exp(s_mx[threadIdx.x], n);
        s_ex[threadIdx.x] = ex;
        xs[v0 + threadIdx.x] = ex;
    }
    __syncthreads();
    // 8 sources of one real vector per thread: one 16-byte chunk per digit
    const int chunks = 4 * nst;
    auto at = [&](int row, int ch) {
        return reinterpret_cast<uint4*>(X + ((size_t)(ch >> 2) * Np + row) * 64 + ((ch & 3) ^ ((row >> 1) & 3)) * 16);
    };
    for (int e = threadIdx.x; e < 4 * chunks; e += blockDim.x) {
        const int ch = e >> 2, v = 2 * v0 + (e & 3), h = (e >> 1) & 1;
        const int ex = s_ex[h];
        const double* src = reinterpret_cast<const double*>(s_v + h * n) + (e & 1);
        unsigned long long d[8];
#pragma unroll
        for (int b = 0; b < 8; ++b) {
            const int j = 8 * ch + b;
            d[b] = j < n ? sl_digits(src[2 * j], ex) : 0x80808080808080ull;
        }
#pragma unroll
        for (int t = 0; t < kSl; ++t) *at(t * V + v, ch) = sl_halves(d, t);
    }
    if (v0 + 2 < V / 2) return;
    for (int e = threadIdx.x; e < (Np - kSl * V) * chunks; e += blockDim.x) {
        const int ch = e / (Np - kSl * V), row = kSl * V + e - ch * (Np - kSl * V);
        *at(row, ch) = make_uint4(0u, 0u, 0u, 0u);
    }
}

// bins: vectors (r, part) of X^[bin][R][2E], r0 <= r < r0 + live (zero above)
__global__ void __launch_bounds__(kSlSplit)
slice_bins_kernel(const double2* __restrict__ Xg, int E, int R, int r0, int live, int nst, int V, int Np,
                  unsigned char* __restrict__ X, int* __restrict__ xs) {
    const size_t bin = blockIdx.x;
    const double2* src = Xg + (bin * R + r0) * 2 * E;
    slice_vectors(
        E, nst, V, Np, 2 * blockIdx.y, [&](int v, int j) { return v < 2 * live ? src[(size_t)v * E + j] : make_double2(0.0, 0.0); },
        X + bin * nst * Np * 64, xs + bin * (V / 2));
}

// macromodels: columns (cell slot, rhs) of an entry's type, x1 = U_o x gathered
__global__ void __launch_bounds__(kSlSplit)
slice_cells_kernel(const double2* __restrict__ x, const int32_t* __restrict__ idx, const int8_t* __restrict__ sgn,
                   const int2* __restrict__ ent, const int32_t* __restrict__ type_ptr,
                   const int32_t* __restrict__ type_cells, int K, int R, int n_unique, int nst, int V, int Np,
                   unsigned char* __restrict__ X, int* __restrict__ xs) {
    const int2 e = ent[blockIdx.x];
    const int c0 = type_ptr[e.x], nt = (type_ptr[e.x + 1] - c0) * R;
    slice_vectors(
        K, nst, V, Np, 2 * blockIdx.y,
        [&](int v, int j) {
            const int col = e.y + v;
            if (col >= nt) return make_double2(0.0, 0.0);
            const size_t at = (size_t)type_cells[c0 + col / R] * K + j;
            const double s = (double)sgn[at];
            const double2 a = x[(size_t)(col % R) * n_unique + idx[at]];
            return make_double2(s * a.x, s * a.y);
        },
        X + (size_t)blockIdx.x * nst * Np * 64, xs + (size_t)blockIdx.x * (V / 2));
}

// columns of a launch of Rg rhs
int sl_bin_v(int Rg) { return (4 * Rg + 7) & ~7; }
int nk16_of(int n) { return (n + 15) / 16; }
// rhs of a launch
int rhs_per(int R) {
    const int groups = (R + kSlRhs - 1) / kSlRhs;
    return (R + groups - 1) / groups;
}
// columns of a macromodel entry: as many as the bins' accumulators have room for
// anyway (an MMA costs the same up to N = 176), at least 8
int cells_of(int R) { return sl_bin_v(rhs_per(R)) == kSlMaxV ? kSlMaxV / 2 : 8; }
int cell_rows(int R) { return sl_up16(kSl * 2 * cells_of(R)); }   // digit rows of an entry
int nst_of(int n) { return (n + kSlK - 1) / kSlK; }
// macromodel entries of R rhs
size_t mm_entries(const emsurf_handle* h, int R) {
    const int per = cells_of(R);
    size_t n = 0;
    for (int t = 0; t < h->T; ++t) n += ((h->h_type_ptr[t + 1] - h->h_type_ptr[t]) * (size_t)R + per - 1) / per;
    return n;
}

// what the macromodel columns of 1..max_rhs rhs take: the most digits and exponents,
// the entries of all
struct CellSizes {
    size_t digits = 0, exps = 0, entries = 0;
};
CellSizes cell_sizes(const emsurf_handle* h) {
    CellSizes z;
    for (int r = 1; r <= h->max_rhs; ++r) {
        const size_t n = mm_entries(h, r);
        z.digits = std::max(z.digits, n * nst_of(h->K) * cell_rows(r) * 64);
        z.exps = std::max(z.exps, n * cells_of(r) * sizeof(int));
        z.entries += n;
    }
    return z;
}

}  // namespace

size_t slice_plane_bytes(size_t mats, int rows, int n) { return mats * rows * (size_t)nk16_of(n) * kSlKbBytes; }

// Digit planes of the FP64 spectrum and of the macromodels, each left out when
// the device-memory budget has no room for it and the work space that goes with
// it (products then use the FP64 blocks).  The spectrum's planes of a shared
// handle are taken over; digits false: nothing else.
int slices_build(emsurf_handle* h, const emsurf_handle* share, bool digits) {
    const int E = h->E, K = h->K;
    const size_t nb = (size_t)h->nbins, grids = nb * (size_t)h->max_rhs * K, cells = (size_t)h->max_rhs * h->M * K;
    const size_t bbytes = slice_plane_bytes(nb, 4 * E, E), brs = nb * 2 * E * sizeof(int);
    const CellSizes cs = cell_sizes(h);
    const size_t zbytes = slice_plane_bytes(h->T, 2 * K, K),
                 zrs = (size_t)h->T * K * sizeof(int) + cs.digits + cs.exps + cs.entries * sizeof(int2);
    if (share ? !share->sl_A : !digits || E > kSlMaxN) return EMSURF_OK;
    cudaStream_t st = h->setup_stream;
    // work space still to come: grids, products, and the partials of the SIMT macromodels
    const size_t work = (2 * grids + cells) * sizeof(double2), split = cells * sizeof(double2);
    auto fits = [&](size_t n) { return h->budget <= 0 || h->device_bytes + (int64_t)n <= h->budget; };
    if (share) {
        h->sl_A = share->sl_A;
        h->sl_rs = share->sl_rs;
    } else {
        if (!fits(bbytes + brs + work + kMmSplit * split) &&
            (K > kSlMaxN || !fits(bbytes + brs + zbytes + zrs + work + split)))
            return EMSURF_OK;
        EMS_TRY(dev_alloc(h, (void**)&h->sl_A, bbytes));
        EMS_TRY(dev_alloc(h, (void**)&h->sl_rs, brs));
        for (size_t m0 = 0; m0 < nb; m0 += 65535) {
            const dim3 grid((4 * E + kSlRows - 1) / kSlRows, (unsigned)std::min<size_t>(65535, nb - m0));
            slice_rows_kernel<false><<<grid, dim3(kSlRows, kSlRowParts), 0, st>>>(h->op64.Bhat, E, 4 * E, nk16_of(E), m0, h->sl_A, h->sl_rs);
            EMS_CUDA(cudaGetLastError());
            h->launches += 1;
        }
    }
    if (!digits || K > kSlMaxN || !fits(zbytes + zrs + work + split)) return EMSURF_OK;
    EMS_TRY(dev_alloc(h, (void**)&h->sl_Z, zbytes));
    EMS_TRY(dev_alloc(h, (void**)&h->sl_zrs, (size_t)h->T * K * sizeof(int)));
    for (size_t m0 = 0; m0 < (size_t)h->T; m0 += 65535) {
        const dim3 grid((2 * K + kSlRows - 1) / kSlRows, (unsigned)std::min<size_t>(65535, h->T - m0));
        slice_rows_kernel<true><<<grid, dim3(kSlRows, kSlRowParts), 0, st>>>(h->op64.Zt, K, 2 * K, nk16_of(K), m0, h->sl_Z, h->sl_zrs);
        EMS_CUDA(cudaGetLastError());
        h->launches += 1;
    }
    return EMSURF_OK;
}

// Vector digits' work space (after the FP64 spectrum is given back); digits as for
// slices_build.
int slices_work(emsurf_handle* h, bool digits) {
    const int R = h->max_rhs, V = sl_bin_v(std::min(R, kSlRhs));
    if (h->sl_Z) {
        const CellSizes cs = cell_sizes(h);
        EMS_TRY(dev_alloc(h, (void**)&h->sl_Xc, cs.digits));
        EMS_TRY(dev_alloc(h, (void**)&h->sl_xcs, cs.exps));
        h->sl_ent.assign(R + 1, nullptr);
        h->sl_nent.assign(R + 1, 0);
        std::vector<int2> e;
        e.reserve(cs.entries);
        int2* dev = nullptr;
        EMS_TRY(dev_alloc(h, (void**)&dev, cs.entries * sizeof(int2)));
        for (int r = 1; r <= R; ++r) {
            h->sl_ent[r] = dev + e.size();
            for (int t = 0; t < h->T; ++t)
                for (int c = 0; c < (h->h_type_ptr[t + 1] - h->h_type_ptr[t]) * r; c += cells_of(r)) e.push_back(make_int2(t, c));
            h->sl_nent[r] = (int)(dev + e.size() - static_cast<int2*>(h->sl_ent[r]));
        }
        EMS_CUDA(cudaMemcpyAsync(dev, e.data(), e.size() * sizeof(int2), cudaMemcpyHostToDevice, h->setup_stream));
        EMS_CUDA(cudaStreamSynchronize(h->setup_stream));     // e goes out of scope
    }
    // bins whose digits are held at a time: all of them up to 512 MiB, fewer under
    // a tight budget (a handle that shares its spectrum gives none back), one at
    // worst where the handle is built without planes of its own
    const size_t per = (size_t)nst_of(h->E) * sl_up16(kSl * V) * 64 + (V / 2) * sizeof(int);
    size_t nb = std::min<size_t>(h->nbins, std::max<size_t>(1, ((size_t)512 << 20) / per));
    while (nb > (digits ? 16u : 1u) && h->budget > 0 && h->device_bytes + (int64_t)(nb * per) > h->budget) nb = (nb + 1) / 2;
    h->sl_bins = (int)nb;
    EMS_TRY(dev_alloc(h, (void**)&h->sl_X, nb * nst_of(h->E) * sl_up16(kSl * V) * 64));
    EMS_TRY(dev_alloc(h, (void**)&h->sl_xs, nb * (V / 2) * sizeof(int)));
    return EMSURF_OK;
}

// Digits of x1 for the macromodel product of R rhs (reads x only).
int slices_cells(emsurf_handle* h, const double2* x, int R, cudaStream_t st) {
    const int V = 2 * cells_of(R);
    EMS_TRY(set_smem_once(slice_cells_kernel, 2 * h->K * sizeof(double2)));
    slice_cells_kernel<<<dim3(h->sl_nent[R], V / 4), kSlSplit, 2 * h->K * sizeof(double2), st>>>(x, h->d_uo_index, h->d_uo_sign,
                                                     static_cast<const int2*>(h->sl_ent[R]), h->d_type_ptr,
                                                     h->d_type_cells, h->K, R, h->n_unique, nst_of(h->K), V,
                                                     cell_rows(R), h->sl_Xc, h->sl_xcs);
    EMS_CUDA(cudaGetLastError());
    h->launches += 1;
    return EMSURF_OK;
}

static_assert(2 * sl_up16(kSl * kSlMaxV) + 2 * (int)kSlAStep <= (int)kSlTmemCols, "TMEM columns");

namespace {
// Launch of rhs r0 .. r0 + Rg - 1 of R and the bins from b0: arguments, blocks, shared memory.
struct SlLaunch {
    SlArgs g;
    int grid;
    size_t smem;
};
SlLaunch sl_launch(const emsurf_handle* h, double2* Yg, double2* Ymm, int R, int r0, int Rg, int b0, const double2* coef) {
    const int E = h->E, K = h->K;
    SlArgs g{};
    SlProb& b = g.p[0];
    b.nk16 = nk16_of(E);
    b.nst = nst_of(E);
    b.rows = 4 * E;
    b.tiles = (b.rows + kSlRows - 1) / kSlRows;
    b.A = h->sl_A + slice_plane_bytes(b0, b.rows, E);
    b.rs = h->sl_rs + (size_t)b0 * 2 * E;
    b.X = h->sl_X;
    b.xs = h->sl_xs;
    b.V = sl_bin_v(Rg);
    b.live = Rg;
    b.Np = sl_up16(kSl * b.V);
    b.xmats = std::min(h->sl_bins, h->nbins - b0);
    b.items = b.xmats * b.tiles;
    SlProb& m = g.p[1];
    m.A = h->sl_Z;
    m.rs = h->sl_zrs;
    m.X = h->sl_Xc;
    m.xs = h->sl_xcs;
    m.nk16 = nk16_of(K);
    m.nst = nst_of(K);
    m.rows = 2 * K;
    m.tiles = (m.rows + kSlRows - 1) / kSlRows;
    m.V = 2 * cells_of(R);
    m.Np = sl_up16(kSl * m.V);
    m.xmats = r0 == 0 && b0 == 0 && h->sl_Z ? h->sl_nent[R] : 0;
    m.items = m.xmats * m.tiles;
    const int dc = std::max(b.Np, m.items ? m.Np : 0), vmax = std::max(b.V, m.items ? m.V : 0);
    g.d_step = dc;
    g.slots = 2 * dc + kSlMaxSlots * (int)kSlAStep <= (int)kSlTmemCols ? kSlMaxSlots : 2;
    g.z_bytes = (kSl - 1) * vmax * 64;
    g.x_bytes = dc * 64;
    const size_t xring = (size_t)kSlXStages * (g.z_bytes + g.x_bytes);
    g.stages = std::min(kSlMaxStages, (int)((kSlSmemMax - 1024 - xring) / kSlABytes));
    g.Y = Yg + (size_t)b0 * R * 2 * E;
    g.E = E;
    g.R = R;
    g.r0 = r0;
    for (int c = 0; c < 4; ++c) g.co[c] = coef[c];
    g.Ymm = Ymm;
    g.ent = h->sl_Z ? static_cast<const int2*>(h->sl_ent[R]) : nullptr;
    g.type_ptr = h->d_type_ptr;
    g.type_cells = h->d_type_cells;
    g.K = K;
    g.M = h->M;
    g.err = h->d_err;
    g.tries = kSlWait;
    return {g, std::min(std::max(1, h->num_sms), b.items + m.items), 1024 + (size_t)g.stages * kSlABytes + xring};
}
}  // namespace

// Y^ = B^ X^ for every bin and Ymm = Z~ x1 for every cell, R rhs: up to kSlRhs rhs of
// sl_bins bins per launch, the macromodels (when their planes are there) with the first.
int slices_multiply(emsurf_handle* h, const double2* Xg, double2* Yg, double2* Ymm, int R, const double2* coef,
                    cudaStream_t st) {
    const int E = h->E, per = rhs_per(R);
    for (int r0 = 0; r0 < R; r0 += per)
        for (int b0 = 0; b0 < h->nbins; b0 += h->sl_bins) {
            const int Rg = std::min(per, R - r0);
            const SlLaunch l = sl_launch(h, Yg, Ymm, R, r0, Rg, b0, coef);
            const SlProb& b = l.g.p[0];
            EMS_TRY(set_smem_once(slice_bins_kernel, 2 * E * sizeof(double2)));
            slice_bins_kernel<<<dim3(b.xmats, b.V / 4), kSlSplit, 2 * E * sizeof(double2), st>>>(
                Xg + (size_t)b0 * R * 2 * E, E, R, r0, Rg, b.nst, b.V, b.Np, h->sl_X, h->sl_xs);
            EMS_CUDA(cudaGetLastError());
            EMS_TRY(set_smem_once(slices_kernel, l.smem));
            EMS_CUDA(launch_after(slices_kernel, dim3(l.grid), kSlThreads, l.smem, st, l.g));
            h->launches += 2;
        }
    return EMSURF_OK;
}

// Products whose vector digits never arrive: every role's wait expires (no output
// is written).
int slices_selftest(emsurf_handle* h, int tries, int* err, cudaStream_t st) {
    SlLaunch l = sl_launch(h, h->op64.Yg, h->op64.Ymm, 1, 0, 1, 0, h->op64.coef);
    l.g.err = err;
    l.g.tries = tries;
    l.g.starve = 1;
    EMS_TRY(set_smem_once(slices_kernel, l.smem));
    slices_kernel<<<l.grid, kSlThreads, l.smem, st>>>(l.g);
    EMS_CUDA(cudaGetLastError());
    h->launches += 1;
    return EMSURF_OK;
}

}  // namespace emsurf
