// SARA dictionary Psi = (1/3) [Dirac, db1, ..., db8] (Section 2.2, Section
// 5.1): separable periodic 2-D DWT, 4 levels, rows then columns per level,
// Mallat quadrant layout per basis; and the prior dual step of Algorithm 3,
// u_i <- (I - S_alpha)(u_i + W_i Psi_i^dagger xt) = clip(u_i + W_i Psi_i^dagger xt, +-alpha),
// fused into the analysis output, with the prior weights W_i of the
// re-weighted scheme (Algorithm 1; W = I unless set) and the clip level
// alpha = kappa ||Psi W||_S^2.  D_b below is the orthonormal DWT of basis b.
//
// The eight wavelet bases run together (grid.y = basis); the filter taps
// sit in registers, the level tiles in shared memory.  Each filter pass
// reads an input window once for every output that uses it: the analysis
// forms the low (h) and high (g) half of a position together, the synthesis
// an even and an odd output sample together (they read the same inputs with
// the even and the odd taps).  Filters are derived on the host by
// minimum-phase spectral factorisation (Daubechies 1988) with a
// Durand-Kerner root finder.
#include <cmath>
#include <algorithm>
#include <complex>

#include "common.cuh"
#include "tma.cuh"

namespace ppd {

__constant__ float c_filt_f[N_WAVELETS][MAX_TAPS];
__constant__ double c_filt_d[N_WAVELETS][MAX_TAPS];

namespace {

// Filter taps of length F (basis db(F/2)) in F registers: h[k], and the
// high-pass g[k] = (-1)^k h[F-1-k] by the sign of an operand.  The asm keeps
// them there: read from the constant bank at each use they cost a load each.
template <typename R, int F> struct Taps {
    R t[F];
    __device__ __forceinline__ Taps() {
#pragma unroll
        for (int k = 0; k < F; ++k) {
            if constexpr (sizeof(R) == 4) {
                t[k] = c_filt_f[F / 2 - 1][k];
                asm volatile("" : "+f"(t[k]));
            } else {
                t[k] = c_filt_d[F / 2 - 1][k];
                asm volatile("" : "+d"(t[k]));
            }
        }
    }
    __device__ __forceinline__ R h(int k) const { return t[k]; }
    __device__ __forceinline__ R g(int k) const { return (k & 1) ? -t[F - 1 - k] : t[F - 1 - k]; }
};

constexpr int NT = 256;

// periodic index i mod n (i may be negative); indices inside [0, n) are
// the common case and skip the division
__device__ __forceinline__ int wrap(int i, int n) {
    if ((unsigned)i < (unsigned)n) return i;
    const int r = i % n;
    return r < 0 ? r + n : r;
}

// One value from global to shared memory in the background.
template <typename R> __device__ __forceinline__ void copy_async(R *dst, const R *src) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], %2;" ::"r"(smem_u32(dst)), "l"(src), "n"(sizeof(R)) : "memory");
}
// 16 bytes of it (both sides 16-byte aligned).
__device__ __forceinline__ void copy_async16(void *dst, const void *src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_u32(dst)), "l"(src) : "memory");
}
__device__ __forceinline__ bool aligned16(const void *p) { return (reinterpret_cast<uintptr_t>(p) & 15) == 0; }
__device__ __forceinline__ void copy_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N> __device__ __forceinline__ void copy_wait() {
    asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

// V consecutive values between shared memory and registers, in pieces of W
// values; the start is aligned to a piece (a load may read past V to the end
// of its piece).
template <typename R, int W> struct Piece;
template <> struct Piece<float, 4> { using T = float4; };
template <> struct Piece<float, 2> { using T = float2; };
template <> struct Piece<double, 2> { using T = double2; };
template <int W, typename R, int V> __device__ __forceinline__ void load_row(const R *p, R (&v)[V]) {
#pragma unroll
    for (int j = 0; j < (V + W - 1) / W; ++j) {
        const auto t = reinterpret_cast<const typename Piece<R, W>::T *>(p)[j];
        R u[W];
        *reinterpret_cast<typename Piece<R, W>::T *>(u) = t;
#pragma unroll
        for (int k = 0; k < W; ++k)
            if (W * j + k < V) v[W * j + k] = u[k];
    }
}
template <int W, typename R, int V> __device__ __forceinline__ void store_row(R *p, const R (&v)[V]) {
    static_assert(V % W == 0, "whole pieces");
#pragma unroll
    for (int j = 0; j < V / W; ++j) {
        R u[W];
#pragma unroll
        for (int k = 0; k < W; ++k) u[k] = v[W * j + k];
        reinterpret_cast<typename Piece<R, W>::T *>(p)[j] = *reinterpret_cast<const typename Piece<R, W>::T *>(u);
    }
}
// widest piece of at most 16 bytes that a run of n values starting at a multiple of n is made of
template <typename R> constexpr int piece(int n) { return n * (int)sizeof(R) >= 16 ? 16 / (int)sizeof(R) : n; }

// ------------------------------------------------------------- tile geometry
// A level kernel's CTA covers TS x TS quadrant positions.  The filters slide
// over registers: a thread forms PS neighbouring outputs of a pass from one
// set of inputs read once (PS = 4: 2 PS + F - 2 inputs for 2 PS F FMAs), where
// a window of F shared reads per output pair left the FMA pipe at a third
// and the issue slots full.  TS = 32 reads 1.5 times its input (halo), TS =
// 16 2.1 times; the small tile serves levels that would not give every SM
// two large ones, and FP64.  Level 0 before -> now: analysis 118 -> 61 us at
// 2048^2 (67 with the Dirac basis, which had a launch of 9), 38 -> 26 us at
// 1024^2, 12.7 -> 9.6 us at 512^2; synthesis 176 -> 101, 47 -> 28, 15.5 -> 10.5
// us.  Issue slots bound the analysis (80 % busy at 2048^2, FMAs under half of
// them).  Row pitches are 4 mod 8 floats with 8 rows in
// distinct banks for 16-byte accesses of lanes in consecutive rows.
template <int TS> struct AnaGeo {
    static constexpr int EXT = 2 * TS + MAX_TAPS - 2;           // input tile side (78 / 46)
    static constexpr int PI = TS == 32 ? 84 : 52;               // its pitch
    static constexpr int PR = 2 * TS + 4;                       // pitch of the row-filtered tile (68 / 36)
    static constexpr int PS = TS == 32 ? 4 : 2;                 // outputs per thread and pass
};
template <typename R, int TS> constexpr size_t ana_smem() {
    return sizeof(R) * AnaGeo<TS>::EXT * (AnaGeo<TS>::PI + AnaGeo<TS>::PR);
}
template <int TS> struct SynGeo {
    static constexpr int EXT = TS + MAX_TAPS / 2 - 1;           // quadrant tile side (39 / 23)
    static constexpr int PQ = TS + 8;                           // its pitch; column 0 is position C0 - 8
    static constexpr int PT = TS == 32 ? 44 : 28;               // pitch of the axis-0 results
    static constexpr int PS = TS == 32 ? 4 : 2;                 // position pairs per thread and pass
    static constexpr int QUADS = 4 * EXT * PQ, HALVES = 2 * 2 * TS * PT;
};
template <typename R, int TS> constexpr size_t syn_smem() {
    return sizeof(R) * (SynGeo<TS>::QUADS + SynGeo<TS>::HALVES);
}

// ------------------------------------------------------------- analysis
// One tile of one level and basis (filter length F): the level input is n0 x
// n1, its quadrants h0 x h1.  Rows (axis 1) are filtered into rowf, then
// columns (axis 0).  Tiles reaching past h0 or h1 skip the positions outside.
template <typename R, int F, int TS, int MODE>
__device__ __forceinline__ void ana_tile(const R *__restrict__ src, int in_pitch, int n0, int n1, int R0, int C0,
                                         R *__restrict__ ll, int last, R *__restrict__ cb,
                                         const R *__restrict__ wb, int L1, R kappa, R *__restrict__ dirac, R *tin,
                                         R *rowf) {
    using G = AnaGeo<TS>;
    constexpr int EXT = 2 * TS + F - 2, PS = G::PS, NR = TS / PS;
    static_assert(2 * TS * NR % NT == 0, "column tasks");
    constexpr int NC = 2 * TS * NR / NT;   // column tasks per thread
    const int h0 = n0 >> 1, h1 = n1 >> 1;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const Taps<R, F> f;
    // input tile: 16-byte pieces where rows are aligned and the columns don't
    // wrap (a fifth of the copy instructions), else value by value
    constexpr int VE = 16 / sizeof(R), NV = (EXT + VE - 1) / VE;
    if (2 * C0 + NV * VE <= n1 && aligned16(src) && in_pitch % VE == 0) {
        for (int e = threadIdx.x; e < EXT * NV; e += NT) {
            const int i = e / NV, v = e - i * NV;
            copy_async16(tin + i * G::PI + v * VE,
                         src + (int64_t)wrap(2 * R0 + i, n0) * in_pitch + 2 * C0 + v * VE);
        }
    } else {
        int jc[3];
#pragma unroll
        for (int q = 0; q < 3; ++q) jc[q] = lane + 32 * q < EXT ? wrap(2 * C0 + lane + 32 * q, n1) : 0;
        for (int i = warp; i < EXT; i += NT / 32) {
            const R *row = src + (int64_t)wrap(2 * R0 + i, n0) * in_pitch;
#pragma unroll
            for (int q = 0; q < 3; ++q)
                if (lane + 32 * q < EXT) copy_async(tin + i * G::PI + lane + 32 * q, row + jc[q]);
        }
    }
    copy_commit();
    // the coefficients this thread clip-updates (and their weights), in
    // flight beside the input tile
    R pu[NC][2 * PS], pw[NC][2 * PS];
    const int64_t high = (int64_t)h0 * L1;
    // of column task t: first output row, rows inside the quadrant, and the
    // coefficient of that row in the low axis-0 half (+ high: the high half)
    auto place = [&](int t, int &r0, int &rows) {
        const int task = threadIdx.x + t * NT, c = task % (2 * TS), cc = c & (TS - 1);
        r0 = (task / (2 * TS)) * PS;
        rows = C0 + cc < h1 ? min(PS, h0 - R0 - r0) : 0;
        return (int64_t)(R0 + r0) * L1 + (c >= TS ? h1 : 0) + C0 + cc;
    };
    auto is_ll = [&](int t) { return !last && (threadIdx.x + t * NT) % (2 * TS) < TS; };   // low half goes to ll
    if constexpr (MODE != 0) {
#pragma unroll
        for (int t = 0; t < NC; ++t) {
            int r0, rows;
            const int64_t off = place(t, r0, rows);
            const bool lo = !is_ll(t);
#pragma unroll
            for (int k = 0; k < PS; ++k) {
                const bool in = k < rows;
                pu[t][2 * k] = in && lo ? cb[off + (int64_t)k * L1] : R(0);
                pu[t][2 * k + 1] = in ? cb[off + high + (int64_t)k * L1] : R(0);
                if constexpr (MODE == 2) {
                    pw[t][2 * k] = in && lo ? wb[off + (int64_t)k * L1] : R(0);
                    pw[t][2 * k + 1] = in ? wb[off + high + (int64_t)k * L1] : R(0);
                }
            }
        }
    }
    copy_wait<0>();
    __syncthreads();
    if constexpr (F == 2 && MODE == 0) {
        // the Dirac basis is the input itself: the shortest filter's CTAs of
        // level 0 write their part of it (a launch of its own was 3 us at
        // 256^2 and 9 us at 2048^2)
        if (dirac)
            for (int e = threadIdx.x; e < 4 * TS * TS; e += NT) {
                const int r = e / (2 * TS), c = e % (2 * TS);
                if (2 * R0 + r < n0 && 2 * C0 + c < n1)
                    dirac[(int64_t)(2 * R0 + r) * L1 + 2 * C0 + c] = R(1.0 / 3.0) * tin[r * G::PI + c];
            }
    }
    // rows: task (row i, PS positions): low halves into column q, high into TS + q
    for (int task = threadIdx.x; task < EXT * NR; task += NT) {
        const int i = task % EXT, q0 = (task / EXT) * PS;
        R v[2 * PS + F - 2], lo[PS], hi[PS];
        load_row<piece<R>(2 * PS)>(tin + i * G::PI + 2 * q0, v);
#pragma unroll
        for (int p = 0; p < PS; ++p) lo[p] = hi[p] = R(0);
#pragma unroll
        for (int k = 0; k < F; ++k)
#pragma unroll
            for (int p = 0; p < PS; ++p) {
                lo[p] = fma(f.h(k), v[2 * p + k], lo[p]);
                hi[p] = fma(f.g(k), v[2 * p + k], hi[p]);
            }
        R *o = rowf + i * G::PR + q0;
        store_row<piece<R>(PS)>(o, lo);
        store_row<piece<R>(PS)>(o + TS, hi);
    }
    __syncthreads();
    // columns: task (column c of the row-filtered tile, PS positions)
#pragma unroll
    for (int t = 0; t < NC; ++t) {
        const int task = threadIdx.x + t * NT, c = task % (2 * TS), r0 = (task / (2 * TS)) * PS;
        const R *col = rowf + 2 * r0 * G::PR + c;
        R lo[PS], hi[PS];
#pragma unroll
        for (int p = 0; p < PS; ++p) lo[p] = hi[p] = R(0);
#pragma unroll
        for (int j = 0; j < 2 * PS + F - 2; ++j) {   // input j serves tap j - 2p of position p
            const R v = col[j * G::PR];
#pragma unroll
            for (int p = 0; p < PS; ++p)
                if (j - 2 * p >= 0 && j - 2 * p < F) {
                    lo[p] = fma(f.h(j - 2 * p), v, lo[p]);
                    hi[p] = fma(f.g(j - 2 * p), v, hi[p]);
                }
        }
        int rr, rows;
        const int64_t off = place(t, rr, rows);
        auto emit = [&](R acc, int k, R *dst) {
            const R cv = acc * R(1.0 / 3.0);
            if constexpr (MODE == 0) {
                *dst = cv;
            } else {
                const R u = pu[t][k] + (MODE == 2 ? pw[t][k] * cv : cv);
                *dst = fmin(fmax(u, -kappa), kappa);
            }
        };
        R *llp = ll + (int64_t)(R0 + rr) * h1 + C0 + c;
#pragma unroll
        for (int k = 0; k < PS; ++k) {
            if (k >= rows) break;
            if (is_ll(t)) llp[(int64_t)k * h1] = lo[k];
            else emit(lo[k], 2 * k, cb + off + (int64_t)k * L1);
            emit(hi[k], 2 * k + 1, cb + off + high + (int64_t)k * L1);
        }
    }
}

// One analysis level for all 8 wavelet bases (grid.y: longest filter first).
//   in:   level input n0 x n1, basis b at in + b*in_bstride, row pitch in_pitch
//   ll:   next level's input (compact, pitch h1) unless last
//   coef: coefficient images (basis b+1 at coef + (b+1)*N, pitch L1), written
//         (MODE 0: c = D x / 3) or clip-updated (1: u = clip(u + D x / 3, kappa);
//         2: u = clip(u + w D x / 3, kappa), w the prior weights wgt, laid out
//         like coef)
//   dirac: MODE 0, level 0: the Dirac basis's coefficients x / 3, or null (in
//         must not overlap them)
//   pmask: active set P of Algorithm 3 (9 flags, Dirac first) or null; in
//         modes 1 and 2 a basis outside P keeps u_b and is skipped at every level
template <typename R, int TS, int MODE>
__global__ void __launch_bounds__(NT) k_sara_ana(const R *__restrict__ in, int in_pitch, int64_t in_bstride, int n0,
                                                 int n1, R *__restrict__ ll, int64_t ll_bstride, int last,
                                                 R *__restrict__ coef, const R *__restrict__ wgt, int L1, int64_t N,
                                                 R kappa, R *__restrict__ dirac,
                                                 const uint8_t *__restrict__ pmask) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    R *tin = reinterpret_cast<R *>(smem_raw), *rowf = tin + AnaGeo<TS>::EXT * AnaGeo<TS>::PI;
    const int b = N_WAVELETS - 1 - blockIdx.y;
    pdl_enter();
    if (MODE != 0 && pmask && !pmask[b + 1]) return;
    const int tpd1 = (n1 / 2 + TS - 1) / TS;
    const int R0 = (blockIdx.x / tpd1) * TS, C0 = (blockIdx.x % tpd1) * TS;
    const R *src = in + (int64_t)b * in_bstride;
    R *lb = ll + (int64_t)b * ll_bstride;
    R *cb = coef + (int64_t)(b + 1) * N;
    const R *wb = MODE == 2 ? wgt + (int64_t)(b + 1) * N : nullptr;
#define PPD_ANA(F) ana_tile<R, F, TS, MODE>(src, in_pitch, n0, n1, R0, C0, lb, last, cb, wb, L1, kappa, dirac, tin, rowf)
    switch (b) {
        case 0: PPD_ANA(2); break;
        case 1: PPD_ANA(4); break;
        case 2: PPD_ANA(6); break;
        case 3: PPD_ANA(8); break;
        case 4: PPD_ANA(10); break;
        case 5: PPD_ANA(12); break;
        case 6: PPD_ANA(14); break;
        default: PPD_ANA(16); break;
    }
#undef PPD_ANA
}

// ------------------------------------------------------------- synthesis
// Inverse of one level (output n0 x n1, quadrants h0 x h1) for one basis on
// one output tile of 2TS x 2TS samples whose quadrant positions start at
// (R0, C0).  The quadrant tiles cover rows R0 - F/2 + 1 ... R0 + TS - 1
// (mod h0) and the same columns (mod h1), TS + F/2 - 1 <= EXT of each.  An
// output pair 2p, 2p + 1 reads quadrant positions p .. p + F/2 - 1 of the
// tile (tap pair kk: position p + F/2 - 1 - kk), the even sample with the
// even taps, the odd one with the odd taps.

// Quadrant tiles of basis filter length F into q (asynchronously; with prior
// weights through registers).
template <typename R, int TS>
__device__ __forceinline__ void syn_load(R *q, const R *__restrict__ cb, const R *__restrict__ wb,
                                         const R *__restrict__ sl, int from_coef, int L1, int h0, int h1, int R0,
                                         int C0, int F) {
    using G = SynGeo<TS>;
    const int ext = TS + F / 2 - 1, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    constexpr int VE = 16 / sizeof(R), NV = (TS + 8) / VE;
    if (!wb && C0 >= 8 && C0 + TS <= h1 && h1 % VE == 0 && L1 % VE == 0 && aligned16(cb) && aligned16(sl)) {
        // whole rows from position C0 - 8 on in 16-byte pieces
        for (int e = threadIdx.x; e < ext * NV; e += NT) {
            const int i = e / NV, v = (e - i * NV) * VE, gi = wrap(R0 - F / 2 + 1 + i, h0);
            const R *c0 = cb + (int64_t)gi * L1 + C0 - 8 + v, *c1 = c0 + (int64_t)h0 * L1;
            const R *l0 = from_coef ? c0 : sl + (int64_t)gi * h1 + C0 - 8 + v;
            R *dst = q + i * G::PQ + v;
            copy_async16(dst, l0);
            copy_async16(dst + G::EXT * G::PQ, c0 + h1);
            copy_async16(dst + 2 * G::EXT * G::PQ, c1);
            copy_async16(dst + 3 * G::EXT * G::PQ, c1 + h1);
        }
        copy_commit();
        return;
    }
    const bool in0 = lane < ext, in1 = lane + 32 < ext;
    const int j0 = in0 ? wrap(C0 - F / 2 + 1 + lane, h1) : 0;
    const int j1 = in1 ? wrap(C0 - F / 2 + 1 + lane + 32, h1) : 0;
    const int64_t high = (int64_t)h0 * L1;
    for (int i = warp; i < ext; i += NT / 32) {   // a warp per row of the four quadrants
        const int gi = wrap(R0 - F / 2 + 1 + i, h0);
        const int64_t off = (int64_t)gi * L1;
        const R *c0 = cb + off, *c1 = c0 + high, *l0 = from_coef ? c0 : sl + (int64_t)gi * h1;
        R *dst = q + i * G::PQ + 9 - F / 2 + lane;
        if (wb) {
            const R *w0 = wb + off, *w1 = w0 + high;
            auto put = [&](int o, int j) {
                dst[o] = from_coef ? l0[j] * w0[j] : l0[j];
                dst[o + G::EXT * G::PQ] = c0[h1 + j] * w0[h1 + j];
                dst[o + 2 * G::EXT * G::PQ] = c1[j] * w1[j];
                dst[o + 3 * G::EXT * G::PQ] = c1[h1 + j] * w1[h1 + j];
            };
            if (in0) put(0, j0);
            if (in1) put(32, j1);
        } else {
            auto put = [&](int o, int j) {
                copy_async(dst + o, l0 + j);
                copy_async(dst + o + G::EXT * G::PQ, c0 + h1 + j);
                copy_async(dst + o + 2 * G::EXT * G::PQ, c1 + j);
                copy_async(dst + o + 3 * G::EXT * G::PQ, c1 + h1 + j);
            };
            if (in0) put(0, j0);
            if (in1) put(32, j1);
        }
    }
    copy_commit();
}

// The low and the high half of a pass are summed apart: in one accumulator every
// addition rounds at the size of the whole sum (error of Psi against 64 bits
// 1.24e-7 of the image, apart 1.18e-7; level 0 at 2048^2 100 and 101 us).
//
// The two filter passes over complete quadrant tiles (a barrier behind them);
// adds the outputs of this thread's tasks to acc: task t = row task % 2TS,
// samples 2 PS (task / 2TS) .. + 2 PS - 1, task = thread + t NT.
template <typename R, int F, int TS, int NO>
__device__ __forceinline__ void syn_compute(const R *q, R *tl, R *th, R (&acc)[NO][2 * SynGeo<TS>::PS]) {
    using G = SynGeo<TS>;
    constexpr int EXT = TS + F / 2 - 1, PS = G::PS, NR = TS / PS, H = F / 2;
    const Taps<R, F> f;
    // axis 0: task (half: columns of the low or of the high axis-1 quadrants,
    // column j, PS positions)
    for (int task = threadIdx.x; task < 2 * EXT * NR; task += NT) {
        const int half = task >= EXT * NR, s = task - half * EXT * NR, j = s % EXT, p0 = (s / EXT) * PS;
        const R *qa = q + (half * G::EXT + p0) * G::PQ + 9 - H + j, *qb = qa + 2 * G::EXT * G::PQ;
        R e[PS], o[PS], eh[PS], oh[PS];
#pragma unroll
        for (int p = 0; p < PS; ++p) e[p] = o[p] = eh[p] = oh[p] = R(0);
#pragma unroll
        for (int i = 0; i < PS + H - 1; ++i) {   // tile row p0 + i serves tap pair kk = p + H - 1 - i
            const R a = qa[i * G::PQ], d = qb[i * G::PQ];
#pragma unroll
            for (int p = 0; p < PS; ++p) {
                const int kk = p + H - 1 - i;
                if (kk >= 0 && kk < H) {
                    e[p] = fma(f.h(2 * kk), a, e[p]);
                    o[p] = fma(f.h(2 * kk + 1), a, o[p]);
                    eh[p] = fma(f.g(2 * kk), d, eh[p]);
                    oh[p] = fma(f.g(2 * kk + 1), d, oh[p]);
                }
            }
        }
        R *dst = (half ? th : tl) + 2 * p0 * G::PT + j;
#pragma unroll
        for (int p = 0; p < PS; ++p) {
            dst[2 * p * G::PT] = e[p] + eh[p];
            dst[(2 * p + 1) * G::PT] = o[p] + oh[p];
        }
    }
    __syncthreads();
    // axis 1: task (row, PS positions)
#pragma unroll
    for (int t = 0; t < NO; ++t) {
        const int task = threadIdx.x + t * NT, m = task % (2 * TS), p0 = (task / (2 * TS)) * PS;
        R a[PS + H - 1], d[PS + H - 1];
        load_row<piece<R>(PS)>(tl + m * G::PT + p0, a);
        load_row<piece<R>(PS)>(th + m * G::PT + p0, d);
        R high[2 * PS] = {};
#pragma unroll
        for (int i = 0; i < PS + H - 1; ++i)
#pragma unroll
            for (int p = 0; p < PS; ++p) {
                const int kk = p + H - 1 - i;
                if (kk >= 0 && kk < H) {
                    acc[t][2 * p] = fma(f.h(2 * kk), a[i], acc[t][2 * p]);
                    acc[t][2 * p + 1] = fma(f.h(2 * kk + 1), a[i], acc[t][2 * p + 1]);
                    high[2 * p] = fma(f.g(2 * kk), d[i], high[2 * p]);
                    high[2 * p + 1] = fma(f.g(2 * kk + 1), d[i], high[2 * p + 1]);
                }
            }
#pragma unroll
        for (int k = 0; k < 2 * PS; ++k) acc[t][k] += high[k];
    }
}

template <typename R, int TS, int NO>
__device__ __forceinline__ void syn_compute_b(int b, const R *q, R *tl, R *th, R (&acc)[NO][2 * SynGeo<TS>::PS]) {
    switch (b) {
        case 0: syn_compute<R, 2, TS, NO>(q, tl, th, acc); break;
        case 1: syn_compute<R, 4, TS, NO>(q, tl, th, acc); break;
        case 2: syn_compute<R, 6, TS, NO>(q, tl, th, acc); break;
        case 3: syn_compute<R, 8, TS, NO>(q, tl, th, acc); break;
        case 4: syn_compute<R, 10, TS, NO>(q, tl, th, acc); break;
        case 5: syn_compute<R, 12, TS, NO>(q, tl, th, acc); break;
        case 6: syn_compute<R, 14, TS, NO>(q, tl, th, acc); break;
        default: syn_compute<R, 16, TS, NO>(q, tl, th, acc); break;
    }
}
// output tasks per thread
template <int TS> constexpr int syn_tasks() { return 2 * TS * (TS / SynGeo<TS>::PS) / NT; }

// The finished output tile through shared memory (over the axis-0 results,
// at least 2TS rows of PW), so that the caller's put(row, column, value)
// writes whole rows: a thread's own outputs are a few samples of one row.
template <typename R, int TS, int NO, typename Put>
__device__ __forceinline__ void syn_emit(R *buf, const R (&acc)[NO][2 * SynGeo<TS>::PS], Put put) {
    using G = SynGeo<TS>;
    constexpr int PS = G::PS, PW = 2 * TS + 4;
    static_assert(2 * TS * PW <= G::HALVES, "output tile fits over the axis-0 results");
    __syncthreads();
#pragma unroll
    for (int t = 0; t < NO; ++t) {
        const int task = threadIdx.x + t * NT;
        store_row<piece<R>(2 * PS)>(buf + (task % (2 * TS)) * PW + 2 * PS * (task / (2 * TS)), acc[t]);
    }
    __syncthreads();
#pragma unroll
    for (int e = threadIdx.x; e < 4 * TS * TS; e += NT) put(e / (2 * TS), e % (2 * TS), buf[e / (2 * TS) * PW + e % (2 * TS)]);
}

// One synthesis level l > 0 for all 8 bases (grid.y: longest filter first):
// out_b (n0 x n1, compact pitch n1) = D_b^T of (LL' block, detail quadrants),
// coefficients times the prior weights when wgt is set.  LL' comes from the
// coefficients at the coarsest level (from_coef) or from the coarser level's
// output sll.
template <typename R, int TS>
__global__ void __launch_bounds__(NT) k_sara_syn(const R *__restrict__ coef, const R *__restrict__ wgt, int L1,
                                                 int64_t N, const R *__restrict__ sll, int from_coef,
                                                 int64_t sll_bstride, int n0, int n1, R *__restrict__ out,
                                                 int64_t out_bstride) {
    using G = SynGeo<TS>;
    constexpr int NO = syn_tasks<TS>(), PS = G::PS;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    R *q = reinterpret_cast<R *>(smem_raw), *tl = q + G::QUADS, *th = tl + G::HALVES / 2;
    const int b = N_WAVELETS - 1 - blockIdx.y;
    const int tpd1 = (n1 / 2 + TS - 1) / TS;
    const int R0 = (blockIdx.x / tpd1) * TS, C0 = (blockIdx.x % tpd1) * TS;
    pdl_enter();
    syn_load<R, TS>(q, coef + (int64_t)(b + 1) * N, wgt ? wgt + (int64_t)(b + 1) * N : nullptr,
                    sll + (int64_t)b * sll_bstride, from_coef, L1, n0 >> 1, n1 >> 1, R0, C0, 2 * b + 2);
    copy_wait<0>();
    __syncthreads();
    R acc[NO][2 * PS] = {};
    syn_compute_b<R, TS, NO>(b, q, tl, th, acc);
    syn_emit<R, TS, NO>(tl, acc, [&](int r, int c, R v) {
        if (2 * R0 + r < n0 && 2 * C0 + c < n1)
            out[(int64_t)b * out_bstride + (int64_t)(2 * R0 + r) * n1 + 2 * C0 + c] = v;
    });
}

// Finest synthesis level, the 8 wavelet bases summed in order per output
// sample: out = scale * (dirac + sum_b D_b^T (w_b c_b)) (dirac may be null).
// A cluster of 8 CTAs per output tile, one per basis: each leaves its samples
// in its shared memory, then sums an eighth of the tile's rows over the
// cluster.  One CTA working through the 8 bases took 8 rounds of copy,
// barrier and cold filter code (21 us at 512^2, 19 us at 256^2, 157 us at
// 2048^2 with these tiles; the cluster takes 10, 6 and 101).  What bounds it
// now is the longest filter of a cluster and its two cluster barriers.
__device__ __forceinline__ void cluster_sync() {
    asm volatile("barrier.cluster.arrive.release.aligned;\nbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
// value at p (this CTA's shared memory) in the CTA of rank r
__device__ __forceinline__ float peer_load(const float *p, int r) {
    float v;
    asm volatile("{\n\t.reg .u32 a;\n\tmapa.shared::cluster.u32 a, %1, %2;\n\tld.shared::cluster.f32 %0, [a];\n\t}"
                 : "=f"(v) : "r"(smem_u32(p)), "r"(r) : "memory");
    return v;
}
__device__ __forceinline__ double peer_load(const double *p, int r) {
    double v;
    asm volatile("{\n\t.reg .u32 a;\n\tmapa.shared::cluster.u32 a, %1, %2;\n\tld.shared::cluster.f64 %0, [a];\n\t}"
                 : "=d"(v) : "r"(smem_u32(p)), "r"(r) : "memory");
    return v;
}
template <typename R, int TS>
__global__ void __cluster_dims__(N_WAVELETS, 1, 1) __launch_bounds__(NT)
    k_sara_syn0(const R *__restrict__ coef, const R *__restrict__ wgt, int L0, int L1, int64_t N,
                const R *__restrict__ sll, int from_coef, int64_t sll_bstride, const R *__restrict__ dirac, R scale,
                R *__restrict__ out) {
    using G = SynGeo<TS>;
    constexpr int NO = syn_tasks<TS>(), PS = G::PS, PW = 2 * TS + 4, ROWS = 2 * TS / N_WAVELETS;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    R *q = reinterpret_cast<R *>(smem_raw), *tl = q + G::QUADS, *th = tl + G::HALVES / 2;
    const int b = blockIdx.x % N_WAVELETS, tile = blockIdx.x / N_WAVELETS;   // rank in the cluster = basis
    const int tpd1 = (L1 / 2 + TS - 1) / TS;
    const int R0 = (tile / tpd1) * TS, C0 = (tile % tpd1) * TS;
    pdl_enter();
    syn_load<R, TS>(q, coef + (int64_t)(b + 1) * N, wgt ? wgt + (int64_t)(b + 1) * N : nullptr,
                    sll + (int64_t)b * sll_bstride, from_coef, L1, L0 >> 1, L1 >> 1, R0, C0, 2 * b + 2);
    copy_wait<0>();
    __syncthreads();
    R acc[NO][2 * PS] = {};
    syn_compute_b<R, TS, NO>(b, q, tl, th, acc);
    // the basis's samples over the quadrant tiles (used up since axis 0)
#pragma unroll
    for (int t = 0; t < NO; ++t) {
        const int task = threadIdx.x + t * NT;
        store_row<piece<R>(2 * PS)>(q + (task % (2 * TS)) * PW + 2 * PS * (task / (2 * TS)), acc[t]);
    }
    cluster_sync();
    for (int e = threadIdx.x; e < ROWS * 2 * TS; e += NT) {
        const int r = b * ROWS + e / (2 * TS), c = e % (2 * TS);
        if (2 * R0 + r < L0 && 2 * C0 + c < L1) {
            const int64_t idx = (int64_t)(2 * R0 + r) * L1 + 2 * C0 + c;
            R v[N_WAVELETS], sum = 0;
#pragma unroll
            for (int k = 0; k < N_WAVELETS; ++k) v[k] = peer_load(q + r * PW + c, k);
#pragma unroll
            for (int k = 0; k < N_WAVELETS; ++k) sum += v[k];
            out[idx] = scale * ((dirac ? dirac[idx] : R(0)) + sum);
        }
    }
    cluster_sync();   // the peers have read this CTA's samples
}

// tiles of ts x ts quadrant positions covering an h0 x h1 quadrant
inline unsigned tiles(int h0, int h1, int ts) { return (unsigned)(((h0 + ts - 1) / ts) * ((h1 + ts - 1) / ts)); }

template <int V> struct Int {
    static constexpr int value = V;
};
// go(tile side) for a level with quadrants of h0 x h1: large tiles once they
// give every SM two CTAs of the eight bases (FP64 keeps the small ones: its
// two FP64 lanes per SM, not the halo, bound it).
template <typename R, typename Go> int with_tile(const ppd_ctx *c, int h0, int h1, Go go) {
    if constexpr (sizeof(R) == 4) {
        if (tiles(h0, h1, 32) * N_WAVELETS >= 2u * c->sms) return go(Int<32>{});
    }
    return go(Int<16>{});
}

// Analysis of all levels (tiled).  mode 0 writes c = D x / 3, mode 1
// clip-updates u with the prior weights and the clip level kappa ||Psi W||^2.
template <typename R> int analysis_all(ppd_ctx *c, const R *x, R *coef, int mode, cudaStream_t s) {
    const R *wgt = mode == 1 ? static_cast<const R *>(c->wgt) : nullptr;
    const uint8_t *pmask = (mode == 1 && c->rand_on) ? c->mask_cur + c->d : nullptr;
    const R alpha = (R)(c->kappa * c->psiw2);
    const int L0 = c->L0, L1 = c->L1;
    const int64_t N = c->N;
    const int64_t ll_stride = (int64_t)(L0 / 2) * (L1 / 2);
    R *ll[2] = {static_cast<R *>(c->wtmp), static_cast<R *>(c->wtmp) + (int64_t)N_WAVELETS * ll_stride};
    int site;
    for (int l = 0; l < c->levels; ++l) {
        const int n0 = L0 >> l, n1 = L1 >> l;
        const bool last = (l == c->levels - 1);
        const R *in = l == 0 ? x : ll[(l - 1) & 1];
        const int pitch = l == 0 ? L1 : n1;
        const int64_t bstride = l == 0 ? 0 : ll_stride;
        // level 0 starts its sequence (in the iteration: after the fork)
        auto go = [&](auto ts) {
            constexpr int TS = decltype(ts)::value;
            auto k = mode == 0 ? k_sara_ana<R, TS, 0> : wgt ? k_sara_ana<R, TS, 2> : k_sara_ana<R, TS, 1>;
            PPD_CHECK(smem_attr((const void *)k, (int)ana_smem<R, TS>()));
            PPD_CHECK(launch_begin(c, "sara_analysis", s, &site));
            launch(c, l > 0, k, dim3(tiles(n0 / 2, n1 / 2, TS), N_WAVELETS), NT, ana_smem<R, TS>(), s, in, pitch,
                   bstride, n0, n1, ll[l & 1], ll_stride, (int)last, coef, wgt, L1, N, alpha,
                   mode == 0 && l == 0 && x != coef ? coef : nullptr, pmask);
            return launch_end(c, site, s);
        };
        PPD_CHECK(with_tile<R>(c, n0 / 2, n1 / 2, go));
    }
    return PPD_OK;
}

// Synthesis of the 8 wavelet bases, levels coarsest .. 1 (tiled); returns
// the buffer holding the LL' block of level 0.
template <typename R>
int synthesis_levels(ppd_ctx *c, const R *coef, const R *wgt, const R **ll0, cudaStream_t s) {
    const int L0 = c->L0, L1 = c->L1;
    const int64_t N = c->N;
    const int64_t st = (int64_t)(L0 / 2) * (L1 / 2);
    R *buf[2] = {static_cast<R *>(c->wtmp2), static_cast<R *>(c->wtmp2) + (int64_t)N_WAVELETS * st};
    const R *prev = nullptr;
    int site, k = 0;
    for (int l = c->levels - 1; l >= 1; --l, ++k) {
        const int n0 = L0 >> l, n1 = L1 >> l;
        const bool coarsest = (l == c->levels - 1);
        auto go = [&](auto ts) {
            constexpr int TS = decltype(ts)::value;
            PPD_CHECK(smem_attr((const void *)k_sara_syn<R, TS>, (int)syn_smem<R, TS>()));
            PPD_CHECK(launch_begin(c, "sara_synthesis", s, &site));
            launch(c, true, k_sara_syn<R, TS>, dim3(tiles(n0 / 2, n1 / 2, TS), N_WAVELETS), NT, syn_smem<R, TS>(), s,
                   coef, wgt, L1, N, coarsest ? coef : prev, coarsest ? 1 : 0, st, n0, n1, buf[k & 1], st);
            return launch_end(c, site, s);
        };
        PPD_CHECK(with_tile<R>(c, n0 / 2, n1 / 2, go));
        prev = buf[k & 1];
    }
    *ll0 = prev;
    return PPD_OK;
}

template <typename R>
int synthesis_final(ppd_ctx *c, const R *coef, const R *wgt, const R *ll0, const R *dirac, R scale, R *out,
                    cudaStream_t s) {
    const int L0 = c->L0, L1 = c->L1;
    const int64_t st = (int64_t)(L0 / 2) * (L1 / 2);
    const bool from_coef = ll0 == nullptr;   // levels == 1: LL' straight from the coefficients
    int site;
    auto go = [&](auto ts) {
        constexpr int TS = decltype(ts)::value;
        PPD_CHECK(smem_attr((const void *)k_sara_syn0<R, TS>, (int)syn_smem<R, TS>()));
        PPD_CHECK(launch_begin(c, "sara_synthesis", s, &site));
        launch(c, true, k_sara_syn0<R, TS>, tiles(L0 / 2, L1 / 2, TS) * N_WAVELETS, NT, syn_smem<R, TS>(), s, coef, wgt,
               L0, L1, c->N, from_coef ? coef : ll0, from_coef ? 1 : 0, st, dirac, scale, out);
        return launch_end(c, site, s);
    };
    return with_tile<R>(c, L0 / 2, L1 / 2, go);
}

// Durand-Kerner roots of the polynomial with real coefficients a (ascending).
std::vector<std::complex<double>> poly_roots(const std::vector<double> &a) {
    using cd = std::complex<double>;
    const int n = (int)a.size() - 1;
    std::vector<cd> r(n);
    const cd seed(0.4, 0.9);
    for (int i = 0; i < n; ++i) r[i] = std::pow(seed, i);
    auto eval = [&](cd z) {
        cd s = 0;
        for (int k = n; k >= 0; --k) s = s * z + a[k];
        return s / a[n];
    };
    for (int it = 0; it < 2000; ++it) {
        double delta = 0;
        for (int i = 0; i < n; ++i) {
            cd den = 1;
            for (int j = 0; j < n; ++j)
                if (j != i) den *= (r[i] - r[j]);
            cd step = eval(r[i]) / den;
            r[i] -= step;
            delta = std::max(delta, std::abs(step));
        }
        if (delta < 1e-15) break;
    }
    // Newton polish on the original polynomial
    for (int i = 0; i < n; ++i) {
        for (int it = 0; it < 5; ++it) {
            cd p = 0, dp = 0;
            for (int k = n; k >= 0; --k) {
                dp = dp * r[i] + p;
                p = p * r[i] + a[k];
            }
            if (std::abs(dp) > 0) r[i] -= p / dp;
        }
    }
    return r;
}

}  // namespace

// db_p low-pass filter: |m0|^2 = cos^{2p} P(sin^2), P(y) = sum_{k<p} C(p-1+k,k) y^k;
// roots y of P -> z from sin^2(xi/2) = (2 - z - 1/z)/4 keeping |z| < 1;
// h = coefficients of (1+z)^p prod (z - z_r), scaled to sum sqrt(2), larger end first.
std::vector<double> daubechies(int p) {
    using cd = std::complex<double>;
    if (p == 1) return {1.0 / std::sqrt(2.0), 1.0 / std::sqrt(2.0)};
    std::vector<double> a(p);
    for (int k = 0; k < p; ++k) {
        double cb = 1.0;   // C(p-1+k, k)
        for (int i = 1; i <= k; ++i) cb = cb * (p - 1 + i) / i;
        a[k] = cb;
    }
    std::vector<cd> poly{1.0};
    auto mul = [&](cd c0, cd c1) {   // poly *= (c0 + c1 X) in coefficient-sequence form
        std::vector<cd> out(poly.size() + 1, 0.0);
        for (size_t i = 0; i < poly.size(); ++i) {
            out[i] += poly[i] * c0;
            out[i + 1] += poly[i] * c1;
        }
        poly.swap(out);
    };
    for (int i = 0; i < p; ++i) mul(1.0, 1.0);
    for (cd y : poly_roots(a)) {
        cd aa = 1.0 - 2.0 * y;
        cd disc = std::sqrt(aa * aa - 1.0);
        cd z1 = aa + disc, z2 = aa - disc;
        cd zr = std::abs(z1) < std::abs(z2) ? z1 : z2;
        mul(1.0, -zr);
    }
    std::vector<double> h(poly.size());
    double sum = 0;
    for (size_t i = 0; i < poly.size(); ++i) {
        h[i] = poly[i].real();
        sum += h[i];
    }
    for (double &v : h) v *= std::sqrt(2.0) / sum;
    if (std::abs(h.front()) < std::abs(h.back())) std::reverse(h.begin(), h.end());
    return h;
}

int make_filters(ppd_ctx *c) {
    (void)c;
    double hd[N_WAVELETS][MAX_TAPS] = {};
    float hf[N_WAVELETS][MAX_TAPS] = {};
    for (int b = 0; b < N_WAVELETS; ++b) {
        std::vector<double> h = daubechies(b + 1);
        for (size_t k = 0; k < h.size(); ++k) {
            hd[b][k] = h[k];
            hf[b][k] = (float)h[k];
        }
    }
    PPD_CUDA(cudaMemcpyToSymbol(c_filt_d, hd, sizeof(hd)));
    PPD_CUDA(cudaMemcpyToSymbol(c_filt_f, hf, sizeof(hf)));
    return PPD_OK;
}

template <typename R> int psi_analysis(ppd_ctx *c, const R *x, R *coef, cudaStream_t s) {
    PPD_CHECK(analysis_all<R>(c, x, coef, 0, s));
    // an image that lies in the Dirac part itself is scaled once every basis has read it
    return x == coef ? scale_copy<R>(c, x, coef, c->N, 1.0 / 3.0, s) : PPD_OK;
}

template <typename R> int psi_synthesis(ppd_ctx *c, const R *coef, R *x, cudaStream_t s) {
    const R *ll0 = nullptr;
    PPD_CHECK(synthesis_levels<R>(c, coef, nullptr, &ll0, s));
    return synthesis_final<R>(c, coef, nullptr, ll0, coef, R(1.0 / 3.0), x, s);
}

// Prior dual step of Algorithm 3 for the 8 wavelet bases up to the level-0
// synthesis: u_b <- clip(u_b + W_b Psi_b^dagger xt, alpha), then the synthesis
// of W_b u_b for levels coarsest .. 1.  Needs only xt and u, so it can run
// beside the data branch of the iteration.
template <typename R> int sara_prior_branch(ppd_ctx *c, const R **ll0, cudaStream_t s) {
    R *u = static_cast<R *>(c->u);
    PPD_CHECK(analysis_all<R>(c, static_cast<const R *>(c->xt), u, 1, s));
    return synthesis_levels<R>(c, u, static_cast<const R *>(c->wgt), ll0, s);
}

// Level-0 synthesis summed over the 8 wavelet bases: ut = sum_b D_b^T (W_b u_b)
// (the Dirac basis and the 1/3 are applied in the primal step).
template <typename R> int sara_level0(ppd_ctx *c, const R *ll0, cudaStream_t s) {
    return synthesis_final<R>(c, static_cast<const R *>(c->u), static_cast<const R *>(c->wgt), ll0, nullptr, R(1),
                              static_cast<R *>(c->ut), s);
}



template int psi_analysis<float>(ppd_ctx *, const float *, float *, cudaStream_t);
template int psi_analysis<double>(ppd_ctx *, const double *, double *, cudaStream_t);
template int psi_synthesis<float>(ppd_ctx *, const float *, float *, cudaStream_t);
template int psi_synthesis<double>(ppd_ctx *, const double *, double *, cudaStream_t);
template int sara_prior_branch<float>(ppd_ctx *, const float **, cudaStream_t);
template int sara_prior_branch<double>(ppd_ctx *, const double **, cudaStream_t);
template int sara_level0<float>(ppd_ctx *, const float *, cudaStream_t);
template int sara_level0<double>(ppd_ctx *, const double *, cudaStream_t);

}  // namespace ppd
