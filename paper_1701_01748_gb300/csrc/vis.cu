// Visibility-side kernels of PPD.
//
//  * binning (Section 2: G's 8 x 8 Kaiser-Bessel taps, Section 5: n = 4
//    oversampling; Section 4.3 / Section 5: sampling density per grid cell)
//  * degridding G with the data step of Algorithm 3 fused in (z = U^-1 v +
//    Theta G a, first forward-backward step of Algorithm 2, block norms)
//  * extra Algorithm 2 sub-iterations and the per-block l2-ball scale
//  * gridding G^dagger Theta^dagger v with the dual update fused in
//    (vbar = U (z - P_B(w))), accumulated per tile in shared memory and
//    summed across work items in a fixed order (deterministic, no atomics)
//
// Work decomposition: visibilities are sorted by (tile of the centred grid
// holding the first tap, block, base cell) and cut into groups of at most 32
// of one tile and block.  Degridding and sub-iterations share the groups out
// to warps; a degridding warp stages the (T+8) x (T+8) extended grid tile of
// its groups in shared memory (TMA for interior tiles, wrapped plain loads at
// the grid edge).  Gridding work items are sequences of groups of one tile; a
// warp or a CTA accumulates one into such a tile.
#include <cmath>
#include <limits>

#include "common.cuh"
#include "tma.cuh"

namespace ppd {

namespace {

template <typename C> __device__ __forceinline__ C cadd(C a, C b) { return C{a.x + b.x, a.y + b.y}; }

// ----------------------------------------------------------------- binning
// kappa = (omega * K) * (1/(2 pi)) with correctly rounded multiplies (no FMA
// contraction possible), f = floor(kappa), first tap (f - 3) mod K, fraction
// kappa - f, nearest cell floor(kappa + 0.5) mod K.
__global__ void k_bin(const double *__restrict__ uv, const int32_t *__restrict__ blk, int64_t M, int K0, int K1,
                      int T, int d, uint64_t *__restrict__ key, int32_t *__restrict__ base,
                      double *__restrict__ frac, int32_t *__restrict__ cell, int32_t *__restrict__ count_grid,
                      int *__restrict__ bad) {
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < M; i += (int64_t)gridDim.x * blockDim.x) {
        const double om0 = uv[2 * i], om1 = uv[2 * i + 1];
        const int b = blk[i];
        if (!(om0 >= -M_PI && om0 <= M_PI && om1 >= -M_PI && om1 <= M_PI) || b < 0 || b >= d) {
            atomicOr(bad, 1);
            key[i] = 0;
            base[2 * i] = base[2 * i + 1] = 0;
            frac[2 * i] = frac[2 * i + 1] = 0.0;
            cell[i] = 0;   // a valid cell for k_cell_count; the call fails on `bad`
            continue;
        }
        const double k0 = __dmul_rn(__dmul_rn(om0, (double)K0), INV_TWO_PI);
        const double k1 = __dmul_rn(__dmul_rn(om1, (double)K1), INV_TWO_PI);
        const double f0 = floor(k0), f1 = floor(k1);
        const int64_t i0 = (int64_t)f0, i1 = (int64_t)f1;
        const int b0 = (int)(((i0 - 3) % K0 + K0) % K0);
        const int b1 = (int)(((i1 - 3) % K1 + K1) % K1);
        const int cb0 = (b0 + K0 / 2) % K0, cb1 = (b1 + K1 / 2) % K1;
        const int64_t n0 = (((int64_t)floor(__dadd_rn(k0, 0.5))) % K0 + K0) % K0;
        const int64_t n1 = (((int64_t)floor(__dadd_rn(k1, 0.5))) % K1 + K1) % K1;
        const uint64_t tile = (uint64_t)(cb0 / T) * (uint64_t)(K1 / T) + (uint64_t)(cb1 / T);
        key[i] = ((tile * (uint64_t)d + (uint64_t)b) * (uint64_t)K0 + (uint64_t)cb0) * (uint64_t)K1 + (uint64_t)cb1;
        base[2 * i] = b0;
        base[2 * i + 1] = b1;
        frac[2 * i] = __dsub_rn(k0, f0);
        frac[2 * i + 1] = __dsub_rn(k1, f1);
        const int c = (int)(n0 * K1 + n1);
        cell[i] = c;
        atomicAdd(&count_grid[c], 1);
    }
}

__global__ void k_cell_count(const int32_t *__restrict__ cell, const int32_t *__restrict__ count_grid, int64_t M,
                             int32_t *__restrict__ out) {
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < M; i += (int64_t)gridDim.x * blockDim.x)
        out[i] = count_grid[cell[i]];
}

// ----------------------------------------------------------------- weights
// Tap j = 0..3 has the weight psi(frac + 3 - j) as a polynomial in t = 2 frac
// - 1, fitted on the host (make_kb_poly) and evaluated as even + t odd part in
// t^2; psi is even, so tap 7 - j is the mirror image even - t odd and the pair
// costs one evaluation (FP32: 32 FMAs an axis instead of 56 for eight Horner
// chains).  The coefficients p[j KB_N + k] of t^k are kernel arguments, so
// with the loops unrolled each is a constant-bank operand: no load.
//
// FP32: 8 coefficients, fit error 4e-8 at most, 1.5e-8 rms.  The constant
// term of the two inner taps (weights up to 1) keeps the part that rounding
// it to FP32 drops (kbl), and is added last: every visibility sees the same
// coefficients, so without it the whole operator's amplitude was 4e-8 low
// (and the weights 2.2e-8 rms off, where eight Horner chains had 2.0e-8; with
// it 1.85e-8, 9.5e-8 at most).  It costs 8 adds a visibility.
// FP64: 16 coefficients reach 2.2e-16 at most, 4e-17 rms for the default
// shape beta = 2.34 J, closer than the Bessel function itself, whose 16
// evaluations a visibility were most of the FP64 visibility kernels' time on
// two FP64 lanes per SM.  A shape the 16 coefficients do not resolve (checked
// on the host) keeps the Bessel function (bessel).
template <typename R> constexpr int KB_N = sizeof(R) == 4 ? 8 : 16;
__device__ __noinline__ double kb_bessel(double frac, int j, double beta, double inv_i0b) {
    const double d = (frac + (double)(3 - j)) * 0.25, x = 1.0 - d * d;
    return x >= 0.0 ? cyl_bessel_i0(beta * sqrt(x)) * inv_i0b : 0.0;
}
template <typename R, typename A> __device__ __forceinline__ void kb_weights(R frac, R (&w)[KB_J], const A &args) {
    constexpr int N = KB_N<R>;
    if constexpr (sizeof(R) == 8) {
        if (args.bessel) {
#pragma unroll
            for (int j = 0; j < KB_J; ++j) w[j] = kb_bessel(frac, j, args.beta, args.inv_i0b);
            return;
        }
    }
    const R t = fma(R(2), frac, R(-1)), s = t * t;
#pragma unroll
    for (int j = 0; j < KB_J / 2; ++j) {
        const bool split = sizeof(R) == 4 && j >= KB_J / 4;   // constant term in two parts
        R e = args.kbp[j * N + N - 2], o = args.kbp[j * N + N - 1];
#pragma unroll
        for (int k = N - 4; k >= 0; k -= 2) {
            e = fma(e, s, split && k == 0 ? args.kbl[j - KB_J / 4] : args.kbp[j * N + k]);
            o = fma(o, s, args.kbp[j * N + k + 1]);
        }
        w[j] = fma(o, t, e);
        w[KB_J - 1 - j] = fma(-o, t, e);
        if (split) {
            w[j] += args.kbp[j * N];
            w[KB_J - 1 - j] += args.kbp[j * N];
        }
    }
}

template <typename R> struct VisArgs {
    const VisRec<R> *rec;
    const R *theta_v;
    R theta_s;
    // gridding work items (sequences of groups of one tile): item k owns the
    // it_grp[k].y groups of gg (groups in the processing order) from
    // it_grp[k].x on; it_order: the items by decreasing size
    const int4 *gg;
    const int2 *it_grp;
    const int32_t *it_order;
    // groups of at most 32 visibilities of one tile and block {start, count,
    // tile, block}: warp w of the degridding and sub-iteration kernels owns
    // groups warp_grp[w] .. warp_grp[w + 1] - 1; its maximal sequences of
    // groups of one block are runs warp_run[w] .. warp_run[w + 1] - 1
    const int4 *grp;
    const int32_t *warp_grp, *warp_run;
    int n_warps;
    int K0, K1, ntile1;
    R kbp[KB_J / 2 * KB_N<R>];   // the weight polynomials (kb_weights)
    R kbl[KB_J / 4];             // FP32: what rounding dropped of the inner taps' constant terms
    int bessel;                  // FP64: the weights come from the Bessel function
    double beta, inv_i0b;
    const cplx_t<R> *y;
    cplx_t<R> *v, *z, *w, *p;
    const R *mu;
    const R *scale;              // per block: the P_B scale of the last step (k_block_scale)
    double *partials;            // norm partials of the runs
    // partials live in block-major slots: run r writes slot run_pos[r]
    const int32_t *run_pos;
    int *err;
    // randomised active sets (null: every block active): the current
    // iteration's block flags, per-block "has a prox output" flags, and the
    // flag that makes the gridding redo the partial tiles of inactive blocks
    const uint8_t *bmask;
    uint8_t *seen;
    const int *regrid;
    // operator mode I/O (caller order through perm when non-null)
    const cplx_t<R> *op_in;
    cplx_t<R> *op_out;
    const int64_t *perm;
    // Algorithm 2 stopping test (inner_tol > 0): this launch's step number
    // (0: the step that forms the start P_B(z); 1 .. n_itr - 1: sub-iterations;
    // n_itr: the gridding), per block the step at which the test held (0:
    // running) and the steps taken
    int tol_on, step, n_itr;
    int *inner_state, *inner_steps;
};

// Kahan-compensated FP32 accumulator of one lane (FP64 accumulation in the FP64
// path).  Only FP64 sums leave it: the sum over the lanes and over runs has
// FP64's precision and range.  A lane whose sum is big() hands it on before
// the next group, so that adding another finite square (at most 2^128, and
// 2^100 is below half its last place) cannot overflow.
template <typename R> struct Acc {
    R s = 0, c = 0;
    __device__ void add(R x) {
        R y = x - c;
        R t = s + y;
        c = (t - s) - y;
        s = t;
    }
    __device__ double get() const { return (double)s - (double)c; }
    __device__ bool big() const { return sizeof(R) == 4 && s > R(0x1p100); }
};

// Warp sums of NV <= 4 values per lane (FP64, fixed order).  The first shuffle
// steps also halve the number of values a lane carries (lanes whose bit is
// set take the upper half), so that NV = 2 costs 5 adds a lane instead of
// 10.  Lane k * warp_sum_step(NV) returns the sum of value k.
__host__ __device__ constexpr int warp_sum_step(int nv) { return nv <= 1 ? 32 : nv <= 2 ? 16 : 8; }
template <int NV> __device__ __forceinline__ double warp_sums(const double (&in)[NV]) {
    constexpr int NP = 32 / warp_sum_step(NV);
    const int lane = threadIdx.x & 31;
    double v[NP];
#pragma unroll
    for (int k = 0; k < NP; ++k) v[k] = k < NV ? in[k < NV ? k : 0] : 0.0;
    auto from = [](double a, int m) { return __shfl_xor_sync(0xffffffffu, a, m); };
    int m = 16;
    if constexpr (NP == 4) {
        const bool hi = lane & m;
#pragma unroll
        for (int k = 0; k < 2; ++k) v[k] = (hi ? v[k + 2] : v[k]) + from(hi ? v[k] : v[k + 2], m);
        m >>= 1;
    }
    if constexpr (NP >= 2) {
        const bool hi = lane & m;
        v[0] = (hi ? v[1] : v[0]) + from(hi ? v[0] : v[1], m);
        m >>= 1;
    }
    for (; m > 0; m >>= 1) v[0] += from(v[0], m);
    return v[0];
}

// a w + c on both components: one instruction on packed pairs in FP32 (the
// same two roundings as two fmaf), half the issue slots of the taps' sums
struct F32x2 {
    unsigned long long v = 0;
};
__device__ __forceinline__ F32x2 pack2(float x, float y) {
    F32x2 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r.v) : "f"(x), "f"(y));
    return r;
}
__device__ __forceinline__ float2 unpack2(F32x2 a) {
    float2 r;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(a.v));
    return r;
}
__device__ __forceinline__ F32x2 fma2(F32x2 a, F32x2 b, F32x2 c) {
    F32x2 r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r.v) : "l"(a.v), "l"(b.v), "l"(c.v));
    return r;
}

// sum_ab w0[a] w1[b] tile[a][b] over an 8 x 8 footprint, row by row
template <int E> __device__ __forceinline__ float2 footprint(const float2 *cell, const float (&w0)[KB_J], const float (&w1)[KB_J]) {
    F32x2 d1[KB_J], q = pack2(0.f, 0.f);
#pragma unroll
    for (int b = 0; b < KB_J; ++b) d1[b] = pack2(w1[b], w1[b]);
#pragma unroll
    for (int a = 0; a < KB_J; ++a) {
        const F32x2 *row = reinterpret_cast<const F32x2 *>(cell + a * E);
        F32x2 r = pack2(0.f, 0.f);
#pragma unroll
        for (int b = 0; b < KB_J; ++b) r = fma2(d1[b], row[b], r);
        q = fma2(pack2(w0[a], w0[a]), r, q);
    }
    return unpack2(q);
}
template <int E> __device__ __forceinline__ double2 footprint(const double2 *cell, const double (&w0)[KB_J], const double (&w1)[KB_J]) {
    double2 q{0, 0};
#pragma unroll
    for (int a = 0; a < KB_J; ++a) {
        const double2 *row = cell + a * E;
        double2 r{0, 0};
#pragma unroll
        for (int b = 0; b < KB_J; ++b) {
            const double2 g = row[b];
            r.x += w1[b] * g.x;
            r.y += w1[b] * g.y;
        }
        q.x += w0[a] * r.x;
        q.y += w0[a] * r.y;
    }
    return q;
}

// ----------------------------------------------------------------- degrid
// mode DG_OP:    op_out[perm[i]] = Theta G a
// mode DG_DUAL:  z = v/U + Theta G a;  w = p - mu U (p - z)
// mode DG_FIRST: z = v/U + Theta G a;  w = z   (Algorithm 2 then starts from P_B(z))
// partials of a run = (||w - y||^2, ||Theta G a - y||^2)
//
// A warp works alone: it owns an equal share of the groups of 32
// visibilities (a lane each; a few pieces spread over the order) and a pair of (T+8)^2 grid tiles in shared
// memory, the one its current groups read and the one TMA fetches for the
// next tile of its share (interior tiles; tiles that wrap around the grid
// edge are loaded with plain loads when they are used).  The next group's
// visibilities are loaded while the current one is computed.  Norms
// accumulate per lane over a run and are summed once at its end.  No CTA
// barrier separates the groups: with a CTA per work item (a tile's
// visibilities of one block) and its barriers, warps waited at barriers for
// 5 of every 14 cycles per issued instruction and small items left most
// lanes idle.  Before -> now, with the dual step: 28.4 -> 17.9 us at 512^2
// (524k visibilities), 159 -> 97 us at 1024^2 (4.2M), 42 -> 23 us at 640 x 480
// (700k); without it 522 -> 223 us at 4096^2 (8.4M).  What bounds it now is
// the shared-memory reads (64 eight-byte reads a visibility, two passes each
// for a warp: 51 % of the SM's data path at 1024^2, 70 % at 4096^2 without the
// dual step) and the issue slots (61 and 46 % busy).
template <typename R> struct VisIn {
    VisRec<R> rc;
    cplx_t<R> v, y, p;
    R th;
};

template <typename R, int MODE>
__device__ __forceinline__ void load_vis(const VisArgs<R> &A, int gi, VisIn<R> &o) {
    o.rc = A.rec[gi];
    o.th = A.theta_v ? A.theta_v[gi] : A.theta_s;
    if (MODE != DG_OP) {
        o.v = A.v[gi];
        o.y = A.y[gi];
        if (MODE == DG_DUAL) o.p = A.p[gi];
    }
}

// Warps per SM the degridding's shared memory and registers allow, and with
// them the shares of the groups (a share per resident warp).  T = 32: one
// tile buffer a warp (the copy is then waited for, with four times the
// visibilities behind each): 125 us with CTA work items and two buffers, 89 with
// one a warp at 1024^2; 27 and 22 at 512^2.
template <typename R, int T> constexpr int dg_warps_per_sm() { return sizeof(R) == 8 ? 8 : T == 16 ? 24 : 16; }
template <int T> constexpr int dg_bufs() { return T == 16 ? 2 : 1; }

// NTD threads per CTA (256 or 128; FP64: 256): the CTA only groups warps.  Which
// is faster follows no rule: an iteration takes 322 us with 256 and 324 with 128
// at 1024^2, 91.1 and 91.0 at 512^2, 60.8 and 62.4 at 256^2, 46.3 and 44.8 at
// 128^2 (8 gridding warps, 4 at 1024^2), and on other coverages the other way.
template <typename R, int T, int MODE, int NTD>
__global__ void __launch_bounds__(NTD, dg_warps_per_sm<R, T>() * 32 / NTD)
    k_degrid(const __grid_constant__ CUtensorMap tmap, int use_tma, const cplx_t<R> *__restrict__ grid, VisArgs<R> A,
             long long spin_first) {
    using C = cplx_t<R>;
    constexpr int E = T + HALO, NB = dg_bufs<T>();
    constexpr int TILE_BYTES = E * E * (int)sizeof(C);
    static_assert(TILE_BYTES % 128 == 0, "TMA destinations stay 128-byte aligned");
    extern __shared__ __align__(128) unsigned char smem_raw[];
    __shared__ uint64_t bars[NTD / 32][NB];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    unsigned char *tiles = smem_raw + warp * NB * TILE_BYTES;
    uint64_t *bar = bars[warp];
    const int gw = blockIdx.x * (NTD / 32) + warp;   // this warp's share
    if (lane == 0)
        for (int k = 0; k < NB; ++k) mbar_init(&bar[k], 1);
    __syncwarp();
    pdl_enter();   // the grid, v and p come from the kernels before
    auto interior = [&](int tile) {
        return use_tma && (tile / A.ntile1) * T + E <= A.K0 && (tile % A.ntile1) * T + E <= A.K1;
    };
    auto issue = [&](int tile, int buf) {   // lane 0 only
        if (interior(tile)) {
            mbar_expect_tx(&bar[buf], (uint32_t)TILE_BYTES);
            tma_load_2d(tiles + buf * TILE_BYTES, &tmap, 2 * (tile % A.ntile1) * T, (tile / A.ntile1) * T, &bar[buf]);
        }
    };
    const int g0 = gw < A.n_warps ? A.warp_grp[gw] : 0, g1 = gw < A.n_warps ? A.warp_grp[gw + 1] : 0;
    if (g0 < g1) {
        uint32_t ph = 0u;   // bit b: parity of the next completion of bar[b]
        int4 D = A.grp[g0], Dn = D;   // {start, count, tile, block} of this group and the next
        if (lane == 0) issue(D.z, 0);
        VisIn<R> cur;
        if (lane < D.y) load_vis<R, MODE>(A, D.x + lane, cur);
        if (g0 + 1 < g1) Dn = A.grp[g0 + 1];
        int buf = 0, run = A.warp_run[gw];
        bool fresh = true;    // the group's tile has not been waited for
        bool begin = true;    // the group starts a run
        bool handed = false;  // the run's slot holds sums of its earlier groups
        bool act = true, first_blk = MODE == DG_FIRST, keep_start = false;
        R mu = 0;
        Acc<R> s_w, s_r;
        for (int g = g0; g < g1; ++g) {
            const bool more = g + 1 < g1, next_tile = more && Dn.z != D.z;
            if (NB == 2 && next_tile && lane == 0) issue(Dn.z, buf ^ 1);
            VisIn<R> nx;
            if (more && lane < Dn.y) load_vis<R, MODE>(A, Dn.x + lane, nx);
            const int4 Dn2 = g + 2 < g1 ? A.grp[g + 2] : Dn;
            if (MODE != DG_OP && begin) {
                const int blk = D.w;
                mu = A.mu[blk];
                // block outside the active set D: z, w untouched (only the
                // residual statistic is formed); block without a prox output
                // yet: w = z, so that the next Algorithm 2 step starts from P_B(z)
                act = !A.bmask || A.bmask[blk];
                first_blk = MODE == DG_FIRST || (A.seen && !A.seen[blk]);
                // with the stopping test the start zbar^(0) = z of a block without
                // a prox output is kept in p, the previous point of the first test
                keep_start = first_blk && A.tol_on;
                if (lane == 0) {
                    if (A.tol_on) A.inner_state[blk] = 0;
                    if (A.inner_steps) A.inner_steps[blk] = act ? A.n_itr : 0;
                }
                begin = false;
            }
            C *tile = reinterpret_cast<C *>(tiles + buf * TILE_BYTES);
            const int row0 = (D.z / A.ntile1) * T, col0 = (D.z % A.ntile1) * T;
            if (fresh) {
                if (interior(D.z)) {
                    // spin_first bounds the first wait (SPIN_LIMIT unless a test shortens
                    // it); the waits for copies in flight before leaving keep SPIN_LIMIT
                    const bool ok = mbar_wait(&bar[buf], (ph >> buf) & 1u, spin_first);
                    if (!__all_sync(0xffffffffu, ok)) {
                        if (lane == 0) atomicOr(A.err, ERR_TMA_TIMEOUT);
                        mbar_wait(&bar[buf], (ph >> buf) & 1u, SPIN_LIMIT);
                        if (NB == 2 && next_tile && interior(Dn.z))
                            mbar_wait(&bar[buf ^ 1], (ph >> (buf ^ 1)) & 1u, SPIN_LIMIT);
                        break;
                    }
                    ph ^= 1u << buf;
                } else {
                    for (int e = lane; e < E * E; e += 32) {
                        const int r = e / E, cc = e % E;
                        tile[e] = grid[(int64_t)((row0 + r) % A.K0) * A.K1 + (col0 + cc) % A.K1];
                    }
                    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");   // a later copy refills the buffer
                    __syncwarp();
                }
                fresh = false;
            }
            if (lane < D.y) {
                const int gi = D.x + lane;
                const int lb0 = (cur.rc.packed & 0xffff) - row0, lb1 = ((cur.rc.packed >> 16) & 0xffff) - col0;
                R w0[KB_J], w1[KB_J];
                kb_weights(cur.rc.f0, w0, A);
                kb_weights(cur.rc.f1, w1, A);
                const C q = footprint<E>(tile + lb0 * E + lb1, w0, w1);
                const C phix{cur.th * q.x, cur.th * q.y};
                if (MODE == DG_OP) {
                    A.op_out[A.perm ? A.perm[gi] : gi] = phix;
                } else {
                    if (act) {
                        const R invU = R(1) / cur.rc.U;
                        const C zz{cur.v.x * invU + phix.x, cur.v.y * invU + phix.y};
                        A.z[gi] = zz;
                        C ww;
                        if (first_blk) {
                            ww = zz;
                            if (keep_start) A.p[gi] = zz;
                        } else {
                            const R mu_u = mu * cur.rc.U;
                            ww = C{cur.p.x - mu_u * (cur.p.x - zz.x), cur.p.y - mu_u * (cur.p.y - zz.y)};
                        }
                        A.w[gi] = ww;
                        const R dx = ww.x - cur.y.x, dy = ww.y - cur.y.y;
                        s_w.add(dx * dx + dy * dy);
                    }
                    const R ex = phix.x - cur.y.x, ey = phix.y - cur.y.y;
                    s_r.add(ex * ex + ey * ey);
                }
            }
            if (MODE != DG_OP) {
                const bool end = !more || Dn.w != D.w;   // the run ends
                if (end || __any_sync(0xffffffffu, s_w.big() || s_r.big())) {
                    const double part[2] = {s_w.get(), s_r.get()};
                    const double t = warp_sums<2>(part);
                    if (lane % 16 == 0) {
                        double *slot = A.partials + NPART * (int64_t)A.run_pos[run] + lane / 16;
                        *slot = handed ? *slot + t : t;
                    }
                    s_w = Acc<R>{};
                    s_r = Acc<R>{};
                    run += end;
                    begin = end;
                    handed = !end;
                }
            }
            if (next_tile) {
                __syncwarp();   // every lane has read the tile: its buffer may be refilled
                if (NB == 2) buf ^= 1;
                else if (lane == 0) issue(Dn.z, 0);
                fresh = true;
            }
            D = Dn;
            Dn = Dn2;
            cur = nx;
        }
    }
}

// ----------------------------------------------------------------- sub-iteration
// Algorithm 2 step with the block scale c of the previous step:
//   p = P_B(w) = y + c (w - y);  w = q - mu U (q - z);  partial ||w - y||^2
// with q = p (Algorithm 2) or, for the accelerated form, the extrapolated
// point q = p + beta (p - p_prev), p_prev read from and p written to the
// warm-start array (beta = 0: p_prev is not read; write_p = 0: p not written).
// only_first: the extra step that moves the start of a block with no prox
// output yet from z to P_B(z) (randomised active sets); groups of other
// blocks, and of blocks outside D, leave their scale as it is.
// Stopping test (inner_tol > 0): p is kept every step; a step k >= 1 also
// forms the partials ||p - p_prev||^2 and ||p||^2; a block whose test held
// for the previous step (or earlier) stops, its p being the prox output.
// The work is split as in the degridding (a warp per share of the groups).
// Groups of a block that a step leaves alone are passed over without a load of
// their data: a launch with every block skipped takes 16 us at 1024^2 (4.2M
// visibilities, 64 blocks; 45 with the loads), a working one 51.
constexpr int SUB_NT = 256;
template <typename R>
__global__ void __launch_bounds__(SUB_NT) k_subiter(VisArgs<R> A, int only_first, R beta, int write_p) {
    using C = cplx_t<R>;
    const int lane = threadIdx.x & 31, gw = blockIdx.x * (SUB_NT / 32) + (threadIdx.x >> 5);
    pdl_enter();
    const bool tol_on = A.tol_on;
    // blocks this step leaves as they are: outside D, not first in an
    // only_first step, or stopped at an earlier step of this iteration
    auto skips = [&](int blk) {
        return (A.bmask && !A.bmask[blk]) || (only_first && !(A.seen && !A.seen[blk])) ||
               (tol_on && A.inner_state[blk]);
    };
    const bool test_out = tol_on && A.step > 0;
    const bool keep = write_p || tol_on, prev = beta != R(0) || test_out;
    const int g0 = gw < A.n_warps ? A.warp_grp[gw] : 0, g1 = gw < A.n_warps ? A.warp_grp[gw + 1] : 0;
    struct In {
        R U;
        C y, w, z, p;
    };
    auto load = [&](int gi, In &o) {
        o.U = A.rec[gi].U;
        o.y = A.y[gi];
        o.w = A.w[gi];
        o.z = A.z[gi];
        if (prev) o.p = A.p[gi];
    };
    if (g0 < g1) {
        int run = A.warp_run[gw];
        int4 D = A.grp[g0], Dn = g0 + 1 < g1 ? A.grp[g0 + 1] : D;   // this group and the next
        In cur;
        bool skip = skips(D.w);   // (looked at before the loads: a block left alone costs none)
        if (!skip && lane < D.y) load(D.x + lane, cur);
        bool begin = true, handed = false;   // handed: as in the degridding
        R c = 0, mu = 0;
        Acc<R> s_w, s_d, s_n;
        for (int g = g0; g < g1; ++g) {
            const bool more = g + 1 < g1;
            const int4 Dn2 = g + 2 < g1 ? A.grp[g + 2] : Dn;
            const bool skip_n = Dn.w == D.w ? skip : skips(Dn.w);
            In nx;
            if (more && !skip_n && lane < Dn.y) load(Dn.x + lane, nx);
            if (begin) {
                c = A.scale[D.w];
                mu = A.mu[D.w];
                begin = false;
            }
            if (!skip && lane < D.y) {
                const int gi = D.x + lane;
                const C yy = cur.y, ww = cur.w, zz = cur.z;
                const C pp{yy.x + c * (ww.x - yy.x), yy.y + c * (ww.y - yy.y)};
                C q = pp;
                if (prev) {
                    const C pm = cur.p;
                    if (beta != R(0)) q = C{pp.x + beta * (pp.x - pm.x), pp.y + beta * (pp.y - pm.y)};
                    if (test_out) {
                        const R ex = pp.x - pm.x, ey = pp.y - pm.y;
                        s_d.add(ex * ex + ey * ey);
                        s_n.add(pp.x * pp.x + pp.y * pp.y);
                    }
                }
                if (keep) A.p[gi] = pp;
                const R mu_u = mu * cur.U;
                const C wn{q.x - mu_u * (q.x - zz.x), q.y - mu_u * (q.y - zz.y)};
                A.w[gi] = wn;
                const R dx = wn.x - yy.x, dy = wn.y - yy.y;
                s_w.add(dx * dx + dy * dy);
            }
            const bool end = !more || Dn.w != D.w;   // the run ends
            if (end || __any_sync(0xffffffffu, s_w.big() || s_d.big() || s_n.big())) {
                if (!skip) {
                    double *slot = A.partials + NPART * (int64_t)A.run_pos[run];
                    // (a warp's FP64 add holds the pipe of the SM's two lanes for 16
                    // cycles: only the sums that are read are formed)
                    if (test_out) {
                        const double part[3] = {s_w.get(), s_d.get(), s_n.get()};
                        const double t = warp_sums<3>(part);
                        // slot 1 keeps the degridding's residual
                        slot += lane ? lane / 8 + 1 : 0;
                        if (lane % 8 == 0 && lane < 24) *slot = handed ? *slot + t : t;
                    } else {
                        const double part[1] = {s_w.get()}, t = warp_sums<1>(part);
                        if (lane == 0) *slot = handed ? *slot + t : t;
                    }
                }
                s_w = s_d = s_n = Acc<R>{};
                run += end;
                begin = end;
                handed = !end;
            }
            D = Dn;
            Dn = Dn2;
            cur = nx;
            skip = skip_n;
        }
    }
}

// ----------------------------------------------------------------- block norms
// P_B scale of every block after the degridding or a sub-iteration (Section
// 3.3, Eq. "proj-L2" as a radial scale): eps / ||w - y|| if that norm exceeds
// eps, else 1, from the block's norm partials summed in FP64 in a fixed
// order, a CTA per block.  After a sub-iteration with the stopping test
// (step > 0): ||zbar^t - zbar^(t-1)|| <= inner_tol ||zbar^t|| in FP64; a block
// whose test holds is marked stopped at this step, its last (a block that stopped
// before, or that the step left alone, keeps what it has: its partials are
// those of its last step).
// A launch of its own: in the prologue of every CTA of the next kernel the
// sums took 19 of the gridding's 46 us at 512^2 with 16 blocks and 45 of a
// sub-iteration's 61 us (640 x 480, 12 blocks), their FP64 adds queueing for
// the SM's two FP64 lanes; in the CTA that counted a block's last run, the
// last CTA found most blocks at once (7 us after the others at 512^2, 35 us
// at 1024^2 with 64 blocks).
constexpr int BS_NT = 256;
template <typename R>
__global__ void __launch_bounds__(BS_NT) k_block_scale(const double *__restrict__ partials,
                                                       const int32_t *__restrict__ blk_ptr,
                                                       const double *__restrict__ eps, double inner_tol, int step,
                                                       R *__restrict__ scale, int *__restrict__ inner_state,
                                                       int *__restrict__ inner_steps, int *__restrict__ err) {
    __shared__ double red[BS_NT / 32][3];
    const int blk = blockIdx.x, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    pdl_enter();
    const int k0 = blk_ptr[blk], k1 = blk_ptr[blk + 1];
    const bool test = inner_tol > 0 && step > 0;
    double v[3] = {0, 0, 0};
#pragma unroll 8
    for (int k = k0 + threadIdx.x; k < k1; k += BS_NT) v[0] += partials[NPART * (int64_t)k];
    if (test)
#pragma unroll 4
        for (int k = k0 + threadIdx.x; k < k1; k += BS_NT) {
            v[1] += partials[NPART * (int64_t)k + 2];
            v[2] += partials[NPART * (int64_t)k + 3];
        }
    const int nw = min(BS_NT / 32, (k1 - k0 + 31) / 32);   // warps with a partial
    if (warp < nw) {
        if (test) {
            const double t = warp_sums<3>(v);
            if (lane % 8 == 0 && lane < 24) red[warp][lane / 8] = t;
        } else {
            const double u[1] = {v[0]}, t = warp_sums<1>(u);
            if (lane == 0) red[warp][0] = t;
        }
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        double a = 0, d = 0, n = 0;
        for (int w = 0; w < nw; ++w) a += red[w][0];
        if (test)
            for (int w = 0; w < nw; ++w) {
                d += red[w][1];
                n += red[w][2];
            }
        const double nrm = sqrt(a);
        if (!isfinite(nrm)) atomicOr(err, ERR_NONFINITE);
        scale[blk] = (R)((nrm > eps[blk]) ? eps[blk] / nrm : 1.0);
        if (test && inner_state[blk] == 0 && inner_steps[blk] != 0 && sqrt(d) <= inner_tol * sqrt(n))
            inner_state[blk] = inner_steps[blk] = step;
    }
}

// One warp per block j: ||Phi_j xt - y_j||^2 of the last data step from the
// block's partials (fixed order), for the statistics and the stopping rule.
__global__ void k_block_norms(const double *__restrict__ partials, const int32_t *__restrict__ blk_ptr, int d,
                              double *__restrict__ resid2, int *__restrict__ err) {
    const int j = blockIdx.x * (blockDim.x / 32) + (threadIdx.x >> 5);
    const int lane = threadIdx.x & 31;
    if (j >= d) return;
    double a = 0, b = 0;
    for (int k = blk_ptr[j] + lane; k < blk_ptr[j + 1]; k += 32) {
        a += partials[NPART * (int64_t)k];
        b += partials[NPART * (int64_t)k + 1];
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        a += __shfl_down_sync(0xffffffffu, a, o);
        b += __shfl_down_sync(0xffffffffu, b, o);
    }
    if (lane == 0) {
        if (!isfinite(sqrt(a))) atomicOr(err, ERR_NONFINITE);
        resid2[j] = b;
    }
}

// ----------------------------------------------------------------- gridding
// A work item is a sequence of groups (up to 32 visibilities of one block) of
// one tile; a warp or the NW warps of a CTA add its footprints into a private
// (T+8)^2 tile per warp, and the sum of the private tiles is the item's
// partial tile.  Per group: each lane stages one visibility (dual update,
// Theta v, the 8 products w0[a] Theta v and the 8 weights w1[b]) in the warp's
// staging area, then the warp adds the footprints one after the other, each
// lane accumulating two cells in registers (columns b and b + 4 of row a =
// lane / 4: 16 staged bytes a lane and visibility, 20 with two rows of a
// column) and adding them to the tile when the base cell changes (the order
// keeps visibilities of one cell together).  GR_DUAL fuses the end of the data step: p = P_B(w) = y + c (w - y), v = U (z - p).
//
// Items of up to `small` groups take one warp, NW of them share a CTA that
// has no CTA barrier; larger ones are spread over the warps of a CTA.  An
// item of one block and a CTA per item left most warps idle (4096^2, 8.4M
// visibilities in 256 blocks: 81k items of 103 on average, 5700
// instructions each, against 36k of 2 to 32 groups now).  Before -> now: 644 ->
// 361 us there (and the combine pass, with half the partial tiles, 138 ->
// 112), 125 -> 107 us at 1024^2 (4.2M visibilities, 64 blocks, dual step), 37
// -> 29 us at 640 x 480 (700k), 27 -> 29 us at 512^2 (524k).  What bounds it
// now: issue slots (73 % busy at 1024^2, 22 instructions a visibility) and
// the shared-memory path (63 %).
// With the private-tile pitch T + 8 = 8 mod 16 (in 8-byte words) rows a and a
// + 2 share banks: lanes of rows 2, 3, 6 and 7 take column b + 4 first.
// A warp's staging area: per visibility w0[a] Theta v and the pairs (w1[b],
// w1[b+4]).  The pitch keeps rows 16-byte aligned and the 8 (4) rows that a
// warp reads at once in distinct banks.
template <typename R> struct GridStage {
    static constexpr int PITCH = sizeof(R) == 4 ? 34 : 33;
    cplx_t<R> p[8][PITCH];
    cplx_t<R> w[4][PITCH];
};
template <typename R, int T> struct __align__(16) GridWarp {
    cplx_t<R> tile[(T + HALO) * (T + HALO)];
    GridStage<R> st;
};

// NW warps per CTA (4 or 8; FP64: 4): eight split an item finer, four
// leave room for more CTAs per SM (the autotuner picks per problem).
template <typename R, int T, int MODE, int NW>
__global__ void __launch_bounds__(NW * 32, sizeof(R) == 8 || T == 32 ? 1 : 28 / NW)
    k_grid(VisArgs<R> A, int n_large, int n_items,
                                                  cplx_t<R> *__restrict__ gpart) {
    using C = cplx_t<R>;
    constexpr int E = T + HALO, P = E, EE = E * E;   // P: pitch of the private tiles (8 mod 16 words)
    static_assert(P % 16 == 8, "private-tile pitch");
    constexpr int VEC = 16 / sizeof(C), NV = EE / VEC;   // 16-byte pieces of a tile
    extern __shared__ __align__(128) unsigned char smem_raw[];
    GridWarp<R, T> *W = reinterpret_cast<GridWarp<R, T> *>(smem_raw);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    // largest items first, so that the last wave holds the small ones
    const bool large = (int)blockIdx.x < n_large;
    const int pos = large ? (int)blockIdx.x : n_large + ((int)blockIdx.x - n_large) * NW + warp;
    const int item = pos < n_items ? A.it_order[pos] : -1;
    const int2 ig = item >= 0 ? A.it_grp[item] : make_int2(0, 0);
    // warps that share the item, at least two groups each, so that only as
    // many private tiles are cleared and summed as get filled
    const int nwu = large ? min(NW, max(1, ig.y / 2)) : 1, w = large ? warp : 0;
    C *mine = W[warp].tile;
    if (w < nwu)
        for (int e = lane; e < NV; e += 32) reinterpret_cast<float4 *>(mine)[e] = make_float4(0.f, 0.f, 0.f, 0.f);
    pdl_enter();
    if (item < 0) return;
    // blocks outside the active set D keep v_j: an item with none inside
    // keeps its partial tile of the last gridding, unless that may be stale
    if (MODE == GR_DUAL && A.bmask && !*A.regrid) {
        bool any = false;
        for (int g = lane; g < ig.y; g += 32) any = any || A.bmask[A.gg[ig.x + g].w];
        if (!__any_sync(0xffffffffu, any)) return;   // (the same for every warp of the item)
    }
    const int arow = lane >> 2, bcol = lane & 3;   // row, and columns bcol and bcol + 4
    const bool swap = arow & 2;
    struct In {
        VisRec<R> rc;
        C a, b, z;   // GR_DUAL active: y, w, z (stopped early: p, -, z); inactive: v; operator modes: input
        R th;
    };
    // of a group's block: inside D, Algorithm 2 stopped early (stopping
    // test: the prox output is the p the stopping step kept, not P_B of the
    // current w), the P_B scale
    struct Blk {
        bool act, done;
        R c;
    };
    auto block_of = [&](int blk) {
        Blk o{true, false, R(0)};
        if (MODE == GR_DUAL) {
            o.act = !A.bmask || A.bmask[blk];
            if (A.tol_on) o.done = A.inner_state[blk] != 0;
            o.c = A.scale[blk];
        }
        return o;
    };
    auto load_in = [&](int gi, const Blk &q, In &o) {
        o.rc = A.rec[gi];
        if (MODE == GR_DUAL && q.act) {
            if (q.done) {
                o.a = A.p[gi];
            } else {
                o.a = A.y[gi];
                o.b = A.w[gi];
            }
            o.z = A.z[gi];
        } else if (MODE == GR_DUAL) {
            o.a = A.v[gi];
        } else {
            o.a = A.op_in[A.perm ? A.perm[gi] : gi];
        }
        o.th = A.theta_v ? A.theta_v[gi] : A.theta_s;
    };
    GridStage<R> &st = W[warp].st;
    const int g0 = ig.x + (w < nwu ? w * ig.y / nwu : 0), g1 = ig.x + (w < nwu ? (w + 1) * ig.y / nwu : 0);
    if (g0 < g1) {
        int4 D = A.gg[g0], Dn = g0 + 1 < g1 ? A.gg[g0 + 1] : D;   // this group and the next
        Blk bk = block_of(D.w);
        In cur;
        if (lane < D.y) load_in(D.x + lane, bk, cur);
        const int row0 = (D.z / A.ntile1) * T, col0 = (D.z % A.ntile1) * T;
        C *cells0 = mine + arow * P + bcol + (swap ? 4 : 0), *cells1 = mine + arow * P + bcol + (swap ? 0 : 4);
        int run = -1;   // base cell (tile offset) of the run being accumulated
        C acc0{0, 0}, acc1{0, 0};   // columns bcol, bcol + 4
        auto flush = [&]() {   // add the run's two cells of this lane into the private tile
            const C t0 = cells0[run], t1 = cells1[run];
            cells0[run] = cadd(t0, swap ? acc1 : acc0);
            cells1[run] = cadd(t1, swap ? acc0 : acc1);
        };
        auto accumulate = [&](C w, C q) {
            acc0.x += w.x * q.x;
            acc0.y += w.x * q.y;
            acc1.x += w.y * q.x;
            acc1.y += w.y * q.y;
        };
        for (int g = g0; g < g1; ++g) {
            const int n = D.y;
            int mylb = -1;
            R w0[KB_J] = {}, w1[KB_J] = {};
            C tv{0, 0};
            if (lane < n) {
                const int gi = D.x + lane;
                const VisRec<R> rc = cur.rc;
                C vv = cur.a;
                if (MODE == GR_DUAL && bk.act) {
                    C pp = cur.a;
                    if (!bk.done) {
                        pp = C{cur.a.x + bk.c * (cur.b.x - cur.a.x), cur.a.y + bk.c * (cur.b.y - cur.a.y)};
                        A.p[gi] = pp;
                    }
                    vv = C{rc.U * (cur.z.x - pp.x), rc.U * (cur.z.y - pp.y)};
                    A.v[gi] = vv;
                } else if (MODE == GR_OP_U) {
                    vv = C{rc.U * vv.x, rc.U * vv.y};
                }
                tv = C{cur.th * vv.x, cur.th * vv.y};
                kb_weights(rc.f0, w0, A);
                kb_weights(rc.f1, w1, A);
                mylb = ((rc.packed & 0xffff) - row0) * P + ((rc.packed >> 16) & 0xffff) - col0;
            }
            // (lanes past the group stage zeros: the loop below works in fours)
#pragma unroll
            for (int a = 0; a < KB_J; ++a) st.p[a][lane] = C{w0[a] * tv.x, w0[a] * tv.y};
#pragma unroll
            for (int j = 0; j < KB_J / 2; ++j) st.w[j][lane] = C{w1[j], w1[j + 4]};
            if (MODE == GR_DUAL && A.seen && lane == 0 && bk.act && !A.seen[D.w]) A.seen[D.w] = 1;
            // the group's visibilities that start a new run: lane 0 compares
            // with the run carried over
            const int prev = __shfl_up_sync(0xffffffffu, mylb, 1);
            const unsigned starts = __ballot_sync(0xffffffffu, lane < n && mylb != (lane == 0 ? run : prev));
            __syncwarp();
            if (g + 1 < g1) {   // the next group, in flight during the sums
                D = Dn;
                bk = block_of(D.w);
                if (lane < D.y) load_in(D.x + lane, bk, cur);
                if (g + 2 < g1) Dn = A.gg[g + 2];
            }
            for (int i = 0; i < n; i += 4) {
                C pq[4], wq[4];
                if constexpr (sizeof(R) == 4) {   // two visibilities per 16-byte read
#pragma unroll
                    for (int q = 0; q < 4; q += 2) {
                        const float4 u = *reinterpret_cast<const float4 *>(&st.p[arow][i + q]);
                        const float4 v = *reinterpret_cast<const float4 *>(&st.w[bcol][i + q]);
                        pq[q] = C{u.x, u.y};
                        pq[q + 1] = C{u.z, u.w};
                        wq[q] = C{v.x, v.y};
                        wq[q + 1] = C{v.z, v.w};
                    }
                } else {
#pragma unroll
                    for (int q = 0; q < 4; ++q) {
                        pq[q] = st.p[arow][i + q];
                        wq[q] = st.w[bcol][i + q];
                    }
                }
                const unsigned m = (starts >> i) & 15u;
                if (m == 0) {   // (m is uniform across the warp)
#pragma unroll
                    for (int q = 0; q < 4; ++q) accumulate(wq[q], pq[q]);
                } else {
#pragma unroll
                    for (int q = 0; q < 4; ++q) {
                        if (m & (1u << q)) {
                            if (run >= 0) flush();
                            run = __shfl_sync(0xffffffffu, mylb, i + q);
                            acc0 = acc1 = C{0, 0};
                        }
                        accumulate(wq[q], pq[q]);
                    }
                }
            }
            __syncwarp();   // the staging is rewritten by the next group
        }
        if (run >= 0) flush();
    }
    float4 *out = reinterpret_cast<float4 *>(gpart + (int64_t)item * EE);
    if (!large) {
        __syncwarp();
        for (int e = lane; e < NV; e += 32) out[e] = reinterpret_cast<const float4 *>(mine)[e];
        return;
    }
    __syncthreads();
    for (int e = threadIdx.x; e < NV; e += NW * 32) {
        C s[VEC];
#pragma unroll
        for (int q = 0; q < VEC; ++q) s[q] = W[0].tile[e * VEC + q];
        for (int k = 1; k < nwu; ++k)
#pragma unroll
            for (int q = 0; q < VEC; ++q) s[q] = cadd(s[q], W[k].tile[e * VEC + q]);
        out[e] = *reinterpret_cast<const float4 *>(s);
    }
}

template <int V> struct Count {
    static constexpr int value = V;
};

// ----------------------------------------------------------------- combine
// One CTA per active tile (a tile with items, or below/right of one):
// grid[r][c] = sum of the partial tiles covering the cell, in a fixed order:
// the cell's own tile's items, then the halo rows/columns of the tiles
// above, left and above-left (periodic grid).  The grid is column-major
// (element (r, c) at c K0 + r, the layout the inverse column pass reads):
// the T x T sums, formed from row-major partial-tile reads, are transposed
// in shared memory and written as whole column segments.  Tiles never
// touched by any visibility stay zero from the initial clear.
//
// NTH threads per tile read the tile's item ranges themselves, no barrier
// before the partial tiles.  Where tiles have about one item each, 64 threads
// with four cells side by side keep four times the loads in flight per
// thread and as many tiles per SM (4096^2, 36k items: 112 -> 52 us; 960 x 400:
// 15.6 -> 8.7; 640 x 480: 8.0 -> 6.6); where a tile has several, a thread per
// cell shortens the sums' chain (1024^2, two items per tile: 64 threads took
// 20 us, 256 take 15).
template <typename R, int T, int NTH>
__global__ void __launch_bounds__(NTH) k_combine(const cplx_t<R> *__restrict__ gpart,
                                                 const int32_t *__restrict__ tile_first,
                                                 const int32_t *__restrict__ tile_n,
                                                 const int32_t *__restrict__ active, int K0, int nt0, int nt1,
                                                 cplx_t<R> *__restrict__ grid) {
    using C = cplx_t<R>;
    constexpr int E = T + HALO, CELLS = T * T / NTH;
    // of a thread's cells the first UPPER lie in the rows above HALO (all or
    // none when it has one cell)
    constexpr int UPPER = CELLS == 1 ? 1 : CELLS * HALO / T;
    static_assert(CELLS == 1 || T * HALO % NTH == 0, "cells split at row HALO");
    __shared__ C tr[T][T + 1];
    const int t = active[blockIdx.x];
    const int t0 = t / nt1, t1 = t - t0 * nt1;
    const int up = t0 == 0 ? nt0 - 1 : t0 - 1, left = t1 == 0 ? nt1 - 1 : t1 - 1;
    const int tt[4] = {t, up * nt1 + t1, t0 * nt1 + left, up * nt1 + left};
    int f[4], n[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        f[q] = __ldg(tile_first + tt[q]);
        n[q] = __ldg(tile_n + tt[q]);
    }
    pdl_enter();
    // cell i of this thread: row lr + i NTH / T, column lc
    const int lr = threadIdx.x / T, lc = threadIdx.x % T;
    C acc[CELLS];
#pragma unroll
    for (int i = 0; i < CELLS; ++i) acc[i] = C{0, 0};
    auto add = [&](int q, int off, bool in, auto cells) {   // the items of tile q at offset `off`
        constexpr int NC = decltype(cells)::value;
        if (!in) return;
        const C *p = gpart + (int64_t)f[q] * E * E + off + lr * E + lc;
        if constexpr (CELLS == 1) {
#pragma unroll 4
            for (int k = 0; k < n[q]; ++k) acc[0] = cadd(acc[0], p[(int64_t)k * (E * E)]);
        } else {
            for (int k = 0; k < n[q]; ++k, p += E * E)
#pragma unroll
                for (int i = 0; i < NC; ++i) acc[i] = cadd(acc[i], p[i * (NTH / T) * E]);
        }
    };
    const bool upper = CELLS > 1 || lr < HALO;
    add(0, 0, true, Count<CELLS>{});
    add(1, T * E, upper, Count<UPPER>{});
    add(2, T, lc < HALO, Count<CELLS>{});
    add(3, T * E + T, upper && lc < HALO, Count<UPPER>{});
#pragma unroll
    for (int i = 0; i < CELLS; ++i) tr[lc][lr + i * (NTH / T)] = acc[i];
    __syncthreads();
#pragma unroll
    for (int i = 0; i < CELLS; ++i) {
        const int e = threadIdx.x + i * NTH, oc = e / T, orow = e % T;
        grid[(int64_t)(t1 * T + oc) * K0 + t0 * T + orow] = tr[oc][orow];
    }
}

template <typename R> VisArgs<R> make_args(ppd_ctx *c) {
    VisArgs<R> A{};
    A.rec = static_cast<const VisRec<R> *>(c->rec);
    A.theta_v = static_cast<const R *>(c->theta_v);
    A.theta_s = (R)c->theta_scalar;
    A.gg = c->ch.gg;
    A.it_grp = c->ch.it_grp;
    A.it_order = c->ch.order;
    A.K0 = c->K0;
    A.K1 = c->K1;
    A.ntile1 = c->K1 / c->T;
    for (int i = 0; i < KB_J / 2 * KB_N<R>; ++i) A.kbp[i] = (R)c->kbpoly_h[i];
    for (int i = 0; i < KB_J / 4; ++i) {
        const int at = (KB_J / 4 + i) * KB_N<R>;
        A.kbl[i] = (R)(c->kbpoly_h[at] - (double)A.kbp[at]);
    }
    A.bessel = c->kb_bessel;
    A.beta = c->beta;
    A.inv_i0b = c->kb_inv_i0b;
    A.y = static_cast<const cplx_t<R> *>(c->y);
    A.v = static_cast<cplx_t<R> *>(c->v);
    A.z = static_cast<cplx_t<R> *>(c->z);
    A.w = static_cast<cplx_t<R> *>(c->w);
    A.p = static_cast<cplx_t<R> *>(c->p);
    A.mu = static_cast<const R *>(c->mu_d);
    A.scale = static_cast<const R *>(c->scale);
    A.partials = c->partials;
    A.run_pos = c->ch.run_pos;
    A.warp_run = c->ch.warp_run;
    A.grp = c->ch.grp;
    A.warp_grp = c->ch.warp_grp;
    A.n_warps = c->ch.n_warps;
    A.err = c->err;
    A.bmask = c->rand_on ? c->mask_cur : nullptr;
    A.seen = c->rand_on ? c->blk_seen : nullptr;
    A.regrid = c->rand_on ? c->regrid_d : nullptr;
    A.tol_on = c->cfg.inner_tol > 0;
    A.step = c->next_step;
    A.n_itr = c->cfg.n_itr;
    A.inner_state = c->inner_state;
    A.inner_steps = c->inner_steps;
    return A;
}

// the blocks' scales from the norm partials of the kernel before
template <typename R> int block_scales(ppd_ctx *c, int step, cudaStream_t s) {
    int site;
    PPD_CHECK(launch_begin(c, "block_scale", s, &site));
    launch(c, true, k_block_scale<R>, (unsigned)c->d, BS_NT, 0, s, (const double *)c->partials,
           (const int32_t *)c->ch.blk_ptr, (const double *)c->eps_d, c->cfg.inner_tol, step,
           static_cast<R *>(c->scale), c->inner_state, c->inner_steps, c->err);
    return launch_end(c, site, s);
}

template <typename R, int T, int NTD>
int degrid_t(ppd_ctx *c, int mode, const cplx_t<R> *grid, cplx_t<R> *out, const int64_t *perm, cudaStream_t s) {
    VisArgs<R> A = make_args<R>(c);
    A.op_out = out;
    A.perm = perm;
    constexpr int E = T + HALO;
    const size_t sh = (size_t)(NTD / 32) * dg_bufs<T>() * E * E * sizeof(cplx_t<R>);
    const int use_tma = (c->tma_ok && grid == c->grid_a) ? 1 : 0;
    if (c->ch.n_grp == 0) return PPD_OK;
    const unsigned nb = (unsigned)((c->ch.n_warps + NTD / 32 - 1) / (NTD / 32));
    auto k = mode == DG_OP     ? k_degrid<R, T, DG_OP, NTD>
             : mode == DG_DUAL ? k_degrid<R, T, DG_DUAL, NTD>
                               : k_degrid<R, T, DG_FIRST, NTD>;
    PPD_CHECK(smem_attr((const void *)k, (int)sh));
    int site;
    PPD_CHECK(launch_begin(c, mode == DG_OP ? "degrid_op" : "degrid_dual", s, &site));
    const long long sf = c->wait_first;
    launch(c, true, k, nb, NTD, sh, s, c->tmap_a, use_tma, grid, A, sf);
    PPD_CHECK(launch_end(c, site, s));
    return mode == DG_OP ? PPD_OK : block_scales<R>(c, 0, s);
}

template <typename R, int T, int NW> int grid_launch(ppd_ctx *c, int mode, const VisArgs<R> &A, cudaStream_t s) {
    const size_t sh = NW * sizeof(GridWarp<R, T>);
    auto k = mode == GR_OP     ? k_grid<R, T, GR_OP, NW>
             : mode == GR_OP_U ? k_grid<R, T, GR_OP_U, NW>
                               : k_grid<R, T, GR_DUAL, NW>;
    PPD_CHECK(smem_attr((const void *)k, (int)sh));
    int site;
    PPD_CHECK(launch_begin(c, mode == GR_DUAL ? "grid_dual" : "grid_op", s, &site));
    const int64_t small = c->ch.n - c->ch.n_large;
    launch(c, true, k, (unsigned)(c->ch.n_large + (small + NW - 1) / NW), NW * 32, sh, s, A, (int)c->ch.n_large,
           (int)c->ch.n, static_cast<cplx_t<R> *>(c->gpart));
    return launch_end(c, site, s);
}

template <typename R, int T>
int grid_t(ppd_ctx *c, int mode, const cplx_t<R> *in, const int64_t *perm, cplx_t<R> *grid, cudaStream_t s,
           bool combine) {
    VisArgs<R> A = make_args<R>(c);
    A.op_in = in;
    A.perm = perm;
    cplx_t<R> *gp = static_cast<cplx_t<R> *>(c->gpart);
    int site;
    if (c->ch.n > 0) {
        if constexpr (sizeof(R) == 4) {
            PPD_CHECK((c->grid_nw == 4 ? grid_launch<R, T, 4>(c, mode, A, s) : grid_launch<R, T, 8>(c, mode, A, s)));
        } else {
            PPD_CHECK((grid_launch<R, T, 4>(c, mode, A, s)));
        }
    }
    if (c->ch.n_active == 0 || !combine) return PPD_OK;
    PPD_CHECK(launch_begin(c, "grid_combine", s, &site));
    constexpr int few = T == 16 ? 64 : 256, many = T == 16 ? 256 : 1024;
    const bool sparse = c->ch.n * 5 < c->ch.n_active * 6;   // under 1.2 items per written tile
    launch(c, true, sparse ? k_combine<R, T, few> : k_combine<R, T, many>, (unsigned)c->ch.n_active,
           sparse ? few : many, 0, s, (const cplx_t<R> *)gp,
           (const int32_t *)c->ch.tile_first, (const int32_t *)c->ch.tile_n, (const int32_t *)c->ch.active, c->K0,
           c->K0 / T, c->K1 / T, grid);
    return launch_end(c, site, s);
}

}  // namespace

int degrid_warps_per_sm(const ppd_ctx *c) {
    if (!c->is_f32) return c->T == 16 ? dg_warps_per_sm<double, 16>() : dg_warps_per_sm<double, 32>();
    return c->T == 16 ? dg_warps_per_sm<float, 16>() : dg_warps_per_sm<float, 32>();
}

// Binning entry used by the API: fills key, base (2 per vis), frac (2 per
// vis), per-visibility cell count.
int bin_all(ppd_ctx *c, const double *uv_d, const int32_t *blk_d, int64_t M, uint64_t *key_d, int32_t *base_d,
            double *frac_d, int32_t *count_d, int *bad_d) {
    int32_t *cell_d = nullptr, *cgrid = nullptr;
    PPD_CUDA(cudaMalloc(&cell_d, M * sizeof(int32_t)));
    PPD_CUDA(cudaMalloc(&cgrid, (size_t)c->K0 * c->K1 * sizeof(int32_t)));
    PPD_CUDA(cudaMemsetAsync(cgrid, 0, (size_t)c->K0 * c->K1 * sizeof(int32_t), c->stream));
    const int nb = (int)std::min<int64_t>((M + 255) / 256, 152 * 32);
    k_bin<<<nb, 256, 0, c->stream>>>(uv_d, blk_d, M, c->K0, c->K1, c->T, c->d, key_d, base_d, frac_d, cell_d, cgrid,
                                     bad_d);
    k_cell_count<<<nb, 256, 0, c->stream>>>(cell_d, cgrid, M, count_d);
    c->launches += 2;
    PPD_CUDA(cudaGetLastError());
    PPD_CUDA(cudaStreamSynchronize(c->stream));
    PPD_CUDA(cudaFree(cell_d));
    PPD_CUDA(cudaFree(cgrid));
    return PPD_OK;
}

// I0(z) by its power series sum_k (z^2/4)^k / (k!)^2 (all terms positive, so
// the sum is as exact as the type).
template <typename X> static X bessel_i0(X z) {
    const X q = z * z / 4;
    X sum = 1, term = 1;
    for (int k = 1; k < 100000; ++k) {
        term *= q / ((X)k * k);
        sum += term;
        if (!(term > sum * std::numeric_limits<X>::epsilon() / 4)) break;
    }
    return sum;
}

// Chebyshev interpolation (in t = 2 frac - 1, n points) of the weights
// psi(frac + 3 - j) of taps 0..3, converted to n monomial coefficients per
// tap, in type X.
template <typename X> static std::vector<X> fit_weights(int n, X beta) {
    const X i0b = bessel_i0<X>(beta), pi = std::acos((X)-1);
    std::vector<X> out((size_t)n * KB_J / 2), node(n), cs((size_t)n * n);
    for (int k = 0; k < n; ++k) {
        node[k] = std::cos(pi * (k + (X)0.5) / n);
        for (int m = 0; m < n; ++m) cs[(size_t)m * n + k] = std::cos(pi * ((m * (2 * k + 1)) % (4 * n)) / (2 * n));
    }
    for (int j = 0; j < KB_J / 2; ++j) {
        std::vector<X> fk(n), cheb(n, 0), mono(n, 0), Tm1(n, 0), Tm(n, 0), Tn(n, 0);
        for (int k = 0; k < n; ++k) {
            const X d = ((node[k] + 1) / 2 + 3 - j) / 4;
            fk[k] = bessel_i0<X>(beta * std::sqrt(1 - d * d)) / i0b;   // |d| < 1 at every node
        }
        for (int m = 0; m < n; ++m) {
            X s = 0;
            for (int k = 0; k < n; ++k) s += fk[k] * cs[(size_t)m * n + k];
            cheb[m] = s * (m == 0 ? 1 : 2) / n;
        }
        // Chebyshev -> monomial: T_0 = 1, T_1 = t, T_{m+1} = 2 t T_m - T_{m-1}
        Tm1[0] = 1;
        Tm[1] = 1;
        for (int k = 0; k < n; ++k) mono[k] = cheb[0] * Tm1[k] + cheb[1] * Tm[k];
        for (int m = 2; m < n; ++m) {
            for (int k = 0; k < n; ++k) Tn[k] = (k > 0 ? 2 * Tm[k - 1] : 0) - Tm1[k];
            for (int k = 0; k < n; ++k) mono[k] += cheb[m] * Tn[k];
            Tm1 = Tm;
            Tm = Tn;
        }
        for (int k = 0; k < n; ++k) out[(size_t)j * n + k] = mono[k];
    }
    return out;
}

// The weight polynomials (KB_N coefficients per tap) and 1 / I0(beta).  The
// FP64 fit runs in long double, so that its coefficients carry only their
// own rounding (a fit in double leaves 3e-15).  FP64: where the polynomials
// are off by more than 1e-15 (a shape far from the default) the kernels keep
// the Bessel function.
int make_kb_poly(ppd_ctx *c) {
    c->kb_bessel = 0;
    if (c->is_f32) {
        c->kbpoly_h = fit_weights<double>(KB_N<float>, c->beta);
        c->kb_inv_i0b = 1.0 / bessel_i0<double>(c->beta);
        return PPD_OK;
    }
    using X = long double;
    const int n = KB_N<double>;
    const X beta = c->beta, i0b = bessel_i0<X>(beta);
    const std::vector<X> fit = fit_weights<X>(n, beta);
    c->kbpoly_h.assign(fit.begin(), fit.end());
    c->kb_inv_i0b = (double)(1 / i0b);
    for (int j = 0; j < KB_J / 2; ++j)
        for (int i = 0; i <= 8; ++i) {
            const double t = i / 4.0 - 1.0;
            double v = 0;
            for (int k = n - 1; k >= 0; --k) v = std::fma(v, t, c->kbpoly_h[(size_t)j * n + k]);
            const X d = (((X)t + 1) / 2 + 3 - j) / 4, x = 1 - d * d;
            const X ref = x >= 0 ? bessel_i0<X>(beta * std::sqrt(x)) / i0b : (X)0;
            // (written so that a value that is not finite also counts)
            if (!(std::abs((X)v - ref) <= (X)1e-15)) c->kb_bessel = 1;
        }
    return PPD_OK;
}

template <typename R>
int degrid(ppd_ctx *c, int mode, const cplx_t<R> *grid, cplx_t<R> *out, const int64_t *perm, cudaStream_t s) {
    if constexpr (sizeof(R) == 4) {
        if (c->degrid_nt == 128)
            return c->T == 16 ? degrid_t<R, 16, 128>(c, mode, grid, out, perm, s)
                              : degrid_t<R, 32, 128>(c, mode, grid, out, perm, s);
    }
    return c->T == 16 ? degrid_t<R, 16, 256>(c, mode, grid, out, perm, s)
                      : degrid_t<R, 32, 256>(c, mode, grid, out, perm, s);
}

template <typename R>
int grid_vis(ppd_ctx *c, int mode, const cplx_t<R> *in, const int64_t *perm, cplx_t<R> *grid, cudaStream_t s,
             bool combine) {
    return c->T == 16 ? grid_t<R, 16>(c, mode, in, perm, grid, s, combine)
                      : grid_t<R, 32>(c, mode, in, perm, grid, s, combine);
}

template <typename R> int subiter(ppd_ctx *c, cudaStream_t s, int only_first, double beta, int write_p) {
    if (c->ch.n_grp == 0) return PPD_OK;
    int site;
    PPD_CHECK(launch_begin(c, "subiter", s, &site));
    const unsigned nb = (unsigned)((c->ch.n_warps + SUB_NT / 32 - 1) / (SUB_NT / 32));
    launch(c, true, k_subiter<R>, nb, SUB_NT, 0, s, make_args<R>(c), only_first, (R)beta, write_p);
    PPD_CHECK(launch_end(c, site, s));
    return block_scales<R>(c, c->next_step, s);
}

int block_norms(ppd_ctx *c, cudaStream_t s) {
    int site;
    PPD_CHECK(launch_begin(c, "block_norms", s, &site));
    const int wpb = 8;
    k_block_norms<<<(c->d + wpb - 1) / wpb, wpb * 32, 0, s>>>(c->partials, c->ch.blk_ptr, c->d, c->resid2, c->err);
    return launch_end(c, site, s);
}

// Same launches as grid_vis, with the per-chunk partial tiles written to a
// caller-supplied device buffer instead of the context's.
template <typename R>
int grid_vis_into(ppd_ctx *c, int mode, const cplx_t<R> *in, const int64_t *perm, cplx_t<R> *grid, void *gpart,
                  cudaStream_t s) {
    void *own = c->gpart;
    c->gpart = gpart;
    const int st = grid_vis<R>(c, mode, in, perm, grid, s);
    c->gpart = own;
    return st;
}

template int grid_vis_into<float>(ppd_ctx *, int, const float2 *, const int64_t *, float2 *, void *, cudaStream_t);
template int grid_vis_into<double>(ppd_ctx *, int, const double2 *, const int64_t *, double2 *, void *,
                                   cudaStream_t);
template int degrid<float>(ppd_ctx *, int, const float2 *, float2 *, const int64_t *, cudaStream_t);
template int degrid<double>(ppd_ctx *, int, const double2 *, double2 *, const int64_t *, cudaStream_t);
template int grid_vis<float>(ppd_ctx *, int, const float2 *, const int64_t *, float2 *, cudaStream_t, bool);
template int grid_vis<double>(ppd_ctx *, int, const double2 *, const int64_t *, double2 *, cudaStream_t, bool);
template int subiter<float>(ppd_ctx *, cudaStream_t, int, double, int);
template int subiter<double>(ppd_ctx *, cudaStream_t, int, double, int);

}  // namespace ppd
