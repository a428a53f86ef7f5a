// Oversampled 2-D FFT with the zero-padding / scaling operator Z fused in
// (Section 2: Phi = Theta G F Z; F is the unnormalised n-oversampled DFT).
//
// Image L0 x L1 (rows x columns), grid K0 x K1 (K = 2L per axis).
// Forward  a = F Z x:  row pass    x (L0 x L1 real) -> tmp (L0 x K1 complex)
//                      column pass tmp              -> grid (K0 x K1 complex)
// Inverse  Re(Z^T F^H grid): column pass grid -> tmp, row pass tmp -> image.
//
// Every pass is a batched Stockham FFT: a CTA takes B sequences of one or two
// whole rows (row pass, length K1) or a strip of W columns (column pass, length
// K0), runs the stages and writes the result.  Only the L nonzero rows / columns of the
// padded image are read or produced; the grid is stored with the zero
// frequency at the centre (plain index k at (k + K/2) mod K).
//
// Two cores: lengths that are powers of two keep a sequence in the registers
// of its threads and cross shared memory once or twice (compile-time radices
// up to 32); any other length whose prime factors are 2, 3 and 5 uses a
// run-time mixed-radix core (radices from a plan made on the host) that
// ping-pongs between two shared buffers.  The pass kernels are templated on
// KT = the length for the first core, 0 for the second.
#include <cmath>
#include <vector>

#include "common.cuh"

namespace ppd {

namespace {

template <typename C> __device__ __forceinline__ C cmul(C a, C b) {
    return C{a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x};
}
template <typename C> __device__ __forceinline__ C cadd(C a, C b) { return C{a.x + b.x, a.y + b.y}; }
template <typename C> __device__ __forceinline__ C csub(C a, C b) { return C{a.x - b.x, a.y - b.y}; }
template <typename C> __device__ __forceinline__ C cconj(C a) { return C{a.x, -a.y}; }

// v mod K for v in [0, 2K)
__device__ __forceinline__ int wrapK(int v, int K) { return v >= K ? v - K : v; }

// threads per CTA of the mixed-radix core's row and column passes
constexpr int NTR = 128, NTC = 256;

template <int V> struct IntC {
    static constexpr int value = V;
};

// ------------------------------------------------------------ power-of-two core
// Forward DFT of N = 2 .. 32 points in registers, in place, natural order.
template <typename R, int N> __device__ __forceinline__ void dft_regs(cplx_t<R> *v);
// v (c - i s) for a fixed rotation (c, s).  FP32 adds the parts of c and s
// that rounding drops: the same few constants turn every transform's data, so
// their rounding (1.7e-8 of the amplitude at 45 degrees) would not average
// out but scale the whole result (adjoint at 4096^2: amplitude 1.3e-7 low and
// error 2.1e-7 without them; 0.9e-7 and 1.8e-7 with radix-4 stages and table
// twiddles only).
template <typename R> __device__ __forceinline__ cplx_t<R> rotate(cplx_t<R> v, double c, double s) {
    using C = cplx_t<R>;
    const R ch = R(c), sh = R(s);
    if constexpr (sizeof(R) == 4) {
        const R cl = R(c - (double)ch), sl = R(s - (double)sh);
        return C{fmaf(v.x, ch, fmaf(v.y, sh, fmaf(v.x, cl, v.y * sl))),
                 fmaf(v.y, ch, fmaf(-v.x, sh, fmaf(v.y, cl, -v.x * sl)))};
    } else {
        return C{v.x * ch + v.y * sh, v.y * ch - v.x * sh};
    }
}
// v w^m, w = exp(-2 pi i / 32), m a compile-time value after unrolling
template <typename R> __device__ __forceinline__ cplx_t<R> rot32(cplx_t<R> v, int m) {
    using C = cplx_t<R>;
    // cos(2 pi m / 32), m = 0 .. 8
    constexpr double c32[9] = {1.0,
                               0.98078528040323044913,
                               0.92387953251128675613,
                               0.83146961230254523708,
                               0.70710678118654752440,
                               0.55557023301960222474,
                               0.38268343236508977173,
                               0.19509032201612826785,
                               0.0};
    m &= 31;
    if (m == 0) return v;
    if (m == 8) return C{v.y, -v.x};
    if (m == 16) return C{-v.x, -v.y};
    if (m == 24) return C{-v.y, v.x};
    const int a = m & 7, quad = m >> 3;
    const C t = rotate<R>(v, c32[a], c32[8 - a]);   // then a quarter turn -i per quadrant
    return quad == 0 ? t : quad == 1 ? C{t.y, -t.x} : quad == 2 ? C{-t.x, -t.y} : C{-t.y, t.x};
}
template <typename R> __device__ __forceinline__ void dft2_regs(cplx_t<R> &a, cplx_t<R> &b) {
    const cplx_t<R> t = a;
    a = cadd(t, b);
    b = csub(t, b);
}
template <typename R>
__device__ __forceinline__ void dft4_regs(cplx_t<R> &a0, cplx_t<R> &a1, cplx_t<R> &a2, cplx_t<R> &a3) {
    using C = cplx_t<R>;
    const C t0 = cadd(a0, a2), t1 = csub(a0, a2), t2 = cadd(a1, a3), t3 = csub(a1, a3);
    a0 = cadd(t0, t2);
    a1 = C{t1.x + t3.y, t1.y - t3.x};   // t1 - i t3
    a2 = csub(t0, t2);
    a3 = C{t1.x - t3.y, t1.y + t3.x};
}
// N = 4 M points: for each residue a mod 4 the M-point DFT of v[a + 4 m],
// rotated by w_N^(a c), then 4-point DFTs over a: X[c + M d]
template <typename R, int N> __device__ __forceinline__ void dft_regs(cplx_t<R> *v) {
    using C = cplx_t<R>;
    if constexpr (N == 2) {
        dft2_regs<R>(v[0], v[1]);
    } else if constexpr (N == 4) {
        dft4_regs<R>(v[0], v[1], v[2], v[3]);
    } else {
        constexpr int M = N / 4;
        C y[4][M];
#pragma unroll
        for (int a = 0; a < 4; ++a) {
#pragma unroll
            for (int m = 0; m < M; ++m) y[a][m] = v[a + 4 * m];
            dft_regs<R, M>(y[a]);
#pragma unroll
            for (int c = 0; c < M; ++c) y[a][c] = rot32<R>(y[a][c], a * c * (32 / N));
        }
#pragma unroll
        for (int c = 0; c < M; ++c) {
            dft4_regs<R>(y[0][c], y[1][c], y[2][c], y[3][c]);
#pragma unroll
            for (int d = 0; d < 4; ++d) v[c + M * d] = y[d][c];
        }
    }
}

// Radices of length K and the layout of a sequence: TPS threads hold EPT
// elements each (largest radices first).  A pass of radix RAD from span Ns: thread t's butterflies j =
// t + b TPS take inputs j + q K/RAD, twiddled by w^(q k K/(Ns RAD)), k = j mod
// Ns, and give outputs (j - k) RAD + k + p Ns.  Inputs and outputs of the
// whole transform that thread t sees are the positions t + m TPS, m < EPT.
// Passes are few (two to four, the last of the radix that is left: 8 8 at K =
// 64, 8 8 8 2 for FP32 rows of 1024, 16 16 32 at 8192) because each crosses
// shared memory: a radix-4 core went through it seven times at K = 8192 with up
// to 4-way bank conflicts and was bound by it (75 % of the data path busy).  PAD adds
// one element per 16, so that the stride-RAD stores of the first pass fall
// in distinct banks.
template <typename R_, int K_, int EPT_> struct Fft {
    using R = R_;
    static constexpr int K = K_, EPT = EPT_, TPS = K / EPT;
    static_assert(K % EPT == 0 && EPT >= 8, "image positions are quarters of a thread's elements");
    // radix of pass p: EPT as long as it divides what is left, then the rest
    __host__ __device__ static constexpr int radix(int p) {
        int left = K, r = 1;
        for (int i = 0; i <= p; ++i) {
            r = left < EPT ? left : EPT == 32 && left > 32 ? 16 : EPT;   // (8192 = 16 16 32)
            left /= r;
        }
        return r;
    }
    __host__ __device__ static constexpr int count() {
        int n = 0, left = K;
        while (left > 1) left /= radix(n++);
        return n;
    }
    static constexpr int PASSES = count();
    __host__ __device__ static constexpr int span(int p) {   // Ns of pass p
        int n = 1;
        for (int i = 0; i < p; ++i) n *= radix(i);
        return n;
    }
    __host__ __device__ static constexpr int tw_offset(int p) {   // its twiddles in the table (none for pass 0)
        int o = 0;
        for (int i = 1; i < p; ++i) o += span(i) * (radix(i) - 1);
        return o;
    }
    __host__ __device__ static constexpr int pad(int i) { return i + (i >> 4); }
    // distance of two sequences in shared memory when W of them are
    // interleaved over the lanes (lane = t W + s; W = 1: sequence after
    // sequence): the lanes of a half-warp in distinct banks
    __host__ __device__ static constexpr int stride(int W) {
        return pad(K) + (W > 1 ? (W < 16 ? 16 / W : 1) : (TPS < 16 ? TPS : 0));
    }
};

// Elements per thread.  Row passes up to K = 1024 (two warps per scheduler at
// most: a warp's instructions are the time) and FP64 (whose lanes need
// warps on all four schedulers): 8.  Longer FP32 rows and the columns: 16, a
// pass through shared memory less; 32 at K = 8192, where it keeps a column
// at 256 threads.
template <typename R> constexpr int row_ept(int K) {
    return sizeof(R) == 8 ? (K <= 2048 ? 8 : 16) : K <= 1024 ? 8 : K == 8192 ? 32 : 16;
}
template <typename R> constexpr int col_ept(int K) {
    return sizeof(R) == 8 ? (K <= 2048 ? 8 : 16) : K <= 64 ? 8 : K == 8192 ? 32 : 16;
}
template <typename R, int K> using RowFft = Fft<R, K, row_ept<R>(K)>;
template <typename R, int K> using ColFft = Fft<R, K, col_ept<R>(K)>;

// One transform: in(m) gives the input at position t + m TPS, out(m, value)
// takes the output there (m compile-time after unrolling).  buf: this
// sequence's padded buffer; tw: the twiddles pass by pass
// (upload_stage_twiddles).  All threads of the CTA call it together; the
// buffer may be read by in() (a barrier follows pass 0's inputs when
// in_smem) and is free again after the caller's next barrier.
template <typename F, bool in_smem, typename In, typename Out>
__device__ __forceinline__ void fft_run(cplx_t<typename F::R> *buf, int t,
                                        const cplx_t<typename F::R> *__restrict__ tw, In in, Out out) {
    using R = typename F::R;
    using C = cplx_t<R>;
    constexpr int K = F::K, EPT = F::EPT, TPS = F::TPS;
    C v[EPT];
    auto pass = [&](auto pc) {
        constexpr int P = decltype(pc)::value, RAD = F::radix(P), NS = F::span(P), NB = EPT / RAD;
        constexpr bool last = P == F::PASSES - 1;
        static_assert(EPT % RAD == 0, "whole butterflies per thread");
#pragma unroll
        for (int b = 0; b < NB; ++b) {
            const int j = t + b * TPS;
#pragma unroll
            for (int q = 0; q < RAD; ++q)
                v[b * RAD + q] = P == 0 ? in(b + q * (K / RAD / TPS)) : buf[F::pad(j + q * (K / RAD))];
        }
        if (P > 0 || in_smem) {
            if (!last) __syncthreads();   // every input is read before the buffer is rewritten
        }
#pragma unroll
        for (int b = 0; b < NB; ++b) {
            const int j = t + b * TPS, k = j & (NS - 1);
            if constexpr (P > 0) {
                const C *w = tw + F::tw_offset(P) + k;
#pragma unroll
                for (int q = 1; q < RAD; ++q) v[b * RAD + q] = cmul(v[b * RAD + q], __ldg(w + (q - 1) * NS));
            }
            dft_regs<R, RAD>(v + b * RAD);
            if constexpr (last) {
#pragma unroll
                for (int q = 0; q < RAD; ++q) out(b + q * (K / RAD / TPS), v[b * RAD + q]);
            } else {
                const int d = (j - k) * RAD + k;
#pragma unroll
                for (int q = 0; q < RAD; ++q) buf[F::pad(d + q * NS)] = v[b * RAD + q];
            }
        }
        if (!last) __syncthreads();
    };
    pass(IntC<0>{});
    pass(IntC<1>{});
    if constexpr (F::PASSES > 2) pass(IntC<2>{});
    if constexpr (F::PASSES > 3) pass(IntC<3>{});
}

// ------------------------------------------------------------ mixed-radix core
// v x + z for a constant v, in FP32 with the part of v that rounding drops
// (see rotate): the radix-5 constants alone left the adjoint at K = 800 an
// amplitude of +1.9e-8.
__device__ __forceinline__ float mad_const(double v, float x, float z) {
    const float h = float(v), l = float(v - (double)h);
    return fmaf(h, x, fmaf(l, x, z));
}
__device__ __forceinline__ double mad_const(double v, double x, double z) { return v * x + z; }

// Forward DFT of RAD points in place (sign -), written out per radix.
template <typename C> __device__ __forceinline__ void dft(C (&a)[2]) {
    const C t = a[0];
    a[0] = cadd(t, a[1]);
    a[1] = csub(t, a[1]);
}
template <typename C> __device__ __forceinline__ void dft(C (&a)[3]) {
    using R = decltype(a[0].x);
    constexpr double h = 0.86602540378443864676;   // sin(2 pi / 3)
    const C s = cadd(a[1], a[2]), d = csub(a[1], a[2]);
    const C m{a[0].x - R(0.5) * s.x, a[0].y - R(0.5) * s.y};
    a[0] = cadd(a[0], s);
    a[1] = C{mad_const(h, d.y, m.x), mad_const(-h, d.x, m.y)};   // m - i sin(2 pi/3) (a1 - a2)
    a[2] = C{mad_const(-h, d.y, m.x), mad_const(h, d.x, m.y)};
}
template <typename C> __device__ __forceinline__ void dft(C (&a)[4]) {
    const C t0 = cadd(a[0], a[2]), t1 = csub(a[0], a[2]);
    const C t2 = cadd(a[1], a[3]), t3 = csub(a[1], a[3]);
    a[0] = cadd(t0, t2);
    a[1] = C{t1.x + t3.y, t1.y - t3.x};
    a[2] = csub(t0, t2);
    a[3] = C{t1.x - t3.y, t1.y + t3.x};
}
template <typename C> __device__ __forceinline__ void dft(C (&a)[5]) {
    using R = decltype(a[0].x);
    constexpr double c1 = 0.30901699437494742410, c2 = -0.80901699437494742410;   // cos(2 pi/5), cos(4 pi/5)
    constexpr double s1 = 0.95105651629515357212, s2 = 0.58778525229247312917;    // sin(2 pi/5), sin(4 pi/5)
    const C t1 = cadd(a[1], a[4]), t2 = cadd(a[2], a[3]);
    const C t3 = csub(a[1], a[4]), t4 = csub(a[2], a[3]);
    // p x + q y (+ z)
    auto lin = [](double p, R x, double q, R y, R z) { return mad_const(q, y, mad_const(p, x, z)); };
    const C u1{lin(c1, t1.x, c2, t2.x, a[0].x), lin(c1, t1.y, c2, t2.y, a[0].y)};
    const C u2{lin(c2, t1.x, c1, t2.x, a[0].x), lin(c2, t1.y, c1, t2.y, a[0].y)};
    const C v1{lin(s1, t3.x, s2, t4.x, R(0)), lin(s1, t3.y, s2, t4.y, R(0))};
    const C v2{lin(s2, t3.x, -s1, t4.x, R(0)), lin(s2, t3.y, -s1, t4.y, R(0))};
    a[0] = cadd(a[0], cadd(t1, t2));
    a[1] = C{u1.x + v1.y, u1.y - v1.x};   // u1 - i v1
    a[4] = C{u1.x - v1.y, u1.y + v1.x};   // u1 + i v1
    a[2] = C{u2.x + v2.y, u2.y - v2.x};
    a[3] = C{u2.x - v2.y, u2.y + v2.x};
}

template <typename C> __device__ __forceinline__ void dft(C (&a)[8]) { dft_regs<decltype(a[0].x), 8>(a); }
template <typename C> __device__ __forceinline__ void dft(C (&a)[16]) { dft_regs<decltype(a[0].x), 16>(a); }
// cos and sin of 2 pi m / N as multiples of 2 pi / 60 (N divides 60; m is a
// compile-time value after unrolling)
__device__ __forceinline__ constexpr double cos60(int m) {
    constexpr double c[16] = {1.0, 0.99452189536827333692, 0.97814760073380563793, 0.95105651629515357212,
                              0.91354545764260089550, 0.86602540378443864676, 0.80901699437494742410,
                              0.74314482547739423501, 0.66913060635885821383, 0.58778525229247312917, 0.5,
                              0.40673664307580020775, 0.30901699437494742410, 0.20791169081775933710,
                              0.10452846326765347140, 0.0};
    m = m % 60;
    if (m > 30) m = 60 - m;
    return m <= 15 ? c[m] : -c[30 - m];
}
__device__ __forceinline__ constexpr double sin60(int m) { return cos60(m + 45); }
// N = A B points (6 = 2 3, 10 = 2 5, 12 = 4 3): B-point DFTs of a[i + A m],
// rotated by w_N^(i c), then A-point DFTs over i: X[c + B d].
template <int A, int B, typename C> __device__ __forceinline__ void dft_ab(C (&v)[A * B]) {
    using R = decltype(v[0].x);
    C y[B][A];
#pragma unroll
    for (int i = 0; i < A; ++i) {
        C t[B];
#pragma unroll
        for (int m = 0; m < B; ++m) t[m] = v[i + A * m];
        dft(t);
#pragma unroll
        for (int c = 0; c < B; ++c) {
            const int m = i * c * (60 / (A * B));
            y[c][i] = m == 0 ? t[c] : rotate<R>(t[c], cos60(m), sin60(m));
        }
    }
#pragma unroll
    for (int c = 0; c < B; ++c) {
        dft(y[c]);
#pragma unroll
        for (int d = 0; d < A; ++d) v[c + B * d] = y[c][d];
    }
}
template <typename C> __device__ __forceinline__ void dft(C (&a)[6]) { dft_ab<2, 3>(a); }
template <typename C> __device__ __forceinline__ void dft(C (&a)[10]) { dft_ab<2, 5>(a); }
template <typename C> __device__ __forceinline__ void dft(C (&a)[12]) { dft_ab<4, 3>(a); }

// Place of element i of sequence s in a buffer of the mixed-radix core: one
// element in 17 is padding (as Fft::pad), sequences one after the other or,
// INTERLEAVED, element by element (nseq = 2^lseq).
__host__ __device__ constexpr int mpad(int i) { return i + (i >> 4); }
template <bool INTERLEAVED> __device__ __forceinline__ int mplace(int s, int i, int K, int lseq) {
    return INTERLEAVED ? (mpad(i) << lseq) + s : s * mpad(K) + mpad(i);
}
// n / d for n < 2^16, 2 <= d <= 2^13, from inv = ceil(2^32 / d)
__device__ __forceinline__ int fast_div(int n, uint32_t inv) { return (int)__umulhi((uint32_t)n, inv); }

// One Stockham stage of radix RAD from src to dst: for butterfly j (k = j mod
// Ns) the inputs j + q K/RAD, twiddled by w^(q k K/(Ns RAD)), go to
// (j - k) RAD + k + p Ns.
template <typename R, int RAD, int NTH, bool INTERLEAVED>
__device__ __forceinline__ void stage_any(const cplx_t<R> *__restrict__ src, cplx_t<R> *__restrict__ dst,
                                          const FftPlan &pl, int st, int nseq, int lseq, int Ns,
                                          const cplx_t<R> *__restrict__ tw) {
    using C = cplx_t<R>;
    const int K = pl.K, m = K / RAD, tstep = pl.tstep[st], nbf = nseq * m;
    for (int bf = threadIdx.x; bf < nbf; bf += NTH) {
        int s, j;
        if (INTERLEAVED) {
            j = bf >> lseq;
            s = bf - (j << lseq);
        } else {
            s = nseq == 1 ? 0 : fast_div(bf, pl.inv_m[st]);
            j = bf - s * m;
        }
        const int k = Ns == 1 ? 0 : j - fast_div(j, pl.inv_ns[st]) * Ns;
        C a[RAD];
#pragma unroll
        for (int q = 0; q < RAD; ++q) a[q] = src[mplace<INTERLEAVED>(s, j + q * m, K, lseq)];
        if (Ns > 1) {
#pragma unroll
            for (int q = 1; q < RAD; ++q) a[q] = cmul(a[q], __ldg(tw + q * k * tstep));
        }
        dft(a);
        const int d = (j - k) * RAD + k;
#pragma unroll
        for (int p = 0; p < RAD; ++p) dst[mplace<INTERLEAVED>(s, d + p * Ns, K, lseq)] = a[p];
    }
}

// Batched mixed-radix FFT of nseq sequences of length pl.K in a (places by
// mplace), ping-ponging with b; returns the buffer holding the result.
// Callers synchronise before (the input is complete) and the last stage
// ends with a barrier.  Radices up to 16: three stages for most lengths up
// to 1920 where radices up to 5 took six, each a trip through shared memory
// and a barrier.
template <typename R, int NTH, bool INTERLEAVED>
__device__ cplx_t<R> *fft_any(cplx_t<R> *a, cplx_t<R> *b, int nseq, int lseq, const FftPlan &pl,
                              const cplx_t<R> *tw) {
    int Ns = 1;
    for (int st = 0; st < pl.ns; ++st) {
        const int r = pl.rad[st];
#define PPD_STAGE(RAD) \
    case RAD: stage_any<R, RAD, NTH, INTERLEAVED>(a, b, pl, st, nseq, lseq, Ns, tw); break
        switch (r) {
            PPD_STAGE(2);
            PPD_STAGE(3);
            PPD_STAGE(4);
            PPD_STAGE(5);
            PPD_STAGE(6);
            PPD_STAGE(8);
            PPD_STAGE(10);
            PPD_STAGE(12);
            PPD_STAGE(16);
        }
#undef PPD_STAGE
        __syncthreads();
        Ns *= r;
        cplx_t<R> *t = a;
        a = b;
        b = t;
    }
    return a;
}

// ------------------------------------------------------------ pass geometry
// Power-of-two core.  Row passes: sequences (two real rows each) per CTA, at
// least 64 threads.  Column passes: W columns per CTA with their lanes
// interleaved, so that a row of the strip is one 32-byte sector where a CTA
// stays within 512 threads (FP32: 4 columns up to K = 2048, 2 beyond; FP64
// half of that).  Two columns at K = 8192 (139 KB, one CTA of 512 threads per
// SM) against one (two CTAs of 256): forward 188 -> 165 us, inverse 214 -> 192.
template <typename R, int K> constexpr int row_seqs() { return RowFft<R, K>::TPS >= 64 ? 1 : 64 / RowFft<R, K>::TPS; }
template <typename R, int K> constexpr int col_width() {
    if (K >= 4096) return sizeof(R) == 4 ? 2 : 1;
    if (K >= 256) return sizeof(R) == 4 ? 4 : 2;
    return 64 / ColFft<R, K>::TPS;
}
template <typename R> int col_width_of(int K) {
    switch (K) {
        case 32: return col_width<R, 32>();
        case 64: return col_width<R, 64>();
        case 128: return col_width<R, 128>();
        case 256: return col_width<R, 256>();
        case 512: return col_width<R, 512>();
        case 1024: return col_width<R, 1024>();
        case 2048: return col_width<R, 2048>();
        case 4096: return col_width<R, 4096>();
        default: return col_width<R, 8192>();
    }
}
// threads per CTA of a row / column pass (mixed-radix core: NT)
template <typename R, int KT> constexpr int row_nt() {
    if constexpr (KT != 0) return row_seqs<R, KT>() * RowFft<R, KT>::TPS;
    else return NTR;
}
template <typename R, int KT> constexpr int col_nt() {
    if constexpr (KT != 0) return col_width<R, KT>() * ColFft<R, KT>::TPS;
    else return NTC;
}

// least CTAs per SM: two of the 32-element threads' (128 registers each)
template <typename R, int KT> constexpr int pass_ctas() { return KT == 8192 && sizeof(R) == 4 ? 2 : 1; }

// Run-time arguments of a pass: the FFT plan of its length and the
// sequences per CTA (used by the mixed-radix core only).
struct PassArgs {
    FftPlan pl;
    int nseq, lseq;   // lseq: log2 of nseq (columns)
};

// Row passes transform two real rows (a, b) as one complex sequence (but for
// the mixed-radix core's k_rows_inv: load_rows_inverse).  Forward: z = a + i b, and after the FFT
// A[k] = (Z[k] + conj(Z[-k]))/2, B[k] = (Z[k] - conj(Z[-k]))/(2i).
template <typename C> __device__ __forceinline__ void split_two_real(C z, C zr, C &A, C &B) {
    using R = decltype(z.x);
    A = C{R(0.5) * (z.x + zr.x), R(0.5) * (z.y - zr.y)};
    B = C{R(0.5) * (z.y + zr.y), R(0.5) * (zr.x - z.x)};
}
// Inverse to real parts: Re(F^H X) = F^H H with H[k] = (X[k] + conj(X[-k]))/2
// (the Hermitian part of X), so the pair is Y = Ha + i Hb, F^H Y = ha + i hb;
// returns Y[k] and Y[-k] from Xa[k], Xa[-k], Xb[k], Xb[-k].
template <typename C> __device__ __forceinline__ void pack_two_real(C xa, C xar, C xb, C xbr, C &y, C &yr) {
    using R = decltype(xa.x);
    const C ha{R(0.5) * (xa.x + xar.x), R(0.5) * (xa.y - xar.y)};
    const C hb{R(0.5) * (xb.x + xbr.x), R(0.5) * (xb.y - xbr.y)};
    y = C{ha.x - hb.y, ha.y + hb.x};    // ha + i hb
    yr = C{ha.x + hb.y, hb.x - ha.y};   // conj(ha) + i conj(hb)
}

// Loads the spectra of rows (row0 + 2s, row0 + 2s + 1), s < NSEQ, of tmp
// (stored centred: natural frequency k at column (k + K/2) mod K) and writes
// conj(Y) in natural order into buf, so that the forward FFT of buf gives
// conj(F^H Y): row a's real inverse in .x, row b's in -.y.
template <typename R, int K, int NSEQ, int NTH>
__device__ __forceinline__ void load_two_real_inverse(const cplx_t<R> *__restrict__ tmp, int row0, int L0,
                                                      cplx_t<R> *buf) {
    using C = cplx_t<R>;
    using F = RowFft<R, K>;
    constexpr int H = K / 2 + 1;   // pairs (k, -k), k = 0 .. K/2
#pragma unroll 4
    for (int e = threadIdx.x; e < NSEQ * H; e += NTH) {
        const int s = e / H, k = e - s * H, kr = (K - k) & (K - 1);
        const int ra = row0 + 2 * s, rb = ra + 1;
        const int ck = (k + K / 2) & (K - 1), ckr = (kr + K / 2) & (K - 1);
        C xa{0, 0}, xar{0, 0}, xb{0, 0}, xbr{0, 0};
        if (ra < L0) {
            xa = tmp[(int64_t)ra * K + ck];
            xar = tmp[(int64_t)ra * K + ckr];
        }
        if (rb < L0) {
            xb = tmp[(int64_t)rb * K + ck];
            xbr = tmp[(int64_t)rb * K + ckr];
        }
        C y, yr;
        pack_two_real(xa, xar, xb, xbr, y, yr);
        buf[s * F::stride(1) + F::pad(k)] = cconj(y);
        buf[s * F::stride(1) + F::pad(kr)] = cconj(yr);
    }
}

// Writes the spectra of rows (row0 + 2s, row0 + 2s + 1) from the FFT of
// a + i b in buf (natural order) to the column-major tmp (column c at
// c L0, stored centred, marked columns): the two rows are adjacent there.
template <typename R, int K, int NSEQ, int NTH>
__device__ __forceinline__ void store_two_real_forward(const cplx_t<R> *out, int row0, int L0,
                                                       const uint8_t *__restrict__ colmask,
                                                       cplx_t<R> *__restrict__ tmp) {
    using C = cplx_t<R>;
    using F = RowFft<R, K>;
#pragma unroll 4
    for (int e = threadIdx.x; e < NSEQ * K; e += NTH) {
        // the sequences of a CTA are adjacent row pairs: side by side in tmp
        const int s = e % NSEQ, c = e / NSEQ, ra = row0 + 2 * s;
        if (!colmask[c] || ra >= L0) continue;
        const int kk = (c + K / 2) & (K - 1), kr = (K - kk) & (K - 1);
        C A, B;
        split_two_real(out[s * F::stride(1) + F::pad(kk)], out[s * F::stride(1) + F::pad(kr)], A, B);
        C *dst = tmp + (int64_t)c * L0 + ra;   // ra and L0 even: rb < L0, 16-byte aligned pair
        if constexpr (sizeof(R) == 4) {
            *reinterpret_cast<float4 *>(dst) = make_float4(A.x, A.y, B.x, B.y);
        } else {
            dst[0] = A;
            dst[1] = B;
        }
    }
}

// The same for the mixed-radix core (any even K).
template <typename R>
__device__ __forceinline__ void load_two_real_any(const cplx_t<R> *__restrict__ tmp, int row0, int L0, int K,
                                                  int nseq, cplx_t<R> *buf) {
    using C = cplx_t<R>;
    const int H = K / 2 + 1;
    for (int s = 0; s < nseq; ++s) {
        const int ra = row0 + 2 * s, rb = ra + 1;
#pragma unroll 4
        for (int k = threadIdx.x; k < H; k += NTR) {
            const int kr = k == 0 ? 0 : K - k, ck = wrapK(k + K / 2, K), ckr = wrapK(kr + K / 2, K);
            C xa{0, 0}, xar{0, 0}, xb{0, 0}, xbr{0, 0};
            if (ra < L0) {
                xa = tmp[(int64_t)ra * K + ck];
                xar = tmp[(int64_t)ra * K + ckr];
            }
            if (rb < L0) {
                xb = tmp[(int64_t)rb * K + ck];
                xbr = tmp[(int64_t)rb * K + ckr];
            }
            C y, yr;
            pack_two_real(xa, xar, xb, xbr, y, yr);
            buf[mplace<false>(s, k, K, 0)] = cconj(y);
            buf[mplace<false>(s, kr, K, 0)] = cconj(yr);
        }
    }
}
// The spectra of rows row0 + s, s < nseq, one to a sequence, conjugated and in
// natural order, so that the real parts of the forward FFT are those of the
// inverse.  The operator's inverse rows go this way: a row's own transform has
// half of its rounding in the imaginary part, which is dropped, where a pair's
// has the other row there (adjoint at 960 x 400, error against 64 bits: 1.55e-7
// in pairs, 1.32e-7 by single rows; 78 and 81 us).  The iteration's fused pass
// keeps pairs: its images are as close either way (1.08e-7 at 160^2, 1.04e-7 at
// 240^2) and 144 x 80 takes 61 us an iteration against 65.
template <typename R>
__device__ __forceinline__ void load_rows_inverse(const cplx_t<R> *__restrict__ tmp, int row0, int L0, int K, int nseq,
                                                  cplx_t<R> *buf) {
    for (int s = 0; s < nseq; ++s) {
        const int r = row0 + s;
#pragma unroll 4
        for (int c = threadIdx.x; c < K; c += NTR)   // column c holds frequency (c + K/2) mod K
            buf[mplace<false>(s, wrapK(c + K / 2, K), K, 0)] =
                r < L0 ? cconj(tmp[(int64_t)r * K + c]) : cplx_t<R>{0, 0};
    }
}
template <typename R>
__device__ __forceinline__ void store_two_real_any(const cplx_t<R> *out, int row0, int L0, int K, int nseq,
                                                   const uint8_t *__restrict__ colmask, cplx_t<R> *__restrict__ tmp) {
    using C = cplx_t<R>;
    for (int s = 0; s < nseq; ++s) {
        const int ra = row0 + 2 * s;
        if (ra >= L0) break;
#pragma unroll 4
        for (int c = threadIdx.x; c < K; c += NTR) {
            if (!colmask[c]) continue;
            const int kk = wrapK(c + K / 2, K), kr = kk == 0 ? 0 : K - kk;
            C A, B;
            split_two_real(out[mplace<false>(s, kk, K, 0)], out[mplace<false>(s, kr, K, 0)], A, B);
            C *dst = tmp + (int64_t)c * L0 + ra;   // ra and L0 even: rb < L0, 16-byte aligned pair
            if constexpr (sizeof(R) == 4) {
                *reinterpret_cast<float4 *>(dst) = make_float4(A.x, A.y, B.x, B.y);
            } else {
                dst[0] = A;
                dst[1] = B;
            }
        }
    }
}

// forward row pass: tmp[n0][c] = FFT_axis1(Z x)[n0][(c + K1/2) mod K1],
// tmp column-major (element (n0, c) at c L0 + n0) for the column pass
template <typename R, int KT>
__global__ void __launch_bounds__(row_nt<R, KT>(), pass_ctas<R, KT>()) k_rows_fwd(const R *__restrict__ x, cplx_t<R> *__restrict__ tmp,
                                                 const cplx_t<R> *__restrict__ tw, const R *__restrict__ s0,
                                                 const R *__restrict__ s1, int L0, int L1,
                                                 const uint8_t *__restrict__ colmask, PassArgs pa) {
    using C = cplx_t<R>;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    C *buf = reinterpret_cast<C *>(smem_raw);
    pdl_enter();
    if constexpr (KT != 0) {   // two rows per sequence
        constexpr int K = KT ? KT : 32;
        using F = RowFft<R, K>;
        constexpr int B = row_seqs<R, K>(), NTH = row_nt<R, K>(), LT = K / 2;
        const int row0 = blockIdx.x * 2 * B, s = threadIdx.x / F::TPS, t = threadIdx.x % F::TPS;
        const int ra = row0 + 2 * s, rb = ra + 1;
        const R fa = ra < L0 ? s0[ra] : R(0), fb = rb < L0 ? s0[rb] : R(0);
        C *mine = buf + s * F::stride(1);
        fft_run<F, false>(mine, t, tw,
            [&](int m) {   // position p: pixel p + L1/2 (p < L1/2) or p - K + L1/2 (p >= K - L1/2), else padding
                if (m >= F::EPT / 4 && m < 3 * F::EPT / 4) return C{0, 0};
                const int n1 = (t + m * F::TPS + LT / 2) & (K - 1);
                R va = 0, vb = 0;
                if (ra < L0) va = fa * s1[n1] * x[(int64_t)ra * LT + n1];
                if (rb < L0) vb = fb * s1[n1] * x[(int64_t)rb * LT + n1];
                return C{va, vb};
            },
            [&](int m, C v) { mine[F::pad(t + m * F::TPS)] = v; });
        __syncthreads();
        store_two_real_forward<R, K, B, NTH>(buf, row0, L0, colmask, tmp);
        return;
    }
    const int K = pa.pl.K, B = pa.nseq, row0 = blockIdx.x * 2 * B;
    C *buf2 = buf + B * mpad(K);
    // one pass over the padded rows: position p holds pixel p + L1/2 (p <
    // L1/2) or p - K + L1/2 (p >= K - L1/2), zero in between
    for (int s = 0; s < B; ++s) {
        const int ra = row0 + 2 * s, rb = ra + 1;
        const R fa = ra < L0 ? s0[ra] : R(0), fb = rb < L0 ? s0[rb] : R(0);
        for (int p = threadIdx.x; p < K; p += NTR) {
            const int n1 = p < L1 / 2 ? p + L1 / 2 : (p >= K - L1 / 2 ? p - K + L1 / 2 : -1);
            R va = 0, vb = 0;
            if (n1 >= 0 && ra < L0) va = fa * s1[n1] * x[(int64_t)ra * L1 + n1];
            if (n1 >= 0 && rb < L0) vb = fb * s1[n1] * x[(int64_t)rb * L1 + n1];
            buf[mplace<false>(s, p, K, 0)] = C{va, vb};
        }
    }
    __syncthreads();
    const C *out = fft_any<R, NTR, false>(buf, buf2, B, 0, pa.pl, tw);
    store_two_real_any<R>(out, row0, L0, K, B, colmask, tmp);
}

// forward column pass: grid[r][c] = FFT_axis0(tmp padded)[(r + K0/2) mod K0][c]
template <typename R, int KT>
__global__ void __launch_bounds__(col_nt<R, KT>()) k_cols_fwd(const cplx_t<R> *__restrict__ tmp,
                                                 cplx_t<R> *__restrict__ grid, const cplx_t<R> *__restrict__ tw,
                                                 int L0, int K1, const int32_t *__restrict__ strips,
                                                 const uint8_t *__restrict__ rowmask, PassArgs pa) {
    using C = cplx_t<R>;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    C *buf = reinterpret_cast<C *>(smem_raw);
    pdl_enter();
    const int c0 = strips[blockIdx.x];
    if constexpr (KT != 0) {
        constexpr int K = KT ? KT : 32, LT = K / 2;
        using F = ColFft<R, K>;
        constexpr int W = col_width<R, K>();
        const int s = threadIdx.x % W, t = threadIdx.x / W;
        const C *col = tmp + (int64_t)(c0 + s) * LT;
        fft_run<F, false>(buf + s * F::stride(W), t, tw,
            [&](int m) {   // position p: image row p + L0/2 (p < L0/2) or p - K + L0/2 (p >= K - L0/2), else padding
                if (m >= F::EPT / 4 && m < 3 * F::EPT / 4) return C{0, 0};
                return col[(t + m * F::TPS + LT / 2) & (K - 1)];
            },
            [&](int m, C v) {
                const int r = (t + m * F::TPS + K / 2) & (K - 1);
                if (rowmask[r]) grid[(int64_t)r * K1 + c0 + s] = v;
            });
        return;
    }
    const int K = pa.pl.K, W = pa.nseq, lw = pa.lseq;
    C *buf2 = buf + W * mpad(K);
    // one pass over the padded strip: position p holds image row p + L0/2
    // (p < L0/2) or p - K + L0/2 (p >= K - L0/2), zero in between; the
    // column-major tmp makes consecutive threads read consecutive rows
    for (int s = 0; s < W; ++s)
        for (int p = threadIdx.x; p < K; p += NTC) {
            const int n0 = p < L0 / 2 ? p + L0 / 2 : (p >= K - L0 / 2 ? p - K + L0 / 2 : -1);
            buf[mplace<true>(s, p, K, lw)] = n0 >= 0 ? tmp[(int64_t)(c0 + s) * L0 + n0] : C{0, 0};
        }
    __syncthreads();
    const C *out = fft_any<R, NTC, true>(buf, buf2, W, lw, pa.pl, tw);
    for (int e = threadIdx.x; e < W * K; e += NTC) {
        const int r = e >> lw, s = e - (r << lw);
        if (rowmask[r]) grid[(int64_t)r * K1 + c0 + s] = out[mplace<true>(s, wrapK(r + K / 2, K), K, lw)];
    }
}

// inverse column pass: tmp[n0][c] = (F^H along axis 0 of grid)[(n0 - L0/2) mod K0][c],
// the grid column-major (element (r, c) at c K0 + r, written by the combine
// pass), so that consecutive threads read consecutive rows
template <typename R, int KT>
__global__ void __launch_bounds__(col_nt<R, KT>()) k_cols_inv(const cplx_t<R> *__restrict__ grid,
                                                 cplx_t<R> *__restrict__ tmp, const cplx_t<R> *__restrict__ tw,
                                                 int L0, int K1, const int32_t *__restrict__ strips,
                                                 const uint8_t *__restrict__ rowmask, PassArgs pa) {
    using C = cplx_t<R>;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    C *buf = reinterpret_cast<C *>(smem_raw);
    pdl_enter();
    const int c0 = strips[blockIdx.x];
    if constexpr (KT != 0) {
        constexpr int K = KT ? KT : 32, LT = K / 2;
        using F = ColFft<R, K>;
        constexpr int W = col_width<R, K>();
        const int s = threadIdx.x % W, t = threadIdx.x / W;
        const C *col = grid + (int64_t)(c0 + s) * K;
        fft_run<F, false>(buf + s * F::stride(W), t, tw,
            [&](int m) {   // natural frequency k is stored (centred) in row (k + K/2) mod K
                const int r = (t + m * F::TPS + K / 2) & (K - 1);
                return rowmask[r] ? cconj(col[r]) : C{0, 0};
            },
            [&](int m, C v) {
                if (m >= F::EPT / 4 && m < 3 * F::EPT / 4) return;   // cropped
                const int n0 = (t + m * F::TPS + LT / 2) & (K - 1);
                tmp[(int64_t)n0 * K1 + c0 + s] = cconj(v);
            });
        return;
    }
    const int K = pa.pl.K, W = pa.nseq, lw = pa.lseq;
    C *buf2 = buf + W * mpad(K);
    for (int s = 0; s < W; ++s)
        for (int r = threadIdx.x; r < K; r += NTC)   // r: stored (centred) row; natural frequency (r + K/2) mod K
            buf[mplace<true>(s, wrapK(r + K / 2, K), K, lw)] =
                rowmask[r] ? cconj(grid[(int64_t)(c0 + s) * K + r]) : C{0, 0};
    __syncthreads();
    const C *out = fft_any<R, NTC, true>(buf, buf2, W, lw, pa.pl, tw);
    for (int e = threadIdx.x; e < W * L0; e += NTC) {
        const int n0 = e >> lw, s = e - (n0 << lw);
        tmp[(int64_t)n0 * K1 + c0 + s] = cconj(out[mplace<true>(s, wrapK(n0 - L0 / 2 + K, K), K, lw)]);
    }
}

// inverse row pass: img[n0][n1] = s0 s1 Re(F^H along axis 1 of tmp)[n0][(n1 - L1/2) mod K1]
template <typename R, int KT>
__global__ void __launch_bounds__(row_nt<R, KT>(), pass_ctas<R, KT>()) k_rows_inv(const cplx_t<R> *__restrict__ tmp, R *__restrict__ img,
                                                 const cplx_t<R> *__restrict__ tw, const R *__restrict__ s0,
                                                 const R *__restrict__ s1, int L0, int L1, PassArgs pa) {
    using C = cplx_t<R>;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    C *buf = reinterpret_cast<C *>(smem_raw);
    pdl_enter();
    if constexpr (KT != 0) {   // two rows per sequence
        constexpr int K = KT ? KT : 32;
        using F = RowFft<R, K>;
        constexpr int B = row_seqs<R, K>(), NTH = row_nt<R, K>(), LT = K / 2;
        const int row0 = blockIdx.x * 2 * B, s = threadIdx.x / F::TPS, t = threadIdx.x % F::TPS;
        const int ra = row0 + 2 * s, rb = ra + 1;
        load_two_real_inverse<R, K, B, NTH>(tmp, row0, L0, buf);
        __syncthreads();
        const R fa = ra < L0 ? s0[ra] : R(0), fb = rb < L0 ? s0[rb] : R(0);
        C *mine = buf + s * F::stride(1);
        fft_run<F, true>(mine, t, tw, [&](int m) { return mine[F::pad(t + m * F::TPS)]; },
            [&](int m, C v) {
                if (m >= F::EPT / 4 && m < 3 * F::EPT / 4) return;   // cropped
                const int n1 = (t + m * F::TPS + LT / 2) & (K - 1);
                if (ra < L0) img[(int64_t)ra * LT + n1] = fa * s1[n1] * v.x;
                if (rb < L0) img[(int64_t)rb * LT + n1] = -fb * s1[n1] * v.y;
            });
        return;
    }
    const int K = pa.pl.K, B = pa.nseq, row0 = blockIdx.x * B;
    C *buf2 = buf + B * mpad(K);
    load_rows_inverse<R>(tmp, row0, L0, K, B, buf);
    __syncthreads();
    const C *out = fft_any<R, NTR, false>(buf, buf2, B, 0, pa.pl, tw);
    for (int s = 0; s < B && row0 + s < L0; ++s) {
        const R f = s0[row0 + s];
        for (int n1 = threadIdx.x; n1 < L1; n1 += NTR)
            img[(int64_t)(row0 + s) * L1 + n1] =
                f * s1[n1] * out[mplace<false>(s, wrapK(n1 - L1 / 2 + K, K), K, 0)].x;
    }
}

// The end of one PPD iteration and the start of the next, B rows per CTA:
// the inverse row pass g = s0 s1 Re(F^H along axis 1 of tmp_inv) (the rows'
// Phi^dagger v, kept on chip), the primal step of Algorithm 3 on those
// pixels (primal_pixel), and the forward row pass of the new xt into
// tmp_fwd (the next iteration's first FFT pass), with the FP64 statistics
// partials of the CTA.  The join of the prior branch precedes it (ut, u0).
template <typename R, int KT>
__global__ void __launch_bounds__(row_nt<R, KT>(), pass_ctas<R, KT>()) k_rows_primal(const cplx_t<R> *__restrict__ tmp_inv,
                                                    cplx_t<R> *__restrict__ tmp_fwd, const cplx_t<R> *__restrict__ tw,
                                                    const R *__restrict__ s0, const R *__restrict__ s1,
                                                    const uint8_t *__restrict__ colmask, PrimalArgs<R> P,
                                                    double *__restrict__ part, int L0, int L1, PassArgs pa) {
    using C = cplx_t<R>;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    C *buf = reinterpret_cast<C *>(smem_raw);
    pdl_enter();
    PrimalSums<R> acc;
    if constexpr (KT != 0) {
        // two rows per sequence (rows row0 + 2s and row0 + 2s + 1); the
        // positions a thread gets from the inverse transform are the ones it
        // gives to the forward one, so the primal step runs on registers
        constexpr int K = KT ? KT : 32;
        using F = RowFft<R, K>;
        constexpr int B = row_seqs<R, K>(), NTH = row_nt<R, K>(), LT = K / 2, EPT = F::EPT, NP = EPT / 2;
        const int row0 = blockIdx.x * 2 * B, s = threadIdx.x / F::TPS, t = threadIdx.x % F::TPS;
        const int ra = row0 + 2 * s, rb = ra + 1;
        // pixel of the i-th position inside the image (i < NP)
        auto pixel = [&](int i) { return (t + (i < NP / 2 ? i : i + NP) * F::TPS + LT / 2) & (K - 1); };
        load_two_real_inverse<R, K, B, NTH>(tmp_inv, row0, L0, buf);
        // the primal step's pixel inputs, in flight during the inverse FFT
        // (up to K = 1024; longer rows have too many CTAs for the registers)
        constexpr bool PRE = K <= 1024;
        PrimalIn<R> ina[PRE ? NP : 1], inb[PRE ? NP : 1];
        if constexpr (PRE) {
#pragma unroll
            for (int i = 0; i < NP; ++i) {
                if (ra < L0) ina[i] = primal_load(P, (int64_t)ra * LT + pixel(i));
                if (rb < L0) inb[i] = primal_load(P, (int64_t)rb * LT + pixel(i));
            }
        }
        __syncthreads();
        const R fa = ra < L0 ? s0[ra] : R(0), fb = rb < L0 ? s0[rb] : R(0);
        C *mine = buf + s * F::stride(1);
        C z[NP];   // conj(F^H Y) there, then the new a + i b
        fft_run<F, true>(mine, t, tw, [&](int m) { return mine[F::pad(t + m * F::TPS)]; },
            [&](int m, C v) {
                if (m < EPT / 4) z[m] = v;
                else if (m >= 3 * EPT / 4) z[m - NP] = v;
            });
#pragma unroll
        for (int i = 0; i < NP; ++i) {
            const int n1 = pixel(i);
            const R f1 = s1[n1];
            const int64_t ea = (int64_t)ra * LT + n1, eb = (int64_t)rb * LT + n1;
            R xa = 0, xb = 0;
            if (ra < L0) xa = primal_pixel(P, ea, fa * f1 * z[i].x, PRE ? ina[PRE ? i : 0] : primal_load(P, ea), acc);
            if (rb < L0) xb = primal_pixel(P, eb, -fb * f1 * z[i].y, PRE ? inb[PRE ? i : 0] : primal_load(P, eb), acc);
            z[i] = C{fa * f1 * xa, fb * f1 * xb};
        }
        __syncthreads();   // the last pass's inputs are read
        fft_run<F, false>(mine, t, tw,
            [&](int m) { return m < EPT / 4 ? z[m] : m >= 3 * EPT / 4 ? z[m - NP] : C{0, 0}; },
            [&](int m, C v) { mine[F::pad(t + m * F::TPS)] = v; });
        __syncthreads();
        store_two_real_forward<R, K, B, NTH>(buf, row0, L0, colmask, tmp_fwd);
        acc.template write<NTH>(part + 3 * (int64_t)blockIdx.x);
        return;
    }
    const int K = pa.pl.K, B = pa.nseq, row0 = blockIdx.x * 2 * B;
    C *buf2 = buf + B * mpad(K);
    load_two_real_any<R>(tmp_inv, row0, L0, K, B, buf);
    __syncthreads();
    C *out = fft_any<R, NTR, false>(buf, buf2, B, 0, pa.pl, tw);
    // the result is in one buffer, the forward input is built in the other
    C *fin = out == buf ? buf2 : buf;
    for (int s = 0; s < B; ++s) {
        const int ra = row0 + 2 * s, rb = ra + 1;
        const R fa = ra < L0 ? s0[ra] : R(0), fb = rb < L0 ? s0[rb] : R(0);
        for (int n1 = threadIdx.x; n1 < L1; n1 += NTR) {
            // the pixel's position, and the padding position K/2 = L1 from it
            const int pos = wrapK(n1 - L1 / 2 + K, K), at = mplace<false>(s, pos, K, 0);
            const C v = out[at];
            const int64_t ea = (int64_t)ra * L1 + n1, eb = ea + L1;
            R xa = 0, xb = 0;
            if (ra < L0) xa = primal_pixel(P, ea, fa * s1[n1] * v.x, acc);
            if (rb < L0) xb = primal_pixel(P, eb, -fb * s1[n1] * v.y, acc);
            fin[at] = C{fa * s1[n1] * xa, fb * s1[n1] * xb};
            fin[mplace<false>(s, wrapK(pos + L1, K), K, 0)] = C{0, 0};
        }
    }
    __syncthreads();
    const C *res = fft_any<R, NTR, false>(fin, out, B, 0, pa.pl, tw);
    store_two_real_any<R>(res, row0, L0, K, B, colmask, tmp_fwd);
    acc.template write<NTR>(part + 3 * (int64_t)blockIdx.x);
}

// ------------------------------------------------------------ launchers
// Sequences per CTA of the mixed-radix passes: rows (pairs): enough for
// ~1024 points; columns: one 32-byte sector per row (4 FP32, 2 FP64) while a
// CTA's two buffers stay within ~90 KB, so powers of two up to 4, which
// divide K1, a multiple of 32.
int any_rows(int K) { return std::max(1, 1024 / K); }
int any_cols(int K, bool fp64) {
    int w = fp64 ? 2 : 4;
    while (w > 1 && w * K * (fp64 ? 2 : 1) > 5400) w /= 2;
    return w;
}
int log2_of(int w) { return w >= 4 ? 2 : w >= 2 ? 1 : 0; }

// Row passes have the row length K1, column passes the column length K0.
// RowPass / ColPass hold the launches of one core (KT) and precision.
template <typename R, int KT> struct RowPass {
    static constexpr int NTH = row_nt<R, KT>();
    static int nseq(const ppd_ctx *c) {   // sequences per CTA
        if constexpr (KT != 0) return row_seqs<R, KT>();
        else return any_rows(c->K1);
    }
    static size_t smem(const ppd_ctx *c) {
        if constexpr (KT != 0) return (size_t)nseq(c) * RowFft<R, KT>::stride(1) * 2 * sizeof(R);
        else return (size_t)2 * nseq(c) * mpad(c->K1) * 2 * sizeof(R);
    }
    static PassArgs args(const ppd_ctx *c) { return PassArgs{c->plan1, nseq(c), 0}; }
    static int rows(const ppd_ctx *c) { return 2 * nseq(c); }   // rows per CTA: two per sequence
    static unsigned blocks(const ppd_ctx *c) { return (unsigned)((c->L0 + rows(c) - 1) / rows(c)); }
    static const cplx_t<R> *tw(const ppd_ctx *c) {
        return static_cast<const cplx_t<R> *>(KT ? c->twst1 : c->tw1);
    }
    static int fwd(ppd_ctx *c, const R *x, cudaStream_t s) {
        const int sh = (int)smem(c);
        PPD_CHECK(smem_attr((const void *)k_rows_fwd<R, KT>, sh));
        int site;
        PPD_CHECK(launch_begin(c, "fft_fwd_rows", s, &site));
        // mostly the first kernel of its sequence: an ordinary launch
        launch(c, false, k_rows_fwd<R, KT>, blocks(c), NTH, sh, s, x, static_cast<cplx_t<R> *>(c->fft_tmp), tw(c),
               static_cast<const R *>(c->deap0), static_cast<const R *>(c->deap1), c->L0, c->L1,
               (const uint8_t *)c->col_fwd, args(c));
        return launch_end(c, site, s);
    }
    static int inv(ppd_ctx *c, R *img, cudaStream_t s) {
        const int sh = (int)smem(c);
        PPD_CHECK(smem_attr((const void *)k_rows_inv<R, KT>, sh));
        int site;
        PPD_CHECK(launch_begin(c, "fft_inv_rows", s, &site));
        // (the mixed-radix core inverts single rows)
        const unsigned n = KT ? blocks(c) : (unsigned)((c->L0 + nseq(c) - 1) / nseq(c));
        launch(c, true, k_rows_inv<R, KT>, n, NTH, sh, s, static_cast<const cplx_t<R> *>(c->fft_tmp_inv),
               img, tw(c), static_cast<const R *>(c->deap0), static_cast<const R *>(c->deap1), c->L0, c->L1,
               args(c));
        return launch_end(c, site, s);
    }
    static int primal(ppd_ctx *c, cudaStream_t s) {
        const int sh = (int)smem(c);
        PPD_CHECK(smem_attr((const void *)k_rows_primal<R, KT>, sh));
        int site;
        PPD_CHECK(launch_begin(c, "rows_primal", s, &site));
        const unsigned n = blocks(c);
        // it follows the join of the two branches: an ordinary launch
        launch(c, false, k_rows_primal<R, KT>, n, NTH, sh, s, static_cast<const cplx_t<R> *>(c->fft_tmp_inv),
               static_cast<cplx_t<R> *>(c->fft_tmp), tw(c), static_cast<const R *>(c->deap0),
               static_cast<const R *>(c->deap1), (const uint8_t *)c->col_fwd, primal_args<R>(c), c->prim_part, c->L0,
               c->L1, args(c));
        c->n_stat_parts = (int)n;
        return launch_end(c, site, s);
    }
};

template <typename R, int KT> struct ColPass {
    static constexpr int NTH = col_nt<R, KT>();
    static int nseq(const ppd_ctx *c) {   // columns per CTA
        if constexpr (KT != 0) return col_width<R, KT>();
        else return any_cols(c->K0, sizeof(R) == 8);
    }
    static size_t smem(const ppd_ctx *c) {
        if constexpr (KT != 0) return (size_t)nseq(c) * ColFft<R, KT>::stride(nseq(c)) * 2 * sizeof(R);
        else return (size_t)2 * nseq(c) * mpad(c->K0) * 2 * sizeof(R);
    }
    static PassArgs args(const ppd_ctx *c) { return PassArgs{c->plan0, nseq(c), log2_of(nseq(c))}; }
    static const cplx_t<R> *tw(const ppd_ctx *c) {
        return static_cast<const cplx_t<R> *>(KT ? c->twst0 : c->tw0);
    }
    static int fwd(ppd_ctx *c, cplx_t<R> *grid, cudaStream_t s) {
        if (c->n_fwd_strips == 0) return PPD_OK;
        const int sh = (int)smem(c);
        PPD_CHECK(smem_attr((const void *)k_cols_fwd<R, KT>, sh));
        int site;
        PPD_CHECK(launch_begin(c, "fft_fwd_cols", s, &site));
        launch(c, true, k_cols_fwd<R, KT>, (unsigned)c->n_fwd_strips, NTH, sh, s,
               static_cast<const cplx_t<R> *>(c->fft_tmp), grid, tw(c), c->L0, c->K1,
               (const int32_t *)c->fwd_strips, (const uint8_t *)c->row_fwd, args(c));
        return launch_end(c, site, s);
    }
    static int inv(ppd_ctx *c, const cplx_t<R> *grid, cudaStream_t s) {
        if (c->n_inv_strips == 0) return PPD_OK;
        const int sh = (int)smem(c);
        PPD_CHECK(smem_attr((const void *)k_cols_inv<R, KT>, sh));
        int site;
        PPD_CHECK(launch_begin(c, "fft_inv_cols", s, &site));
        launch(c, true, k_cols_inv<R, KT>, (unsigned)c->n_inv_strips, NTH, sh, s, grid,
               static_cast<cplx_t<R> *>(c->fft_tmp_inv), tw(c), c->L0, c->K1, (const int32_t *)c->inv_strips,
               (const uint8_t *)c->row_inv, args(c));
        return launch_end(c, site, s);
    }
};

}  // namespace

// Power-of-two lengths take the compile-time core; other 5-smooth lengths
// the mixed-radix one (KT = 0).
#define PPD_FFT_DISPATCH(KLEN, PASS, CALL)                  \
    switch (KLEN) {                                         \
        case 32: return PASS<R, 32>::CALL;                  \
        case 64: return PASS<R, 64>::CALL;                  \
        case 128: return PASS<R, 128>::CALL;                \
        case 256: return PASS<R, 256>::CALL;                \
        case 512: return PASS<R, 512>::CALL;                \
        case 1024: return PASS<R, 1024>::CALL;              \
        case 2048: return PASS<R, 2048>::CALL;              \
        case 4096: return PASS<R, 4096>::CALL;              \
        case 8192: return PASS<R, 8192>::CALL;              \
        default: return PASS<R, 0>::CALL;                   \
    }

// forward row pass of x into the FFT temporary (first half of F Z x)
template <typename R> int fft_forward_rows(ppd_ctx *c, const R *x, cudaStream_t s) {
    c->xt_rows_valid = false;
    PPD_FFT_DISPATCH(c->K1, RowPass, fwd(c, x, s))
}

// forward column pass from the FFT temporary to the grid (second half of F Z x)
template <typename R> int fft_forward_cols(ppd_ctx *c, cplx_t<R> *grid, cudaStream_t s) {
    PPD_FFT_DISPATCH(c->K0, ColPass, fwd(c, grid, s))
}

// inverse column pass of a combined grid into the inverse temporary
template <typename R> int fft_inverse_cols(ppd_ctx *c, const cplx_t<R> *grid, cudaStream_t s) {
    PPD_FFT_DISPATCH(c->K0, ColPass, inv(c, grid, s))
}

// inverse row pass into an image (second half of Z^T F^H)
template <typename R> int fft_inverse_rows(ppd_ctx *c, R *img, cudaStream_t s) {
    PPD_FFT_DISPATCH(c->K1, RowPass, inv(c, img, s))
}

// inverse row pass + primal step + forward row pass of the new xt
template <typename R> int rows_primal(ppd_ctx *c, cudaStream_t s) {
    PPD_FFT_DISPATCH(c->K1, RowPass, primal(c, s))
}

template <typename R> int fft_forward(ppd_ctx *c, const R *x, cplx_t<R> *grid, cudaStream_t s) {
    PPD_CHECK(fft_forward_rows<R>(c, x, s));
    return fft_forward_cols<R>(c, grid, s);
}

template <typename R> int fft_inverse(ppd_ctx *c, const cplx_t<R> *grid, R *img, cudaStream_t s) {
    PPD_CHECK(fft_inverse_cols<R>(c, grid, s));
    return fft_inverse_rows<R>(c, img, s);
}

#undef PPD_FFT_DISPATCH

#define PPD_FFT_INST(R)                                                                                         \
    template int fft_forward<R>(ppd_ctx *, const R *, cplx_t<R> *, cudaStream_t);                              \
    template int fft_inverse<R>(ppd_ctx *, const cplx_t<R> *, R *, cudaStream_t);                              \
    template int fft_forward_rows<R>(ppd_ctx *, const R *, cudaStream_t);                                       \
    template int fft_forward_cols<R>(ppd_ctx *, cplx_t<R> *, cudaStream_t);                                     \
    template int fft_inverse_cols<R>(ppd_ctx *, const cplx_t<R> *, cudaStream_t);                              \
    template int fft_inverse_rows<R>(ppd_ctx *, R *, cudaStream_t);                                             \
    template int rows_primal<R>(ppd_ctx *, cudaStream_t);
PPD_FFT_INST(float)
PPD_FFT_INST(double)
#undef PPD_FFT_INST

// Fewest stages for `left` points with radices up to `most`; of those the
// smallest sum of radices (r: the current choice, best: the result).
static void fewest_stages(int left, int most, std::vector<int> &r, std::vector<int> &best) {
    if (left == 1) {
        auto sum = [](const std::vector<int> &v) {
            int t = 0;
            for (int x : v) t += x;
            return t;
        };
        if (best.empty() || r.size() < best.size() || (r.size() == best.size() && sum(r) < sum(best))) best = r;
        return;
    }
    if (!best.empty() && r.size() >= best.size()) return;
    for (int k : {16, 12, 10, 8, 6, 5, 4, 3, 2})
        if (k <= most && left % k == 0) {
            r.push_back(k);
            fewest_stages(left / k, k, r, best);
            r.pop_back();
        }
}

// FFT plan of length K (an empty plan if K has a prime factor above 5).
FftPlan make_fft_plan(int K) {
    FftPlan p{};
    p.K = K;
    int k = K;
    for (int f : {2, 3, 5})
        while (k % f == 0) k /= f;
    if (K < 2 || k != 1) return p;
    std::vector<int> r, best;
    fewest_stages(K, 16, r, best);
    if ((int)best.size() > FftPlan::MAX_STAGES) return p;
    int Ns = 1;
    for (int rad : best) {
        p.rad[p.ns] = rad;
        p.tstep[p.ns] = K / (Ns * rad);
        // reciprocals of fast_div (a divisor of 1 is never used)
        auto inv = [](int d) { return d > 1 ? (uint32_t)(((1ull << 32) + d - 1) / d) : 0u; };
        p.inv_ns[p.ns] = inv(Ns);
        p.inv_m[p.ns] = inv(K / rad);
        ++p.ns;
        Ns *= rad;
    }
    return p;
}

bool fft_length_supported(int K, bool fp64) {
    if (K < 32 || K > 8192 || make_fft_plan(K).ns == 0) return false;
    const bool pow2 = (K & (K - 1)) == 0;
    // two buffers of the mixed-radix core per CTA: at most 128 KB
    return pow2 || (size_t)2 * K * 2 * (fp64 ? 8 : 4) <= 128 * 1024;
}

// Column strips (W columns each, W as the column passes use) that contain a
// marked column, and the row / column masks, uploaded for the pruned passes.
int fft_plan_pruning(ppd_ctx *c, const std::vector<char> &rows_fwd, const std::vector<char> &cols_fwd,
                     const std::vector<char> &rows_inv, const std::vector<char> &cols_inv) {
    const int K0 = c->K0, K1 = c->K1;
    const bool p2 = (K0 & (K0 - 1)) == 0;
    const int W = !p2 ? any_cols(K0, !c->is_f32) : c->is_f32 ? col_width_of<float>(K0) : col_width_of<double>(K0);
    std::vector<int32_t> fs, is;
    for (int s0 = 0; s0 < K1; s0 += W) {
        bool f = false, i = false;
        for (int j = s0; j < s0 + W && j < K1; ++j) {
            f = f || cols_fwd[j];
            i = i || cols_inv[j];
        }
        if (f) fs.push_back(s0);
        if (i) is.push_back(s0);
    }
    std::vector<uint8_t> rf(rows_fwd.begin(), rows_fwd.end()), ri(rows_inv.begin(), rows_inv.end()),
        cf(cols_fwd.begin(), cols_fwd.end());
    c->n_fwd_strips = (int)fs.size();
    c->n_inv_strips = (int)is.size();
    if (!fs.empty()) PPD_CUDA(cudaMemcpy(c->fwd_strips, fs.data(), fs.size() * 4, cudaMemcpyHostToDevice));
    if (!is.empty()) PPD_CUDA(cudaMemcpy(c->inv_strips, is.data(), is.size() * 4, cudaMemcpyHostToDevice));
    PPD_CUDA(cudaMemcpy(c->row_fwd, rf.data(), K0, cudaMemcpyHostToDevice));
    PPD_CUDA(cudaMemcpy(c->row_inv, ri.data(), K0, cudaMemcpyHostToDevice));
    PPD_CUDA(cudaMemcpy(c->col_fwd, cf.data(), K1, cudaMemcpyHostToDevice));
    // the inverse column pass writes only its strips: the rest of its output
    // stays zero; the forward row pass writes only marked columns
    PPD_CUDA(cudaMemset(c->fft_tmp_inv, 0, (size_t)c->L0 * K1 * 2 * c->rsz));
    PPD_CUDA(cudaMemset(c->fft_tmp, 0, (size_t)c->L0 * K1 * 2 * c->rsz));
    return PPD_OK;
}

// Twiddles exp(-2 pi i m / K), m < K, computed in double on the host, for
// the column length K0 (tw0) and the row length K1 (tw1).
static int upload_twiddles(ppd_ctx *c, int K, void *dst) {
    std::vector<double> t(2 * (size_t)K);
    for (int m = 0; m < K; ++m) {
        double a = -2.0 * M_PI * (double)m / (double)K;
        t[2 * m] = std::cos(a);
        t[2 * m + 1] = std::sin(a);
    }
    if (c->is_f32) {
        std::vector<float> f(t.begin(), t.end());
        PPD_CUDA(cudaMemcpy(dst, f.data(), f.size() * sizeof(float), cudaMemcpyHostToDevice));
    } else {
        PPD_CUDA(cudaMemcpy(dst, t.data(), t.size() * sizeof(double), cudaMemcpyHostToDevice));
    }
    return PPD_OK;
}

// Twiddles of the power-of-two core pass by pass (K entries, zero padded):
// for each pass after the first, of span Ns and radix RAD, w^(q k K/(Ns RAD))
// at (q - 1) Ns + k, q = 1 .. RAD - 1, k < Ns: the lanes' consecutive k read
// consecutive words.
template <typename F> static std::vector<double> pass_twiddles() {
    constexpr int K = F::K;
    std::vector<double> t;
    t.reserve(2 * (size_t)K);
    for (int p = 1; p < F::PASSES; ++p) {
        const int Ns = F::span(p), rad = F::radix(p);
        for (int q = 1; q < rad; ++q)
            for (int k = 0; k < Ns; ++k) {
                const double a = -2.0 * M_PI * ((double)q * k / ((double)Ns * rad));
                t.push_back(std::cos(a));
                t.push_back(std::sin(a));
            }
    }
    t.resize(2 * (size_t)K, 0.0);
    return t;
}
template <typename R> static std::vector<double> pass_twiddles_of(int K, bool rows) {
    switch (K) {
        case 32: return rows ? pass_twiddles<RowFft<R, 32>>() : pass_twiddles<ColFft<R, 32>>();
        case 64: return rows ? pass_twiddles<RowFft<R, 64>>() : pass_twiddles<ColFft<R, 64>>();
        case 128: return rows ? pass_twiddles<RowFft<R, 128>>() : pass_twiddles<ColFft<R, 128>>();
        case 256: return rows ? pass_twiddles<RowFft<R, 256>>() : pass_twiddles<ColFft<R, 256>>();
        case 512: return rows ? pass_twiddles<RowFft<R, 512>>() : pass_twiddles<ColFft<R, 512>>();
        case 1024: return rows ? pass_twiddles<RowFft<R, 1024>>() : pass_twiddles<ColFft<R, 1024>>();
        case 2048: return rows ? pass_twiddles<RowFft<R, 2048>>() : pass_twiddles<ColFft<R, 2048>>();
        case 4096: return rows ? pass_twiddles<RowFft<R, 4096>>() : pass_twiddles<ColFft<R, 4096>>();
        case 8192: return rows ? pass_twiddles<RowFft<R, 8192>>() : pass_twiddles<ColFft<R, 8192>>();
        default: return std::vector<double>(2 * (size_t)K, 0.0);
    }
}
static int upload_stage_twiddles(ppd_ctx *c, int K, bool rows, void *dst) {
    if (c->is_f32) {
        const std::vector<double> t = pass_twiddles_of<float>(K, rows);
        const std::vector<float> f(t.begin(), t.end());
        PPD_CUDA(cudaMemcpy(dst, f.data(), f.size() * sizeof(float), cudaMemcpyHostToDevice));
    } else {
        const std::vector<double> t = pass_twiddles_of<double>(K, rows);
        PPD_CUDA(cudaMemcpy(dst, t.data(), t.size() * sizeof(double), cudaMemcpyHostToDevice));
    }
    return PPD_OK;
}

int make_twiddles(ppd_ctx *c) {
    c->plan0 = make_fft_plan(c->K0);
    c->plan1 = make_fft_plan(c->K1);
    PPD_CHECK(upload_twiddles(c, c->K0, c->tw0));
    PPD_CHECK(upload_twiddles(c, c->K1, c->tw1));
    PPD_CHECK(upload_stage_twiddles(c, c->K0, false, c->twst0));
    return upload_stage_twiddles(c, c->K1, true, c->twst1);
}

// Z's scaling s(n) = 1 / psi_hat((n - L/2)/K), psi_hat(f) = (J / I0(beta)) sinh(q)/q,
// q = sqrt(beta^2 - (pi J f)^2): the Fourier transform of the Kaiser-Bessel kernel.
static int upload_deapodisation(ppd_ctx *c, int L, int K, void *dst) {
    // 1/I0(beta) as the weights have it (make_kb_poly), so that its rounding cancels
    const double J = KB_J, beta = c->beta, inv_i0b = c->kb_inv_i0b;
    std::vector<double> s(L);
    for (int n = 0; n < L; ++n) {
        double f = ((double)n - L / 2) / (double)K;
        double q = std::sqrt(beta * beta - (M_PI * J * f) * (M_PI * J * f));
        s[n] = 1.0 / ((J * inv_i0b) * std::sinh(q) / q);
    }
    if (c->is_f32) {
        std::vector<float> f(s.begin(), s.end());
        PPD_CUDA(cudaMemcpy(dst, f.data(), L * sizeof(float), cudaMemcpyHostToDevice));
    } else {
        PPD_CUDA(cudaMemcpy(dst, s.data(), L * sizeof(double), cudaMemcpyHostToDevice));
    }
    return PPD_OK;
}

int make_deapodisation(ppd_ctx *c) {
    PPD_CHECK(upload_deapodisation(c, c->L0, c->K0, c->deap0));
    return upload_deapodisation(c, c->L1, c->K1, c->deap1);
}

}  // namespace ppd
