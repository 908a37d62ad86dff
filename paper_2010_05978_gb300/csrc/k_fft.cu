// Hand-written 2D FFT for the NUFFT fine grid: batched 1D mixed-radix Stockham
// transforms held in shared memory, one pass along rows (contiguous) and one
// along columns (a CTA takes several adjacent columns so global accesses stay
// coalesced).  Forward sign e^{-2 pi i k l / n}, unnormalised.
//
// The FFT is the middle step of the type-1 and type-3 NUFFTs used by the
// paper's fast algorithm (arXiv:2010.05978, Secs. 3.2-3.3; "under the hood the
// NUFFT uses FFTs", Sec. 4.1).  Both passes are pruned to what the path needs:
// the type-1 row pass keeps only the n1 wanted modes; the type-1 column pass
// keeps n2 modes and applies the fused output epilogue (deconvolution, target
// chirp, 1/(i lz), Babinet); the type-3 passes read only the nonzero central
// block of the zero-padded grid and fuse the inner type-2 deconvolution.
//
// Each Stockham stage with radix r and p = product of earlier radices maps
// butterfly i (k = i mod p) from inputs x[i + q n/r] (twiddled by
// w_{p r}^{q k}) to outputs y[(i - k) r + k + t p].  A thread keeps up
// to 16 values (FP64: 8): several butterflies of a small radix, read into registers
// before a barrier and written back in place after it, so one buffer per line
// is enough and the threads (64 registers) and lines resident at once cover
// the passes' grids in one wave.  These passes are short and bound by latency:
// fewer stages (radices up to 16 with the composite 15, 12, 10 and 9, which
// need no inner twiddles but 9's and 16's) and twiddles read consecutively from a table
// per stage matter more than operations, and so does the code a block
// runs once: in the FP32 single passes one body per radix serves every stage,
// with the pruning, factors and epilogue in the short loops that fill and empty
// the lines (fused into the first and last stages they made 33 KB of
// straight-line code, whose fetching took up to half of a pass: 29 against 19
// us cold for the star's 928 rows of 2048; rows of 256 and 640 points 2 us more).  The four-step passes are short
// transforms over gigabytes: there the code stays fetched, and they read and
// store in their first and last stages (17,280^2 points: 3.6 against 4.8 ms).
#include <algorithm>

#include "internal.cuh"

namespace fres {

namespace {

// Radices, and the butterflies of a radix that a thread keeps: 16 values in
// FP32; 8 in FP64 (9 and 10 for the radices 3 and 5, so that lines of up to
// 6,834 points need no more than 1024 threads whatever their factors; 16
// values and the larger radices save a quarter of FP64's twiddles, but leave
// a short line too few warps: 720 points 49 against 41 us).
constexpr int kRadicesF[] = {16, 15, 12, 10, 9, 8, 5, 4, 3, 2};
constexpr int kRadicesD[] = {8, 6, 5, 4, 3, 2};
__host__ __device__ constexpr int butterflies(int r, bool dbl) {
    return dbl ? (r == 3 ? 3 : (r == 5 ? 2 : 8 / r > 0 ? 8 / r : 1)) : 16 / r;
}

template <typename T> struct Ops {
    using C = cx_t<T>;
    static __device__ __forceinline__ C mk(T a, T b) { C c; c.x = a; c.y = b; return c; }
    static __device__ __forceinline__ C add(C a, C b) { return mk(a.x + b.x, a.y + b.y); }
    static __device__ __forceinline__ C sub(C a, C b) { return mk(a.x - b.x, a.y - b.y); }
    static __device__ __forceinline__ C mul(C a, C b) {
        return mk(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);
    }
    static __device__ __forceinline__ C scale(C a, T s) { return mk(a.x * s, a.y * s); }
    static __device__ __forceinline__ C mul_negi(C a) { return mk(a.y, -a.x); }   // -i a
};

// In-register DFTs y_t = sum_q u_q e^{-2 pi i q t / R}.  Radix 8 is two
// radix-4 halves joined by w_8^k; radix 16 is 4 x 4 with w_16^{n2 k1}
// twiddles between the two radix-4 layers (Cooley-Tukey in registers).
template <typename T, int R> struct Dft;
template <typename T> struct Dft<T, 2> {
    using C = cx_t<T>;
    static __device__ __forceinline__ void run(const C* u, C* y) {
        y[0] = Ops<T>::add(u[0], u[1]);
        y[1] = Ops<T>::sub(u[0], u[1]);
    }
};
template <typename T> struct Dft<T, 4> {
    using C = cx_t<T>;
    static __device__ __forceinline__ void run(const C* u, C* y) {
        using O = Ops<T>;
        C t0 = O::add(u[0], u[2]), t1 = O::sub(u[0], u[2]);
        C t2 = O::add(u[1], u[3]), t3 = O::mul_negi(O::sub(u[1], u[3]));
        y[0] = O::add(t0, t2);
        y[2] = O::sub(t0, t2);
        y[1] = O::add(t1, t3);
        y[3] = O::sub(t1, t3);
    }
};
template <typename T> struct Dft<T, 3> {
    using C = cx_t<T>;
    static __device__ __forceinline__ void run(const C* u, C* y) {
        using O = Ops<T>;
        const T c3 = (T)-0.5, s3 = (T)0.86602540378443864676372317075294;
        C s = O::add(u[1], u[2]), d = O::sub(u[1], u[2]);
        C a = O::add(u[0], O::scale(s, c3));
        C b = O::mul_negi(O::scale(d, s3));   // -i s3 (u1 - u2)
        y[0] = O::add(u[0], s);
        y[1] = O::add(a, b);
        y[2] = O::sub(a, b);
    }
};
template <typename T> struct Dft<T, 5> {
    using C = cx_t<T>;
    static __device__ __forceinline__ void run(const C* u, C* y) {
        using O = Ops<T>;
        const T c1 = (T)0.30901699437494742410229341718282;   // cos(2 pi/5)
        const T s1 = (T)0.95105651629515357211643933337938;   // sin(2 pi/5)
        const T c2 = (T)-0.80901699437494742410229341718282;  // cos(4 pi/5)
        const T s2 = (T)0.58778525229247312916870595463907;   // sin(4 pi/5)
        C a14 = O::add(u[1], u[4]), d14 = O::sub(u[1], u[4]);
        C a23 = O::add(u[2], u[3]), d23 = O::sub(u[2], u[3]);
        C r1 = O::add(u[0], O::add(O::scale(a14, c1), O::scale(a23, c2)));
        C r2 = O::add(u[0], O::add(O::scale(a14, c2), O::scale(a23, c1)));
        C i1 = O::mul_negi(O::add(O::scale(d14, s1), O::scale(d23, s2)));
        C i2 = O::mul_negi(O::sub(O::scale(d14, s2), O::scale(d23, s1)));
        y[0] = O::add(u[0], O::add(a14, a23));
        y[1] = O::add(r1, i1);
        y[4] = O::sub(r1, i1);
        y[2] = O::add(r2, i2);
        y[3] = O::sub(r2, i2);
    }
};
template <typename T> struct Dft<T, 8> {
    using C = cx_t<T>;
    static __device__ __forceinline__ void run(const C* u, C* y) {
        using O = Ops<T>;
        const T r = (T)0.70710678118654752440084436210485;   // 1/sqrt(2)
        C e[4] = {u[0], u[2], u[4], u[6]}, o[4] = {u[1], u[3], u[5], u[7]}, a[4], b[4];
        Dft<T, 4>::run(e, a);
        Dft<T, 4>::run(o, b);
        // w8^1 = (1 - i)/sqrt2, w8^2 = -i, w8^3 = -(1 + i)/sqrt2
        b[1] = O::mk(r * (b[1].x + b[1].y), r * (b[1].y - b[1].x));
        b[2] = O::mul_negi(b[2]);
        b[3] = O::mk(r * (b[3].y - b[3].x), -r * (b[3].x + b[3].y));
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            y[k] = O::add(a[k], b[k]);
            y[k + 4] = O::sub(a[k], b[k]);
        }
    }
};
template <typename T> struct Dft<T, 16> {
    using C = cx_t<T>;
    static __device__ __forceinline__ void run(const C* u, C* y) {
        using O = Ops<T>;
        // cos / sin of 2 pi j / 16, j = 0..9
        const T cs[10] = {(T)1, (T)0.92387953251128675612818318939679,
                          (T)0.70710678118654752440084436210485,
                          (T)0.38268343236508977172845998403040, (T)0,
                          (T)-0.38268343236508977172845998403040,
                          (T)-0.70710678118654752440084436210485,
                          (T)-0.92387953251128675612818318939679, (T)-1,
                          (T)-0.92387953251128675612818318939679};
        const T sn[10] = {(T)0, (T)0.38268343236508977172845998403040,
                          (T)0.70710678118654752440084436210485,
                          (T)0.92387953251128675612818318939679, (T)1,
                          (T)0.92387953251128675612818318939679,
                          (T)0.70710678118654752440084436210485,
                          (T)0.38268343236508977172845998403040, (T)0,
                          (T)-0.38268343236508977172845998403040};
        C A[4][4];
#pragma unroll
        for (int n2 = 0; n2 < 4; ++n2) {
            C v[4] = {u[n2], u[4 + n2], u[8 + n2], u[12 + n2]};
            Dft<T, 4>::run(v, A[n2]);
#pragma unroll
            for (int k1 = 1; k1 < 4; ++k1) {
                const int j = n2 * k1;
                if (j > 0) A[n2][k1] = O::mul(A[n2][k1], O::mk(cs[j], -sn[j]));
            }
        }
#pragma unroll
        for (int k1 = 0; k1 < 4; ++k1) {
            C v[4] = {A[0][k1], A[1][k1], A[2][k1], A[3][k1]}, d[4];
            Dft<T, 4>::run(v, d);
#pragma unroll
            for (int k2 = 0; k2 < 4; ++k2) y[k1 + 4 * k2] = d[k2];
        }
    }
};

// Coprime composites N = N1 N2 by the prime-factor map: input (N2 a + N1 b)
// mod N, output k at (k mod N1, k mod N2), no twiddles.
template <typename T, int N1, int N2> struct DftPfa {
    using C = cx_t<T>;
    static __device__ __forceinline__ void run(const C* u, C* y) {
        constexpr int N = N1 * N2;
        C A[N2][N1];
#pragma unroll
        for (int b = 0; b < N2; ++b) {
            C v[N1];
#pragma unroll
            for (int a = 0; a < N1; ++a) v[a] = u[(N2 * a + N1 * b) % N];
            Dft<T, N1>::run(v, A[b]);
        }
#pragma unroll
        for (int k1 = 0; k1 < N1; ++k1) {
            C v[N2], d[N2];
#pragma unroll
            for (int b = 0; b < N2; ++b) v[b] = A[b][k1];
            Dft<T, N2>::run(v, d);
#pragma unroll
            for (int k = 0; k < N; ++k)
                if (k % N1 == k1) y[k] = d[k % N2];
        }
    }
};
template <typename T> struct Dft<T, 6> : DftPfa<T, 2, 3> {};
template <typename T> struct Dft<T, 10> : DftPfa<T, 2, 5> {};
template <typename T> struct Dft<T, 12> : DftPfa<T, 4, 3> {};
template <typename T> struct Dft<T, 15> : DftPfa<T, 3, 5> {};
template <typename T> struct Dft<T, 9> {
    using C = cx_t<T>;
    static __device__ __forceinline__ void run(const C* u, C* y) {
        using O = Ops<T>;
        // cos / sin of 2 pi j / 9, j = 0..4 (j = n2 k1 takes 1, 2, 4)
        const T cs[5] = {(T)1, (T)0.76604444311897803520239265055542,
                         (T)0.17364817766693034885171662676931, (T)-0.5,
                         (T)-0.93969262078590838405410927732473};
        const T sn[5] = {(T)0, (T)0.64278760968653932632264340990726,
                         (T)0.98480775301220805936674302458952,
                         (T)0.86602540378443864676372317075294,
                         (T)0.34202014332566873304409961468226};
        C A[3][3];
#pragma unroll
        for (int n2 = 0; n2 < 3; ++n2) {
            C v[3] = {u[n2], u[3 + n2], u[6 + n2]};
            Dft<T, 3>::run(v, A[n2]);
#pragma unroll
            for (int k1 = 1; k1 < 3; ++k1)
                if (n2 > 0) A[n2][k1] = O::mul(A[n2][k1], O::mk(cs[n2 * k1], -sn[n2 * k1]));
        }
#pragma unroll
        for (int k1 = 0; k1 < 3; ++k1) {
            C v[3] = {A[0][k1], A[1][k1], A[2][k1]}, d[3];
            Dft<T, 3>::run(v, d);
#pragma unroll
            for (int k2 = 0; k2 < 3; ++k2) y[k1 + 3 * k2] = d[k2];
        }
    }
};

// Shared-memory element index with one padding slot per 16 elements, so the
// stride-R writes of the early Stockham stages spread over all banks.
__host__ __device__ __forceinline__ int pad(int e) { return e + (e >> 4); }
__host__ __device__ __forceinline__ int padded_len(int n) { return n + (n >> 4) + 1; }

// A thread's place: its line (c: offset of the line's element 0 in S, element
// e at c + (pad(e) << ls)) and its butterflies or elements t, t + tr, ...
struct Place {
    int c, t, tr, ls;
};

// The input side of a fused transform: load(e) reads natural input e, use(e,
// v) turns the value read into the value transformed.  Apart, so that a
// butterfly's loads are all in flight before a store that may alias them.
template <class L, class U>
struct Input {
    L l;
    U u;
    __device__ __forceinline__ auto load(int e) const { return l(e); }
    template <class C> __device__ __forceinline__ C use(int e, C v) const { return u(e, v); }
};
template <class L, class U> __device__ __forceinline__ Input<L, U> make_input(L l, U u) { return {l, u}; }
struct NoIo {
    template <class C> __device__ __forceinline__ void operator()(int, C) const {}
};

// One stage, in place: every butterfly of the line is read before any is
// written.  kStage: from S to S; kFirst: from `in` (p = 1) to S; kLast: from S
// to `out` (output i + t p of butterfly i).
enum { kStage = 0, kFirst = 1, kLast = 2 };
template <typename T, int R, int WHERE, class In, class Out>
__device__ __forceinline__ void stage(cx_t<T>* __restrict__ S, const Place pl, int nb, int p,
                                      unsigned pmagic, const cx_t<T>* __restrict__ tw, In& in,
                                      Out& out) {
    using O = Ops<T>;
    using C = cx_t<T>;
    constexpr int K = butterflies(R, sizeof(T) == 8);
    C u[K][R];
#pragma unroll
    for (int kk = 0; kk < K; ++kk) {
        const int i = pl.t + kk * pl.tr;
        if (i < nb) {
#pragma unroll
            for (int q = 0; q < R; ++q) {
                if constexpr (WHERE == kFirst) u[kk][q] = in.load(i + q * nb);
                else u[kk][q] = S[pl.c + (pad(i + q * nb) << pl.ls)];
            }
        } else {   // defined on every path: else a value carried round the stage loop, and spilled
#pragma unroll
            for (int q = 0; q < R; ++q) u[kk][q] = O::mk(0, 0);
        }
    }
    if constexpr (WHERE != kFirst) __syncthreads();
#pragma unroll
    for (int kk = 0; kk < K; ++kk) {
        const int i = pl.t + kk * pl.tr;
        if (i < nb) {
            int k = 0;
            if constexpr (WHERE == kFirst) {
#pragma unroll
                for (int q = 0; q < R; ++q) u[kk][q] = in.use(i + q * nb, u[kk][q]);
            } else if (WHERE == kLast || p > 1) {
                k = WHERE == kLast ? i : i - (int)__umulhi((unsigned)i, pmagic) * p;
#pragma unroll
                for (int q = 1; q < R; ++q) {
                    // 32-bit offsets from a uniform base keep the addresses out of register pairs
                    const unsigned off = (unsigned)((q - 1) * p + k) * (unsigned)sizeof(C);
                    u[kk][q] = O::mul(u[kk][q], __ldg(reinterpret_cast<const C*>(
                                                    reinterpret_cast<const char*>(tw) + off)));
                }
            }
            C y[R];
            Dft<T, R>::run(u[kk], y);
            const int j = (i - k) * R + k;
#pragma unroll
            for (int t = 0; t < R; ++t) {
                if constexpr (WHERE == kLast) out(i + t * p, y[t]);
                else S[pl.c + (pad(j + t * p) << pl.ls)] = y[t];
            }
        }
    }
    if constexpr (WHERE != kLast) __syncthreads();
}

template <typename T, int WHERE, class In, class Out>
__device__ __forceinline__ void stage_dispatch(int s, const FftPlan& fp, cx_t<T>* S, const Place pl,
                                               const cx_t<T>* tw, In& in, Out& out) {
    const int nb = fp.nb[s], p = fp.p[s];
    const unsigned mg = fp.pmagic[s];
    const cx_t<T>* t = tw + fp.toff[s];
#define FRES_RADIX(RR)                                                     \
    case RR: stage<T, RR, WHERE>(S, pl, nb, p, mg, t, in, out); break;
    if constexpr (sizeof(T) == 4) {
        switch (fp.radix[s]) {
            FRES_RADIX(16) FRES_RADIX(15) FRES_RADIX(12) FRES_RADIX(10) FRES_RADIX(9)
            FRES_RADIX(8) FRES_RADIX(5) FRES_RADIX(4) FRES_RADIX(3) FRES_RADIX(2)
        }
    } else {
        switch (fp.radix[s]) {
            FRES_RADIX(8) FRES_RADIX(6) FRES_RADIX(5) FRES_RADIX(4) FRES_RADIX(3) FRES_RADIX(2)
        }
    }
#undef FRES_RADIX
}

// The transform of the lines in S.  Every thread of the block must call it
// (it holds barriers).  A block transforms its lines once: in a loop over
// lines the compiler keeps the stages' invariant twiddles in registers, and
// spills.
template <typename T>
__device__ __forceinline__ void fft_line(cx_t<T>* S, const FftPlan& fp, const Place pl,
                                         const cx_t<T>* tw) {
    NoIo none;
    for (int s = 0; s < fp.nstages; ++s) stage_dispatch<T, kStage>(s, fp, S, pl, tw, none, none);
}
// The same from `in` to `out`, the first stage at place pf.
template <typename T, class In, class Out>
__device__ __forceinline__ void fft_fused(cx_t<T>* S, const FftPlan& fp, const Place pf,
                                          const Place pl, const cx_t<T>* tw, In& in, Out& out) {
    stage_dispatch<T, kFirst>(0, fp, S, pf, tw, in, out);
    for (int s = 1; s < fp.nstages - 1; ++s) stage_dispatch<T, kStage>(s, fp, S, pl, tw, in, out);
    stage_dispatch<T, kLast>(fp.nstages - 1, fp, S, pl, tw, in, out);
}

// Natural index of input i of len (centred: modes i - len/2), and of kept
// output kp (centred order over len).
__device__ __forceinline__ int in_natural(int i, int len, int n, int centered) {
    if (!centered) return i;
    return i < len / 2 ? n - len / 2 + i : i - len / 2;
}
__device__ __forceinline__ int out_natural(int kp, int len, int n) {
    return kp < len / 2 ? n - len / 2 + kp : kp - len / 2;
}

// items t, t + tr, ... below count, kBatch at a time: read all, then use all,
// so that a batch's loads are in flight together.
template <typename C, class Read, class Use>
__device__ __forceinline__ void batched(const Place pl, int count, Read read, Use use) {
    constexpr int kBatch = sizeof(C) == 8 ? 8 : 4;
#pragma unroll 1
    for (int i0 = pl.t; i0 < count; i0 += kBatch * pl.tr) {
        C v[kBatch];
#pragma unroll
        for (int b = 0; b < kBatch; ++b) {
            const int i = i0 + b * pl.tr;
            if (i < count) v[b] = read(i);
        }
#pragma unroll
        for (int b = 0; b < kBatch; ++b) {
            const int i = i0 + b * pl.tr;
            if (i < count) use(i, v[b]);
        }
    }
}

// The line's elements that no input fills: [in natural order] after the
// inputs, or between the centred inputs' two halves.
template <typename C>
__device__ __forceinline__ void zero_rest(C* S, const Place pl, int len, int n, int centered) {
    C z;
    z.x = z.y = 0;
    const int lo = centered ? len - len / 2 : len, hi = centered ? n - len / 2 : n;
    for (int e = lo + pl.t; e < hi; e += pl.tr) S[pl.c + (pad(e) << pl.ls)] = z;
}

// Natural input index e of a length-n transform whose len inputs hold modes
// i - len/2 (centred) or index i itself: the input index, or -1 (zero).
__device__ __forceinline__ int in_src(int e, int len, int n, int centered) {
    if (!centered) return e < len ? e : -1;
    const int hi = len - len / 2;
    if (e < hi) return e + len / 2;
    if (e >= n - len / 2) return e - n + len / 2;
    return -1;
}
// Kept output slot of natural output index k (centred order over len), or -1.
__device__ __forceinline__ int out_slot(int k, int len, int n) {
    if (k < len - len / 2) return k + len / 2;
    if (k >= n - len / 2) return k - n + len / 2;
    return -1;
}

// Rows: a block takes `lines` rows, tr threads each.
template <typename T>
__global__ void __launch_bounds__(1024, 1)
k_fft_rows(FftPlan fp, RowPassArgs a, int lines, int tr) {
    using C = cx_t<T>;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    C* S = (C*)smem_raw;
    kernel_begin();
    const int n = fp.n;
    const C* tw = (const C*)a.twiddle;
    const T* dcol = (const T*)a.deconv_col;
    int line = threadIdx.x / tr;
    Place pl{line * padded_len(n), (int)threadIdx.x - line * tr, tr, 0};
    const int total = a.row_list ? a.nlist : a.nrows;
    int row = blockIdx.x * lines + line;
    bool on = line < lines && row < total;
    if (a.row_list) {
        row = on ? a.row_list[row] : 0;
    } else if (a.live && on) {
        // rows of dead tile rows are zero in and out of the transform: skipped
        on = a.live[(row / a.batch_rows) * a.nty + (row % a.batch_rows) / kTile] != 0;
        if (lines == 1 && !on) return;   // the same for the whole block
    }
    if (!on) {   // no line: no elements, no butterflies
        pl.t = n;
        pl.c = 0;
        row = 0;
    }
    C* in = (C*)a.in + (long long)row * a.in_stride;
    C* out = (C*)a.out + (long long)row * a.out_stride;
    const T rowf = a.deconv_row ? ((const T*)a.deconv_row)[row] : (T)1;
    auto use = [&](int i, C v) {   // input i, read as v
        if (a.clear_in && nonzero(v)) in[i] = Ops<T>::mk(0, 0);
        if (a.centered_in) v = Ops<T>::scale(v, rowf * (dcol ? __ldg(&dcol[i]) : (T)1));
        return v;
    };
    if constexpr (sizeof(T) == 8) {
        // few radices, so little code: reads and stores in the first and last
        // stages (us, from start over short loops to fused: 500 x 500 nodes' rows
        // of 1024 33.4, 37.5, 35.5; of 2048 66.2, 70.3, 66.2)
        auto input = make_input(
            [&](int e) {
                const int i = in_src(e, a.in_len, n, a.centered_in);
                return i < 0 ? Ops<T>::mk(0, 0) : in[i];
            },
            [&](int e, C v) {
                const int i = in_src(e, a.in_len, n, a.centered_in);
                return i < 0 ? v : use(i, v);
            });
        auto store = [&](int k, C v) {
            const int kp = out_slot(k, a.out_len, n);
            if (kp >= 0) out[kp] = v;
        };
        fft_fused<T>(S, fp, pl, pl, tw, input, store);
    } else {
        batched<C>(
            pl, a.in_len, [&](int i) { return in[i]; },
            [&](int i, C v) { S[pl.c + pad(in_natural(i, a.in_len, n, a.centered_in))] = use(i, v); });
        zero_rest(S, pl, a.in_len, n, a.centered_in);
        __syncthreads();
        fft_line<T>(S, fp, pl, tw);
        for (int kp = pl.t; kp < a.out_len; kp += tr)
            out[kp] = S[pl.c + pad(out_natural(kp, a.out_len, n))];
    }
}

// Columns: a block takes 2^ls adjacent columns.
template <typename T, int MODE>
__global__ void __launch_bounds__(1024, 1)
k_fft_cols(FftPlan fp, ColPassArgs a, int ls) {
    using C = cx_t<T>;
    using O = Ops<T>;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ unsigned s_live[kMaxTileRows / 32];
    C* S = (C*)smem_raw;
    kernel_begin();
    const int n = fp.n;
    const C* tw = (const C*)a.twiddle;
    const int ncol = 1 << ls, ngroups = (a.ncols + ncol - 1) >> ls;
    const int tr = blockDim.x >> ls;
    const int c = threadIdx.x & (ncol - 1);        // this thread's column
    const Place pl{c, (int)threadIdx.x >> ls, tr, ls};
    const int o = blockIdx.x / ngroups, col = ((int)(blockIdx.x - o * ngroups) << ls) + c;
    const bool on = col < a.ncols;
    auto at = [&](int e) -> C& { return S[c + (pad(e) << ls)]; };
    if constexpr (MODE == kFftPlain) {
        const C* in = (const C*)a.in + (long long)o * a.in_bstride + col;
        C* out = (C*)a.out + (long long)o * a.out_bstride + col;
        if (a.live) {   // live tile rows of this transform as a bit mask
            for (int t = threadIdx.x; t < kMaxTileRows / 32; t += blockDim.x) s_live[t] = 0u;
            __syncthreads();
            for (int t = threadIdx.x; t < a.nty; t += blockDim.x)
                if (a.live[(long long)o * a.nty + t]) atomicOr(&s_live[t >> 5], 1u << (t & 31));
            __syncthreads();
        }
        batched<C>(
            pl, a.in_len,
            [&](int i) {
                const int r = i / kTile;
                const bool live = on && (!a.live || ((s_live[r >> 5] >> (r & 31)) & 1u));
                return live ? in[(long long)i * a.ncols] : O::mk(0, 0);
            },
            [&](int i, C v) { at(in_natural(i, a.in_len, n, a.centered_in)) = v; });
        zero_rest(S, pl, a.in_len, n, a.centered_in);
        __syncthreads();
        fft_line<T>(S, fp, pl, tw);
        if (!on) return;
        const C axc = a.ax ? ((const C*)a.ax)[(long long)o * a.ncols + col] : O::mk(1, 0);
        const C* ay = a.ax ? (const C*)a.ay + (long long)o * a.out_len : nullptr;
        for (int kp = pl.t; kp < a.out_len; kp += tr) {
            C v = at(out_natural(kp, a.out_len, n));
            if (ay) {
                v = O::mul(O::mul(v, axc), __ldg(&ay[kp]));
                if (a.occulter) v = O::mk((T)1 - v.x, -v.y);
            }
            out[(long long)kp * a.ncols] = v;
        }
    } else if constexpr (MODE == kFftRowStep1) {
        // grid row o viewed as fa x fb (element e = fb a + b at column b = col)
        C* in = (C*)a.in + (long long)o * a.in_stride;
        C* out = (C*)a.out + (long long)o * a.fN + col;
        const T rowf = a.deconv_row ? ((const T*)a.deconv_row)[o] : (T)1;
        const T* dcol = (const T*)a.deconv_col;
        auto src = [&](int ea) {
            return on ? in_src(a.fb * ea + col, a.in_len, a.fN, a.centered_in) : -1;
        };
        auto input = make_input(
            [&](int ea) {
                const int i = src(ea);
                return i < 0 ? O::mk(0, 0) : in[i];
            },
            [&](int ea, C v) {
                const int i = src(ea);
                if (i < 0) return v;
                if (a.clear_in && nonzero(v)) in[i] = O::mk(0, 0);
                if (a.centered_in) v = O::scale(v, rowf * (dcol ? __ldg(&dcol[i]) : (T)1));
                return v;
            });
        auto store = [&](int k1, C v) {
            if (on) out[(long long)k1 * a.fb] = v;
        };
        fft_fused<T>(S, fp, pl, pl, tw, input, store);
    } else if constexpr (MODE == kFftColStep1) {
        // outer index o = b: rows e = fb a + b of the grid columns
        const C* in = (const C*)a.in + col;
        C* out = (C*)a.out + (long long)o * a.ncols + col;
        auto input = make_input(
            [&](int ea) {
                const int i = on ? in_src(a.fb * ea + o, a.in_len, a.fN, a.centered_in) : -1;
                return i < 0 ? O::mk(0, 0) : in[(long long)i * a.ncols];
            },
            [](int, C v) { return v; });
        auto store = [&](int k1, C v) {
            if (on) out[(long long)k1 * a.fb * a.ncols] = v;
        };
        fft_fused<T>(S, fp, pl, pl, tw, input, store);
    } else if constexpr (MODE == kFftRowStep2) {
        // transform (l = o, k1 = col): scratch row (o fa + k1), b contiguous.
        // The first stage's neighbouring threads take neighbouring b, the
        // others' neighbouring columns, whose outputs are adjacent
        const int cf = threadIdx.x / tr;
        const Place pf{cf, (int)threadIdx.x - cf * tr, tr, ls};
        const int colf = col - c + cf;
        const bool onf = colf < a.ncols;
        const C* in = (const C*)a.in + ((long long)o * a.fa + colf) * a.fb;
        C* out = (C*)a.out + (long long)o * a.out_stride;
        const C* twN = (const C*)a.twN;
        auto input = make_input([&](int b) { return onf ? in[b] : O::mk(0, 0); },
                                [&](int b, C v) {
                                    return onf ? O::mul(v, __ldg(&twN[b * colf])) : v;
                                });
        auto store = [&](int k2, C v) {
            const int kp = out_slot(col + a.fa * k2, a.out_len, a.fN);
            if (kp >= 0 && on) out[kp] = v;
        };
        fft_fused<T>(S, fp, pf, pl, tw, input, store);
    } else {   // kFftColStep2: outer index o = k1
        const C* in = (const C*)a.in + (long long)o * a.fb * a.ncols + col;
        C* out = (C*)a.out + col;
        const C* twN = (const C*)a.twN;
        C axc = O::mk(1, 0);
        if (a.ax && on) axc = ((const C*)a.ax)[col];
        auto input = make_input(
            [&](int b) { return on ? in[(long long)b * a.ncols] : O::mk(0, 0); },
            [&](int b, C v) { return O::mul(v, __ldg(&twN[b * o])); });
        auto store = [&](int k2, C v) {
            const int kp = out_slot(o + a.fa * k2, a.out_len, a.fN);
            if (kp < 0 || !on) return;
            if (a.ax) {
                v = O::mul(O::mul(v, axc), __ldg(&((const C*)a.ay)[kp]));
                if (a.occulter) v = O::mk((T)1 - v.x, -v.y);
            }
            out[(long long)kp * a.ncols] = v;
        };
        fft_fused<T>(S, fp, pl, pl, tw, input, store);
    }
}

// Fewest stages, then fewest threads per line (at most 1024), then the larger
// radices first.
void search_radices(int m, int n, bool dbl, int first, int depth, int threads, int* cur, int* best,
                    int* best_stages, int* best_threads) {
    if (m == 1) {
        if (depth >= 2 && (depth < *best_stages ||
                           (depth == *best_stages && threads < *best_threads))) {
            std::copy(cur, cur + depth, best);
            *best_stages = depth;
            *best_threads = threads;
        }
        return;
    }
    if (depth >= *best_stages || depth >= kMaxRadixStages) return;
    const int nr = (int)((dbl ? sizeof(kRadicesD) : sizeof(kRadicesF)) / sizeof(int));
    for (int i = first; i < nr; ++i) {
        const int r = dbl ? kRadicesD[i] : kRadicesF[i];
        if (m % r) continue;
        const int k = butterflies(r, dbl), t = std::max(threads, (n / r + k - 1) / k);
        if (t > 1024) continue;
        cur[depth] = r;
        search_radices(m / r, n, dbl, i, depth + 1, t, cur, best, best_stages, best_threads);
    }
}

}  // namespace

// FP32 with `plain`: the radices 16, 8, 4, 2, 3, 5, each as often as it divides
// what is left (the same stages as the search's for powers of two).  The order
// of the radices decides the rounding, and a starshade's field u = 1 - u^ap and
// its gradient carry it magnified: 288 points in three stages of 12, 12 and 2
// round less (9.4e-8 against 1.06e-7 of the output) but moved the gradient by
// 3e-7 of itself, three times the distance between two runs.  Plans that can
// be differentiated in their petals' profile keep the plain order.
FftPlan make_fft_plan(int n, int is_double, bool plain) {
    FftPlan fp{};
    fp.n = n;
    int cur[kMaxRadixStages], best = kMaxRadixStages + 1, threads = 1 << 30;
    int m = n;
    for (int f : {2, 3, 5})
        while (m % f == 0) m /= f;
    const bool smooth = m == 1 && n >= 4;
    if (smooth && plain && !is_double) {
        best = 0;
        threads = 1;
        m = n;
        for (int r : {16, 8, 4, 2, 3, 5})
            for (; m % r == 0 && best < kMaxRadixStages; m /= r) {
                fp.radix[best++] = r;
                const int k = butterflies(r, false);
                threads = std::max(threads, (n / r + k - 1) / k);
            }
        if (m > 1 || best < 2 || threads > 1024) best = kMaxRadixStages + 1;
    }
    if (smooth && best > kMaxRadixStages)
        search_radices(n, n, is_double != 0, 0, 0, 1, cur, fp.radix, &best, &threads);
    if (best > kMaxRadixStages) {
        fp.nstages = -1;
        return fp;
    }
    fp.nstages = best;
    fp.threads = threads;
    long long p = 1, off = 0;
    for (int s = 0; s < fp.nstages; ++s) {
        fp.nb[s] = n / fp.radix[s];
        fp.p[s] = (int)p;
        fp.pmagic[s] = p == 1 ? 0u : (unsigned)(((1ULL << 32) + (unsigned long long)p - 1) / p);
        fp.toff[s] = (int)off;
        if (s > 0) off += p * (fp.radix[s] - 1);
        p *= fp.radix[s];
    }
    fp.ntw = (int)off;
    return fp;
}

// One pass: up to 13,671 points in FP32, 6,834 in FP64 (half the shared
// memory): a longer line leaves one block per SM, and four steps are faster.
bool fft_supported(int n, int is_double) {
    return make_fft_plan(n, is_double).nstages >= 2 &&
           2LL * padded_len(n) * (is_double ? 16 : 8) <= 227 * 1024;
}

// FP64 passes are bound by the FP64 pipe, so their time is the fullest SM's
// share of the lines.  Three blocks per SM (by the shared memory asked for),
// one line each, hand out the last lines evenly (the star's 1,000 columns of
// 2048: 190 us with two columns per block, 168 with one).
template <typename T>
size_t fft_smem(size_t bytes) {
    return sizeof(T) == 8 ? std::max(bytes, (size_t)60 * 1024) : bytes;
}

template <typename T>
void launch_fft_rows(const FftPlan& fp, const RowPassArgs& a, cudaStream_t st) {
    const int nwork = a.row_list ? a.nlist : a.nrows;
    // short rows: several per block, as long as the blocks still cover the SMs
    int lines = 1;
    while (lines < 8 && 2 * lines * fp.threads <= 128 && nwork / (2 * lines) >= 152 * 2) lines *= 2;
    const int tr = lines > 1 ? fp.threads : (fp.threads + 31) / 32 * 32;
    const int threads = (lines * tr + 31) / 32 * 32;
    const size_t smem = fft_smem<T>((size_t)lines * padded_len(fp.n) * sizeof(cx_t<T>));
    const int blocks = std::max(1, (nwork + lines - 1) / lines);
    if (smem > 48 * 1024)   // below, none is needed
        cudaFuncSetAttribute(k_fft_rows<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    launch_after(k_fft_rows<T>, blocks, threads, smem, st, fp, a, lines, tr);
}

template <typename T, int MODE>
void launch_cols_mode(const FftPlan& fp, const ColPassArgs& a, cudaStream_t st) {
    const int nouter = MODE == kFftPlain ? (a.batch > 1 ? a.batch : 1) : a.nouter;
    const size_t line = (size_t)padded_len(fp.n) * sizeof(cx_t<T>);
    auto items = [&](int ls) { return (long long)((a.ncols + (1 << ls) - 1) >> ls) * nouter; };
    // columns per block: 4 fill a 32-byte sector in FP32, short transforms take
    // up to 16; two blocks per SM, and enough blocks for the SMs.  FP64: one
    // long column (256 threads), see fft_smem
    int ls = 4;
    while (ls > 0 && ((fp.threads << ls) > (ls > 2 || sizeof(T) == 8 ? 256 : 512) ||
                      (line << ls) > 110 * 1024 || (ls > 1 && items(ls) < 152)))
        --ls;
    const int threads = ((fp.threads << ls) + 31) / 32 * 32;
    const size_t smem = fft_smem<T>(line << ls);
    const int blocks = (int)std::max(1LL, items(ls));
    if (smem > 48 * 1024)
        cudaFuncSetAttribute(k_fft_cols<T, MODE>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)smem);
    // FP64 plainly where the blocks fill the SMs: placed early, by the room that
    // the row pass leaves, they load them unevenly (800-point columns of a star's
    // field 139 -> 121 us a call, its gradient at 512 points 614 -> 602)
    if (sizeof(T) == 8 && blocks >= 152)
        k_fft_cols<T, MODE><<<blocks, threads, smem, st>>>(fp, a, ls);
    else
        launch_after(k_fft_cols<T, MODE>, blocks, threads, smem, st, fp, a, ls);
}

// FP32 column passes of square type-3 grids, start (two buffers, radix-16/8/4/
// 2/3/5 stages) -> single pass here -> four steps (us): 1920: 37 -> 31; 2560:
// 70 -> 57 in four steps; 3200: 109 -> 86; 3456: 170 -> 109; 5120: 406 -> 178
// (single pass -> four steps from 2560 on): the line lies at 2400.
template <typename T>
void launch_fft_cols(const FftPlan& fp, const ColPassArgs& a, cudaStream_t st) {
    switch (a.mode) {
        case kFftRowStep1: launch_cols_mode<T, kFftRowStep1>(fp, a, st); break;
        case kFftColStep1: launch_cols_mode<T, kFftColStep1>(fp, a, st); break;
        case kFftColStep2: launch_cols_mode<T, kFftColStep2>(fp, a, st); break;
        case kFftRowStep2: launch_cols_mode<T, kFftRowStep2>(fp, a, st); break;
        default: launch_cols_mode<T, kFftPlain>(fp, a, st); break;
    }
}

// n = fa * fb with both factors single-pass lengths, fa the divisor closest
// to sqrt(n) from below that works.
bool fft_split(int n, int is_double, int* fa, int* fb) {
    int best = 0;
    for (int d = 2; (long long)d * d <= n; ++d) {
        if (n % d) continue;
        if (fft_supported(d, is_double) && fft_supported(n / d, is_double)) best = d;
    }
    if (!best) return false;
    *fa = best;
    *fb = n / best;
    return true;
}

template void launch_fft_rows<float>(const FftPlan&, const RowPassArgs&, cudaStream_t);
template void launch_fft_rows<double>(const FftPlan&, const RowPassArgs&, cudaStream_t);
template void launch_fft_cols<float>(const FftPlan&, const ColPassArgs&, cudaStream_t);
template void launch_fft_cols<double>(const FftPlan&, const ColPassArgs&, cudaStream_t);

// ------------------------------------------------------------------ direct column DFT
// When only a narrow band of the type-1 grid's rows holds nodes (a starshade
// a few grid cells across on a pupil-sized grid), the column transform of the
// kept outputs is a small dense product: for problem b, kept output slot kp
// (natural index k) and column c,
//   out[kp][c] = sum_{r live} w_n^{k r} in[r][c],
// i.e. (n_out x R) x (R x ncols) with R live rows.  A block takes 64
// columns and up to four 64-output tiles; it stages 32 (FP64: 16) live rows
// at a time of the input (once for all its tiles when they fit one chunk)
// and of the twiddle matrix (from the exact n-point table, index k r mod n:
// a mask for power-of-two n) in shared memory, and each thread accumulates a 4 x 4 tile (outputs
// ty + 16 i, columns tx + 16 j: conflict-free shared reads, coalesced stores)
// before the output epilogue of the FFT path.
namespace {

constexpr int kDftTile = 64;

template <typename T>
__global__ void __launch_bounds__(256)
k_col_dft(ColPassArgs a, int n, unsigned nmask, unsigned* __restrict__ status) {
    using C = cx_t<T>;
    using O = Ops<T>;
    constexpr int kDftChunk = sizeof(T) == 4 ? 32 : 16;   // live rows staged at a time
    __shared__ C sX[kDftChunk][kDftTile];
    __shared__ C sW[kDftChunk][kDftTile];
    __shared__ int s_rows[kDftMaxRows];
    __shared__ int s_nt;
    const int b = blockIdx.z;
    const int c0 = blockIdx.x * kDftTile;
    const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
    // the problem's live tile rows in increasing order (one warp, ballots):
    // a fixed summation order, so the outputs repeat bit for bit
    if (tid < 32) {
        int cnt = 0;
        for (int t0 = 0; t0 < a.nty; t0 += 32) {
            const int t = t0 + tid;
            const bool on = t < a.nty && a.live[(long long)b * a.nty + t] != 0;
            const unsigned m = __ballot_sync(0xffffffffu, on);
            const int q = cnt + __popc(m & ((1u << tid) - 1u));
            if (on && q < kDftMaxRows / kTile)
                for (int i = 0; i < kTile; ++i) s_rows[q * kTile + i] = t * kTile + i;
            cnt += __popc(m);
        }
        if (tid == 0) s_nt = cnt;
    }
    __syncthreads();
    int R = s_nt * kTile;
    if (R > kDftMaxRows) {
        if (tid == 0) atomicOr(status, kStatusOverflow);
        R = kDftMaxRows;
    }
    const int len = a.out_len;
    const C* in = (const C*)a.in + (long long)b * a.in_bstride;
    const C* tw = (const C*)a.twiddle;
    C* out = (C*)a.out + (long long)b * a.out_bstride;
    const C* ax = a.ax ? (const C*)a.ax + (long long)b * a.ncols : nullptr;
    const C* ay = a.ax ? (const C*)a.ay + (long long)b * len : nullptr;
    // live rows fitting one chunk are staged once for all the block's output tiles
    const bool one = R <= kDftChunk;
    auto stage_x = [&](int r0, int rc) {
        for (int e = tid; e < kDftChunk * kDftTile; e += blockDim.x) {
            const int r = e / kDftTile, c = e % kDftTile, col = c0 + c;
            C x = O::mk(0, 0);
            if (r < rc && col < a.ncols) x = in[(long long)s_rows[r0 + r] * a.ncols + col];
            sX[r][c] = x;
        }
    };
    if (one) stage_x(0, R);
    const int nkt = (len + kDftTile - 1) / kDftTile;
    for (int kt = blockIdx.y; kt < nkt; kt += gridDim.y) {
        const int k0 = kt * kDftTile;
        C acc[4][4];
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int j = 0; j < 4; ++j) acc[i][j] = O::mk(0, 0);
        for (int r0 = 0; r0 < R; r0 += kDftChunk) {
            const int rc = min(kDftChunk, R - r0);
            __syncthreads();   // the previous tile's or chunk's values are consumed
            if (!one) stage_x(r0, rc);
            for (int e = tid; e < kDftChunk * kDftTile; e += blockDim.x) {
                // twiddle row r, output kk = c
                const int r = e / kDftTile, c = e % kDftTile, kp = k0 + c;
                C w = O::mk(0, 0);
                if (r < rc && kp < len) {
                    const unsigned k = kp >= len / 2 ? kp - len / 2 : kp - len / 2 + n;
                    const unsigned kr = k * (unsigned)s_rows[r0 + r];   // < 2^26
                    w = __ldg(&tw[nmask ? (kr & nmask) : kr % (unsigned)n]);
                }
                sW[r][c] = w;
            }
            __syncthreads();
            for (int r = 0; r < rc; ++r) {
                C w[4], x[4];
#pragma unroll
                for (int i = 0; i < 4; ++i) w[i] = sW[r][ty + 16 * i];
#pragma unroll
                for (int j = 0; j < 4; ++j) x[j] = sX[r][tx + 16 * j];
#pragma unroll
                for (int i = 0; i < 4; ++i)
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        acc[i][j].x = fma(w[i].x, x[j].x, fma(-w[i].y, x[j].y, acc[i][j].x));
                        acc[i][j].y = fma(w[i].x, x[j].y, fma(w[i].y, x[j].x, acc[i][j].y));
                    }
            }
        }
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const int kp = k0 + ty + 16 * i;
            if (kp >= len) continue;
            const C yv = ay ? __ldg(&ay[kp]) : O::mk(1, 0);
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const int col = c0 + tx + 16 * j;
                if (col >= a.ncols) continue;
                C v = acc[i][j];
                if (ax) {
                    v = O::mul(O::mul(v, __ldg(&ax[col])), yv);
                    if (a.occulter) v = O::mk((T)1 - v.x, -v.y);
                }
                out[(long long)kp * a.ncols + col] = v;
            }
        }
    }
}

// In-register 32-point DFT, y_t = sum_q u_q e^{-2 pi i q t / 32}, in place:
// q = 4 m + q2, t = t1 + 8 t2 (Cooley-Tukey): 8-point DFTs over m, twiddles
// w_32^{q2 t1}, then 4-point DFTs over q2.
template <typename T>
__device__ __forceinline__ void dft32(cx_t<T>* y) {
    using C = cx_t<T>;
    using O = Ops<T>;
    // cos (2 pi j / 32), j = 0..8; sin (2 pi j / 32) = cos (2 pi (8 - j) / 32)
    const T c[9] = {(T)1, (T)0.98078528040323044912618223613424,
                    (T)0.92387953251128675612818318939679,
                    (T)0.83146961230254523707878837761791,
                    (T)0.70710678118654752440084436210485,
                    (T)0.55557023301960222474283081394853,
                    (T)0.38268343236508977172845998403040,
                    (T)0.19509032201612826784828486847702, (T)0};
    C A[4][8];
#pragma unroll
    for (int q2 = 0; q2 < 4; ++q2) {
        C v[8];
#pragma unroll
        for (int m = 0; m < 8; ++m) v[m] = y[4 * m + q2];
        Dft<T, 8>::run(v, A[q2]);
#pragma unroll
        for (int t1 = 1; t1 < 8; ++t1) {
            const int j = q2 * t1;   // < 32: w_32^j = (cos, -sin) of 2 pi j / 32
            if (j == 0) continue;
            const int jq = j & 7, quad = j >> 3;   // j = 8 quad + jq
            // (cos, sin) of 2 pi j / 32 from the first quadrant
            T cs = c[jq], sn = c[8 - jq];
            if (quad == 1) { const T t = cs; cs = -sn; sn = t; }
            else if (quad == 2) { cs = -cs; sn = -sn; }
            else if (quad == 3) { const T t = cs; cs = sn; sn = -t; }
            A[q2][t1] = O::mul(A[q2][t1], O::mk(cs, -sn));
        }
    }
#pragma unroll
    for (int t1 = 0; t1 < 8; ++t1) {
        C v[4] = {A[0][t1], A[1][t1], A[2][t1], A[3][t1]}, d[4];
        Dft<T, 4>::run(v, d);
#pragma unroll
        for (int t2 = 0; t2 < 4; ++t2) y[t1 + 8 * t2] = d[t2];
    }
}

// Type-1 column pass over one live tile row by a pruned FFT.  A problem
// whose nodes occupy the 32 grid rows row0 .. row0 + 31 has, for the
// natural output index k = P a + b (P = n / 32, a < 32, b < P),
//   sum_j w_n^{k (row0 + j)} x_j = w_n^{k row0} sum_j w_32^{a j} (w_n^{b j} x_j):
// a 32-point DFT per b of the inputs twiddled by w_n^{b j}, about 30
// operations per output instead of the direct sum's 32 multiply-adds, then
// the epilogue (ax[c] folded into the staged inputs, ay[k] and Babinet).
// A warp takes 32 adjacent columns and one b; the block's 8 warps (8 b)
// share the staged 32 x 32 input block.  Stores: each output row segment of
// a warp is 32 adjacent columns.
template <typename T>
__global__ void __launch_bounds__(256)
k_col_pfft(ColPassArgs a, int n, unsigned nmask, unsigned* __restrict__ status) {
    using C = cx_t<T>;
    using O = Ops<T>;
    __shared__ C xs[kTile][kTile + 1];
    __shared__ int s_nt, s_row0;
    const int pb = blockIdx.z, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int c0 = blockIdx.x * kTile, col = c0 + lane;
    const int P = n / kTile;
    const int bb = blockIdx.y * 8 + warp;   // this warp's b
    const int len = a.out_len;
    if (tid == 0) {
        s_nt = 0;
        s_row0 = 0;
    }
    __syncthreads();
    for (int t = tid; t < a.nty; t += blockDim.x)
        if (a.live[(long long)pb * a.nty + t]) {
            atomicAdd(&s_nt, 1);
            s_row0 = t * kTile;
        }
    __syncthreads();
    const int nt = s_nt, row0 = s_row0;
    const C* in = (const C*)a.in + (long long)pb * a.in_bstride;
    C* out = (C*)a.out + (long long)pb * a.out_bstride;
    const C* tw = (const C*)a.twiddle;
    const C* ax = a.ax ? (const C*)a.ax + (long long)pb * a.ncols : nullptr;
    const C* ay = a.ax ? (const C*)a.ay + (long long)pb * len : nullptr;
    const bool bab = ay && a.occulter;
    if (nt != 1) {   // no nodes: u^ap = 0 (u^oc = 1); several live tile rows: flagged
        if (nt > 1 && tid == 0) atomicOr(status, kStatusOverflow);
        if (nt == 0 && bb < P && col < a.ncols)
            for (int aa = 0; aa < kTile; ++aa) {
                const int kp = out_slot(P * aa + bb, len, n);
                if (kp >= 0) out[(long long)kp * a.ncols + col] = O::mk(bab ? (T)1 : (T)0, 0);
            }
        return;
    }
    for (int e = tid; e < kTile * kTile; e += blockDim.x) {
        const int r = e / kTile, cc = e % kTile, cg = c0 + cc;
        C x = O::mk(0, 0);
        if (cg < a.ncols) {
            x = in[(long long)(row0 + r) * a.ncols + cg];
            if (ax) x = O::mul(x, ax[cg]);
        }
        xs[r][cc] = x;
    }
    __syncthreads();
    if (bb >= P || col >= a.ncols) return;
    C y[kTile];
#pragma unroll
    for (int j = 0; j < kTile; ++j) {
        const C x = xs[j][lane];
        y[j] = j == 0 ? x : O::mul(x, __ldg(&tw[bb * j]));   // bb j < n
    }
    dft32<T>(y);
#pragma unroll
    for (int aa = 0; aa < kTile; ++aa) {
        const int k = P * aa + bb;
        const int kp = out_slot(k, len, n);
        if (kp >= 0) {
            const unsigned kr = (unsigned)k * (unsigned)row0;   // < n^2 <= 2^30
            C v = O::mul(y[aa], __ldg(&tw[nmask ? (kr & nmask) : kr % (unsigned)n]));
            if (ay) {
                v = O::mul(v, __ldg(&ay[kp]));
                if (a.occulter) v = O::mk((T)1 - v.x, -v.y);
            }
            out[(long long)kp * a.ncols + col] = v;
        }
    }
}

}  // namespace

template <typename T>
void launch_col_dft(const ColPassArgs& a, int n, unsigned* status, cudaStream_t st) {
    // each block takes up to four 64-output tiles of its 64 columns
    const int nkt = (a.out_len + kDftTile - 1) / kDftTile;
    const dim3 grid((a.ncols + kDftTile - 1) / kDftTile, (nkt + 3) / 4, a.batch > 1 ? a.batch : 1);
    // power-of-two n: the index reduction is a mask instead of a division
    const unsigned nmask = (n & (n - 1)) == 0 ? (unsigned)(n - 1) : 0u;
    k_col_dft<T><<<grid, 256, 0, st>>>(a, n, nmask, status);
}
template void launch_col_dft<float>(const ColPassArgs&, int, unsigned*, cudaStream_t);
template void launch_col_dft<double>(const ColPassArgs&, int, unsigned*, cudaStream_t);

bool col_pfft_supported(int n, int live_rows) {
    return live_rows == kTile && n % kTile == 0 && n <= 32768;
}

void launch_col_pfft_d(const ColPassArgs& a, int n, unsigned* status, cudaStream_t st) {
    const int P = n / kTile;
    const dim3 grid((a.ncols + kTile - 1) / kTile, (P + 7) / 8, a.batch > 1 ? a.batch : 1);
    const unsigned nmask = (n & (n - 1)) == 0 ? (unsigned)(n - 1) : 0u;
    k_col_pfft<double><<<grid, 256, 0, st>>>(a, n, nmask, status);
}

}  // namespace fres
