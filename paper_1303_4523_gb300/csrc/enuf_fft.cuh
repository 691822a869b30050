// enuf_fft.cuh -- batched shared-memory FFT of length n = 2^a 3^b 5^c (n <= 1024).
//
// The 3-D transforms of the NFFT (the plain FFT step of Sec. 3.3 inside the
// transposed and conjugated NFFT, Eq. 13-14) are done one dimension at a time;
// each CTA loads a batch of lines into shared memory and runs this Stockham
// auto-sort FFT on all of them. Stage s with radix R combines R sub-transforms
// of length Ns (product of the earlier radices): butterfly j of a line reads
// x[j + r n/R], twiddles element r by w^{r k n/(Ns R)} (k = j mod Ns,
// w = e^{-+2 pi i/n}), does an R-point DFT and writes the results to
// (j - k) R + k + m Ns. After the last stage the line is in natural order.
// Radices 2, 3, 4, 5, 8 and the composites 6, 10, 12, 16, 20 (two small DFTs
// in registers with compile-time twiddles), so most lengths take two stages
// (9, 15 and 18 serve the two-factor transform below only).
#pragma once
#include <cuda_runtime.h>

#include <type_traits>
#include <utility>

namespace enuf {

template <typename R> struct Cx;
template <> struct Cx<float> { using T = float2; };
template <> struct Cx<double> { using T = double2; };

struct FftPlanDev {
    int n;
    int nst;
    int rad[8];
    int f1, f2;   // two-factor split n = f1 f2 of the FP32 two-factor kernels (0: none)
};

// a / b for 0 <= a < 2^23, b >= 1, given rb = 1/b in float: the float quotient
// of a + 1/2 is within one of the true one, and one integer step corrects it.
__device__ __forceinline__ int qdiv(int a, int b, float rb) {
    int q = (int)(((float)a + 0.5f) * rb);
    const int r = a - q * b;
    q += (r >= b ? 1 : 0) - (r < 0 ? 1 : 0);
    return q;
}

// Shared-memory layout of the line buffers. A bank row holds 128 B, i.e. B
// complex values (16 float2 or 8 double2). The index inside a line is
// swizzled, i -> i XOR (row of i mod B), so that both unit-stride accesses
// and the strided writes of the early Stockham stages spread over all banks;
// lines are padded to whole bank rows plus one value, which skews consecutive
// lines for the accesses that run across lines.
template <typename C> struct SwzBits;
template <> struct SwzBits<float2> { static constexpr int v = 4; };
template <> struct SwzBits<double2> { static constexpr int v = 3; };
template <typename C>
__device__ __forceinline__ int swz(int i) {
    constexpr int b = SwzBits<C>::v;
    return i ^ ((i >> b) & ((1 << b) - 1));
}
template <typename C>
__host__ __device__ constexpr int line_stride(int n) {
    return ((n + (1 << SwzBits<C>::v) - 1) >> SwzBits<C>::v << SwzBits<C>::v) + 1;
}

template <typename C>
__device__ __forceinline__ C cmul(C a, C b) {
    C r;
    r.x = a.x * b.x - a.y * b.y;
    r.y = a.x * b.y + a.y * b.x;
    return r;
}
template <typename C>
__device__ __forceinline__ C cadd(C a, C b) { C r; r.x = a.x + b.x; r.y = a.y + b.y; return r; }
template <typename C>
__device__ __forceinline__ C csub(C a, C b) { C r; r.x = a.x - b.x; r.y = a.y - b.y; return r; }
// multiply by -i (forward) or +i (inverse): the rotation of the 4-point DFT
template <typename C, bool INV>
__device__ __forceinline__ C rot_i(C a) {
    C r;
    if (INV) { r.x = -a.y; r.y = a.x; }   // +i a
    else     { r.x = a.y;  r.y = -a.x; }  // -i a
    return r;
}

template <typename R, int RAD, bool INV> struct SmallDft;

template <typename R, bool INV> struct SmallDft<R, 2, INV> {
    template <typename C> __device__ __forceinline__ static void run(C* v) {
        C a = cadd(v[0], v[1]), b = csub(v[0], v[1]);
        v[0] = a; v[1] = b;
    }
};

template <typename R, bool INV> struct SmallDft<R, 4, INV> {
    template <typename C> __device__ __forceinline__ static void run(C* v) {
        C s02 = cadd(v[0], v[2]), d02 = csub(v[0], v[2]);
        C s13 = cadd(v[1], v[3]), d13 = rot_i<C, INV>(csub(v[1], v[3]));
        v[0] = cadd(s02, s13);
        v[2] = csub(s02, s13);
        v[1] = cadd(d02, d13);
        v[3] = csub(d02, d13);
    }
};

template <typename R, bool INV> struct SmallDft<R, 8, INV> {
    template <typename C> __device__ __forceinline__ static void run(C* v) {
        // even / odd 4-point DFTs, then combine with w8^m
        C e[4] = {v[0], v[2], v[4], v[6]};
        C o[4] = {v[1], v[3], v[5], v[7]};
        SmallDft<R, 4, INV>::run(e);
        SmallDft<R, 4, INV>::run(o);
        combine(v, e, o);
    }
    template <typename C> __device__ __forceinline__ static void combine(C* v, const C* e, const C* o) {
        const R h = (R)0.70710678118654752440;
        C t1, t3;
        // w8 = (1 -+ i)/sqrt2 ; w8^2 = -+ i ; w8^3 = (-1 -+ i)/sqrt2
        if (INV) {
            t1.x = h * (o[1].x - o[1].y); t1.y = h * (o[1].x + o[1].y);
            t3.x = -h * (o[3].x + o[3].y); t3.y = h * (o[3].x - o[3].y);
        } else {
            t1.x = h * (o[1].x + o[1].y); t1.y = h * (o[1].y - o[1].x);
            t3.x = h * (o[3].y - o[3].x); t3.y = -h * (o[3].x + o[3].y);
        }
        C t2 = rot_i<C, INV>(o[2]);
        v[0] = cadd(e[0], o[0]); v[4] = csub(e[0], o[0]);
        v[1] = cadd(e[1], t1);   v[5] = csub(e[1], t1);
        v[2] = cadd(e[2], t2);   v[6] = csub(e[2], t2);
        v[3] = cadd(e[3], t3);   v[7] = csub(e[3], t3);
    }
};

template <typename R, bool INV> struct SmallDft<R, 3, INV> {
    template <typename C> __device__ __forceinline__ static void run(C* v) {
        const R s3 = (R)0.86602540378443864676;  // sqrt(3)/2
        C t = cadd(v[1], v[2]);
        C d = csub(v[1], v[2]);
        C m;
        m.x = v[0].x - (R)0.5 * t.x;
        m.y = v[0].y - (R)0.5 * t.y;
        // forward: y1 = m - i s3 d, y2 = m + i s3 d ; inverse swaps the sign of i
        C id = rot_i<C, INV>(d);   // -i d (fwd) or +i d (inv)
        v[0] = cadd(v[0], t);
        v[1].x = m.x + s3 * id.x; v[1].y = m.y + s3 * id.y;
        v[2].x = m.x - s3 * id.x; v[2].y = m.y - s3 * id.y;
    }
};

template <typename R, bool INV> struct SmallDft<R, 5, INV> {
    template <typename C> __device__ __forceinline__ static void run(C* v) {
        const R c1 = (R)0.30901699437494742410, c2 = (R)-0.80901699437494742410;
        const R s1 = (R)0.95105651629515357212, s2 = (R)0.58778525229247312917;
        C a1 = cadd(v[1], v[4]), b1 = csub(v[1], v[4]);
        C a2 = cadd(v[2], v[3]), b2 = csub(v[2], v[3]);
        C m1, m2, u1, u2;
        m1.x = v[0].x + c1 * a1.x + c2 * a2.x; m1.y = v[0].y + c1 * a1.y + c2 * a2.y;
        m2.x = v[0].x + c2 * a1.x + c1 * a2.x; m2.y = v[0].y + c2 * a1.y + c1 * a2.y;
        u1.x = s1 * b1.x + s2 * b2.x; u1.y = s1 * b1.y + s2 * b2.y;
        u2.x = s2 * b1.x - s1 * b2.x; u2.y = s2 * b1.y - s1 * b2.y;
        C iu1 = rot_i<C, INV>(u1), iu2 = rot_i<C, INV>(u2);  // -i u (fwd)
        v[0].x = v[0].x + a1.x + a2.x; v[0].y = v[0].y + a1.y + a2.y;
        v[1] = cadd(m1, iu1); v[4] = csub(m1, iu1);
        v[2] = cadd(m2, iu2); v[3] = csub(m2, iu2);
    }
};

// The same DFTs of inputs whose middle half is zero (v[N/4] .. v[3N/4 - 1], not
// read): the first stage of an inverse transform whose spectrum is kept for
// |k| < n/4 only. 8 of 16 and 36 of 52 additions.
template <typename R, int RAD, bool INV> struct HalfDft;
template <typename R, bool INV> struct HalfDft<R, 4, INV> {
    template <typename C> __device__ __forceinline__ static void run(C* v) {
        const C a = v[0], b = v[3], rb = rot_i<C, INV>(v[3]);
        v[0] = cadd(a, b);
        v[2] = csub(a, b);
        v[1] = csub(a, rb);
        v[3] = cadd(a, rb);
    }
};
template <typename R, bool INV> struct HalfDft<R, 8, INV> {
    template <typename C> __device__ __forceinline__ static void run(C* v) {
        C e[4], o[4];
        e[0] = v[0]; e[3] = v[6];
        o[0] = v[1]; o[3] = v[7];
        HalfDft<R, 4, INV>::run(e);
        HalfDft<R, 4, INV>::run(o);
        SmallDft<R, 8, INV>::combine(v, e, o);
    }
};

// Compile-time loop: f(std::integral_constant<int, i>) for i = 0 .. N-1.
template <typename F, int... I>
__device__ __forceinline__ void sfor_(F&& f, std::integer_sequence<int, I...>) {
    (f(std::integral_constant<int, I>{}), ...);
}
template <int N, typename F>
__device__ __forceinline__ void sfor(F&& f) {
    sfor_(f, std::make_integer_sequence<int, N>{});
}

// cos and sin of 2 pi m / N, evaluated by the compiler: the angle is reduced
// to [0, pi/2) by its quadrant (exact integer arithmetic), then Taylor series
// to 30 terms (the last term is below 1e-60 there).
struct Root {
    double c, s;
};
__host__ __device__ constexpr double taylor_cos(double x) {
    double sum = 1.0, t = 1.0;
    for (int k = 1; k < 30; ++k) {
        t *= -x * x / ((2.0 * k - 1.0) * (2.0 * k));
        sum += t;
    }
    return sum;
}
__host__ __device__ constexpr double taylor_sin(double x) {
    double sum = x, t = x;
    for (int k = 1; k < 30; ++k) {
        t *= -x * x / ((2.0 * k) * (2.0 * k + 1.0));
        sum += t;
    }
    return sum;
}
__host__ __device__ constexpr Root unit_root(int m, int N) {
    m = ((m % N) + N) % N;
    const int q = 4 * m / N;            // quadrant
    const int rn = 4 * m - q * N;       // remaining angle (pi/2) rn / N in [0, pi/2)
    const double r = 1.57079632679489661923 * rn / N;
    const double c = taylor_cos(r), sn = taylor_sin(r);
    return q == 0 ? Root{c, sn} : q == 1 ? Root{-sn, c} : q == 2 ? Root{-c, -sn} : Root{sn, -c};
}

// a omega^M with omega = e^{-2 pi i/N} (forward) or e^{+2 pi i/N} (inverse);
// the quarter turns are exact rotations.
template <int M, int N, bool INV, typename R, typename C>
__device__ __forceinline__ C twiddle_const(C a) {
    constexpr int m = M % N;
    if constexpr (m == 0) {
        return a;
    } else if constexpr (4 * m == N) {
        return rot_i<C, INV>(a);
    } else if constexpr (2 * m == N) {
        a.x = -a.x;
        a.y = -a.y;
        return a;
    } else if constexpr (4 * m == 3 * N) {
        return rot_i<C, !INV>(a);
    } else {
        constexpr Root w = unit_root(m, N);
        const R c = (R)w.c, sn = INV ? (R)w.s : (R)-w.s;
        C r;
        r.x = a.x * c - a.y * sn;
        r.y = a.x * sn + a.y * c;
        return r;
    }
}

// Composite radix N1 N2 in registers (Cooley-Tukey): input index N2 n1 + n2,
// N2 DFTs of length N1 over n1, twiddle omega_{N1 N2}^{n2 k1}, N1 DFTs of
// length N2 over n2; output index k1 + N1 k2 (natural order).
template <typename R, int N1, int N2, bool INV>
struct CompositeDft {
    template <typename C>
    __device__ __forceinline__ static void run(C* v) {
        constexpr int RR = N1 * N2;
        C y[RR];   // y[n2 N1 + k1]
        sfor<N2>([&](auto n2c) {
            constexpr int n2 = decltype(n2c)::value;
            C a[N1];
#pragma unroll
            for (int n1 = 0; n1 < N1; ++n1) a[n1] = v[N2 * n1 + n2];
            SmallDft<R, N1, INV>::run(a);
            sfor<N1>([&](auto k1c) {
                constexpr int k1 = decltype(k1c)::value;
                y[n2 * N1 + k1] = twiddle_const<n2 * k1, RR, INV, R>(a[k1]);
            });
        });
#pragma unroll
        for (int k1 = 0; k1 < N1; ++k1) {
            C b[N2];
#pragma unroll
            for (int n2 = 0; n2 < N2; ++n2) b[n2] = y[n2 * N1 + k1];
            SmallDft<R, N2, INV>::run(b);
#pragma unroll
            for (int k2 = 0; k2 < N2; ++k2) v[k1 + N1 * k2] = b[k2];
        }
    }
};
template <typename R, bool INV> struct SmallDft<R, 6, INV> : CompositeDft<R, 2, 3, INV> {};
template <typename R, bool INV> struct SmallDft<R, 9, INV> : CompositeDft<R, 3, 3, INV> {};
template <typename R, bool INV> struct SmallDft<R, 10, INV> : CompositeDft<R, 2, 5, INV> {};
template <typename R, bool INV> struct SmallDft<R, 12, INV> : CompositeDft<R, 4, 3, INV> {};
template <typename R, bool INV> struct SmallDft<R, 15, INV> : CompositeDft<R, 3, 5, INV> {};
template <typename R, bool INV> struct SmallDft<R, 16, INV> : CompositeDft<R, 4, 4, INV> {};
template <typename R, bool INV> struct SmallDft<R, 18, INV> : CompositeDft<R, 2, 9, INV> {};
template <typename R, bool INV> struct SmallDft<R, 20, INV> : CompositeDft<R, 4, 5, INV> {};

// One Stockham stage over nlines lines (line l at offset l*ls, swizzled inside).
// HALF: a first stage (Ns = 1) whose inputs are zero from n/4 to 3n/4; that half
// of src is not read.
template <typename R, int RAD, bool INV, bool HALF = false>
__device__ __forceinline__ void fft_stage(const typename Cx<R>::T* __restrict__ src,
                                          typename Cx<R>::T* __restrict__ dst,
                                          const typename Cx<R>::T* __restrict__ tw,
                                          int n, int Ns, int nlines, int ls) {
    using C = typename Cx<R>::T;
    const int m = n / RAD;
    const int tstep = n / (Ns * RAD);
    const int total = nlines * m;
    const float rm = 1.0f / (float)m, rNs = 1.0f / (float)Ns;
    for (int idx = threadIdx.x; idx < total; idx += blockDim.x) {
        const int line = qdiv(idx, m, rm);
        const int j = idx - line * m;
        const int k = j - qdiv(j, Ns, rNs) * Ns;
        const C* s = src + line * ls;
        C* d = dst + line * ls;
        C v[RAD];
#pragma unroll
        for (int r = 0; r < RAD; ++r)
            if (!HALF || r < RAD / 4 || r >= RAD - RAD / 4) v[r] = s[swz<C>(j + r * m)];
        if (!HALF && k != 0) {
#pragma unroll
            for (int r = 1; r < RAD; ++r) {
                C w = tw[r * k * tstep];
                if (INV) w.y = -w.y;
                v[r] = cmul(v[r], w);
            }
        }
        if constexpr (HALF) HalfDft<R, RAD, INV>::run(v);
        else SmallDft<R, RAD, INV>::run(v);
        const int base = (j - k) * RAD + k;
#pragma unroll
        for (int r = 0; r < RAD; ++r) d[swz<C>(base + r * Ns)] = v[r];
    }
}

// Transform nlines lines held in b0; b1 is scratch of the same size. Returns
// the buffer holding the result. Contains __syncthreads (call from all threads).
// CR: the composite radices 6, 10, 12, 16, 20 are compiled in (the plan's
// radix list decides which instance runs; they raise the kernels' register
// count, so plans without them run the CR = false instance).
// HALF: the inverse of a spectrum kept for |k| < n/4: the stage of fft_half, where
// there is one, runs first and skips the empty half (which it does not read).
// FP64 additions bound these passes (the FP64 pipe 65-79% busy): with the z pass's
// two fields instead of three a whole call at n = 160 (375,000 beads) takes 1057 us
// instead of 1147, four steps at n = 96 1265 instead of 1337.
__device__ __forceinline__ int fft_half(const FftPlanDev& fp) {   // first radix 8 or 4, -1: none
    for (int st = 0; st < fp.nst; ++st)
        if (fp.rad[st] == 8 || fp.rad[st] == 4) return st;
    return -1;
}
template <typename R, bool INV, bool CR = false, bool HALF = false>
__device__ typename Cx<R>::T* fft_lines(typename Cx<R>::T* b0, typename Cx<R>::T* b1,
                                        const typename Cx<R>::T* tw, const FftPlanDev& fp,
                                        int nlines, int ls) {
    using C = typename Cx<R>::T;
    C* src = b0;
    C* dst = b1;
    int Ns = 1;
    const int sh = HALF ? fft_half(fp) : -1;
    if (HALF && sh >= 0) {
        Ns = fp.rad[sh];
        if (Ns == 8) fft_stage<R, 8, INV, true>(src, dst, tw, fp.n, 1, nlines, ls);
        else fft_stage<R, 4, INV, true>(src, dst, tw, fp.n, 1, nlines, ls);
        __syncthreads();
        C* t = src; src = dst; dst = t;
    }
    for (int st = 0; st < fp.nst; ++st) {
        if (HALF && st == sh) continue;
        const int rad = fp.rad[st];
        if constexpr (CR) {
            switch (rad) {
                case 16: fft_stage<R, 16, INV>(src, dst, tw, fp.n, Ns, nlines, ls); break;
                case 20: fft_stage<R, 20, INV>(src, dst, tw, fp.n, Ns, nlines, ls); break;
                case 12: fft_stage<R, 12, INV>(src, dst, tw, fp.n, Ns, nlines, ls); break;
                case 10: fft_stage<R, 10, INV>(src, dst, tw, fp.n, Ns, nlines, ls); break;
                case 6: fft_stage<R, 6, INV>(src, dst, tw, fp.n, Ns, nlines, ls); break;
                default: break;
            }
        }
        switch (rad) {
            case 8: fft_stage<R, 8, INV>(src, dst, tw, fp.n, Ns, nlines, ls); break;
            case 4: fft_stage<R, 4, INV>(src, dst, tw, fp.n, Ns, nlines, ls); break;
            case 2: fft_stage<R, 2, INV>(src, dst, tw, fp.n, Ns, nlines, ls); break;
            case 3: fft_stage<R, 3, INV>(src, dst, tw, fp.n, Ns, nlines, ls); break;
            case 5: fft_stage<R, 5, INV>(src, dst, tw, fp.n, Ns, nlines, ls); break;
            default: break;
        }
        __syncthreads();
        C* t = src; src = dst; dst = t;
        Ns *= rad;
    }
    return src;
}

}  // namespace enuf

namespace enuf {

// ---------------------------------------------------------------------------
// Two-factor line FFT for lengths n = f1 f2 with both factors among the
// radices above: the Cooley-Tukey split of the n-point DFT into f2 DFTs of
// length f1, one twiddle per element, and f1 DFTs of length f2. With
// element m = t + f2 j of a line (t < f2, j < f1) and output k = k1 + f1 k2,
//   X[k1 + f1 k2] = sum_t w_n^{t k1} w_f2^{t k2} sum_j x[t + f2 j] w_f1^{j k1}.
// Phase A (one task per line and t): loads its f1 elements (through the
//   caller's loader, usually straight from global memory), the f1-point DFT
//   in registers, the twiddles w_n^{t k1} from the shared table, and stores
//   row k1 of the line's buffer at k1 (f2 + 1) + t (rows padded by one value:
//   phase B reads a row per lane, and the odd stride spreads those reads
//   over the banks).
// Phase B (one task per line and k1): the f2-point DFT of row k1 in
//   registers; the caller's storer receives X[k1 + f1 k2].
// The factors are compile-time (the DFTs and every offset inside a task are
// constants); n, f1, f2 and the line count are runtime values, so one kernel
// serves every length with such a factorization. Per element this is one
// load, the DFT arithmetic of two radices, one twiddle multiply and two
// shared-memory accesses, against the runtime-radix Stockham stages'
// per-stage quotients, swizzles and twiddle indices.
// ---------------------------------------------------------------------------
// Row stride of a phase-A line buffer, and of a buffer of natural-order
// results. A two-factor pass with L lines per CTA holds the twiddle table (n
// values), L phase-A rows and L result rows in shared memory.
__host__ __device__ constexpr int fft2_lsa(int f1, int f2) { return f1 * (f2 + 1); }
__host__ __device__ constexpr int fft2_lsb(int n) { return n + 1; }

// The lengths a two-factor kernel works with. FftLen<F1, F2>: compile-time, so
// that every offset, quotient and loop bound of a pass is a constant (the
// runtime form spends two thirds of its instructions on them: ~95 per complex
// point in the inverse x pass at n = 320, of which ~30 are the transform);
// FftLen<0, 0>: from the plan, for line passes of lengths without an instance of
// their own (up to n = 100 with fft_path = 1) and the fused brick spreading.
template <int F1, int F2>
struct FftLen {
    static constexpr int kF1 = F1, kF2 = F2;
    static constexpr int n = F1 * F2, f1 = F1, f2 = F2, nc = n / 4 - 1, nc1 = nc + 1, K = 2 * nc + 1;
    static constexpr int lsa = fft2_lsa(F1, F2), lsb = fft2_lsb(n);
    __device__ __forceinline__ FftLen(int, int, int) {}
    static __device__ __forceinline__ int by_n(int a) { return (int)((unsigned)a / (unsigned)n); }
    static __device__ __forceinline__ int by_f1(int a) { return (int)((unsigned)a / (unsigned)F1); }
    static __device__ __forceinline__ int by_f2(int a) { return (int)((unsigned)a / (unsigned)F2); }
    static __device__ __forceinline__ int by_K(int a) { return (int)((unsigned)a / (unsigned)K); }
    static __device__ __forceinline__ int by_nc1(int a) { return (int)((unsigned)a / (unsigned)nc1); }
};
template <>
struct FftLen<0, 0> {
    static constexpr int kF1 = 0, kF2 = 0;
    int n, f1, f2, nc, nc1, K, lsa, lsb;
    __device__ __forceinline__ FftLen(int f1_, int f2_, int nc_)
        : n(f1_ * f2_), f1(f1_), f2(f2_), nc(nc_), nc1(nc_ + 1), K(2 * nc_ + 1), lsa(fft2_lsa(f1_, f2_)),
          lsb(fft2_lsb(f1_ * f2_)) {}
    __device__ __forceinline__ int by_n(int a) const { return qdiv(a, n, 1.0f / (float)n); }
    __device__ __forceinline__ int by_f1(int a) const { return qdiv(a, f1, 1.0f / (float)f1); }
    __device__ __forceinline__ int by_f2(int a) const { return qdiv(a, f2, 1.0f / (float)f2); }
    __device__ __forceinline__ int by_K(int a) const { return qdiv(a, K, 1.0f / (float)K); }
    __device__ __forceinline__ int by_nc1(int a) const { return qdiv(a, nc1, 1.0f / (float)nc1); }
};

template <typename R, int F1, bool INV, typename Len, typename Load>
__device__ __forceinline__ void fft2_phase_a(typename Cx<R>::T* __restrict__ buf, const Len& L, int nlines,
                                             const typename Cx<R>::T* __restrict__ tw, Load& load) {
    using C = typename Cx<R>::T;
    const int f2 = L.f2, total = nlines * f2;
    for (int task = threadIdx.x; task < total; task += blockDim.x) {
        const int line = L.by_f2(task), t = task - line * f2;
        C v[F1];
#pragma unroll
        for (int j = 0; j < F1; ++j) v[j] = load(line, t + f2 * j);
        SmallDft<R, F1, INV>::run(v);
#pragma unroll
        for (int k = 1; k < F1; ++k) {
            C w = tw[k * f2 + t];   // w_n^{t k}: lanes over t read consecutive values
            if (INV) w.y = -w.y;
            v[k] = cmul(v[k], w);
        }
        C* d = buf + line * L.lsa + t;
#pragma unroll
        for (int k = 0; k < F1; ++k) d[k * (f2 + 1)] = v[k];
    }
}

template <typename R, int F2, bool INV, typename Len, typename Store>
__device__ __forceinline__ void fft2_phase_b(const typename Cx<R>::T* __restrict__ buf, const Len& L, int nlines,
                                             Store& store) {
    using C = typename Cx<R>::T;
    const int f1 = L.f1, total = nlines * f1;
    for (int task = threadIdx.x; task < total; task += blockDim.x) {
        const int line = L.by_f1(task), k1 = task - line * f1;
        const C* s = buf + line * L.lsa + k1 * (F2 + 1);
        C u[F2];
#pragma unroll
        for (int t = 0; t < F2; ++t) u[t] = s[t];
        SmallDft<R, F2, INV>::run(u);
#pragma unroll
        for (int k2 = 0; k2 < F2; ++k2) store(line, k1 + f1 * k2, u[k2]);
    }
}

// The twiddle table of phase A in shared memory, tw[k f2 + t] = w_n^{t k}
// (t < f2, k < f1; forward sign), from the table twg[m] = w_n^m: the lanes of
// a phase-A step read consecutive values (the natural table, read at t k,
// puts lanes of an even k on few banks).
template <typename C, typename Len>
__device__ __forceinline__ void fft2_twiddles(C* __restrict__ tw, const C* __restrict__ twg, const Len& L) {
    for (int e = threadIdx.x; e < L.n; e += blockDim.x) {
        const int k = L.by_f2(e), t = e - k * L.f2;
        tw[e] = twg[t * k];
    }
}

// The whole two-factor transform of nlines lines: load(line, m) gives element
// m of a line, store(line, k, X_k) takes the results; tw is the table that
// fft2_twiddles fills. buf holds nlines rows of L.lsa values. Contains
// __syncthreads (call from all threads); the caller synchronises before
// reading what store wrote to shared memory.
template <typename R, bool INV, typename Len, typename Load, typename Store>
__device__ __forceinline__ void fft2_lines(typename Cx<R>::T* __restrict__ buf, const typename Cx<R>::T* tw,
                                           const Len& L, int nlines, Load&& load, Store&& store) {
    if constexpr (Len::kF1 > 0) {
        fft2_phase_a<R, Len::kF1, INV>(buf, L, nlines, tw, load);
        __syncthreads();
        fft2_phase_b<R, Len::kF2, INV>(buf, L, nlines, store);
    } else {
        switch (L.f1) {
            case 4: fft2_phase_a<R, 4, INV>(buf, L, nlines, tw, load); break;
            case 5: fft2_phase_a<R, 5, INV>(buf, L, nlines, tw, load); break;
            case 6: fft2_phase_a<R, 6, INV>(buf, L, nlines, tw, load); break;
            case 8: fft2_phase_a<R, 8, INV>(buf, L, nlines, tw, load); break;
            case 10: fft2_phase_a<R, 10, INV>(buf, L, nlines, tw, load); break;
            case 12: fft2_phase_a<R, 12, INV>(buf, L, nlines, tw, load); break;
            case 16: fft2_phase_a<R, 16, INV>(buf, L, nlines, tw, load); break;
            case 20: fft2_phase_a<R, 20, INV>(buf, L, nlines, tw, load); break;
            default: break;
        }
        __syncthreads();
        switch (L.f2) {
            case 4: fft2_phase_b<R, 4, INV>(buf, L, nlines, store); break;
            case 5: fft2_phase_b<R, 5, INV>(buf, L, nlines, store); break;
            case 6: fft2_phase_b<R, 6, INV>(buf, L, nlines, store); break;
            case 8: fft2_phase_b<R, 8, INV>(buf, L, nlines, store); break;
            case 10: fft2_phase_b<R, 10, INV>(buf, L, nlines, store); break;
            case 12: fft2_phase_b<R, 12, INV>(buf, L, nlines, store); break;
            case 16: fft2_phase_b<R, 16, INV>(buf, L, nlines, store); break;
            case 20: fft2_phase_b<R, 20, INV>(buf, L, nlines, store); break;
            default: break;
        }
    }
}

// Lines per CTA of the passes: what fits a shared-memory budget beside the
// twiddle table. ab: transforms held per line (phase-A and result rows);
// extra: further bytes per line (input buffers of the persistent passes).
__host__ __device__ constexpr int fft2_lines_for(int f1, int f2, int csz, int ab, int extra, int budget, int cap) {
    const int n = f1 * f2, per = ab * (fft2_lsa(f1, f2) + fft2_lsb(n)) * csz + extra;
    const int l = (budget - n * csz - 16) / per;
    return l < 1 ? 1 : (l > cap ? cap : l);
}
constexpr int kFftPipe = 72 * 1024;   // persistent passes: three CTAs per SM
constexpr int kFftLine = 64 * 1024;
// x: input rows double buffered; inverse x: LP line pairs of each of nf fields,
// Hermitian rows double buffered
__host__ __device__ constexpr int fft2_lx(int f1, int f2) { return fft2_lines_for(f1, f2, 8, 1, 16 * f1 * f2, kFftPipe, 64); }
__host__ __device__ constexpr int fft2_lz(int f1, int f2, int ni) {
    return fft2_lines_for(f1, f2, 8, ni, 16 * f1 * f2, kFftPipe, 64);
}
__host__ __device__ constexpr int fft2_lix(int f1, int f2, int nf) {
    return fft2_lines_for(f1, f2, 8, nf, nf * 32 * (f1 * f2 / 4), kFftPipe, 64);
}

// Lines per CTA of the y passes: runs of a multiple of 4 values (32-byte
// sectors) in the transposed output.
__host__ __device__ constexpr int fft2_ly(int f1, int f2) {
    const int l = fft2_lines_for(f1, f2, 8, 1, 0, kFftLine, 16);
    return l >= 4 ? l / 4 * 4 : l;
}

// Field a's spectrum after the z pass: which array of spec3 holds it and the
// factor of the mode (kx, ky). With three fields the z pass transforms back G
// and kz G; x and y are kx G and ky G.
__device__ __forceinline__ int spec3_array(int nf, int a) { return nf == 3 && a == 2 ? 1 : 0; }
template <typename R>
__device__ __forceinline__ R spec3_factor(int nf, int a, int kx, int ky) {
    return nf == 3 && a < 2 ? (R)(a == 0 ? kx : ky) : (R)1;
}

// Lengths with instances of their own: every n <= 112 of two radices (plane
// passes), every larger one up to 400, and 108 in both forms.
#define ENUF_FFT2_PLANES_A(X) X(4, 4) X(4, 5) X(4, 6) X(4, 8) X(6, 6) X(5, 8) X(6, 8)
#define ENUF_FFT2_PLANES_B(X) X(6, 10) X(8, 8) X(6, 12) X(8, 10) X(8, 12) X(10, 10) X(9, 12)
#define ENUF_FFT2_LINES_A(X) X(9, 12) X(10, 12) X(8, 16) X(12, 12) X(10, 16)
#define ENUF_FFT2_LINES_B(X) X(12, 15) X(12, 16) X(10, 20) X(12, 18)
#define ENUF_FFT2_LINES_C(X) X(12, 20) X(16, 16) X(16, 18) X(15, 20)
#define ENUF_FFT2_LINES_D(X) X(16, 20) X(18, 18) X(18, 20) X(20, 20)
#define ENUF_FFT2_PLANES(X) ENUF_FFT2_PLANES_A(X) ENUF_FFT2_PLANES_B(X)
#define ENUF_FFT2_LINES(X) ENUF_FFT2_LINES_A(X) ENUF_FFT2_LINES_B(X) ENUF_FFT2_LINES_C(X) ENUF_FFT2_LINES_D(X)

// Two-factor split n = f1 f2: both factors in the radix set of the any-length
// kernels; the most balanced split, ties to the larger f2 (phase A reads f2
// consecutive elements per line and load). Lengths without such a split (108,
// 180, 216, 288, 300, 324, 360) take radices 9, 15 and 18 as well (ext), which only
// kernels of single lengths have. f1 = 0: none.
struct Fft2Split {
    int f1, f2;
    bool ext;
};
constexpr Fft2Split fft2_split(int n) {
    constexpr int set[] = {4, 5, 6, 8, 10, 12, 16, 20, 9, 15, 18};   // the first eight: any length
    Fft2Split best{0, 0, false};
    for (int k = 8; k <= 11 && !best.f1; k += 3)
        for (int i = 0; i < k; ++i)
            for (int j = 0; j < k; ++j) {
                const int a = set[i], b = set[j];
                if (a * b != n) continue;
                const int m = a < b ? a : b, mb = best.f1 < best.f2 ? best.f1 : best.f2;
                if (!best.f1 || m > mb || (m == mb && b > best.f2)) best = Fft2Split{a, b, k > 8};
            }
    return best;
}

// The plane passes hold the twiddles, the n/2 phase-A rows and n/2 result rows of
// a z-plane; taken up to this size.
constexpr int kFftPlaneSmem = 100 * 1024;
__host__ __device__ constexpr int fft2_smem_xy(int f1, int f2, int csz) {
    return (f1 * f2 + (f1 * f2 / 2) * (fft2_lsa(f1, f2) + fft2_lsb(f1 * f2))) * csz;
}

// Every split that a plan (n = 2 M, M even, n <= 1024) can take has its kernels:
// plane passes of that length where they are chosen, line passes of that length
// where a factor is 9, 15 or 18 (the any-length kernels would leave such lines
// untransformed).
constexpr bool fft2_splits_covered() {
#define ENUF_IS(a, b) || (s.f1 == a && s.f2 == b)
    for (int n = 8; n <= 1024; n += 4) {
        const Fft2Split s = fft2_split(n);
        if (!s.f1) continue;
        if (fft2_smem_xy(s.f1, s.f2, 8) <= kFftPlaneSmem && !(false ENUF_FFT2_PLANES(ENUF_IS))) return false;
        if (s.ext && !(false ENUF_FFT2_LINES(ENUF_IS))) return false;
    }
#undef ENUF_IS
    return true;
}
static_assert(fft2_splits_covered(), "a two-factor split without kernels");

// body(f1, f2) with the split of fp as constants: every split of the plane passes is
// in the list (fft2_splits_covered), the default is never taken. It stays because the
// compiler's layout of these kernels without it is slower, though with fewer registers
// and no spill: 40 systems of 3000 to 20,000 beads 301 us against 293, 16 systems 281
// against 277 (64 systems the same).
template <typename Body>
__device__ __forceinline__ void fft2_by_length(const FftPlanDev& fp, Body body) {
    switch (32 * fp.f1 + fp.f2) {
#define ENUF_CASE(a, b) \
    case 32 * a + b: body(std::integral_constant<int, a>{}, std::integral_constant<int, b>{}); break;
        ENUF_FFT2_PLANES(ENUF_CASE)
#undef ENUF_CASE
        default: body(std::integral_constant<int, 0>{}, std::integral_constant<int, 0>{});
    }
}

}  // namespace enuf
