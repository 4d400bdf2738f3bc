// ss_fft.cuh -- batched complex FFTs of lines held in shared memory (Sec. II-A: the dipole field as a
// zero-padded convolution evaluated with FFTs).
//
// Lines of length P (P = 2^a 3^b) sit in shared memory with stride LS = fft_line_stride(P); element i
// of a line is stored at fft_pad(i) (one padding slot per 16 elements against bank conflicts).  The
// transform is a mixed-radix Stockham autosort FFT (radices 8, 4, 3, 2) done in place: in each stage
// every thread reads its butterflies' inputs into registers, the block synchronises, and the outputs
// are written to their autosorted positions.  Twiddles W_P^k = exp(-2 pi i k / P) come from a table in
// shared memory that the host computed in FP64.  Forward transforms only; an inverse is obtained by
// conjugating on load and on store.
#pragma once
#include "ss_internal.h"

namespace ss {

template <typename C> __device__ __forceinline__ C cadd(C a, C b) { return C{a.x + b.x, a.y + b.y}; }
template <typename C> __device__ __forceinline__ C csub(C a, C b) { return C{a.x - b.x, a.y - b.y}; }
template <typename C> __device__ __forceinline__ C cmul(C a, C b) {
    return C{a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x};
}
// FP32 sums as one paired (two-lane) FP32 instruction each
__device__ __forceinline__ float2 cadd(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float2 csub(float2 a, float2 b) { return __fadd2_rn(a, make_float2(-b.x, -b.y)); }
template <typename C> __device__ __forceinline__ C cconj(C a) { return C{a.x, -a.y}; }
// multiply by -i
template <typename C> __device__ __forceinline__ C cmi(C a) { return C{a.y, -a.x}; }

// Size-R forward DFTs in registers.
template <int R, typename C> struct Dft;

template <typename C> struct Dft<2, C> {
    static __device__ __forceinline__ void run(C* v) {
        C a = v[0];
        v[0] = cadd(a, v[1]);
        v[1] = csub(a, v[1]);
    }
};

template <typename C> struct Dft<3, C> {
    static __device__ __forceinline__ void run(C* v) {
        using R = decltype(v[0].x);
        const R h = R(0.8660254037844386467637231707529362);  // sqrt(3)/2
        C s = cadd(v[1], v[2]);
        C d = csub(v[1], v[2]);
        C m = C{v[0].x - R(0.5) * s.x, v[0].y - R(0.5) * s.y};
        C r = cmi(d);  // -i d
        v[0] = cadd(v[0], s);
        v[1] = C{m.x + h * r.x, m.y + h * r.y};
        v[2] = C{m.x - h * r.x, m.y - h * r.y};
    }
};

template <typename C> struct Dft<4, C> {
    static __device__ __forceinline__ void run(C* v) {
        C a = cadd(v[0], v[2]), b = csub(v[0], v[2]);
        C c = cadd(v[1], v[3]), d = cmi(csub(v[1], v[3]));
        v[0] = cadd(a, c);
        v[2] = csub(a, c);
        v[1] = cadd(b, d);
        v[3] = csub(b, d);
    }
};

template <typename C> struct Dft<8, C> {
    static __device__ __forceinline__ void run(C* v) {
        using R = decltype(v[0].x);
        const R q = R(0.7071067811865475244008443621048490);  // sqrt(2)/2
        C e[4] = {v[0], v[2], v[4], v[6]};
        C o[4] = {v[1], v[3], v[5], v[7]};
        Dft<4, C>::run(e);
        Dft<4, C>::run(o);
        // twiddles W8^k, k = 0..3: 1, (q,-q), -i, (-q,-q)
        C t1 = C{q * (o[1].x + o[1].y), q * (o[1].y - o[1].x)};
        C t2 = cmi(o[2]);
        C t3 = C{q * (o[3].y - o[3].x), -q * (o[3].x + o[3].y)};
        v[0] = cadd(e[0], o[0]);
        v[4] = csub(e[0], o[0]);
        v[1] = cadd(e[1], t1);
        v[5] = csub(e[1], t1);
        v[2] = cadd(e[2], t2);
        v[6] = csub(e[2], t2);
        v[3] = cadd(e[3], t3);
        v[7] = csub(e[3], t3);
    }
};

// Size 6 and 12 by Cooley-Tukey over 3 x 2 and 3 x 4 (n = M n1 + n2, k = k1 + 3 k2 with M = 2 or 4):
// 3-point DFTs over n1 for each n2, the twiddles W_N^{n2 k1}, then 2- or 4-point DFTs over n2.
template <typename C> struct Dft<6, C> {
    static __device__ __forceinline__ void run(C* v) {
        using R = decltype(v[0].x);
        const R h = R(0.8660254037844386467637231707529362);  // sqrt(3)/2
        C a[3] = {v[0], v[2], v[4]}, b[3] = {v[1], v[3], v[5]};
        Dft<3, C>::run(a);
        Dft<3, C>::run(b);
        b[1] = cmul(b[1], C{R(0.5), -h});    // W_6^1
        b[2] = cmul(b[2], C{R(-0.5), -h});   // W_6^2
#pragma unroll
        for (int k1 = 0; k1 < 3; ++k1) {
            v[k1] = cadd(a[k1], b[k1]);
            v[k1 + 3] = csub(a[k1], b[k1]);
        }
    }
};

template <typename C> struct Dft<12, C> {
    static __device__ __forceinline__ void run(C* v) {
        using R = decltype(v[0].x);
        const R h = R(0.8660254037844386467637231707529362);  // sqrt(3)/2
        C a[4][3];
#pragma unroll
        for (int n2 = 0; n2 < 4; ++n2) {
            a[n2][0] = v[n2];
            a[n2][1] = v[4 + n2];
            a[n2][2] = v[8 + n2];
            Dft<3, C>::run(a[n2]);
        }
        // W_12^{n2 k1}: n2 k1 in {1, 2, 2, 3, 4, 6}
        a[1][1] = cmul(a[1][1], C{h, R(-0.5)});      // W_12^1
        a[1][2] = cmul(a[1][2], C{R(0.5), -h});      // W_12^2
        a[2][1] = cmul(a[2][1], C{R(0.5), -h});      // W_12^2
        a[2][2] = cmul(a[2][2], C{R(-0.5), -h});     // W_12^4
        a[3][1] = cmi(a[3][1]);                      // W_12^3 = -i
        a[3][2] = C{-a[3][2].x, -a[3][2].y};         // W_12^6 = -1
#pragma unroll
        for (int k1 = 0; k1 < 3; ++k1) {
            C q[4] = {a[0][k1], a[1][k1], a[2][k1], a[3][k1]};
            Dft<4, C>::run(q);
#pragma unroll
            for (int k2 = 0; k2 < 4; ++k2) v[k1 + 3 * k2] = q[k2];
        }
    }
};

// ---- further DFT sizes of the two-pass transforms: primes 5 and 7, and composites by Cooley-Tukey -------
// cos(2 pi k / n) and sin(2 pi k / n) at compile time: the angle reduced exactly to [0, pi/4] in integers,
// then the Taylor series (its terms fall below 1e-19 well before the loop ends).
struct CxCs {
    double c, s;
};
__host__ __device__ constexpr CxCs cx_cos_sin(int k, int n) {
    long m = 4L * (((k % n) + n) % n);  // angle = 2 pi m / D, D = 4 n
    const long D = 4L * n;
    bool neg_s = false, neg_c = false, swap = false;
    if (2 * m > D) m = D - m, neg_s = true;
    if (4 * m > D) m = D / 2 - m, neg_c = true;
    if (8 * m > D) m = D / 4 - m, swap = true;
    const double x = 6.283185307179586476925286766559 * (double)m / (double)D;
    double c = 0.0, s = 0.0, t = 1.0;
    for (int i = 0; i < 24; ++i) {  // t = x^i / i! with the sign of the series' pairs
        if (i % 2 == 0)
            c += (i % 4 == 0) ? t : -t;
        else
            s += (i % 4 == 1) ? t : -t;
        t *= x / (double)(i + 1);
    }
    const double cc = swap ? s : c, ss = swap ? c : s;
    return CxCs{neg_c ? -cc : cc, neg_s ? -ss : ss};
}
// y + a x with a real
template <typename C> __device__ __forceinline__ C caxpy(decltype(C{}.x) a, C x, C y) {
    return C{y.x + a * x.x, y.y + a * x.y};
}
__device__ __forceinline__ float2 caxpy(float a, float2 x, float2 y) { return __ffma2_rn(make_float2(a, a), x, y); }

// y + a x for scalars and pairs alike
template <typename T> __device__ __forceinline__ T caxpy_v(T a, T x, T y) { return y + a * x; }
__device__ __forceinline__ float2 caxpy_v(float a, float2 x, float2 y) { return caxpy(a, x, y); }
// v with its sign flipped where the top bit of s is set
__device__ __forceinline__ float flip_sign(float v, unsigned s) { return __uint_as_float(__float_as_uint(v) ^ s); }
__device__ __forceinline__ double flip_sign(double v, unsigned s) {
    return __hiloint2double(__double2hiint(v) ^ (int)s, __double2loint(v));
}
// f v, or conj(f v), for a real f = +-1 given as its sign bit: one paired multiplication in FP32, bit operations in
// FP64, whose pipe is the narrow one
__device__ __forceinline__ float2 sign_mul(float2 v, unsigned f, bool conj) {
    const float a = flip_sign(1.f, f);
    return __fmul2_rn(make_float2(a, conj ? -a : a), v);
}
__device__ __forceinline__ double2 sign_mul(double2 v, unsigned f, bool conj) {
    return make_double2(flip_sign(v.x, f), flip_sign(v.y, conj ? f ^ 0x80000000u : f));
}

template <int I> struct ic {
    static constexpr int v = I;
};
template <int I, int N, typename F> __device__ __forceinline__ void static_for(F f) {
    if constexpr (I < N) {
        f(ic<I>{});
        static_for<I + 1, N>(f);
    }
}
// a * W_N^K, W_N = exp(-2 pi i / N)
template <int K, int N, typename C> __device__ __forceinline__ C mul_w(C a) {
    using R = decltype(a.x);
    constexpr int k = K % N;
    if constexpr (k == 0) {
        return a;
    } else if constexpr (4 * k == N) {
        return cmi(a);
    } else if constexpr (2 * k == N) {
        return C{-a.x, -a.y};
    } else if constexpr (4 * k == 3 * N) {
        return C{-a.y, a.x};
    } else {
        constexpr CxCs w = cx_cos_sin(k, N);
        return cmul(a, C{R(w.c), R(-w.s)});
    }
}

template <typename C> struct Dft<1, C> {
    static __device__ __forceinline__ void run(C*) {}
};

// Odd prime R: with s_j = v_j + v_{R-j} and d_j = v_j - v_{R-j}, X_k and X_{R-k} are
// v_0 + sum_j s_j cos(2 pi j k / R) -+ i sum_j d_j sin(2 pi j k / R), 1 <= j, k <= (R-1)/2.
template <int R, typename C> struct DftPrime {
    static __device__ __forceinline__ void run(C* v) {
        using Re = decltype(v[0].x);
        constexpr int M = (R - 1) / 2;
        C s[M], d[M];
#pragma unroll
        for (int j = 0; j < M; ++j) {
            s[j] = cadd(v[1 + j], v[R - 1 - j]);
            d[j] = csub(v[1 + j], v[R - 1 - j]);
        }
        const C v0 = v[0];
#pragma unroll
        for (int j = 0; j < M; ++j) v[0] = cadd(v[0], s[j]);
        static_for<1, M + 1>([&](auto kk) {
            constexpr int k = decltype(kk)::v;
            C a = v0, b = C{Re(0), Re(0)};
            static_for<1, M + 1>([&](auto jj) {
                constexpr int j = decltype(jj)::v;
                constexpr CxCs w = cx_cos_sin(j * k, R);
                a = caxpy(Re(w.c), s[j - 1], a);
                b = caxpy(Re(w.s), d[j - 1], b);
            });
            const C r = cmi(b);
            v[k] = cadd(a, r);
            v[R - k] = csub(a, r);
        });
    }
};
template <typename C> struct Dft<5, C> : DftPrime<5, C> {};
template <typename C> struct Dft<7, C> : DftPrime<7, C> {};

// N = N1 N2 by Cooley-Tukey (n = N2 n1 + n2, k = k1 + N1 k2): N1-point DFTs over n1 for each n2, the
// twiddles W_N^{n2 k1}, then N2-point DFTs over n2.
template <int N1, int N2, typename C> struct DftCt {
    static __device__ __forceinline__ void run(C* v) {
        constexpr int N = N1 * N2;
        C a[N2][N1];
        static_for<0, N2>([&](auto nn) {
            constexpr int n2 = decltype(nn)::v;
#pragma unroll
            for (int n1 = 0; n1 < N1; ++n1) a[n2][n1] = v[N2 * n1 + n2];
            Dft<N1, C>::run(a[n2]);
            static_for<0, N1>([&](auto kk) {
                constexpr int k1 = decltype(kk)::v;
                a[n2][k1] = mul_w<n2 * k1, N>(a[n2][k1]);
            });
        });
#pragma unroll
        for (int k1 = 0; k1 < N1; ++k1) {
            C q[N2];
#pragma unroll
            for (int n2 = 0; n2 < N2; ++n2) q[n2] = a[n2][k1];
            Dft<N2, C>::run(q);
#pragma unroll
            for (int k2 = 0; k2 < N2; ++k2) v[k1 + N1 * k2] = q[k2];
        }
    }
};
template <typename C> struct Dft<9, C> : DftCt<3, 3, C> {};
template <typename C> struct Dft<10, C> : DftCt<5, 2, C> {};
template <typename C> struct Dft<14, C> : DftCt<7, 2, C> {};
template <typename C> struct Dft<16, C> : DftCt<4, 4, C> {};
template <typename C> struct Dft<18, C> : DftCt<3, 6, C> {};
template <typename C> struct Dft<20, C> : DftCt<5, 4, C> {};
template <typename C> struct Dft<24, C> : DftCt<3, 8, C> {};

// Host-side plan: radices 8, 4, 2 first (largest first), then 3s, 5s and 7s (the last two only in the setup
// transforms of the tensor spectrum: padded_lengths gives a length with those factors to two-pass kernels alone).
inline FftPlan fft_make_plan(int P) {
    FftPlan p{};
    p.P = P;
    int a = 0, b = 0, c5 = 0, c7 = 0, q = P;
    while (q % 2 == 0) q /= 2, ++a;
    while (q % 3 == 0) q /= 3, ++b;
    while (q % 5 == 0) q /= 5, ++c5;
    while (q % 7 == 0) q /= 7, ++c7;
    int n = 0;
    const int n8 = a / 3, rem = a % 3;
    if (rem == 1 && n8 == 0) {
        p.radix[n++] = 2;
    } else {
        const int eights = rem == 1 ? n8 - 1 : n8;
        for (int i = 0; i < eights; ++i) p.radix[n++] = 8;
        if (rem == 1) {
            p.radix[n++] = 4;
            p.radix[n++] = 4;
        }
        if (rem == 2) p.radix[n++] = 4;
    }
    for (int i = 0; i < b; ++i) p.radix[n++] = 3;
    for (int i = 0; i < c5; ++i) p.radix[n++] = 5;
    for (int i = 0; i < c7; ++i) p.radix[n++] = 7;
    p.nstages = n;
    int ns = 1;
    for (int s = 0; s < n; ++s) {
        const int R = p.radix[s];
        p.q[s] = P / R;
        p.ns[s] = ns;
        p.tw[s] = P / (ns * R);
        p.ns_mask[s] = (ns & (ns - 1)) == 0 ? ns - 1 : -1;
        ns *= R;
    }
    return p;
}

// The kernels of the runtime plans have stages for the plan's radices: fft_lines without R57.
inline bool fft_plan_2348(const FftPlan& p) {
    for (int s = 0; s < p.nstages; ++s)
        if (p.radix[s] == 5 || p.radix[s] == 7) return false;
    return true;
}

// Elements each thread holds in registers per stage: 8 (9 for radix 3).  Lines are transformed in
// passes of fft_lines_per_pass() lines, so any block of at least P/8 threads can transform any number
// of lines.
template <int R> struct StageCap { static constexpr int B = R == 2 ? 4 : R == 3 ? 3 : R == 8 ? 1 : 2; };
constexpr int kFftElemsPerThread = 8;

__host__ __device__ inline int fft_lines_per_pass(int nthr, int P) { return (nthr * kFftElemsPerThread) / P; }
// Smallest block that can transform lines of length P.
__host__ __device__ inline int fft_min_threads(int P) { return (P + kFftElemsPerThread - 1) / kFftElemsPerThread; }

template <int R, typename C>
__device__ __forceinline__ void fft_stage(C* buf, const C* tw, int LS, int L, int Q, int Ns, int twstep, int ns_mask,
                                          int tid, int nthr) {
    constexpr int B = StageCap<R>::B;
    // butterfly b = tid + i*nthr of the pass: line = b / Q, j = b % Q, advanced without divisions
    int line = tid / Q;
    int j = tid - line * Q;
    const int dl = nthr / Q, dj = nthr - dl * Q;
    C v[B][R];
    int dline[B], de[B];
#pragma unroll
    for (int i = 0; i < B; ++i) {
        dline[i] = -1;
        de[i] = 0;
        if (line < L) {
            const int jm = ns_mask >= 0 ? (j & ns_mask) : (j % Ns);
            const C* src = buf + line * LS;
#pragma unroll
            for (int r = 0; r < R; ++r) {
                C x = src[fft_pad(j + r * Q)];
                if (r > 0) x = cmul(x, tw[jm * r * twstep]);
                v[i][r] = x;
            }
            Dft<R, C>::run(v[i]);
            dline[i] = line * LS;
            de[i] = (j - jm) * R + jm;
        }
        j += dj;
        line += dl;
        if (j >= Q) {
            j -= Q;
            ++line;
        }
    }
    __syncthreads();
#pragma unroll
    for (int i = 0; i < B; ++i) {
        if (dline[i] >= 0) {
#pragma unroll
            for (int r = 0; r < R; ++r) buf[dline[i] + fft_pad(de[i] + r * Ns)] = v[i][r];
        }
    }
    __syncthreads();
}

// Forward FFT of L lines (stride LS, elements at fft_pad positions) in shared memory.  Must be called
// by every thread of the block, with blockDim.x >= fft_min_threads(P).  Ends synchronised.  R57: the plan
// may hold radices 5 and 7 (setup).  Kernels without them are compiled without their cases: empty ones in the switch cost
// the runtime-plan y/z kernel 2 to 3% (481x450x1 x 9 images, 1024 points: 306.4 us with, 301.0 without on one GB300;
// 168x9x4 x 40: 187.9 and 181.5).
template <bool R57 = false, typename C>
__device__ __forceinline__ void fft_lines(C* buf, const C* tw, const FftPlan& plan, int LS, int L, int tid, int nthr) {
    const int lpp = max(1, fft_lines_per_pass(nthr, plan.P));  // the host guarantees >= 1; never loop forever
    for (int l0 = 0; l0 < L; l0 += lpp) {
        const int nl = min(lpp, L - l0);
        C* b = buf + l0 * LS;
        for (int st = 0; st < plan.nstages; ++st) {
            const int Q = plan.q[st], Ns = plan.ns[st], tws = plan.tw[st], msk = plan.ns_mask[st];
            if constexpr (R57) {
                if (plan.radix[st] == 5) {
                    fft_stage<5>(b, tw, LS, nl, Q, Ns, tws, msk, tid, nthr);
                    continue;
                }
                if (plan.radix[st] == 7) {
                    fft_stage<7>(b, tw, LS, nl, Q, Ns, tws, msk, tid, nthr);
                    continue;
                }
            }
            switch (plan.radix[st]) {
                case 8: fft_stage<8>(b, tw, LS, nl, Q, Ns, tws, msk, tid, nthr); break;
                case 4: fft_stage<4>(b, tw, LS, nl, Q, Ns, tws, msk, tid, nthr); break;
                case 3: fft_stage<3>(b, tw, LS, nl, Q, Ns, tws, msk, tid, nthr); break;
                default: fft_stage<2>(b, tw, LS, nl, Q, Ns, tws, msk, tid, nthr); break;
            }
        }
    }
}

// ---- multiplications by 16th roots of unity
// a * W_16^J for a compile-time J < 8, W_16 = exp(-2 pi i / 16)
template <int J, typename C> __device__ __forceinline__ C mul_w16(C a) {
    using R = decltype(a.x);
    constexpr double c1 = 0.923879532511286756128183189396788933;  // cos(pi/8)
    constexpr double s1 = 0.382683432365089771728459984030398866;  // sin(pi/8)
    constexpr double h = 0.707106781186547524400844362104849039;   // cos(pi/4)
    if constexpr (J == 0) {
        return a;
    } else if constexpr (J == 4) {
        return cmi(a);
    } else if constexpr (J == 2) {
        return C{R(h) * (a.x + a.y), R(h) * (a.y - a.x)};
    } else if constexpr (J == 6) {
        return C{R(h) * (a.y - a.x), R(-h) * (a.x + a.y)};
    } else {
        constexpr double cr = J == 1 ? c1 : J == 3 ? s1 : J == 5 ? -s1 : -c1;
        constexpr double ci = J == 1 ? -s1 : J == 3 ? -c1 : J == 5 ? -c1 : -s1;
        return cmul(a, C{R(cr), R(ci)});
    }
}
template <typename C> __device__ __forceinline__ void mul_w16_ramp(C (&u)[8]) {
    u[1] = mul_w16<1>(u[1]);
    u[2] = mul_w16<2>(u[2]);
    u[3] = mul_w16<3>(u[3]);
    u[4] = mul_w16<4>(u[4]);
    u[5] = mul_w16<5>(u[5]);
    u[6] = mul_w16<6>(u[6]);
    u[7] = mul_w16<7>(u[7]);
}

// ---- lengths P = 16 R2 (R2 = 2..32: 32 to 512) in two register passes ------------------------------------
// A line of P elements is held in shared memory as R2 rows of 16 at row stride kT2Row = 17 (element
// (r, c) at r * 17 + c; a line takes kT2Row * R2 slots).  With n = R2 n1 + n2, k = k1 + 16 k2 (n1, k1 < 16;
// n2, k2 < R2) the forward transform is
//   X[k1 + 16 k2] = sum_{n2} W_R2^{n2 k2} Z[n2][k1],   Z[n2][k1] = W_P^{n2 k1} sum_{n1} W_16^{n1 k1} x[R2 n1 + n2]:
// pass 1, role n2, inputs x[R2 j + n2], j < 8 (the upper half of the line is zero): the 16-point DFT as two
//   8-point ones of x W_16^{j par}, par = 0, 1 -> row n2 of Z (k1 = 2m + par);
// pass 2, role k1, column k1 of Z: the R2-point DFT -> X[k1 + 16 k2], written back in place into column k1
//   (row k2), so X[ky] sits at (ky >> 4) * 17 + (ky & 15).
// The inverse direction (a forward transform of the conjugate) starts from that column layout: with
// y = y2 + R2 y1,
//   Y[y2 + R2 y1] = sum_{k1} W_16^{k1 y1} T[k1][y2],   T[k1][y2] = W_P^{k1 y2} sum_{k2} W_R2^{k2 y2} V[k1 + 16 k2];
// pass A, role k1, column k1: the R2-point DFT as in pass 2, times W_P^{k1 y2}, back into column k1 (row y2);
// pass B, role y2, row y2: the outputs below P/2, Y[y2 + R2 y1], y1 = 2m + par < 8, from 8-point DFTs of
//   (T[j][y2] +- T[j+8][y2]) W_16^{j par}.
// So every element crosses shared memory once per pass.  (Roles of one parity each, with half the registers,
// read every element twice: the y/z kernel of 64x64x8 spent 75% of its time's L1 wavefronts there.)  From
// R2 = 28 on a whole column takes too many registers, and passes 2 and A take two roles per column, par2 = 0
// and 1, with the R2/2-point DFTs of the outputs of one parity.  The twiddles of pass 1 and pass A come from
// the tables of GroupArgs::t2x / t2y (t1 = the pass-1 half, ta = the pass-A half, indexed so that a warp's lanes
// read consecutive entries); the ramp W_R2^j = W_P^{16 j} of the split columns from the flat table tw (the
// same entry across a warp).
__device__ __forceinline__ int t2_at(int r, int c) { return r * kT2Row + c; }
__device__ __forceinline__ int t2_pos(int ky) { return t2_at(ky >> 4, ky & 15); }

// Pass 1 of a line whose upper half is zero: u[j] = x[R2 j + n2] (j < 8) on entry; writes row n2 of Z.
template <int P, typename C>
__device__ __forceinline__ void t2_pass1(C (&u)[8], int n2, const C* __restrict__ t1, C* line) {
    C w[8];
#pragma unroll
    for (int j = 0; j < 8; ++j) w[j] = u[j];
    mul_w16_ramp(w);
    Dft<8, C>::run(u);
#pragma unroll
    for (int m = 0; m < 8; ++m) line[t2_at(n2, 2 * m)] = cmul(u[m], t1[2 * m * (P / 16) + n2]);  // W_P^{2 m n2}
    Dft<8, C>::run(w);
#pragma unroll
    for (int m = 0; m < 8; ++m)
        line[t2_at(n2, 2 * m + 1)] = cmul(w[m], t1[(2 * m + 1) * (P / 16) + n2]);  // W_P^{(2 m + 1) n2}
}

// Roles per column of passes 2 and A (2: the output rows split by parity) and outputs per role.
template <int P> struct T2 {
    static constexpr int R2 = P / 16, NP = R2 > 24 ? 2 : 1, H = R2 / NP;
};

// The H-point DFTs of pass 2 (TW_OUT = false) or pass A (TW_OUT = true) for column k1 and parity par2:
// a[m] = the output of row NP m + par2 (times W_P^{k1 (NP m + par2)} in pass A).  col(j) returns the column's
// row j (from shared or global memory).
template <int P, bool TW_OUT, typename C, typename Col>
__device__ __forceinline__ void t2_col_vals(C (&a)[T2<P>::H], Col col, int k1, int par2, const C* __restrict__ tw,
                                            const C* __restrict__ ta) {
    constexpr int H = T2<P>::H, NP = T2<P>::NP;
    if constexpr (NP == 2) {
#pragma unroll
        for (int j = 0; j < H; ++j) {
            const C lo = col(j), hi = col(j + H);
            a[j] = par2 ? csub(lo, hi) : cadd(lo, hi);
        }
        if (par2) {
#pragma unroll
            for (int j = 1; j < H; ++j) a[j] = cmul(a[j], tw[16 * j]);  // W_R2^j
        }
    } else {
#pragma unroll
        for (int j = 0; j < H; ++j) a[j] = col(j);
    }
    Dft<H, C>::run(a);
    if constexpr (TW_OUT) {
#pragma unroll
        for (int m = 0; m < H; ++m) a[m] = cmul(a[m], ta[(NP * m + par2) * 16 + k1]);  // W_P^{k1 (NP m + par2)}
    }
}

// Pass 2 / pass A in place on a shared line: reads column k1, writes rows NP m + par2 of the same column.
// The caller pairs the roles par2 = 0 and 1 of a column in one warp; the column is read whole before
// either writes (a __syncwarp between the reads and the writes).
template <int P, bool TW_OUT, typename C>
__device__ __forceinline__ void t2_cols(C* line, int k1, int par2, const C* __restrict__ tw, const C* __restrict__ ta) {
    constexpr int H = T2<P>::H, NP = T2<P>::NP;
    C a[H];
    t2_col_vals<P, TW_OUT>(a, [&](int j) { return line[t2_at(j, k1)]; }, k1, par2, tw, ta);
    if constexpr (NP == 2) __syncwarp();
#pragma unroll
    for (int m = 0; m < H; ++m) line[t2_at(NP * m + par2, k1)] = a[m];
}

// Pass B of row y2: v[y1] = Y[y2 + R2 y1] for y1 < 8 (the outputs below P/2).
template <typename C>
__device__ __forceinline__ void t2_passB(C (&v)[8], const C* line, int y2) {
    C s[8], d[8];
#pragma unroll
    for (int j = 0; j < 8; ++j) {
        const C lo = line[t2_at(y2, j)], hi = line[t2_at(y2, j + 8)];
        s[j] = cadd(lo, hi);
        d[j] = csub(lo, hi);
    }
    Dft<8, C>::run(s);
    mul_w16_ramp(d);
    Dft<8, C>::run(d);
#pragma unroll
    for (int m = 0; m < 4; ++m) {
        v[2 * m] = s[m];
        v[2 * m + 1] = d[m];
    }
}

}  // namespace ss
