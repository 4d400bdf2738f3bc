// ss_twopass.cuh -- the y/z and x kernels whose transforms take two register passes (lengths P = 16 R2 of
// SS_T2_LENGTHS; ss_fft.cuh has the passes) and their launchers.  Each length is a translation unit of its
// own (ss_twopass.cu compiled with SS_T2_P defined), so that they compile in parallel.
#pragma once
#include "ss_kernels.cuh"

namespace ss {

// yz for a two-pass length Py = P (ny <= P/2), NZ layers, KXB kx columns per CTA: the y-transforms
// in two register passes each way (t2_pass1 / t2_cols / t2_passB, ss_fft.cuh) on lines held in the
// 17-strided row layout, the z-convolution in place between them.  One shared line per (column, component,
// layer): 3 NZ KXB lines of t2_line(P) complex elements, read from the spectrum in pass 1 and written back
// (rows y < ny) in pass B; one shared-memory round trip per pass instead of one per Stockham stage.
// Pass 2 and pass A take half a warp per line (16 columns; a warp with two roles per column from P = 448 on).
//
// The z-convolution works on sums and differences of mirrored layers.  A component of the tensor is even
// in z (t) or odd (G), so with n = NZ, e_i = s_i + s_{n-1-i}, o_i = s_i - s_{n-1-i} (i < n/2; the middle layer
// of an odd n is an e of its own) and the same for the field (a factor 2, taken into dhat), even components
// map e to e and o to o, odd ones e to o and o to e: two independent systems, (x, y in e; z in o) and
// (x, y in o; z in e), each a real symmetric matrix of a quarter of the elements.  With sg = +1 or -1 for the
// two, its blocks are t(|i-j|) + sg t(n-1-i-j) between x and y, t(|i-j|) - sg t(n-1-i-j) for zz, and
// G(i-j) + sg G(n-1-i-j) between x or y (row i) and i times z (row j), so every product is a real
// coefficient times a complex number.  Half the multiply-adds of the direct sum (144 instead of 192 + 96 per
// frequency and system at 8 layers), and each spectrum element is read from shared memory once instead of
// three times; the transforms are linear, so e and o are formed when pass 1 reads the layers and undone
// when pass B writes them.  Kernel times on one GB300 before and after: 192x192x8 x 128 images 1420 -> 1214 us,
// 128x128x8 x 192 788 -> 703, 128x128x4 x 384 733 -> 610, 100x100x5 x 32 79 -> 67, 112x112x1 x 60 (xz = yz = 0
// left out) 40.5 -> 28.6; with roles of whole columns and rows and small CTAs 928, 561, 481, 54 and 22.3.
template <int NZ, int PAR> struct ZSys {  // PAR 0: (x, y in e; z in o), 1: (x, y in o; z in e)
    static constexpr int ME = (NZ + 1) / 2, MO = NZ / 2;
    static constexpr int NXY = PAR == 0 ? ME : MO, NZC = PAR == 0 ? MO : ME;  // elements of x (and y), and of z
};

// One system at one frequency: A points at the frequency's element of line 0 (line stride LS), load(c, t) gets
// its coefficients of component c, |dz| = 0 .. NZ - 1; par the system; fx, fy the parity signs of kx, ky
// as sign bits (the tensor's xy, xz, yz are odd in them: flip x and y going in and coming out).  The result
// replaces the inputs, conjugated (the inverse transform is the conjugate of the forward transform of the conjugate).
template <int NZ, int PAR, int LS, typename T, typename C, typename LOAD>
__device__ __forceinline__ void zconv_sys(C* A, const LOAD& load, int par, unsigned fx, unsigned fy) {
    using S = ZSys<NZ, PAR>;  // the shape; for even NZ both systems share it and par picks one at run time
    constexpr int NA = S::NXY, NB = S::NZC;
    constexpr int NA1 = NA > 0 ? NA : 1, NB1 = NB > 0 ? NB : 1;
    const T sg = par ? T(-1) : T(1);
    C* Ax = A + (par ? S::ME : 0) * LS;
    C* Ay = Ax + NZ * LS;
    C* Az = A + (2 * NZ + (par ? 0 : S::ME)) * LS;
    C X[NA1], Y[NA1], Z[NB1], HX[NA1], HY[NA1], W[NB1];
    const C zero = C{T(0), T(0)};
#pragma unroll
    for (int i = 0; i < NA; ++i) {
        X[i] = sign_mul(Ax[i * LS], fx, false);
        Y[i] = sign_mul(Ay[i * LS], fy, false);
        HX[i] = HY[i] = zero;
    }
#pragma unroll
    for (int i = 0; i < NB; ++i) {
        const C z = Az[i * LS];
        Z[i] = C{-z.y, z.x};  // i z
        W[i] = zero;
    }
    // t(|i-j|) + s t(n-1-i-j) for an even component
    auto even = [&](const T (&t)[NZ], T s, int i, int j) {
        return t[i > j ? i - j : j - i] + s * t[NZ - 1 - i - j];
    };
    T t[NZ];
    if constexpr (NA > 0) {
        load(0, t);  // xx
#pragma unroll
        for (int i = 0; i < NA; ++i)
#pragma unroll
            for (int j = 0; j <= i; ++j) {
                const T c = even(t, sg, i, j);
                HX[i] = caxpy(c, X[j], HX[i]);
                if (j < i) HX[j] = caxpy(c, X[i], HX[j]);
            }
        load(3, t);  // xy
#pragma unroll
        for (int i = 0; i < NA; ++i)
#pragma unroll
            for (int j = 0; j <= i; ++j) {
                const T c = even(t, sg, i, j);
                HX[i] = caxpy(c, Y[j], HX[i]);
                HY[i] = caxpy(c, X[j], HY[i]);
                if (j < i) {
                    HX[j] = caxpy(c, Y[i], HX[j]);
                    HY[j] = caxpy(c, X[i], HY[j]);
                }
            }
        load(1, t);  // yy
#pragma unroll
        for (int i = 0; i < NA; ++i)
#pragma unroll
            for (int j = 0; j <= i; ++j) {
                const T c = even(t, sg, i, j);
                HY[i] = caxpy(c, Y[j], HY[i]);
                if (j < i) HY[j] = caxpy(c, Y[i], HY[j]);
            }
    }
    if constexpr (NA > 0 && NB > 0) {
        // G(i-j) + sg G(n-1-i-j), G(0) = 0: xz, then yz
        auto odd = [&](const T (&t)[NZ], int i, int j) {
            const int p = NZ - 1 - i - j;
            const T hank = p > 0 ? t[p] : p < 0 ? -t[-p] : T(0);
            return i == j ? sg * hank : (i > j ? t[i - j] : -t[j - i]) + sg * hank;
        };
        load(4, t);
#pragma unroll
        for (int i = 0; i < NA; ++i)
#pragma unroll
            for (int j = 0; j < NB; ++j) {
                const T c = odd(t, i, j);
                HX[i] = caxpy(c, Z[j], HX[i]);
                W[j] = caxpy(c, X[i], W[j]);
            }
        load(5, t);
#pragma unroll
        for (int i = 0; i < NA; ++i)
#pragma unroll
            for (int j = 0; j < NB; ++j) {
                const T c = odd(t, i, j);
                HY[i] = caxpy(c, Z[j], HY[i]);
                W[j] = caxpy(c, Y[i], W[j]);
            }
    }
#pragma unroll
    for (int i = 0; i < NA; ++i) {
        Ax[i * LS] = sign_mul(HX[i], fx, true);
        Ay[i * LS] = sign_mul(HY[i], fy, true);
    }
    if constexpr (NB > 0) {
        load(2, t);  // zz
#pragma unroll
        for (int i = 0; i < NB; ++i)
#pragma unroll
            for (int j = 0; j <= i; ++j) {
                const T c = even(t, -sg, i, j);
                W[i] = caxpy(c, Z[j], W[i]);
                if (j < i) W[j] = caxpy(c, Z[i], W[j]);
            }
#pragma unroll
        for (int i = 0; i < NB; ++i) Az[i * LS] = C{W[i].y, W[i].x};  // conj(-i W)
    }
}

// The z-convolution at one frequency of one column, in place.  par: the system, for the layer counts that take
// one item each (kZBoth: one item for both).
template <int NZ, typename T> constexpr bool kZBoth = sizeof(T) == 4 && NZ >= 2 && NZ <= 4;
template <int NZ, int P, typename T, typename C>
__device__ __forceinline__ void zconv_item(C* A, int kx, int ky, int par, int Px, const T* dslab) {
    constexpr int LS = t2_line(P), DQ = P / 2 + 1;
    const unsigned fx = kx > Px / 2 ? 0x80000000u : 0u;  // the parity signs of kx, ky, as sign bits
    const unsigned fy = ky > P / 2 ? 0x80000000u : 0u;
    const T* d = dslab + min(ky, P - ky);
    C* a = A + t2_pos(ky);
    if constexpr (NZ == 1) {  // xz and yz vanish
        const C X = a[0], Y = a[LS], Z = a[2 * LS];
        const T xx = d[0], yy = d[DQ], zz = d[2 * DQ], xy = flip_sign(d[3 * DQ], fx ^ fy);
        a[0] = C{xx * X.x + xy * Y.x, -(xx * X.y + xy * Y.y)};
        a[LS] = C{xy * X.x + yy * Y.x, -(xy * X.y + yy * Y.y)};
        a[2 * LS] = C{zz * Z.x, -zz * Z.y};
    } else {
        auto load = [&](int c, T (&t)[NZ]) {
#pragma unroll
            for (int q = 0; q < NZ; ++q) t[q] = d[(q * 6 + c) * DQ];
        };
        if constexpr (kZBoth<NZ, T>) {
            T all[6][NZ];
#pragma unroll
            for (int c = 0; c < 6; ++c) load(c, all[c]);
            auto kept = [&](int c, T (&t)[NZ]) {
#pragma unroll
                for (int q = 0; q < NZ; ++q) t[q] = all[c][q];
            };
            zconv_sys<NZ, 0, LS, T>(a, kept, 0, fx, fy);
            zconv_sys<NZ, 1, LS, T>(a, kept, 1, fx, fy);
        } else if constexpr (NZ % 2 == 0) {  // the two systems have the same shape
            zconv_sys<NZ, 0, LS, T>(a, load, par, fx, fy);
        } else if (par == 0) {
            zconv_sys<NZ, 0, LS, T>(a, load, 0, fx, fy);
        } else {
            zconv_sys<NZ, 1, LS, T>(a, load, 1, fx, fy);
        }
    }
}
// The z-convolution of the columns kx0 .. kx0 + KXB - 1.  FP32, two to four layers: an item takes both systems, so
// that the tensor's coefficients, as many bytes as the spectrum elements, are read once, and the columns' items
// run on in one loop.  Before and after on one GB300: 128x128x4 x 384 images 482 -> 462 us, 96x96x4 x 192 148 ->
// 141.  With more layers the coefficients do not fit in the registers, and one loop over the columns changed nothing
// at one layer and cost 9% at eight (28.2 -> 30.9 us, 64x64x8 x 32).
template <int NZ, int KXB, int P, typename T, typename C>
__device__ __forceinline__ void zconv_t2(C* A, int kx0, int Px, const T* dhat, int tid, int nthr) {
    constexpr int LS = t2_line(P), SLAB = (P / 2 + 1) * NZ * 6;
    if constexpr (kZBoth<NZ, T>) {
#pragma unroll 1
        for (int it = tid; it < KXB * P; it += nthr) {
            const int b = it / P, kx = kx0 + b;
            zconv_item<NZ, P>(A + b * 3 * NZ * LS, kx, it % P, 0, Px, dhat + (size_t)min(kx, Px - kx) * SLAB);
        }
    } else {
#pragma unroll 1
        for (int b = 0; b < KXB; ++b) {
            const int kx = kx0 + b;
            const T* dslab = dhat + (size_t)min(kx, Px - kx) * SLAB;
            for (int it = tid; it < (NZ == 1 ? P : 2 * P); it += nthr) {
                const int par = it >= P ? 1 : 0;
                zconv_item<NZ, P>(A + b * 3 * NZ * LS, kx, it - par * P, par, Px, dslab);
            }
        }
    }
}

template <typename T, int P, int NZ, int KXB>
__global__ void __launch_bounds__(yz2p_threads(sizeof(T), P), yz2p_blocks(sizeof(T), P)) yz2p_kernel(GroupArgs<T> g) {
    using C = cplx<T>;
    constexpr int R2 = P / 16, LS = t2_line(P), L = 3 * NZ * KXB, RC = 16 * T2<P>::NP;  // RC: roles per line
    constexpr int ME = (NZ + 1) / 2, MO = NZ / 2, LP = 3 * ME * KXB;                    // LP: pairs of mirrored layers
    extern __shared__ __align__(16) unsigned char smem_raw[];
    C* A = reinterpret_cast<C*>(smem_raw);  // line (b * 3 + c) * NZ + q: e_q for q < ME, o_{q - ME} above
    const int tid = threadIdx.x, nthr = yz2p_threads(sizeof(T), P);
    const int kx = blockIdx.x * KXB, p = blockIdx.y;
    const int ny = g.ny;
    if (sizeof(T) == 8 && g.pair_on && !g.pair_on[p]) return;  // uniform over the CTA
    C* blk = g.spec + ((size_t)p * g.Px + kx) * 3 * NZ * ny;  // KXB consecutive columns are contiguous
    const C* __restrict__ tw = g.twy;                         // W_P^k
    const C* __restrict__ t1 = g.t2y;                         // pass 1
    const C* __restrict__ ta = g.t2y + P;                     // pass A
    griddep_wait();
    griddep_launch_dependents();
    // pass 1, role (n2, mirrored pair of lines), n2 fastest: the zero-padded spectrum lines in, rows of Z of
    // their sum and difference out
    for (int r = tid; r < R2 * LP; r += nthr) {
        const int n2 = r % R2, lp = r / R2, bc = lp / ME, i = lp % ME;
        const C* src = blk + (size_t)(bc * NZ + i) * ny + n2;
        C u[8];
        if (MO == ME || i < MO) {
            const C* src2 = blk + (size_t)(bc * NZ + NZ - 1 - i) * ny + n2;
            C v[8];
#pragma unroll
            for (int j = 0; j < 8; ++j) {
                const bool in = R2 * j + n2 < ny;
                u[j] = in ? src[R2 * j] : C{T(0), T(0)};
                v[j] = in ? src2[R2 * j] : C{T(0), T(0)};
            }
#pragma unroll
            for (int j = 0; j < 8; ++j) {
                const C a = u[j];
                u[j] = cadd(a, v[j]);
                v[j] = csub(a, v[j]);
            }
            t2_pass1<P>(v, n2, t1, A + (bc * NZ + ME + i) * LS);
        } else {
#pragma unroll
            for (int j = 0; j < 8; ++j) u[j] = R2 * j + n2 < ny ? src[R2 * j] : C{T(0), T(0)};
        }
        t2_pass1<P>(u, n2, t1, A + (bc * NZ + i) * LS);
    }
    __syncthreads();
    // pass 2: half a warp per line (lanes = 16 columns; a warp where a column takes two roles)
    for (int r = tid; r < RC * L; r += nthr) t2_cols<P, false>(A + r / RC * LS, r & 15, r % RC / 16, tw, ta);
    __syncthreads();
    zconv_t2<NZ, KXB, P>(A, kx, g.Px, g.dhat, tid, nthr);
    __syncthreads();
    // pass A (the inverse transform of the conjugated field spectra, in place by columns)
    for (int r = tid; r < RC * L; r += nthr) t2_cols<P, true>(A + r / RC * LS, r & 15, r % RC / 16, tw, ta);
    __syncthreads();
    // pass B, role (y2, mirrored pair of lines): rows y < ny of both layers back to the spectrum, conjugated
    for (int r = tid; r < R2 * LP; r += nthr) {
        const int y2 = r % R2, lp = r / R2, bc = lp / ME, i = lp % ME;
        C v[8];
        t2_passB(v, A + (bc * NZ + i) * LS, y2);
        C* dst = blk + (size_t)(bc * NZ + i) * ny;
        if (MO == ME || i < MO) {
            C w[8];
            t2_passB(w, A + (bc * NZ + ME + i) * LS, y2);
            C* dst2 = blk + (size_t)(bc * NZ + NZ - 1 - i) * ny;
#pragma unroll
            for (int m = 0; m < 8; ++m) {
                const int y = y2 + R2 * m;
                if (y < ny) {
                    dst[y] = cconj(cadd(v[m], w[m]));
                    dst2[y] = cconj(csub(v[m], w[m]));
                }
            }
        } else {
#pragma unroll
            for (int m = 0; m < 8; ++m)
                if (y2 + R2 * m < ny) dst[y2 + R2 * m] = cconj(v[m]);
        }
    }
}

// ------------------------------------------------------------------------------------------------
// Dipole energies without the field (FP64): by Parseval's theorem sum_sites conv.s is the sum over frequencies of
// conj(S).(T S), so an evaluation that wants no field stops at the spectrum: no inverse transforms, and the step
// kernel in evaluation mode has no spectrum to read.  The spectrum of an image pair is Z = A + i B with A and B those
// of real functions: A(k) = (Z(k) + conj Z(-k)) / 2, i B(k) = (Z(k) - conj Z(-k)) / 2, which needs the columns kx and
// Px - kx side by side: both live in the CTA's shared memory, and it does both images at kx (weight 2 where the
// columns differ).  Every real vector v (real and imaginary part of A and of B) takes v^T M v of the real symmetric
// matrix M of its system (ZSys above) by its lower triangle: 90 multiply-adds at 8 layers where T v takes 144.
// Bound by the FP64 pipe.  On one GB300, y/z and step kernel in evaluation mode before and now: 64x64x8 x 32 images
// 815 + 220 -> 483 + 80 us, 64x64x4 x 16 194 + 60 -> 116 + 25, one image pair of 64x64x8 183 + 36 -> 139 + 26.
// Errors against the oracle are unchanged (8e-15 of the largest energy at most; the w terms move by 4e-16).

// Half of v^T M v summed over real and imaginary part of image A (qa) and image B (qb), each twice the spectrum, for
// one system at one frequency: A0 and A1 point at the elements of line 0 at k and -k; d, par, fx, fy as for zconv_sys.
template <int NZ, int PAR, int LS, int DQ>
__device__ __forceinline__ void zquad_sys(const double2* A0, const double2* A1, const double* __restrict__ d, int par,
                                          unsigned fx, unsigned fy, double& qa, double& qb) {
    using S = ZSys<NZ, PAR>;
    constexpr int NA = S::NXY, NB = S::NZC;
    constexpr int NA1 = NA > 0 ? NA : 1, NB1 = NB > 0 ? NB : 1;
    const double sg = par ? -1.0 : 1.0;
    const int lx = (par ? S::ME : 0) * LS, lz = (2 * NZ + (par ? 0 : S::ME)) * LS;
    struct V {  // the four real vectors' components
        double v[4];
    };
    auto load2 = [&](int at, unsigned f) {  // f: sign of the component's real couplings
        const double2 a = A0[at], b = A1[at];
        return V{{flip_sign(a.x + b.x, f), flip_sign(a.y - b.y, f), flip_sign(a.x - b.x, f), flip_sign(a.y + b.y, f)}};
    };
    V X[NA1], Y[NA1], Z[NB1], h;  // h: a row of M's lower triangle times the vectors
#pragma unroll
    for (int i = 0; i < NA; ++i) {
        X[i] = load2(lx + i * LS, fx);
        Y[i] = load2(lx + (NZ + i) * LS, fy);
    }
#pragma unroll
    for (int i = 0; i < NB; ++i) {  // i z
        const V z = load2(lz + i * LS, 0u);
        Z[i] = V{{-z.v[1], z.v[0], -z.v[3], z.v[2]}};
    }
    auto load = [&](int c, double (&t)[NZ]) {
#pragma unroll
        for (int q = 0; q < NZ; ++q) t[q] = d[(q * 6 + c) * DQ];
    };
    auto even = [&](const double (&t)[NZ], double s, int i, int j) {
        return t[i > j ? i - j : j - i] + s * t[NZ - 1 - i - j];
    };
    auto odd = [&](const double (&t)[NZ], int i, int j) {
        const int p = NZ - 1 - i - j;
        const double hank = p > 0 ? t[p] : p < 0 ? -t[-p] : 0.0;
        return i == j ? sg * hank : (i > j ? t[i - j] : -t[j - i]) + sg * hank;
    };
    auto axpy = [&](double c, const V& x) {
#pragma unroll
        for (int k = 0; k < 4; ++k) h.v[k] = fma(c, x.v[k], h.v[k]);
    };
    auto zero = [&] {
#pragma unroll
        for (int k = 0; k < 4; ++k) h.v[k] = 0.0;
    };
    auto dot = [&](const V& x) {
        qa = fma(x.v[0], h.v[0], fma(x.v[1], h.v[1], qa));
        qb = fma(x.v[2], h.v[2], fma(x.v[3], h.v[3], qb));
    };
    // rows i of a diagonal block t (sign s), lower triangle with half its diagonal
    auto block = [&](const double (&t)[NZ], double s, const auto& x, int i) {
#pragma unroll
        for (int j = 0; j <= i; ++j) axpy(j < i ? even(t, s, i, j) : 0.5 * even(t, s, i, j), x[j]);
    };
    double t[NZ], u[NZ];
    if constexpr (NA > 0) {
        load(0, t);  // xx
#pragma unroll
        for (int i = 0; i < NA; ++i) {
            zero();
            block(t, sg, X, i);
            dot(X[i]);
        }
        load(1, t);  // yy, and xy with every x
        load(3, u);
#pragma unroll
        for (int i = 0; i < NA; ++i) {
            zero();
            block(t, sg, Y, i);
#pragma unroll
            for (int j = 0; j < NA; ++j) axpy(even(u, sg, i, j), X[j]);
            dot(Y[i]);
        }
    }
    if constexpr (NB > 0) {
        load(2, t);  // zz
#pragma unroll
        for (int i = 0; i < NB; ++i) {
            zero();
            block(t, -sg, Z, i);
            dot(Z[i]);
        }
    }
    if constexpr (NA > 0 && NB > 0) {
        load(4, t);  // xz, yz
        load(5, u);
#pragma unroll
        for (int j = 0; j < NB; ++j) {
            zero();
#pragma unroll
            for (int i = 0; i < NA; ++i) {
                axpy(odd(t, i, j), X[i]);
                axpy(odd(u, i, j), Y[i]);
            }
            dot(Z[j]);
        }
    }
}

// grid (Px / 2 + 1, pairs): columns kx and Px - kx of a pair; -(1/2) sum conv.s over them, per image, replaces the
// first spectrum element of column kx (its two parts), where the evaluation's reduction finds it.
template <int P, int NZ>
__global__ void __launch_bounds__(kYzqThreads, 2) yzq2p_kernel(GroupArgs<double> g) {
    using C = double2;
    constexpr int R2 = P / 16, LS = t2_line(P), L = 6 * NZ, RC = 16 * T2<P>::NP;
    constexpr int ME = (NZ + 1) / 2, MO = NZ / 2, LP = 6 * ME, DQ = P / 2 + 1;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ double red[kYzqThreads / 32 * 2];
    C* A = reinterpret_cast<C*>(smem_raw);  // line (b * 3 + c) * NZ + q of column b: e_q for q < ME, o_{q - ME} above
    const int tid = threadIdx.x, nthr = kYzqThreads;
    const int kx = blockIdx.x, p = blockIdx.y, kx1 = kx ? g.Px - kx : 0;
    const int ny = g.ny;
    if (g.pair_on && !g.pair_on[p]) return;  // uniform over the CTA
    const size_t col = (size_t)3 * NZ * ny;
    C* blk0 = g.spec + ((size_t)p * g.Px + kx) * col;
    const C* blk1 = g.spec + ((size_t)p * g.Px + kx1) * col;
    const C* __restrict__ tw = g.twy;
    const C* __restrict__ t1 = g.t2y;
    const C* __restrict__ ta = g.t2y + P;
    griddep_wait();
    griddep_launch_dependents();
    // pass 1 and pass 2 as in yz2p_kernel
    for (int r = tid; r < R2 * LP; r += nthr) {
        const int n2 = r % R2, lp = r / R2, bc = lp / ME, i = lp % ME;
        const C* src = (bc < 3 ? blk0 + bc * NZ * ny : blk1 + (bc - 3) * NZ * ny) + n2;
        const bool two = MO == ME || i < MO;
        const C* s0 = src + i * ny;
        const C* s1 = src + (NZ - 1 - i) * ny;
        C u[8], v[8];
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            const bool in = R2 * j + n2 < ny;
            u[j] = in ? s0[R2 * j] : C{0.0, 0.0};
            v[j] = in && two ? s1[R2 * j] : C{0.0, 0.0};
        }
        if (two) {
#pragma unroll
            for (int j = 0; j < 8; ++j) {
                const C a = u[j];
                u[j] = cadd(a, v[j]);
                v[j] = csub(a, v[j]);
            }
            t2_pass1<P>(v, n2, t1, A + (bc * NZ + ME + i) * LS);
        }
        t2_pass1<P>(u, n2, t1, A + (bc * NZ + i) * LS);
    }
    __syncthreads();
    for (int r = tid; r < RC * L; r += nthr) t2_cols<P, false>(A + r / RC * LS, r & 15, r % RC / 16, tw, ta);
    __syncthreads();
    const double* dslab = g.dhat + (size_t)kx * DQ * NZ * 6;
    double q[2] = {0.0, 0.0};
    for (int it = tid; it < 2 * P; it += nthr) {
        const int par = it >= P ? 1 : 0, ky = it - par * P;
        const unsigned fy = ky > P / 2 ? 0x80000000u : 0u;  // (kx <= Px / 2: no sign of its own)
        const double* d = dslab + min(ky, P - ky);
        const C* a = A + t2_pos(ky);
        const C* b = A + 3 * NZ * LS + t2_pos(ky ? P - ky : 0);
        if constexpr (NZ % 2 == 0) {
            zquad_sys<NZ, 0, LS, DQ>(a, b, d, par, 0u, fy, q[0], q[1]);
        } else if (par == 0) {
            zquad_sys<NZ, 0, LS, DQ>(a, b, d, 0, 0u, fy, q[0], q[1]);
        } else {
            zquad_sys<NZ, 1, LS, DQ>(a, b, d, 1, 0u, fy, q[0], q[1]);
        }
    }
    block_reduce_d<2>(q, red);
    // -(1/2) times 1/4 (A and B doubled) times 2 (half of the form), once more for the column Px - kx; a tensor without
    // the factor of mirrored layers (dhat_factor) counts half
    const double f = (kx1 == kx ? -0.25 : -0.5) * (NZ == 1 || !g.yz2 ? 0.5 : 1.0);
    if (tid == 0) blk0[0] = C{f * q[0], f * q[1]};
}

// ------------------------------------------------------------------------------------------------
// x kernels for a two-pass length Px = P (nx <= P/2): the x-transforms in two register passes
// (ss_fft.cuh) on x2_rows rows of one layer of an image pair per CTA.  Every role order puts the rows
// fastest across a warp: the spectrum's rows of one (kx, c) are contiguous in global memory, and with
// line strides = 16 / rows (mod 16) the lanes of a half-warp (rows x 16 / rows consecutive
// columns or rows of a line) hit distinct shared-memory banks.
// x sits at row x mod R2, column x / R2 of its line, which is where pass 1 reads its role's inputs and pass B
// leaves its outputs: both work in place, and the space of separate x-space lines stays with the L1 cache
// that serves the stencil's neighbours.  Roles of whole columns and rows and lines in place: x-forward and
// step kernel of 128x128x4 x 384 images 298 -> 253 us and 438 -> 311, of 192x192x8 x 128 437 -> 441 and
// 662 -> 540, of 64x64x8 x 32 17.0 -> 16.4 and 22.5 -> 18.4 (one GB300).  They are bound by load latency and L1.
// xfwd: the gather (Eq. 12), pass 1 in place, pass 2 straight to the spectrum spec[p][kx][c][z][y].
template <typename T, int P>
__global__ void __launch_bounds__(x2_threads(sizeof(T), P), x2_blocks(sizeof(T), P)) xfwd2p_kernel(GroupArgs<T> g) {
    using C = cplx<T>;
    constexpr int R2 = P / 16, H = T2<P>::H, NP = T2<P>::NP, ROWS = x2_rows(sizeof(T), P), L = 3 * ROWS,
                  LSX = x2_lsx(sizeof(T), P);
    extern __shared__ __align__(16) unsigned char smem_raw[];
    C* A = reinterpret_cast<C*>(smem_raw);  // line c * ROWS + yy: the pair at x, then rows of Z
    const int tid = threadIdx.x, nthr = blockDim.x;
    const int p = blockIdx.z, z = blockIdx.y, y0 = blockIdx.x * ROWS;
    const int rows = min(ROWS, g.ny - y0), nx = g.nx;
    if (sizeof(T) == 8 && g.pair_on && !g.pair_on[p]) return;  // uniform over the CTA
    const C* __restrict__ tw = g.twx;  // W_P^k
    const C* __restrict__ t1 = g.t2x;  // pass 1
    griddep_wait();
    griddep_launch_dependents();
    xfwd_gather(g, A, LSX, ROWS, p, z, y0, rows, tid, nthr, T2Pos<R2>{});
    __syncthreads();
    // pass 1, role (yy, n2, c)
    for (int r = tid; r < R2 * L; r += nthr) {
        const int yy = r % ROWS, q = r / ROWS, n2 = q % R2, c = q / R2;
        if (yy >= rows) continue;
        C* line = A + (c * ROWS + yy) * LSX;
        C u[8];
#pragma unroll
        for (int j = 0; j < 8; ++j) u[j] = R2 * j + n2 < nx ? line[t2_at(n2, j)] : C{T(0), T(0)};
        t2_pass1<P>(u, n2, t1, line);
    }
    __syncthreads();
    // pass 2, role (yy, k1, par2, c): X[k1 + 16 (NP m + par2)] to the spectrum
    const size_t kstride = (size_t)3 * g.nz * g.ny;  // between consecutive kx
    C* outp = g.spec + (size_t)p * P * kstride + (size_t)z * g.ny + y0;
    for (int r = tid; r < 16 * NP * L; r += nthr) {
        const int yy = r % ROWS, q = r / ROWS, k1 = q & 15, par2 = (q >> 4) % NP, c = q / (16 * NP);
        if (yy >= rows) continue;
        const C* col = A + (c * ROWS + yy) * LSX + k1;
        C a[H];
        t2_col_vals<P, false>(a, [&](int j) { return col[j * kT2Row]; }, k1, par2, tw, tw);
        C* o = outp + (size_t)c * g.nz * g.ny + yy;
#pragma unroll
        for (int m = 0; m < H; ++m) o[(size_t)(k1 + 16 * (NP * m + par2)) * kstride] = a[m];
    }
}

// xinv: pass A straight from the spectrum (conjugated), pass B in place, then the per-site work of xinv_sites
// in mode MODE.
template <typename T, int P, int MODE>
__global__ void __launch_bounds__(x2_threads(sizeof(T), P), x2_blocks(sizeof(T), P)) xinv2p_kernel(GroupArgs<T> g, T dt,
                                                                                                   T* hout) {
    using C = cplx<T>;
    constexpr int R2 = P / 16, H = T2<P>::H, NP = T2<P>::NP, ROWS = x2_rows(sizeof(T), P), L = 3 * ROWS,
                  LSX = x2_lsx(sizeof(T), P);
    extern __shared__ __align__(16) unsigned char smem_raw[];
    C* A = reinterpret_cast<C*>(smem_raw);  // line c * ROWS + yy: columns of T, then the field convolution at x
    double* red = reinterpret_cast<double*>(A + L * LSX);
    const int tid = threadIdx.x, nthr = blockDim.x;
    const int p = blockIdx.z, z = blockIdx.y, y0 = blockIdx.x * ROWS;
    const int rows = min(ROWS, g.ny - y0);
    if (sizeof(T) == 8 && g.pair_on && !g.pair_on[p]) return;  // uniform over the CTA
    const size_t kstride = (size_t)3 * g.nz * g.ny;
    const C* inp = g.spec + (size_t)p * P * kstride + (size_t)z * g.ny + y0;
    const C* __restrict__ tw = g.twx;
    const C* __restrict__ ta = g.t2x + P;  // pass A
    griddep_wait();
    griddep_launch_dependents();
    // pass A, role (yy, k1, par2, c): column k1 of the conjugated spectrum line (c, yy)
    for (int r = tid; r < 16 * NP * L; r += nthr) {
        const int yy = r % ROWS, q = r / ROWS, k1 = q & 15, par2 = (q >> 4) % NP, c = q / (16 * NP);
        if (yy >= rows) continue;
        const C* sc = inp + (size_t)c * g.nz * g.ny + yy + (size_t)k1 * kstride;
        C a[H];
        t2_col_vals<P, true>(a, [&](int j) { return cconj(sc[(size_t)16 * j * kstride]); }, k1, par2, tw, ta);
        C* o = A + (c * ROWS + yy) * LSX + k1 + par2 * kT2Row;
#pragma unroll
        for (int m = 0; m < H; ++m) o[NP * m * kT2Row] = a[m];
    }
    __syncthreads();
    // pass B, role (yy, y2, c): x = y2 + R2 m at (y2, m)
    for (int r = tid; r < R2 * L; r += nthr) {
        const int yy = r % ROWS, q = r / ROWS, y2 = q % R2, c = q / R2;
        if (yy >= rows) continue;
        C* line = A + (c * ROWS + yy) * LSX;
        C v[8];
        t2_passB(v, line, y2);
#pragma unroll
        for (int m = 0; m < 8; ++m) line[t2_at(y2, m)] = v[m];
    }
    __syncthreads();
    xinv_sites<T, true, MODE>(g, dt, hout, A, LSX, ROWS, red, p, z, y0, rows, tid, nthr, T2Pos<R2>{});
}

// ---- launchers of one length --------------------------------------------------------------------------
// FP64 per iteration on one GB300, runtime Stockham plans before and these kernels: 64x64x4 x 16
// 432 -> 353 us, 72x60x8 x 8 625 -> 415, 70x70x1 x 32 356 -> 223, 128x128x8 x 4 1226 -> 815, 20x20x2 x 16 77 -> 75.
template <typename T, int P> void t2_xfwd(const GroupArgs<T>& g, cudaStream_t st) {
    const dim3 grid((g.ny + g.ty_a - 1) / g.ty_a, g.nz, g.n_pairs);  // ty_a = x2_rows (set by the host)
    const int thr = x2_launch_threads(sizeof(T), P, g.nx, (long)grid.x * grid.y * grid.z);
    launch_ex(xfwd2p_kernel<T, P>, grid, dim3(thr), x2_smem(sizeof(T), P, false), st, pdl_fft(g), g);
}

template <typename T, int P>
void t2_xinv(const GroupArgs<T>& g, int mode, T dt, T* hout, bool pdl, cudaStream_t st) {
    const dim3 grid((g.ny + g.ty_c - 1) / g.ty_c, g.nz, g.n_pairs);
    const dim3 blk(x2_launch_threads(sizeof(T), P, g.nx, (long)grid.x * grid.y * grid.z));
    const size_t sm = x2_smem(sizeof(T), P, true);
    switch (mode) {
#define SS_CASE(M) \
    case M: launch_ex(xinv2p_kernel<T, P, M>, grid, blk, sm, st, pdl && pdl_fft(g), g, dt, hout); break;
        SS_CASE(0) SS_CASE(1) SS_CASE(2) SS_CASE(3) SS_CASE(4) SS_CASE(5)
#undef SS_CASE
    }
}

// (layers, columns per CTA) of the y/z kernel: yz2p_columns
#define SS_T2_YZ(X) \
    X(1, 8) X(1, 4) X(1, 2) X(2, 4) X(2, 1) X(3, 2) X(3, 1) X(4, 2) X(4, 1) X(5, 1) X(6, 1) X(7, 1) X(8, 1)
template <typename T, int P> void t2_yz(const GroupArgs<T>& g, cudaStream_t st) {
    const int kxb = yz2p_kxb_use(sizeof(T), g.nz, g.yz_kxb);  // divides Px: yz2p_ok, and the counts divide the first
    const size_t sm = yz2p_smem(sizeof(T), P, g.nz, kxb);
    const dim3 grid(g.Px / kxb, g.n_pairs);
#define SS_CASE(Z, B) \
    if (g.nz == Z && kxb == B) launch_ex(yz2p_kernel<T, P, Z, B>, grid, dim3(yz2p_threads(sizeof(T), P)), sm, st, pdl_fft(g), g);
    SS_T2_YZ(SS_CASE)
#undef SS_CASE
}

// (layer counts whose two columns fit: yzq2p_ok)
template <typename T, int P> void t2_yzq(const GroupArgs<T>& g, cudaStream_t st) {
    if constexpr (sizeof(T) == 8) {
        const dim3 grid(g.Px / 2 + 1, g.n_pairs);
        const size_t sm = yz2p_smem(8, P, g.nz, 2);
#define SS_CASE(Z)                    \
    if constexpr (yzq2p_fits(P, Z)) { \
        if (g.nz == Z) launch_ex(yzq2p_kernel<P, Z>, grid, dim3(kYzqThreads), sm, st, false, g); \
    }
        SS_CASE(1) SS_CASE(2) SS_CASE(3) SS_CASE(4) SS_CASE(5) SS_CASE(6) SS_CASE(7) SS_CASE(8)
#undef SS_CASE
    }
}

template <typename T, int P> void t2_smem_limits(int bytes) {
    constexpr int carve = sizeof(T) == 8 || P <= 384 ? carve_kb<T>() : P <= 448 ? 196 : 228;  // two FP32 y/z CTAs
    set_dyn_smem(xfwd2p_kernel<T, P>, bytes, carve);
#define SS_CASE(M) set_dyn_smem(xinv2p_kernel<T, P, M>, bytes, carve);
    SS_CASE(0) SS_CASE(1) SS_CASE(2) SS_CASE(3) SS_CASE(4) SS_CASE(5)
#undef SS_CASE
#define SS_CASE(Z, B) set_dyn_smem(yz2p_kernel<T, P, Z, B>, bytes, carve);
    SS_T2_YZ(SS_CASE)
#undef SS_CASE
    if constexpr (sizeof(T) == 8) {
#define SS_CASE(Z) \
    if constexpr (yzq2p_fits(P, Z)) set_dyn_smem(yzq2p_kernel<P, Z>, bytes, carve);
        SS_CASE(1) SS_CASE(2) SS_CASE(3) SS_CASE(4) SS_CASE(5) SS_CASE(6) SS_CASE(7) SS_CASE(8)
#undef SS_CASE
    }
}

#define SS_T2_INSTANTIATE(T, P)                                                                  \
    template void t2_xfwd<T, P>(const GroupArgs<T>&, cudaStream_t);                               \
    template void t2_xinv<T, P>(const GroupArgs<T>&, int, T, T*, bool, cudaStream_t);             \
    template void t2_yz<T, P>(const GroupArgs<T>&, cudaStream_t);                                 \
    template void t2_yzq<T, P>(const GroupArgs<T>&, cudaStream_t);                                \
    template void t2_smem_limits<T, P>(int);

}  // namespace ss
