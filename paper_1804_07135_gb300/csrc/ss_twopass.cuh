// ss_twopass.cuh -- the y/z and x kernels whose transforms take two register passes (lengths P = 16 R2 of
// SS_T2_LENGTHS; ss_fft.cuh has the passes) and their launchers.  Each length is a translation unit of its
// own (ss_twopass.cu compiled with SS_T2_P defined), so that they compile in parallel.
#pragma once
#include "ss_kernels.cuh"

namespace ss {

// yz for a two-pass length Py = P (ny <= P/2), FP32, NZ layers, KXB kx columns per CTA: the y-transforms
// in two register passes each way (t2_pass1 / t2_cols / t2_passB, ss_fft.cuh) on lines held in the
// 17-strided row layout, the z-convolution in place between them.  One shared line per (column, component,
// layer): 3 NZ KXB lines of t2_line(P) complex elements, read from the spectrum in pass 1 and written back
// (rows y < ny) in pass B; one shared-memory round trip per pass instead of one per Stockham stage.
// 384 threads; pass 2 and pass A take one warp per line (16 columns x 2 parities), or half a warp (odd P/16).
// Three CTAs per SM, two from P = 384 on (its 78 KB lines; there the kernel keeps 80 registers, which runs a
// batch of size groups faster than three CTAs of 56 registers would, although one group alone runs faster
// with three).
template <int NZ, int P>
__device__ __forceinline__ void zconv_t2(float2* A, int kx, int Px, const float* dslab, int tid, int nthr) {
    constexpr int LS = t2_line(P), hy = P / 2, dq = P / 2 + 1;
    const float sxg = kx > Px / 2 ? -1.f : 1.f;
    const int nk = nthr / 3;
    // rounds of nk frequencies; a round reads and writes only its own ky, so one barrier (between its
    // reads and its writes) orders it against every other round
    for (int k0 = 0; k0 < P; k0 += nk) {
        const int a = tid / nk;
        const int ky = k0 + (tid - a * nk);
        const bool act = a < 3 && ky < P;
        float2 out[NZ];
        int pky = 0;
        if (act) {
            const int kyo = min(ky, P - ky);
            const float syg = ky > hy ? -1.f : 1.f;
            const float* d = dslab + kyo;
            pky = t2_pos(ky);
            const int i0 = a == 0 ? 0 : (a == 1 ? 3 : 4);
            const int i1 = a == 0 ? 3 : (a == 1 ? 1 : 5);
            const int i2 = a == 0 ? 4 : (a == 1 ? 5 : 2);
            const float f0 = a == 0 ? 1.f : (a == 1 ? sxg * syg : sxg);
            const float f1 = a == 0 ? sxg * syg : (a == 1 ? 1.f : syg);
            const float f2 = a == 0 ? sxg : (a == 1 ? syg : 1.f);
            float e0[NZ], e1[NZ], e2[NZ];
#pragma unroll
            for (int q = 0; q < NZ; ++q) {
                e0[q] = d[(q * 6 + i0) * dq] * f0;
                e1[q] = d[(q * 6 + i1) * dq] * f1;
                e2[q] = d[(q * 6 + i2) * dq] * f2;
            }
#pragma unroll
            for (int z = 0; z < NZ; ++z) out[z] = make_float2(0.f, 0.f);
            // paired FP32 form as in zconv_c: out += (e, e) * S and (g, g) * (i S), i S = (-S.y, S.x)
            if (a < 2) {
#pragma unroll
                for (int zp = 0; zp < NZ; ++zp) {
                    const float2 sx = A[(0 * NZ + zp) * LS + pky];
                    const float2 sy = A[(1 * NZ + zp) * LS + pky];
                    const float2 sz = A[(2 * NZ + zp) * LS + pky];
                    const float2 isz = make_float2(-sz.y, sz.x), nisz = make_float2(sz.y, -sz.x);
#pragma unroll
                    for (int z = 0; z < NZ; ++z) {
                        const int q = z >= zp ? z - zp : zp - z;
                        out[z] = __ffma2_rn(make_float2(e0[q], e0[q]), sx, out[z]);
                        out[z] = __ffma2_rn(make_float2(e1[q], e1[q]), sy, out[z]);
                        out[z] = __ffma2_rn(make_float2(e2[q], e2[q]), z >= zp ? isz : nisz, out[z]);
                    }
                }
            } else {
#pragma unroll
                for (int zp = 0; zp < NZ; ++zp) {
                    const float2 sx = A[(0 * NZ + zp) * LS + pky];
                    const float2 sy = A[(1 * NZ + zp) * LS + pky];
                    const float2 sz = A[(2 * NZ + zp) * LS + pky];
                    const float2 isx = make_float2(-sx.y, sx.x), nisx = make_float2(sx.y, -sx.x);
                    const float2 isy = make_float2(-sy.y, sy.x), nisy = make_float2(sy.y, -sy.x);
#pragma unroll
                    for (int z = 0; z < NZ; ++z) {
                        const int q = z >= zp ? z - zp : zp - z;
                        out[z] = __ffma2_rn(make_float2(e0[q], e0[q]), z >= zp ? isx : nisx, out[z]);
                        out[z] = __ffma2_rn(make_float2(e1[q], e1[q]), z >= zp ? isy : nisy, out[z]);
                        out[z] = __ffma2_rn(make_float2(e2[q], e2[q]), sz, out[z]);
                    }
                }
            }
        }
        __syncthreads();
        if (act) {
#pragma unroll
            for (int z = 0; z < NZ; ++z) A[(a * NZ + z) * LS + pky] = cconj(out[z]);
        }
    }
}

template <int P, int NZ, int KXB>
__global__ void __launch_bounds__(kYz2Threads, P >= 384 ? 2 : 3) yz2p_kernel(GroupArgs<float> g) {
    using C = float2;
    constexpr int R2 = P / 16, LS = t2_line(P), L = 3 * NZ * KXB, RC = 16 * T2<P>::NP;  // RC: roles per line
    extern __shared__ __align__(16) unsigned char smem_raw[];
    C* A = reinterpret_cast<C*>(smem_raw);
    const int tid = threadIdx.x, nthr = blockDim.x;
    const int kx = blockIdx.x * KXB, p = blockIdx.y;
    const int ny = g.ny;
    C* blk = g.spec + ((size_t)p * g.Px + kx) * 3 * NZ * ny;  // KXB consecutive columns are contiguous
    const C* __restrict__ tw = g.twy;                         // W_P^k
    const C* __restrict__ t1 = g.t2y;                         // pass 1
    const C* __restrict__ ta = g.t2y + P;                     // pass A
    griddep_wait();
    griddep_launch_dependents();
    // pass 1, role (n2, line, par), n2 fastest: the zero-padded spectrum lines in, rows of Z out
    for (int r = tid; r < 2 * R2 * L; r += nthr) {
        const int n2 = r % R2, q = r / R2, line = q % L, par = q / L;
        const C* src = blk + (size_t)line * ny + n2;
        C u[8];
#pragma unroll
        for (int j = 0; j < 8; ++j) u[j] = R2 * j + n2 < ny ? src[R2 * j] : make_float2(0.f, 0.f);
        t2_pass1<P>(u, n2, par, t1, A + line * LS);
    }
    __syncthreads();
    // pass 2: one warp per line (lanes = 16 columns x 2 parities; half a warp for odd P/16)
    for (int r = tid; r < RC * L; r += nthr) t2_cols<P, false>(A + r / RC * LS, r & 15, r % RC / 16, tw, ta);
    __syncthreads();
#pragma unroll 1
    for (int b = 0; b < KXB; ++b) {
        const int kxb = kx + b, kxo = min(kxb, g.Px - kxb);
        zconv_t2<NZ, P>(A + b * 3 * NZ * LS, kxb, g.Px, g.dhat + (size_t)kxo * (P / 2 + 1) * NZ * 6, tid, nthr);
    }
    __syncthreads();
    // pass A (the inverse transform of the conjugated field spectra, in place by columns)
    for (int r = tid; r < RC * L; r += nthr) t2_cols<P, true>(A + r / RC * LS, r & 15, r % RC / 16, tw, ta);
    __syncthreads();
    // pass B, role (y2, line, par): rows y < ny back to the spectrum, conjugated
    for (int r = tid; r < 2 * R2 * L; r += nthr) {
        const int y2 = r % R2, q = r / R2, line = q % L, par = q / L;
        C v[8];
        t2_passB(v, A + line * LS, y2, par);
        C* dst = blk + (size_t)line * ny;
#pragma unroll
        for (int m = 0; m < 4; ++m) {
            const int y = y2 + R2 * (2 * m + par);
            if (y < ny) dst[y] = cconj(v[m]);
        }
    }
}

// ------------------------------------------------------------------------------------------------
// x kernels for a two-pass length Px = P (nx <= P/2), FP32: the x-transforms in two register passes
// (ss_fft.cuh) on kX2Rows rows of one layer of an image pair per CTA.  Every role order puts the rows
// fastest across a warp: the spectrum's rows of one (kx, c) are contiguous in global memory, and with
// line strides = 16 / kX2Rows (mod 16) the lanes of a half-warp (kX2Rows rows x 16 / kX2Rows consecutive
// columns or rows of a line) hit distinct shared-memory banks.
// xfwd: the gather (Eq. 12) into x-space lines, pass 1 into the transform lines, pass 2 straight to the
// spectrum spec[p][kx][c][z][y].
// Resident CTAs the x kernels are compiled for: about 1100 threads per SM, less where their lines take more
// shared memory (78 KB at P = 512).
constexpr int x2_blocks(int P) { return P >= 512 ? 2 : 1152 / x2_threads(P); }
template <int P>
__global__ void __launch_bounds__(x2_threads(P), x2_blocks(P)) xfwd2p_kernel(GroupArgs<float> g) {
    using C = float2;
    constexpr int R2 = P / 16, H = T2<P>::H, NP = T2<P>::NP, ROWS = kX2Rows, L = 3 * ROWS, LSX = x2_lsx(P), LB = x2_lb(P);
    extern __shared__ __align__(16) unsigned char smem_raw[];
    C* xb = reinterpret_cast<C*>(smem_raw);  // line c * ROWS + yy: the pair at x, fft_pad positions
    C* A = xb + L * LB;                       // line c * ROWS + yy: rows of Z
    const int tid = threadIdx.x, nthr = blockDim.x;
    const int p = blockIdx.z, z = blockIdx.y, y0 = blockIdx.x * ROWS;
    const int rows = min(ROWS, g.ny - y0), nx = g.nx;
    const C* __restrict__ tw = g.twx;  // W_P^k
    const C* __restrict__ t1 = g.t2x;  // pass 1
    griddep_wait();
    griddep_launch_dependents();
    xfwd_gather(g, xb, LB, ROWS, p, z, y0, rows, tid, nthr);
    __syncthreads();
    // pass 1, role (yy, n2, c, par)
    for (int r = tid; r < 2 * R2 * L; r += nthr) {
        const int yy = r % ROWS, q = r / ROWS, n2 = q % R2, q2 = q / R2, c = q2 % 3, par = q2 / 3;
        if (yy >= rows) continue;
        const C* b = xb + (c * ROWS + yy) * LB;
        C u[8];
#pragma unroll
        for (int j = 0; j < 8; ++j) u[j] = R2 * j + n2 < nx ? b[fft_pad(R2 * j + n2)] : make_float2(0.f, 0.f);
        t2_pass1<P>(u, n2, par, t1, A + (c * ROWS + yy) * LSX);
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

// xinv: pass A straight from the spectrum (conjugated) into the transform lines, pass B into x-space
// lines (fft_pad positions, line c * rows + yy), then the per-site work of xinv_sites in mode MODE.
template <int P, int MODE>
__global__ void __launch_bounds__(x2_threads(P), x2_blocks(P)) xinv2p_kernel(GroupArgs<float> g, float dt, float* hout) {
    using C = float2;
    constexpr int R2 = P / 16, H = T2<P>::H, NP = T2<P>::NP, ROWS = kX2Rows, L = 3 * ROWS, LSX = x2_lsx(P), LB = x2_lb(P);
    extern __shared__ __align__(16) unsigned char smem_raw[];
    C* A = reinterpret_cast<C*>(smem_raw);  // line c * ROWS + yy: columns of T
    C* xb = A + L * LSX;                     // line c * rows + yy: the field convolution at x
    double* red = reinterpret_cast<double*>(xb + L * LB);
    const int tid = threadIdx.x, nthr = blockDim.x;
    const int p = blockIdx.z, z = blockIdx.y, y0 = blockIdx.x * ROWS;
    const int rows = min(ROWS, g.ny - y0), nx = g.nx;
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
    // pass B, role (yy, y2, c, par): x = y2 + R2 (2m + par) < nx
    for (int r = tid; r < 2 * R2 * L; r += nthr) {
        const int yy = r % ROWS, q = r / ROWS, y2 = q % R2, q2 = q / R2, c = q2 % 3, par = q2 / 3;
        if (yy >= rows) continue;
        C v[8];
        t2_passB(v, A + (c * ROWS + yy) * LSX, y2, par);
        C* b = xb + (c * rows + yy) * LB;
#pragma unroll
        for (int m = 0; m < 4; ++m) {
            const int x = y2 + R2 * (2 * m + par);
            if (x < nx) b[fft_pad(x)] = v[m];
        }
    }
    __syncthreads();
    xinv_sites<float, true, MODE>(g, dt, hout, xb, LB, red, p, z, y0, rows, tid, nthr);
}

// ---- launchers of one length --------------------------------------------------------------------------
template <typename T, int P> void t2_xfwd(const GroupArgs<T>& g, cudaStream_t st) {
    const dim3 grid((g.ny + g.ty_a - 1) / g.ty_a, g.nz, g.n_pairs);  // ty_a = kX2Rows (set by the host)
    launch_pdl(xfwd2p_kernel<P>, grid, dim3(x2_threads(P)), x2_smem(P, false), st, g);
}

template <typename T, int P>
void t2_xinv(const GroupArgs<T>& g, int mode, T dt, T* hout, bool pdl, cudaStream_t st) {
    const dim3 grid((g.ny + g.ty_c - 1) / g.ty_c, g.nz, g.n_pairs), blk(x2_threads(P));
    const size_t sm = x2_smem(P, true);
    switch (mode) {
#define SS_CASE(M) \
    case M: launch_ex(xinv2p_kernel<P, M>, grid, blk, sm, st, pdl, g, dt, hout); break;
        SS_CASE(0) SS_CASE(1) SS_CASE(2) SS_CASE(3) SS_CASE(4) SS_CASE(5)
#undef SS_CASE
    }
}

// (layers, columns per CTA) of the y/z kernel: yz2p_kxb and yz2p_kxb_alt
#define SS_T2_YZ(X) X(1, 8) X(1, 4) X(2, 4) X(3, 2) X(4, 2) X(4, 1) X(5, 1) X(6, 1) X(7, 1) X(8, 1)
template <typename T, int P> void t2_yz(const GroupArgs<T>& g, cudaStream_t st) {
    int kxb = yz2p_kxb_use(g.nz, g.yz_kxb);
    if (g.Px % kxb) kxb = yz2p_kxb(g.nz);
    const size_t sm = yz2p_smem(P, g.nz, kxb);
    const dim3 grid(g.Px / kxb, g.n_pairs), blk(kYz2Threads);
#define SS_CASE(Z, B) \
    if (g.nz == Z && kxb == B) launch_pdl(yz2p_kernel<P, Z, B>, grid, blk, sm, st, g);
    SS_T2_YZ(SS_CASE)
#undef SS_CASE
}

template <typename T, int P> void t2_smem_limits(int bytes) {
    set_dyn_smem(xfwd2p_kernel<P>, bytes);
#define SS_CASE(M) set_dyn_smem(xinv2p_kernel<P, M>, bytes);
    SS_CASE(0) SS_CASE(1) SS_CASE(2) SS_CASE(3) SS_CASE(4) SS_CASE(5)
#undef SS_CASE
#define SS_CASE(Z, B) set_dyn_smem(yz2p_kernel<P, Z, B>, bytes);
    SS_T2_YZ(SS_CASE)
#undef SS_CASE
}

#define SS_T2_INSTANTIATE(T, P)                                                                  \
    template void t2_xfwd<T, P>(const GroupArgs<T>&, cudaStream_t);                               \
    template void t2_xinv<T, P>(const GroupArgs<T>&, int, T, T*, bool, cudaStream_t);             \
    template void t2_yz<T, P>(const GroupArgs<T>&, cudaStream_t);                                 \
    template void t2_smem_limits<T, P>(int);

}  // namespace ss
