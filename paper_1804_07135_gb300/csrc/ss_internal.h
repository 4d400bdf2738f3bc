// ss_internal.h -- types shared by the host runtime (ss_api.cu) and the kernels (ss_kernels.cuh).
//
// Data layout in device memory, per size group (strings whose lattices have the same dimensions):
//   s, sp   [image][3][N]            spins before / after the step (SoA planes, x fastest), N = nx*ny*nz
//   spec    [pair][Px][3][nz][ny]    complex spectra of image pairs after the x transform (y fastest);
//                                    the y/z kernel overwrites them in place with the field spectra
//   dhat    [Px/2+1][nz*6][Py/2+1]   one octant of the dipole-tensor spectrum (real coefficients),
//                                    [kxo][|dz|*6 + comp][kyo]
// Two images (2p, 2p+1) share one complex field (real part = image 2p, imaginary part = image 2p+1):
// the dipole kernel is real in real space, so one complex convolution serves both images.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

namespace ss {

template <typename T> struct cplx_of;
template <> struct cplx_of<float> { using type = float2; };
template <> struct cplx_of<double> { using type = double2; };
template <typename T> using cplx = typename cplx_of<T>::type;

constexpr int kMaxStages = 16;
constexpr int kMaxThreadsX = 512;   // largest block of the x-transform kernels (256 or 512, autotuned)
constexpr int kMinBlocksX = 2;      // resident 512-thread blocks per SM they are compiled for (64 registers)
constexpr int kMaxThreadsYz = 384;  // block size of the y/z kernel (3 x 128: one z-convolution row per warp)
constexpr int kMinBlocksYz = 2;
constexpr int kArcMaxChunk = 8;     // image differences one arc CTA accumulates
constexpr int kArcMaxK = 1024;      // images per string

// Mixed-radix (2, 3, 4, 8; 5 and 7 in the setup transforms) plan of a length-P complex FFT, stages in Stockham order
// (powers of two first, so the stride Ns of every power-of-two stage and of the first radix-3 stage is a power of two).
// Per stage: q = P/R butterflies per line, ns = product of the earlier radices, tw = P/(ns*R) (twiddle
// index step); ns_mask = ns - 1 when ns is a power of two, else -1.
struct FftPlan {
    int P;
    int nstages;
    int radix[kMaxStages];
    int q[kMaxStages];
    int ns[kMaxStages];
    int tw[kMaxStages];
    int ns_mask[kMaxStages];
};

// Shared-memory position of element i of a line: one padding slot per 16 elements, which spreads the
// strided stores of the early FFT stages over all banks.
__host__ __device__ constexpr int fft_pad(int i) { return i + (i >> 4); }
// Line stride (in elements) for lines of length P: padded length, made odd so that a column read
// across consecutive lines touches distinct banks.
__host__ __device__ constexpr int fft_line_stride(int P) { return (P + (P >> 4) + 1) | 1; }

// Reparametrisation source of one image: normalise((1 - t) sp[src0] + t sp[src1]), or an exact copy
// of sp[src0] when copy != 0.  Image indices are local to the size group.
struct InterpEntry {
    int src0, src1;
    double t;          // FP64 weight (Eq. 12)
    float tf, omtf;    // t and 1 - t rounded once, for the FP32 blend
    int copy;
    int pad;
};

// n / d by a multiplication, m = fast_div_m(d), exact for n d < 2^32 (m = ceil(2^32 / d), 0 stands for d = 1: the
// product n m exceeds n 2^32 / d by less than n d / d)
inline unsigned fast_div_m(unsigned d) { return d <= 1 ? 0u : (unsigned)(((1ull << 32) + d - 1) / d); }
#ifdef __CUDACC__
__device__ __forceinline__ int fast_div(int n, unsigned m) { return m ? (int)__umulhi((unsigned)n, m) : n; }
#endif

// Constants of the string an image belongs to.
template <typename T> struct ImgParam {
    T J, D, K, w;
};

struct RkString;
// Runge-Kutta stages: where and how the x-inverse kernel in force mode forms the next stage's state
// (ss_kernels.cuh, rk_next_state); out null: it does not.
template <typename T> struct RkNext {
    const T* y0;
    const T* k;        // earlier stages' forces, `stride` apart
    size_t stride;
    T* out;            // [image][3][N]
    int n;             // earlier stages
    T a[6], a_cur;     // their weights and this stage's
    const RkString* st;
    const int* img_sys;
};

template <typename T> struct GroupArgs {
    int nx, ny, nz, N;
    int Px, Py;
    int n_img, n_pairs;
    unsigned m_nx, m_hx;  // fast_div multipliers of nx and nx / 2
    int lsx, lsy;  // shared-memory line strides (complex elements) of the x and y transforms
    T* s;
    T* sp;
    cplx<T>* spec;
    const T* dhat;
    const cplx<T>* twx;   // flat twiddle tables W_P^k
    const cplx<T>* twy;
    // two-pass transforms (P a multiple of 16), 2P entries each, laid out so that the lanes of a warp
    // read consecutive entries: [0, P) pass 1, W_P^{n2 (2m + par)} at (2m + par) * P/16 + n2; [P, 2P) pass A,
    // W_P^{k1 (2m + par2)} at P + (2m + par2) * 16 + k1
    const cplx<T>* t2x;
    const cplx<T>* t2y;
    FftPlan planx, plany;
    const ImgParam<T>* prm;
    const InterpEntry* interp;
    double* epart;  // energy partials, [n_eblk][image] (step) or [n_eblk][image][4] (eval)
    int n_eblk;     // = nz * ceil(ny / ty_c)
    int ty_a, ty_c; // y rows per CTA in the x-forward and x-inverse kernels
    int* err;       // sticky error word (bit 1: invalid input spin, bit 2: non-finite value)
    const int* climb_img;  // [n_img] nonzero for the image that climbs this iteration (climbing mode only)
    T llg_a, llg_b;        // precessional dynamics (Eq. 9): 1 / (1 + alpha^2) and alpha / (1 + alpha^2)
    const T* hdir;         // [image][3][N] direct dipole sums (SS_DIPOLE_DIRECT), or null
    const int* pair_on;    // [n_pairs] evaluate only the pairs flagged here (generic kernels), or null: all
    RkNext<T> rk;          // force modes only
    unsigned char w_spec;  // evaluation: the dipole term per (column <= Px / 2, pair) is in the spectrum (FP64)
    // the x kernels and the y/z kernel are the two-pass ones (x2_use, yz2_use); bytes, since eight more bytes of arguments
    // cost the four launches of a 16x16x1 iteration 1% (13.60 and 13.73 us on one GB300)
    unsigned char x2, yz2;
    int yz_kxb;            // kx columns per CTA of the two-pass y/z kernel (autotuned; 0: the default)
};
// Energy partials per image of the evaluation mode: the four terms of Eq. 1 (J, D, K, w with the constant
// set to 1) and the squared norm of the dipole convolution (for the FP32 round-off bound of the w term).
constexpr int kEvalTerms = 5;

// Arc-length / reparametrisation bookkeeping of one size group.
struct ArcArgs {
    int n_str;             // strings in the group
    const int* str_img0;   // [n_str] first group-local image of each string
    const int* str_K;      // [n_str] images per string
    const double* str_inv; // [n_str] 1 / (images - 1)
    int maxK;
    int n_tiles;           // spatial tiles of the 3N component vector
    int tile_elems;        // components per tile
    int kchunk;            // image differences per CTA along the string
    int n_kchunks;
    double* dpart;         // [n_str][maxK][n_tiles] squared-distance partials
    double* e_last;        // [n_str][maxK] energies of the state before the step
    unsigned* cnt;         // [n_str] tile CTAs finished; zero between launches
    int reparam;           // 0: keep images where they are
    // variants (Sec. III leaves the interpolation open and names the climbing image as a refinement)
    int climb;             // climbing image on: the energy CTAs also take tickets, the finisher picks the next one
    int* kc;               // [n_str] image climbing in the current iteration, or -1
    int* climb_img;        // [n_img] flag per image for the next iteration's x-inverse kernel
    double* cpart;         // [n_str][c_tiles][2] (F.tau, tau.tau) partials of the climbing image
    int c_tiles;           // site tiles of kClimbTile per image
    int spline;            // natural cubic spline: the finisher writes W, the apply kernel moves the images
    double* W;             // [n_str][maxK][w_stride] interpolation weights phi_k = sum_q W_kq phi*_q, [q][k], in T
    int w_stride;          // spline_w_stride(maxK)
    double* P;             // [n_str][maxK + 1][maxK] scratch: d m_i / d y_q of the spline (in T), column q contiguous
    int* wcopy;            // [n_str][maxK] row k is the identity (image kept as it is)
    int p_dim;             // spline operator columns kept in the finisher's dynamic shared memory (0: none)
};

constexpr int kClimbTile = 256;   // sites per CTA of the climbing-image kernels (one per thread)
constexpr int kSplineMaxK = 256;  // longest string the spline variant accepts
constexpr int kSplineRows = 8;    // rows of W a thread of the FP32 apply kernel takes at once
inline int spline_w_stride(int maxK) { return (maxK + kSplineRows - 1) / kSplineRows * kSplineRows + 4; }
// columns of the spline operator P the arc kernel keeps on chip (66 KB of FP32 or 33 KB of FP64)
inline int spline_p_dim(int real_bytes, int maxK) { const int cap = real_bytes == 4 ? 128 : 64; return maxK + 1 < cap ? maxK + 1 : cap; }

// Adaptive Runge-Kutta evolution (Sec. III, Dormand-Prince 5(4)): controller state of one ODE system
// (a whole string, or one image under per-image step control).
struct RkString {
    double t;           // reduced time reached within the current interval
    double step;        // step carried between attempts and intervals
    double hs;          // step of the current attempt (step cut to end at the interval's end)
    double err;         // error norm of the last attempt
    long long acc, rej; // accepted and rejected attempts since the path was set
    int done;           // the interval is complete
    int accepted;       // the last attempt was accepted
    int attempts;       // attempts in the current interval
    int pad;
};

// An embedded Runge-Kutta pair in the path's precision: `stages` stage rows a (stage i uses a[i][0..i-1]),
// the weights b of the solution carried forward and the error weights e (difference of the two
// solutions' weights).  method 0: Dormand-Prince 5(4) (Dormand and Prince, 1980; 7 stages, the
// fifth-order solution carried); method 1: Runge-Kutta-Fehlberg 4(5) (Fehlberg, 1969; 6 stages, the
// fourth-order solution carried).
template <typename T> struct DpCoef {
    int stages;
    T a[7][6];
    T b[7];
    T e[7];
};
template <typename T> DpCoef<T> dp_coefficients(int method);

// Device buffers and constants of the Runge-Kutta evolution of one size group.
template <typename T> struct RkArgs {
    T* y0;            // [image][3][N] state at the start of the attempt
    T* k;             // [7][image][3][N] stage forces
    T* y5;            // [image][3][N] fifth-order solution of the attempt
    double* errp;     // [image][tile] squared scaled-error partials
    int n_tiles;      // tiles of 1024 components per image
    RkString* st;     // [n_sys]
    const int* img_sys;   // [n_img] system of each image
    const int* sys_img0;  // [n_sys] first image of each system (its images are consecutive)
    const int* sys_cnt;   // [n_sys] images of each system
    int n_sys;
    int* active;      // any system still inside its interval (written by the controller)
    double T_int, rtol, atol;
    DpCoef<T> dp;
};

enum { kErrInvalidSpin = 1, kErrNonFinite = 2, kErrStepCollapse = 4 };

// Lengths P = 16 R2 in two register passes (ss_fft.cuh, ss_twopass.cuh): a line is R2 = P/16 rows of 16
// at row stride kT2Row; the y/z kernel for those Py with 1 to 8 layers, the x kernels for those Px with
// x2_rows rows per CTA.  The list covers lattices of up to 256 sites a side; each length is a multiple of 16
// whose passes need DFTs of at most 16 points.
#define SS_T2_LENGTHS(X) \
    X(32) X(48) X(64) X(80) X(96) X(112) X(128) X(144) X(160) X(192) X(224) X(256) X(288) X(320) X(384) X(448) X(512)
inline bool t2_length(int P) {
    switch (P) {
#define SS_CASE(L) case L:
        SS_T2_LENGTHS(SS_CASE)
#undef SS_CASE
        return true;
        default: return false;
    }
}
// The smallest two-pass length >= m, or 0.
inline int t2_length_from(int m) {
    for (int P = (m + 15) / 16 * 16; P <= 512; P += 16)
        if (t2_length(P)) return P;
    return 0;
}
constexpr int kT2Row = 17;
constexpr int kT2MaxNz = 8;
__host__ __device__ constexpr int t2_line(int P) { return kT2Row * (P / 16); }
// kx columns per CTA, the counts with a kernel, largest first (15 to 24 lines, then fewer): the autotuner
// picks one by time; untuned FP32 launches take the first, FP64 ones the last, whose work spreads most evenly
// over the SMs (an FP64 launch is bound by each SM's FP64 pipe).  Empty when nz has no two-pass kernel.
struct YzColumns {
    int n, v[3];
};
inline YzColumns yz2p_columns(int nz) {
    if (nz == 1) return {3, {8, 4, 2}};
    if (nz == 2) return {2, {4, 1, 0}};
    if (nz <= 4) return {2, {2, 1, 0}};
    return {nz <= kT2MaxNz ? 1 : 0, {1, 0, 0}};
}
__host__ __device__ constexpr size_t yz2p_smem(int real_bytes, int Py, int nz, int kxb) { return (size_t)3 * nz * kxb * t2_line(Py) * 2 * real_bytes; }
inline bool yz2p_ok(int Py, int nz, int Px) {
    if (!t2_length(Py)) return false;
    const YzColumns k = yz2p_columns(nz);
    return k.n > 0 && Px % k.v[0] == 0;
}
// threads and resident CTAs of the y/z kernel: small CTAs, so that several per SM are in different passes, of
// 80 registers per thread (64 spill in the z-convolution and the mirrored pass 1); as many as registers and
// shared memory (24 lines: 26 KB at 128, 78 KB at 384) allow
// (FP64: the pipe issues two lane-operations per clock and SM, so a few warps with all the registers they want)
__host__ __device__ constexpr int yz2p_threads(int real_bytes, int P) {
    if (real_bytes == 8) return P <= 32 ? 64 : P <= 256 ? 128 : 256;
    return P <= 128 ? 128 : P <= 256 ? 192 : P <= 320 ? 256 : 384;
}
__host__ __device__ constexpr int yz2p_blocks(int real_bytes, int P) {
    if (real_bytes == 8) return P <= 32 ? 6 : P <= 192 ? 3 : P <= 256 ? 2 : 1;
    return P <= 128 ? 6 : P <= 256 ? 4 : P <= 320 ? 3 : 2;
}
// The FP64 energy kernel keeps two columns in shared memory (227 KB, less its reduction's): 8 layers up to 256 points
constexpr int kYzqThreads = 128;
__host__ __device__ constexpr bool yzq2p_fits(int P, int nz) { return yz2p_smem(8, P, nz, 2) <= 226 * 1024; }
inline bool yzq2p_ok(int Py, int nz, int Px) { return yz2p_ok(Py, nz, Px) && yzq2p_fits(Py, nz); }
// columns per CTA a launch uses: the tuned count when it is one of them
inline int yz2p_kxb_use(int real_bytes, int nz, int tuned) {
    const YzColumns k = yz2p_columns(nz);
    for (int i = 0; i < k.n; ++i)
        if (k.v[i] == tuned) return tuned;
    return k.n == 0 ? 0 : k.v[real_bytes == 8 ? k.n - 1 : 0];
}
// Dynamic shared memory of the runtime-plan y/z kernel: twiddles, the 3 nz lines of one kx, and the kx slab of the tensor
// spectrum when it is small enough to stage.
inline size_t yz_smem(int real_bytes, int Py, int nz) {
    const size_t slab = (size_t)(Py / 2 + 1) * nz * 6 * real_bytes;
    return (size_t)(Py + 3 * nz * fft_line_stride(Py)) * 2 * real_bytes + (slab <= 24 * 1024 ? slab : 0);
}
// Whether a group's y/z kernel is the two-pass one: wherever it has a form, but for FP64 films of two to five layers on
// a grid of little more than one round of the runtime-plan kernel (two CTAs per SM), at lengths that one can transform.
// The two-pass kernel's roles leave lanes idle that the FP64 pipe still spends its time on, and its CTA takes 32 to 39 us
// where the other's takes 18 to 30.  Per iteration on one GB300, two-pass and runtime-plan, Px n_pairs CTAs in brackets:
// 15x15x2 x 8 images (128) 67 and 56 us, 16x24x2 x 4 (64) 66 and 51, 30x32x2 x 6 (192) 72 and 62, 21x15x2 x 12 (288) 68
// and 66, 30x29x2 x 12 (384) 76 and 84; 15x16x3 x 8 (128) 70 and 56, 12x24x3 x 16 (192) 74 and 66, 12x24x3 x 24 (288) 76
// and 88; with four and five layers at 32 points alone: 30x16x4 x 4 (128) 72 and 60, 4x16x5 x 50 (200) 74 and 70,
// 12x15x4 x 22 (264) 72 and 74, but 48 points 21x21x4 x 8 (192) 78 and 80; one layer 12x24x1 x 24 (288) 51 and 57, eight
// 12x16x8 x 4 (48) 78 and 90.
inline bool yz2_use(int real_bytes, int Px, int Py, int nz, int n_pairs) {
    if (!yz2p_ok(Py, nz, Px)) return false;
    const bool few = nz == 2 ? (long)Px * n_pairs <= 256 : (nz == 3 || ((nz == 4 || nz == 5) && Py == 32)) && (long)Px * n_pairs <= 200;
    return !(real_bytes == 8 && few && Py % 5 != 0 && Py % 7 != 0);
}
// Factor of the stored tensor spectrum besides 4 pi / (Px Py): the two-pass y/z kernel convolves sums and
// differences of mirrored layers, which leaves a factor 2 to be taken out (exact)
inline double dhat_factor(bool yz2, int nz) { return yz2 && nz > 1 ? 0.5 : 1.0; }
// rows per CTA of the two-pass x kernels: 4, from 384 points on 8 (64-byte instead of 32-byte pieces of the spectrum,
// fewer rows shared with neighbouring CTAs: 192x192x8 x 128 images x-forward 425 -> 379 us, step kernel 527 -> 462;
// at 256 points the step kernel loses, 310 -> 322 on 128x128x4 x 384).  FP64: more, smaller CTAs, as for the y/z kernel
__host__ __device__ constexpr int x2_rows(int real_bytes, int P) { return real_bytes == 8 ? 2 : P >= 384 ? 8 : 4; }
// x CTAs: pass 2 has 48 roles per row (up to P = 384), pass 1 has 3 P/16 per row, the sites of four rows take 4 nx
// (even nx) or 8 nx items.
// The kernels are compiled for up to x2_threads threads in x2_blocks CTAs per SM (64 registers, 80 from P = 288
// on) and launched with x2_launch_threads of them: on a grid of many waves the smaller block, of which more fit
// on an SM (128x128x4 x 384 images: step kernel 311 us with 192 threads, 333 with 256); on a small grid the
// larger one where it takes fewer rounds over the sites (112x112x1 x 60: iteration 56.2 us with 192, 53.7 with
// 256).
__host__ __device__ constexpr int x2_threads(int real_bytes, int P) {
    return real_bytes == 8 ? 128 : P <= 64 ? 128 : P <= 128 ? 192 : P <= 320 ? 256 : 384;
}
__host__ __device__ constexpr int x2_blocks(int real_bytes, int P) {
    if (real_bytes == 8) return P <= 256 ? 3 : 2;
    return P <= 64 ? 8 : P <= 128 ? 5 : P <= 256 ? 4 : P <= 320 ? 3 : 2;
}
inline int x2_launch_threads(int real_bytes, int P, int nx, long ctas) {
    if (real_bytes == 8) return x2_threads(8, P);
    const int hi = x2_threads(4, P), lo = P > 64 && P <= 256 ? hi - 64 : hi;
    const int items = nx % 2 == 0 ? 4 * nx : 8 * nx;
    return ctas < 10L * 152 && (items + hi - 1) / hi < (items + lo - 1) / lo ? hi : lo;
}
// Whether a group's x kernels are the two-pass ones: every length that has them, but for FP64 at 32 points on a large
// grid.  There pass 1 has 12 roles per CTA (2 rows x 3 components x R2 = 2) and a warp's FP64 instruction takes as long
// for 12 lanes as for 32, which shows once the grid is several CTAs per SM deep; the runtime-plan kernels at their tuned
// rows fill their warps.  Per iteration on one GB300, two-pass and runtime-plan: 16x60x1 x 40 images (600 CTAs) 90.3 and
// 94.4 us, 15x40x1 x 80 (800) 109 and 105, 14x20x3 x 60 (900) 162 and 162, 14x64x4 x 16 (1024) 129 and 111, 14x40x2 x 100
// (2000) 209 and 176, 14x22x3 x 130 (2145) 281 and 257.  (At 48 points neither is better by more than 6%.)
constexpr long kX2Grid32 = 700;
inline bool x2_use(int real_bytes, int Px, int ny, int nz, int n_pairs) {
    return t2_length(Px) && !(real_bytes == 8 && Px == 32 && (long)((ny + 1) / 2) * nz * n_pairs > kX2Grid32);
}
// Whether SS_X_CONFIG may pin the x kernels to `thr` threads and `rows` rows per CTA: the runtime-plan kernels take 256 or
// 512 threads; the two-pass ones have one shape per length, whatever it names.
inline bool x_shape_ok(bool two_pass, int thr, int rows, int ny) {
    return rows >= 1 && rows <= ny && (two_pass || thr == 256 || thr == 512);
}
// line stride of the x kernels: 16 / rows (mod 16)
__host__ __device__ constexpr int x2_lsx(int real_bytes, int P) {
    const int v = t2_line(P) - 1;
    return v + ((16 / x2_rows(real_bytes, P) - v % 16) + 16) % 16;
}
inline size_t x2_smem(int real_bytes, int P, bool inverse) {
    return (size_t)3 * x2_rows(real_bytes, P) * x2_lsx(real_bytes, P) * 2 * real_bytes + (inverse ? 32 * 2 * kEvalTerms * 8 : 0);
}
// Padded transform length for n sites: the smallest 2^a 3^b >= 2n - 1, or the power of two >= 2n - 1 when that
// is at most 1/8 longer.
inline int padded_smooth(int n) {
    auto smooth = [](int m) {
        while (m % 2 == 0) m /= 2;
        while (m % 3 == 0) m /= 3;
        return m == 1;
    };
    int m = n > 1 ? 2 * n - 1 : 1;
    while (!smooth(m)) ++m;
    int p2 = 1;
    while (p2 < 2 * n - 1) p2 <<= 1;
    return 8 * p2 <= 9 * m ? p2 : m;
}
// Padded transform length for n sites, enough for the linear (non-circular) convolution with offsets
// -(n-1)..(n-1) (Sec. II-A, the zero-padded kernel), where the kernels along the axis have a two-pass form:
// padded_smooth(n), except that a length without two-pass kernels is exchanged for the next one that has them.
// Lattices of up to 12 sites a side keep the short length: one CTA transforms all of their lines at once either way.
inline int padded_len(int n) {
    const int m = padded_smooth(n);
    if (n <= 12 || t2_length(m)) return m;
    const int t = t2_length_from(2 * n - 1);
    return t ? t : m;
}

// The padded lengths of a lattice, Px first: the two-pass x kernels take every t2_length, but the two-pass y/z kernel
// takes Py only together with a Px that its columns per CTA divide (yz2p_ok).  Where it does not (Px = 18 at one
// layer, say), the runtime-plan kernel transforms y, and that one has stages of radix 2, 3, 4 and 8 alone: a two-pass
// length with a factor 5 or 7 is then exchanged for padded_smooth(ny).  The others stay, which have fewer radix-3 stages
// (5x81x1 x 40 images, Py 192 and 162: 30.8 and 34.5 us per iteration on one GB300).
// That kernel's time goes with its columns, in rounds of two CTAs per SM: with a two-pass Px a third longer (17 and 18
// sites, 48 for 36 points) the x kernels gain less than it loses as soon as it takes more rounds (four or more with up to
// eight layers, where a round is short), or two and more of long lines (400 sites and up per column), which share the
// SM's L1 and issue.  FP32, per iteration on one GB300 with 36 and 48 points, rounds in brackets:
// 18x12x1 x 40 images (3, 4) 35.0 and 33.9 us, x 64 (4, 6) 41.1 and 43.2, x 256 (16, 21) 104 and 119; 18x25x20 x 6 (1, 1)
// 65.7 and 47.2, x 16 (1, 2) 71.8 and 86.8, x 24 (2, 2) 103 and 109, 18x40x9 x 24 (2, 2) 59.6 and 59.5.  A two-pass Px up to 1.19 times the short one (13,
// 14, 25 to 27, 41, 81, 161, 162 sites) gains 5 to 15%, except on strips, where the x kernels have little to gain: about 5 us
// a round for the columns it adds against 10 us and 60 per million sites that the x kernels save.  162x3x1 x 200 images,
// 324 and 384 points: 553 and 643 us, 162x3x8 x 40 181 and 199, 162x12x8 x 100 545 and 533; 81x6x1 x 200 284 and 321,
// 81x3x8 x 40 103 and 109, 81x30x9 x 24 142 and 122; 26x6x1 x 200 115 and 123, 26x12x8 x 100 115 and 101.
//
// FP64 kernels' time goes with the work they issue to the FP64 pipe.  The two-pass y/z kernel leaves lanes idle at
// short lengths, which a grid of one or two CTAs per SM does not hide: up to kYz64Few of them the short lengths (and
// yz2_use).  And
// its time goes with Px: a two-pass Px more than a tenth above the short one does not pay where the y/z kernel is the
// same with either.  Per iteration on one GB300, two-pass and short lengths: 13x17x2 x 11 images (192 CTAs) 68 and
// 54 us, 14x22x3 x 10 (160) 74 and 60, 17x17x1 x 11 (144) 56 and 52, 50x26x1 x 8 (224) 64 and 77, 13x17x1 x 30 (240)
// 56 and 64; short Px alone: 25x32x8 x 44 (64 or 54) 510 and 446, 25x25x8 x 40 430 and 399.  13 and 14 sites along y (27
// or 32 points, where the two-pass kernel has 12 of 64 threads at work in two of its passes) take the short lengths
// for longer: to about one round of the runtime-plan kernel, two CTAs per SM, with two layers, less with three and four,
// whose lines take that kernel longer.  In sx n_pairs CTAs of it, two-pass and short: 14x14x2 x 16 (216) 68 and 51,
// 8x14x2 x 36 (288) 64 and 55, 34x13x2 x 10 (360) 70 and 70; 14x14x3 x 18 (243) 70 and 60, 17x14x3 x 16 (288) 71 and
// 74; 14x13x4 x 16 (216) 72 and 66, 10x14x4 x 20 (240) 70 and 75.
constexpr long kYz64Few = 200;
inline long yz64_few_27(int nz) { return nz == 2 ? 304 : nz == 3 ? 256 : nz == 4 ? 224 : 0; }
inline void padded_lengths(int real_bytes, int nx, int ny, int nz, int n_pairs, int* Px, int* Py) {
    const int sx = padded_smooth(nx), sy = padded_smooth(ny);
    const int tx = padded_len(nx), ty = nz <= kT2MaxNz ? padded_len(ny) : sy;
    *Px = tx;
    *Py = ty;
    if (real_bytes == 8) {
        const int kxb = yz2p_kxb_use(8, nz, 0);
        if ((kxb > 0 && (long)(tx / kxb) * n_pairs <= kYz64Few) ||
            (ty == 32 && sy == 27 && (long)sx * n_pairs <= yz64_few_27(nz))) {
            *Px = sx;
            *Py = sy;
        } else if (10 * tx > 11 * sx && yz2p_ok(ty, nz, sx) == yz2p_ok(ty, nz, tx)) {
            *Px = sx;
        }
    } else if (10 * tx > 11 * sx && !yz2p_ok(ty, nz, sx) && !yz2p_ok(ty, nz, tx)) {
        const long round = 2 * 152, rs = (sx * (long)n_pairs + round - 1) / round, rt = (tx * (long)n_pairs + round - 1) / round;
        const bool more = rt > rs ? nz > kT2MaxNz || rs >= 4 : nz > kT2MaxNz && rs >= 2 && ny * nz >= 400;
        const bool strip = 5.0 * (tx - sx) * n_pairs / round > 10.0 + 60e-6 * 2.0 * n_pairs * nx * ny * nz;
        if (strip || (4 * tx > 5 * sx && more)) *Px = sx;
    }
    if (!yz2p_ok(*Py, nz, *Px) && (*Py % 5 == 0 || *Py % 7 == 0)) *Py = sy;
}


// ---- launchers (defined in ss_kernels.cuh, instantiated for float and double) ----
template <typename T> void launch_xfwd(const GroupArgs<T>& g, bool do_fft, int nthr, size_t smem, cudaStream_t st);
template <typename T> void launch_yz(const GroupArgs<T>& g, int nthr, size_t smem, cudaStream_t st);
template <typename T>
void launch_xinv_step(const GroupArgs<T>& g, bool do_fft, T dt, int nthr, size_t smem, cudaStream_t st);
void launch_yzq(const GroupArgs<double>& g, cudaStream_t st);  // where yzq2p_ok
template <typename T>
void launch_xinv_eval(const GroupArgs<T>& g, bool do_fft, T* hout, int nthr, size_t smem, cudaStream_t st);
// Runge-Kutta stage: the force of Eq. 13 (or with llg the right-hand side of Eq. 9) at the state in s
// into kout; energy partials when energies
template <typename T>
void launch_xinv_force(const GroupArgs<T>& g, bool do_fft, T* kout, bool energies, bool llg, int nthr, size_t smem,
                       cudaStream_t st);
template <typename T> void launch_xinv_step_climb(const GroupArgs<T>& g, bool do_fft, T dt, T* hc, int nthr, size_t smem,
                                                  cudaStream_t st);
template <typename T> void launch_xinv_step_llg(const GroupArgs<T>& g, bool do_fft, T dt, int nthr, size_t smem,
                                                cudaStream_t st);
// dtab: the tensor table of the direct sum, [6][N] over (|dz|, |dy|, |dx|)
template <typename T> void launch_dipole_direct(const GroupArgs<T>& g, T* hdir, const T* dtab, cudaStream_t st);
template <typename T> void launch_climb(const GroupArgs<T>& g, const ArcArgs& a, T dt, const T* hc, cudaStream_t st);
template <typename T> void launch_spline_apply(const GroupArgs<T>& g, const ArcArgs& a, int maxK, cudaStream_t st);
template <typename T> void launch_rk_finish(const GroupArgs<T>& g, const RkArgs<T>& r, cudaStream_t st);
template <typename T>
void launch_rk_control(const GroupArgs<T>& g, const RkArgs<T>& r, int begin, cudaStream_t st);
template <typename T> void launch_rk_commit(const GroupArgs<T>& g, const RkArgs<T>& r, cudaStream_t st);
void launch_rk_condition(cudaGraphConditionalHandle h, const int* active, cudaStream_t st);
template <typename T> void launch_arc(const GroupArgs<T>& g, const ArcArgs& a, int nthr, cudaStream_t st);
template <typename T>
void launch_eval_reduce(const GroupArgs<T>& g, const ArcArgs& a, double* terms, double* energies, double* cnorm2,
                        cudaStream_t st);
template <typename T, typename Tin>
void launch_aos_to_soa(const Tin* src, T* dst, int K, int N, int* err, cudaStream_t st);
template <typename T, typename Tout>
void launch_soa_to_aos(const T* src, Tout* dst, int K, int N, Tout scale, cudaStream_t st);
// Two-pass kernels of one length P (ss_twopass.cuh, one translation unit per length): the x kernels for
// g.Px = P (the x-inverse kernel in the given mode of xinv_sites), the y/z kernel for g.Py = P, and the
// dynamic shared-memory limit of all of them.
template <typename T, int P> void t2_xfwd(const GroupArgs<T>& g, cudaStream_t st);
template <typename T, int P> void t2_xinv(const GroupArgs<T>& g, int mode, T dt, T* hout, bool pdl, cudaStream_t st);
template <typename T, int P> void t2_yz(const GroupArgs<T>& g, cudaStream_t st);
template <typename T, int P> void t2_yzq(const GroupArgs<T>& g, cudaStream_t st);  // double only
template <typename T, int P> void t2_smem_limits(int bytes);
// The limits of the two-pass kernels of lengths Px and Py (those that have some).
template <typename T> void set_t2_smem_limits(int Px, int Py, int bytes);
void launch_interp_identity(InterpEntry* tab, int img0, int K, cudaStream_t st);
// the FP32 state [K][3][N] handed to the FP64 energy evaluation: every spin renormalised in FP64
void launch_widen_unit(const float* src, double* dst, int K, int N, const int* pair_on, cudaStream_t st);
// FP64 setup of the dipole-tensor spectrum: x then y transforms of the padded real-space tensor
// (data [6*nz][Py][Px] complex, in place), then the octant extraction into dhat.
void launch_fft_strided_f64(double2* data, const double2* tw, const FftPlan& plan, int n_lines, long elem_stride,
                            int inner_count, long inner_stride, long outer_stride, cudaStream_t st);
template <typename T> void set_smem_limits(int bytes);
template <typename T>
void launch_extract_octant(const double2* spec, T* dhat, int Px, int Py, int nz, double scale, cudaStream_t st);

}  // namespace ss
