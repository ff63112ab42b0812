// k_operator.cu -- operator and exact-inverse kernels for the convection-diffusion family.
//
// W = (tA)^{-1} V replaces the paper's "LU once, then U \ (L \ w)" (Section 4.1,
// Section 5) by an exact structured solve: tA = t (T_x (+) T_y (+) T_z) (Kronecker sum)
// with T_d = D_d^{-1} Q Lambda_d Q D_d (diagonal similarity D_d = diag(rho^j),
// rho = sqrt(u/l); Q the orthonormal DST-I, symmetric, Q Q = I).  Transform every axis
// except x with (D_d, Q), solve one tridiagonal system along x per transformed mode with
// the shift lambda_y + lambda_z, transform back.  The transforms are small dense GEMMs
// (DST-I for N + 1 prime or odd has no cheap power-of-two FFT), the line solves use a
// Thomas factorisation built once per mode at plan creation.
#include "df.cuh"
#include "internal.h"

namespace expm {
namespace {

constexpr int BK = 16;

// C = A * B, FP64.  256 threads, TM x TM outputs per thread (tiles of 16 TM).  CM selects the thread
// layout so that the fastest-varying thread index walks C's contiguous dimension.  The FP64 pipe (2 FMAs
// per SM and clock) is the bound, whatever the tile: a 64 x 64 tile keeps one SM busy for 100 us at
// K = 99, so small problems take smaller tiles and spread over the SMs (launch_gemm picks the tile with
// the least work on the fullest SM; 99 x 99, 3 columns: 127 us with 12 CTAs, 14 us with 147).
template <bool CM, int TM>
__global__ void __launch_bounds__(256) k_gemm(GemmArgs g) {
    constexpr int BM = 16 * TM, BN = 16 * TM;
    __shared__ double As[BK][BM + 1];
    __shared__ double Bs[BK][BN];
    const int b1 = blockIdx.z % g.nb1, b2 = blockIdx.z / g.nb1;
    const double* A = g.A + b1 * g.a_b1 + b2 * g.a_b2;
    double* C = g.C + b1 * g.c_b1 + b2 * g.c_b2;
    const int m0 = blockIdx.x * BM, n0 = blockIdx.y * BN;
    const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
    const bool a_mfast = (g.a_rs == 1);
    double acc[TM][TM];
#pragma unroll
    for (int i = 0; i < TM; ++i)
#pragma unroll
        for (int j = 0; j < TM; ++j) acc[i][j] = 0.0;
    for (int k0 = 0; k0 < g.K; k0 += BK) {
#pragma unroll
        for (int q = 0; q < TM; ++q) {
            const int e = tid + q * 256;
            int mm, kk;
            if (a_mfast) { mm = e % BM; kk = e / BM; }
            else { kk = e % BK; mm = e / BK; }
            const int gm = m0 + mm, gk = k0 + kk;
            As[kk][mm] = (gm < g.M && gk < g.K) ? A[(int64_t)gm * g.a_rs + (int64_t)gk * g.a_cs] : 0.0;
        }
#pragma unroll
        for (int q = 0; q < TM; ++q) {
            const int e = tid + q * 256;
            const int nn = e % BN, kk = e / BN;
            const int gn = n0 + nn, gk = k0 + kk;
            Bs[kk][nn] = (gn < g.N && gk < g.K) ? g.B[(int64_t)gk * g.ldb + gn] : 0.0;
        }
        __syncthreads();
#pragma unroll
        for (int kk = 0; kk < BK; ++kk) {
            double a[TM], b[TM];
#pragma unroll
            for (int i = 0; i < TM; ++i) a[i] = As[kk][(CM ? tx : ty) + 16 * i];
#pragma unroll
            for (int j = 0; j < TM; ++j) b[j] = Bs[kk][(CM ? ty : tx) + 16 * j];
#pragma unroll
            for (int i = 0; i < TM; ++i)
#pragma unroll
                for (int j = 0; j < TM; ++j) acc[i][j] = fma(a[i], b[j], acc[i][j]);
        }
        __syncthreads();
    }
#pragma unroll
    for (int i = 0; i < TM; ++i)
#pragma unroll
        for (int j = 0; j < TM; ++j) {
            const int m = m0 + (CM ? tx : ty) + 16 * i, nn = n0 + (CM ? ty : tx) + 16 * j;
            if (m < g.M && nn < g.N) C[(int64_t)m * g.c_rs + (int64_t)nn * g.c_cs] = acc[i][j];
        }
}

// Line solves along x with the precomputed Thomas factors of tridiag(l, c + lambda_mode, u):
// forward  y_x = (f_x / t - l y_{x-1}) m_x,  backward  z_x = y_x - c'_x z_{x+1} (z_L = 0).
// Both are first-order linear recurrences, i.e. compositions of affine maps v -> a v + b, so
// each line is split into TSEG segments handled by TSEG lanes of one warp: every lane composes
// its segment's map, the segments' entry values are passed lane to lane with shuffles, and
// every lane then reruns its segment from the right entry value.  Lanes of a warp hold
// 32 / TSEG consecutive modes of the same segment position, so each warp-wide load touches
// TSEG fully used 32-byte sectors (the layout is mode-fastest).  in may equal out: every
// element is read and written by the one lane that owns its segment.
constexpr int TSEG = 8;
constexpr int TUNR = 8;    // loads issued ahead inside a segment

template <typename T>
__device__ inline void tridiag_seg(const T* f, T* y, int L, int64_t nm, int64_t k, T l_sub,
                                   const T* __restrict__ thm, const T* __restrict__ thc, T inv_t, int seg,
                                   bool active) {
    const int seglen = (L + TSEG - 1) / TSEG;
    const int x0 = min(L, seg * seglen), x1 = min(L, x0 + seglen);
    const unsigned full = 0xffffffffu;
    // forward: compose y_out = A y_in + B over the segment
    T A = 1, B = 0;
    if (active)
        for (int xb = x0; xb < x1; xb += TUNR) {
            T fv[TUNR], mv[TUNR];
#pragma unroll
            for (int q = 0; q < TUNR; ++q)
                if (xb + q < x1) {
                    fv[q] = f[(int64_t)(xb + q) * nm];
                    mv[q] = thm[(int64_t)(xb + q) * nm + k];
                }
#pragma unroll
            for (int q = 0; q < TUNR; ++q)
                if (xb + q < x1) {
                    const T a = -l_sub * mv[q];
                    B = a * B + fv[q] * inv_t * mv[q];
                    A = a * A;
                }
        }
    T yin = 0;
    for (int sgi = 1; sgi < TSEG; ++sgi) {
        const T v = __shfl_up_sync(full, A * yin + B, 1);
        if (seg == sgi) yin = v;
    }
    if (active) {
        T prev = yin;
        for (int xb = x0; xb < x1; xb += TUNR) {
            T fv[TUNR], mv[TUNR];
#pragma unroll
            for (int q = 0; q < TUNR; ++q)
                if (xb + q < x1) {
                    fv[q] = f[(int64_t)(xb + q) * nm];
                    mv[q] = thm[(int64_t)(xb + q) * nm + k];
                }
#pragma unroll
            for (int q = 0; q < TUNR; ++q)
                if (xb + q < x1) {
                    prev = (fv[q] * inv_t - l_sub * prev) * mv[q];
                    y[(int64_t)(xb + q) * nm] = prev;
                }
        }
    }
    // backward: z_out(x0) = A z_in(x1) + B over the segment, from x1 - 1 down to x0
    A = 1;
    B = 0;
    if (active)
        for (int xb = x1 - 1; xb >= x0; xb -= TUNR) {
            T yv[TUNR], cv[TUNR];
#pragma unroll
            for (int q = 0; q < TUNR; ++q)
                if (xb - q >= x0) {
                    yv[q] = y[(int64_t)(xb - q) * nm];
                    cv[q] = (xb - q < L - 1) ? thc[(int64_t)(xb - q) * nm + k] : T(0);
                }
#pragma unroll
            for (int q = 0; q < TUNR; ++q)
                if (xb - q >= x0) {
                    B = yv[q] - cv[q] * B;
                    A = -cv[q] * A;
                }
        }
    T zin = 0;
    for (int sgi = TSEG - 2; sgi >= 0; --sgi) {
        const T v = __shfl_down_sync(full, A * zin + B, 1);
        if (seg == sgi) zin = v;
    }
    if (active) {
        T next = zin;
        for (int xb = x1 - 1; xb >= x0; xb -= TUNR) {
            T yv[TUNR], cv[TUNR];
#pragma unroll
            for (int q = 0; q < TUNR; ++q)
                if (xb - q >= x0) {
                    yv[q] = y[(int64_t)(xb - q) * nm];
                    cv[q] = (xb - q < L - 1) ? thc[(int64_t)(xb - q) * nm + k] : T(0);
                }
#pragma unroll
            for (int q = 0; q < TUNR; ++q)
                if (xb - q >= x0) {
                    next = yv[q] - cv[q] * next;
                    y[(int64_t)(xb - q) * nm] = next;
                }
        }
    }
}

// line index of a lane: warp-major groups of 32 / TSEG lines, TSEG segment lanes per line
__device__ inline int64_t seg_line(int& seg) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    seg = lane % TSEG;
    return ((int64_t)blockIdx.x * (blockDim.x >> 5) + warp) * (32 / TSEG) + lane / TSEG;
}

__global__ void k_tridiag_lines(const double* in, int64_t ld_in, double* out, int64_t ld_out,
                                int p, int L, int64_t nmodes, double l_sub,
                                const double* __restrict__ thm, const double* __restrict__ thc,
                                double inv_t) {
    int seg;
    const int64_t line = seg_line(seg);
    const bool active = line < nmodes * p;
    const int64_t k = active ? line % nmodes : 0;
    const int c = active ? (int)(line / nmodes) : 0;
    tridiag_seg<double>(in + c * ld_in + k, out + c * ld_out + k, L, nmodes, k, l_sub, thm, thc, inv_t, seg,
                        active);
}

// A single long line per column (1-D problems): one CTA per line.  Thread t owns kLineE consecutive
// points of each chunk of kLineT kLineE; it composes their affine maps keeping the partial results, the
// CTA scans the threads' maps, and each point is corrected with the value that enters its segment
// (y = y_local + P y_in), so every point is read once per sweep and costs nine FP64 operations.  With the
// warp-per-four-lines kernel above, 2000 points were 250 dependent FP64 steps per lane: 178 us a solve,
// now 13 us, most of it the one SM's FP64 pipe.
constexpr int kLineT = 256, kLineE = 8;

struct Affine {
    double a, b;     // v -> a v + b
};

// exclusive scan over the CTA of the maps in thread order (rev: descending), the total in *tot; red:
// one slot per warp
__device__ inline Affine line_scan(Affine m, bool rev, Affine* red, Affine* tot) {
    const unsigned full = 0xffffffffu;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, pos = rev ? 31 - lane : lane;
    const int nw = kLineT / 32, wpos = rev ? nw - 1 - warp : warp;
    Affine x = m;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        const int src = rev ? lane + d : lane - d;
        const double pa = __shfl_sync(full, x.a, src & 31), pb = __shfl_sync(full, x.b, src & 31);
        if (pos >= d) {
            x.b = fma(x.a, pb, x.b);
            x.a = x.a * pa;
        }
    }
    __syncthreads();
    if (pos == 31) red[wpos] = x;
    const int prev = rev ? lane + 1 : lane - 1;
    Affine e;
    e.a = __shfl_sync(full, x.a, prev & 31);
    e.b = __shfl_sync(full, x.b, prev & 31);
    if (pos == 0) e = Affine{1.0, 0.0};
    __syncthreads();
    Affine w{1.0, 0.0}, all{1.0, 0.0};
    for (int k = 0; k < nw; ++k) {
        if (k == wpos) w = all;
        all = Affine{red[k].a * all.a, fma(red[k].a, all.b, red[k].b)};
    }
    *tot = all;
    return Affine{e.a * w.a, fma(e.a, w.b, e.b)};
}

__global__ void __launch_bounds__(kLineT) k_line_solve(const double* in, int64_t ld_in, double* out, int64_t ld_out,
                                                       int L, double l_sub, const double* __restrict__ thm,
                                                       const double* __restrict__ thc, double inv_t) {
    __shared__ Affine red[kLineT / 32];
    const double* f = in + (int64_t)blockIdx.x * ld_in;
    double* y = out + (int64_t)blockIdx.x * ld_out;
    constexpr int CH = kLineT * kLineE;
    const int nch = (L + CH - 1) / CH;
    double yv[kLineE], pv[kLineE];
    double carry = 0.0;
    for (int ch = 0; ch < nch; ++ch) {
        const int x0 = ch * CH + threadIdx.x * kLineE;
        double mv[kLineE];
#pragma unroll
        for (int q = 0; q < kLineE; ++q) {
            yv[q] = x0 + q < L ? f[x0 + q] : 0.0;
            mv[q] = x0 + q < L ? thm[x0 + q] : 0.0;
        }
        Affine m{1.0, 0.0};
#pragma unroll
        for (int q = 0; q < kLineE; ++q) {
            const double a = -l_sub * mv[q];
            m.b = fma(a, m.b, yv[q] * inv_t * mv[q]);
            m.a *= a;
            yv[q] = m.b;
            pv[q] = m.a;
        }
        Affine tot;
        const Affine ex = line_scan(m, false, red, &tot);
        const double yin = fma(ex.a, carry, ex.b);
        carry = fma(tot.a, carry, tot.b);
#pragma unroll
        for (int q = 0; q < kLineE; ++q) {
            yv[q] = fma(pv[q], yin, yv[q]);
            if (x0 + q < L && ch + 1 < nch) y[x0 + q] = yv[q];      // the last chunk stays in registers
        }
    }
    carry = 0.0;
    for (int ch = nch - 1; ch >= 0; --ch) {
        const int x0 = ch * CH + threadIdx.x * kLineE;
        double cv[kLineE];
#pragma unroll
        for (int q = 0; q < kLineE; ++q) {
            if (ch + 1 < nch) yv[q] = x0 + q < L ? y[x0 + q] : 0.0;
            else if (x0 + q >= L) yv[q] = 0.0;
            cv[q] = x0 + q < L - 1 ? thc[x0 + q] : 0.0;
        }
        Affine m{1.0, 0.0};
#pragma unroll
        for (int q = kLineE - 1; q >= 0; --q) {
            m.b = fma(-cv[q], m.b, yv[q]);
            m.a *= -cv[q];
            yv[q] = m.b;
            pv[q] = m.a;
        }
        Affine tot;
        const Affine ex = line_scan(m, true, red, &tot);
        const double zin = fma(ex.a, carry, ex.b);
        carry = fma(tot.a, carry, tot.b);
#pragma unroll
        for (int q = 0; q < kLineE; ++q)
            if (x0 + q < L) y[x0 + q] = fma(pv[q], zin, yv[q]);
    }
}

// Thomas factors for every mode (one thread per mode): pivots b - l c'_{x-1}, stored as
// reciprocals, and c'_x = u / pivot_x.
__global__ void k_thomas_setup(double* thm, double* thc, int L, int64_t nmodes, double l,
                               double c, double u, const double* lam_y, int Ny,
                               const double* lam_z, int Nz) {
    const int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= nmodes) return;
    double shift = 0.0;
    if (lam_y) shift += lam_y[k % Ny];
    if (lam_z) shift += lam_z[k / Ny];
    const double b = c + shift;
    double cp = 0.0;
    for (int x = 0; x < L; ++x) {
        const double piv = b - (x > 0 ? l * cp : 0.0);
        const double mi = 1.0 / piv;
        cp = u * mi;
        thm[(int64_t)x * nmodes + k] = mi;
        thc[(int64_t)x * nmodes + k] = cp;
    }
}

// Axis eigen-data: Q[j][k] = sqrt(2/(N+1)) sin(pi (j+1)(k+1)/(N+1)) (DST-I, exact
// integer argument reduction), Qf = diag(rho^j) Q, Qi = Q diag(rho^-j),
// lambda_k = c + 2 s cos(pi (k+1)/(N+1)), s = sign(l) sqrt(l u).
__global__ void k_axis_setup(double* Qf, double* Qi, double* lam, int N, double l, double c,
                             double u) {
    const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= (int64_t)N * N) return;
    const int j = (int)(e / N), k = (int)(e % N);
    const int64_t arg = ((int64_t)(j + 1) * (k + 1)) % (2 * (int64_t)(N + 1));
    const double q = sqrt(2.0 / (N + 1)) * sinpi((double)arg / (double)(N + 1));
    const double rho = sqrt(u / l);
    Qf[e] = pow(rho, (double)j) * q;              // row j (grid index), column k (mode)
    Qi[e] = q * pow(rho, -(double)k);             // row j (mode), column k (grid index)
    if (j == 0) {
        const double s = (l > 0 ? 1.0 : -1.0) * sqrt(l * u);
        lam[k] = c + 2.0 * s * cospi((double)(k + 1) / (double)(N + 1));
    }
}

// W = t (A V) + beta Y, 3/5/7-point stencil with Dirichlet zeros outside the grid.
// (beta = 0, Y = null: the operator apply; t -> -t, beta = 1: the residual Y - tA V.)
// Stencil coefficients with t folded in (computed on the host): tc = t (c_x + c_y + c_z),
// tl[d] = t l_d, tu[d] = t u_d; 5 (2-D) or 7 (3-D) FP64 multiply-adds per point.
struct StencilT {
    double tc, tl[3], tu[3];
};

// W = tA V (+ beta Y): one thread per grid point and column; grid index arithmetic in 32 bits
// (n < 2^31 is checked by the launcher).  With W32 set, the result is stored rounded to FP32 there (same
// leading dimension), and in W as well when that is given: the refinement residual, whose FP32 copy the
// transforms read and whose FP64 value the next residual starts from.
__global__ void k_cd_apply(const double* __restrict__ V, int64_t ldv, double* __restrict__ W,
                           int64_t ldw, int ndim, int nx, int ny, int nz, StencilT k,
                           const double* __restrict__ Y, int64_t ldy, double beta, float* __restrict__ W32) {
    const unsigned n = (unsigned)nx * (unsigned)ny * (unsigned)nz;
    const unsigned i = blockIdx.x * blockDim.x + threadIdx.x;
    const int c = blockIdx.y;
    if (i >= n) return;
    const double* v = V + c * ldv;
    const unsigned q = i / (unsigned)nx;
    const unsigned ix = i - q * (unsigned)nx;
    double acc = k.tc * v[i];
    if (ix > 0) acc = fma(k.tl[0], v[i - 1], acc);
    if (ix < (unsigned)nx - 1) acc = fma(k.tu[0], v[i + 1], acc);
    if (ndim > 1) {
        const unsigned iz = q / (unsigned)ny, iy = q - iz * (unsigned)ny;
        if (iy > 0) acc = fma(k.tl[1], v[i - nx], acc);
        if (iy < (unsigned)ny - 1) acc = fma(k.tu[1], v[i + nx], acc);
        if (ndim > 2) {
            const unsigned st = (unsigned)nx * (unsigned)ny;
            if (iz > 0) acc = fma(k.tl[2], v[i - st], acc);
            if (iz < (unsigned)nz - 1) acc = fma(k.tu[2], v[i + st], acc);
        }
    }
    const double r = Y ? fma(beta, Y[c * ldy + i], acc) : acc;
    if (W32) W32[c * ldw + i] = f32_rn_i(r);   // integer rounding: no FP64-pipe conversion
    if (W) W[c * ldw + i] = r;
}

// The next residual of a 3-D grid's refined inverse from the last one: R1 - tA D for the FP32 correction D that was
// added to x, in float pairs (coefficients as pairs, D exact floats), rounded to FP32.  D is ~1e-7 of x, so
// the pairs' 2^-48 of |tA||D| lies far below what FP64 resolves of the residual formed from x itself
// (2^-53 |tA||x|); the FP64 pipe, which bounds that form (8 operations a point, 201 us at 96^3, p = 16; both
// residuals of a step 410 -> 313 us), is not used.
struct StencilDF {
    float ch, cl, lh[3], ll[3], uh[3], ul[3];
};

__device__ __forceinline__ void df_term32(float& sh, float& sl, float v, float ch, float cl) {
    const float pr = v * ch;
    const float e = fmaf(v, cl, fmaf(v, ch, -pr));
    df_add(sh, sl, pr);
    sl += e;
}

__global__ void k_cd_next_residual(const double* __restrict__ R1, int64_t ldr, const float* __restrict__ D, int64_t ldd,
                                   float* __restrict__ R2, int64_t ld2, int nx, int ny, int nz, StencilDF k) {
    const unsigned n = (unsigned)nx * (unsigned)ny * (unsigned)nz;
    const unsigned i = blockIdx.x * blockDim.x + threadIdx.x;
    const int c = blockIdx.y;
    if (i >= n) return;
    const float* v = D + c * ldd;
    const unsigned q = i / (unsigned)nx;
    const unsigned ix = i - q * (unsigned)nx;
    float sh, sl;
    split_df_i(R1[c * ldr + i], sh, sl);
    const unsigned iz = q / (unsigned)ny, iy = q - iz * (unsigned)ny;
    const unsigned st = (unsigned)nx * (unsigned)ny;
    df_term32(sh, sl, v[i], k.ch, k.cl);
    if (ix > 0) df_term32(sh, sl, v[i - 1], k.lh[0], k.ll[0]);
    if (ix < (unsigned)nx - 1) df_term32(sh, sl, v[i + 1], k.uh[0], k.ul[0]);
    if (iy > 0) df_term32(sh, sl, v[i - nx], k.lh[1], k.ll[1]);
    if (iy < (unsigned)ny - 1) df_term32(sh, sl, v[i + nx], k.uh[1], k.ul[1]);
    if (iz > 0) df_term32(sh, sl, v[i - st], k.lh[2], k.ll[2]);
    if (iz < (unsigned)nz - 1) df_term32(sh, sl, v[i + st], k.uh[2], k.ul[2]);
    R2[c * ld2 + i] = sh + sl;
}

// The same stencil in double-float arithmetic on the FP32 pipe, for mixed-precision plans:
// coefficients as float pairs (host-split), every value split from its bit pattern
// (split_df_i), products and sums as in the double-float row kernels.  GB300 retires about two
// FP64 FMAs per SM per clock, so the FP64 stencil (5 or 7 per point) is bound by the FP64
// pipe, not by memory; the pair arithmetic is ~2^-48 accurate, the level of the mixed path's
// other double-float kernels.  Y (the refinement's right-hand side) enters with beta = 1.

__device__ __forceinline__ void df_term(float& sh, float& sl, double v, float ch, float cl) {
    float vh, vl;
    split_df_i(v, vh, vl);
    df_fma(sh, sl, vh, vl, ch, cl);
}

__global__ void k_cd_apply_df(const double* __restrict__ V, int64_t ldv, double* __restrict__ W,
                              int64_t ldw, int ndim, int nx, int ny, int nz, StencilDF k,
                              const double* __restrict__ Y, int64_t ldy, float* __restrict__ W32) {
    const unsigned n = (unsigned)nx * (unsigned)ny * (unsigned)nz;
    const unsigned i = blockIdx.x * blockDim.x + threadIdx.x;
    const int c = blockIdx.y;
    if (i >= n) return;
    const double* v = V + c * ldv;
    const unsigned q = i / (unsigned)nx;
    const unsigned ix = i - q * (unsigned)nx;
    float sh = 0.f, sl = 0.f;
    df_term(sh, sl, v[i], k.ch, k.cl);
    if (ix > 0) df_term(sh, sl, v[i - 1], k.lh[0], k.ll[0]);
    if (ix < (unsigned)nx - 1) df_term(sh, sl, v[i + 1], k.uh[0], k.ul[0]);
    if (ndim > 1) {
        const unsigned iz = q / (unsigned)ny, iy = q - iz * (unsigned)ny;
        if (iy > 0) df_term(sh, sl, v[i - nx], k.lh[1], k.ll[1]);
        if (iy < (unsigned)ny - 1) df_term(sh, sl, v[i + nx], k.uh[1], k.ul[1]);
        if (ndim > 2) {
            const unsigned st = (unsigned)nx * (unsigned)ny;
            if (iz > 0) df_term(sh, sl, v[i - st], k.lh[2], k.ll[2]);
            if (iz < (unsigned)nz - 1) df_term(sh, sl, v[i + st], k.uh[2], k.ul[2]);
        }
    }
    if (Y) {
        float yh, yl;
        split_df_i(Y[c * ldy + i], yh, yl);
        df_add(sh, sl, yh);
        sl += yl;
    }
    if (W32) W32[c * ldw + i] = sh + sl;
    if (W) W[c * ldw + i] = f64_of_f32_i(sh) + f64_of_f32_i(sl);
}

// ---------------------------------------------------------------- mixed precision
// FP32 line solves of the exact inverse (its transforms are in k_transform.cu); the result is refined in
// FP64 by the caller (residual with the FP64 stencil, Theorem 4.3 bounds what an inexact inverse costs).
// The FP32 line solves with the lines staged in shared memory: a CTA takes TK consecutive
// modes of one column (16 x L values of f, thm and thc, loaded once with coalesced reads),
// runs the same segmented affine scans as tridiag_seg from shared memory and writes y back.
// Each mode's line is stored contiguously with one pad element per segment, so the TSG lanes
// of a line read distinct banks (segment stride seglen + 1, odd for L = 256).
constexpr int TK = 16;
constexpr int TSG = 32;    // segments per line in the tile kernel (one line per warp)
constexpr size_t kTridiagTileSmemMax = 110 * 1024;
__host__ __device__ constexpr size_t tridiag_tile_smem(int L) { return sizeof(float) * 3 * (size_t)TK * (L + TSG); }

__global__ void __launch_bounds__(TK * TSG) k_tridiag_tile32(float* y_io, int64_t ld, int L, int64_t nmodes,
                                                             float l_sub, const float* __restrict__ thm,
                                                             const float* __restrict__ thc, float inv_t) {
    extern __shared__ float smt[];
    const int Lp = L + TSG;
    const int seglen = (L + TSG - 1) / TSG;
    float* F = smt;                  // TK x Lp: f, then y in place
    float* Mt = F + TK * Lp;
    float* Ct = Mt + TK * Lp;
    const int c = blockIdx.y;
    const int64_t k0 = (int64_t)blockIdx.x * TK;
    float* y = y_io + (int64_t)c * ld;
    constexpr int NT = TK * TSG, UB = 8;   // UB elements (3 UB loads) in flight per thread
    const int tot = L * TK;
    for (int e0 = threadIdx.x; e0 < tot; e0 += UB * NT) {
        float fv[UB], mv[UB], cv[UB];
#pragma unroll
        for (int u = 0; u < UB; ++u) {
            const int e = e0 + u * NT, x = e / TK, kk = e - x * TK;
            const int64_t k = k0 + kk;
            const bool ok = e < tot && k < nmodes;
            fv[u] = ok ? y[(int64_t)x * nmodes + k] : 0.f;
            mv[u] = ok ? thm[(int64_t)x * nmodes + k] : 0.f;
            cv[u] = ok ? thc[(int64_t)x * nmodes + k] : 0.f;
        }
#pragma unroll
        for (int u = 0; u < UB; ++u) {
            const int e = e0 + u * NT, x = e / TK, kk = e - x * TK;
            if (e < tot) {
                const int si = kk * Lp + x + x / seglen;
                F[si] = fv[u];
                Mt[si] = mv[u];
                Ct[si] = cv[u];
            }
        }
    }
    __syncthreads();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int seg = lane % TSG, kk = warp * (32 / TSG) + lane / TSG;
    const int x0 = min(L, seg * seglen), x1 = min(L, x0 + seglen);
    float* f = F + kk * Lp + seg;          // element x of the line at f[x] (x in this segment)
    const float* m = Mt + kk * Lp + seg;
    const float* cc = Ct + kk * Lp + seg;
    const unsigned full = 0xffffffffu;
    float A = 1.f, B = 0.f;
    for (int x = x0; x < x1; ++x) {
        const float a = -l_sub * m[x];
        B = a * B + f[x] * inv_t * m[x];
        A = a * A;
    }
    // inclusive scan of the segment maps y -> A y + B over the line's TSG lanes (log2 TSG
    // steps; the composition is associative), then the value entering each segment is the
    // previous segment's prefix applied to 0
#pragma unroll
    for (int d = 1; d < TSG; d <<= 1) {
        const float Ap = __shfl_up_sync(full, A, d, TSG), Bp = __shfl_up_sync(full, B, d, TSG);
        if (seg >= d) {
            B = fmaf(A, Bp, B);
            A = A * Ap;
        }
    }
    float yin = __shfl_up_sync(full, B, 1, TSG);
    if (seg == 0) yin = 0.f;
    float prev = yin;
    for (int x = x0; x < x1; ++x) {
        prev = (f[x] * inv_t - l_sub * prev) * m[x];
        f[x] = prev;
    }
    A = 1.f;
    B = 0.f;
    for (int x = x1 - 1; x >= x0; --x) {
        const float cv = (x < L - 1) ? cc[x] : 0.f;
        B = f[x] - cv * B;
        A = -cv * A;
    }
#pragma unroll
    for (int d = 1; d < TSG; d <<= 1) {
        const float An = __shfl_down_sync(full, A, d, TSG), Bn = __shfl_down_sync(full, B, d, TSG);
        if (seg + d < TSG) {
            B = fmaf(A, Bn, B);
            A = A * An;
        }
    }
    float zin = __shfl_down_sync(full, B, 1, TSG);
    if (seg == TSG - 1) zin = 0.f;
    float next = zin;
    for (int x = x1 - 1; x >= x0; --x) {
        const float cv = (x < L - 1) ? cc[x] : 0.f;
        next = f[x] - cv * next;
        f[x] = next;
    }
    __syncthreads();
    for (int e = threadIdx.x; e < L * TK; e += blockDim.x) {
        const int x = e / TK, kk2 = e - x * TK;
        const int64_t k = k0 + kk2;
        if (k < nmodes) y[(int64_t)x * nmodes + k] = F[kk2 * Lp + x + x / seglen];
    }
}

// Short lines with many modes (the x lines of a 3-D grid, L <= 128, ny nz modes): one thread
// per (mode, column) runs both sweeps of the factored solve over its line, consecutive
// threads on consecutive modes (coalesced: the layout is mode-fastest).  The sweeps' loads do
// not depend on the recurrence, but they may alias the stores as far as the compiler knows,
// so each sweep reads its line in explicit batches of TB elements into registers and issues
// the next batch's loads before it stores the current one.
constexpr int TB = 8;
__global__ void __launch_bounds__(256) k_tridiag_thread32(float* y_io, int64_t ld, int L, int64_t nmodes,
                                                          float l_sub, const float* __restrict__ thm,
                                                          const float* __restrict__ thc, float inv_t) {
    const int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= nmodes) return;
    float* y = y_io + (int64_t)blockIdx.y * ld + k;
    const float* m = thm + k;
    const float* cc = thc + k;
    float yv[TB], mv[TB], out[TB];
    // forward sweep, x ascending
#pragma unroll
    for (int u = 0; u < TB; ++u) {
        yv[u] = u < L ? y[(int64_t)u * nmodes] : 0.f;
        mv[u] = u < L ? m[(int64_t)u * nmodes] : 0.f;
    }
    float prev = 0.f;
    for (int x0 = 0; x0 < L; x0 += TB) {
#pragma unroll
        for (int u = 0; u < TB; ++u) {
            if (x0 + u < L) prev = (yv[u] * inv_t - l_sub * prev) * mv[u];
            out[u] = prev;
        }
        if (x0 + TB < L) {
#pragma unroll
            for (int u = 0; u < TB; ++u) {
                const int x = x0 + TB + u;
                yv[u] = x < L ? y[(int64_t)x * nmodes] : 0.f;
                mv[u] = x < L ? m[(int64_t)x * nmodes] : 0.f;
            }
        }
#pragma unroll
        for (int u = 0; u < TB; ++u)
            if (x0 + u < L) y[(int64_t)(x0 + u) * nmodes] = out[u];
    }
    // backward sweep, x descending from L - 1 (whose value the forward sweep left final)
    int xb = L - 2;
#pragma unroll
    for (int u = 0; u < TB; ++u) {
        yv[u] = xb - u >= 0 ? y[(int64_t)(xb - u) * nmodes] : 0.f;
        mv[u] = xb - u >= 0 ? cc[(int64_t)(xb - u) * nmodes] : 0.f;
    }
    float next = prev;
    for (; xb >= 0; xb -= TB) {
#pragma unroll
        for (int u = 0; u < TB; ++u) {
            next = yv[u] - mv[u] * next;
            out[u] = next;
        }
        if (xb - TB >= 0) {
#pragma unroll
            for (int u = 0; u < TB; ++u) {
                const int x = xb - TB - u;
                yv[u] = x >= 0 ? y[(int64_t)x * nmodes] : 0.f;
                mv[u] = x >= 0 ? cc[(int64_t)x * nmodes] : 0.f;
            }
        }
#pragma unroll
        for (int u = 0; u < TB; ++u)
            if (xb - u >= 0) y[(int64_t)(xb - u) * nmodes] = out[u];
    }
}

__global__ void k_tridiag_lines32(float* y_io, int64_t ld, int p, int L, int64_t nmodes,
                                  float l_sub, const float* __restrict__ thm,
                                  const float* __restrict__ thc, float inv_t) {
    int seg;
    const int64_t line = seg_line(seg);
    const bool active = line < nmodes * p;
    const int64_t k = active ? line % nmodes : 0;
    const int c = active ? (int)(line / nmodes) : 0;
    float* y = y_io + c * ld + k;
    tridiag_seg<float>(y, y, L, nmodes, k, l_sub, thm, thc, inv_t, seg, active);
}

// Certify mode: partial sums of ||B - (tA - tau_i I) X_i||_F^2 per pole, X_i = Xr + i Xi stored
// as columns [i 2p + c] (real) and [i 2p + p + c] (imaginary) of X.  One partial per CTA and
// pole; the host adds them.
__global__ void k_true_resid(const double* __restrict__ X, int64_t ldx, const double* __restrict__ B,
                             int64_t ldb, int p, int npoles, int ndim, int nx, int ny, int nz, Axis ax0,
                             Axis ax1, Axis ax2, double t, const double* __restrict__ tau_re,
                             const double* __restrict__ tau_im, double* __restrict__ part,
                             const double* __restrict__ AX, int64_t ldax) {
    __shared__ double red[256];
    const int64_t n = (int64_t)nx * ny * nz;
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int pole = blockIdx.y;
    double acc = 0.0;
    if (i < n) {
        const int ix = (int)(i % nx);
        const int iy = (int)((i / nx) % ny);
        const int iz = (int)(i / ((int64_t)nx * ny));
        const double dc = ax0.c + (ndim > 1 ? ax1.c : 0.0) + (ndim > 2 ? ax2.c : 0.0);
        const double tr = tau_re[pole], ti = tau_im[pole];
        for (int c = 0; c < p; ++c) {
            double ax[2];
            for (int part_ = 0; part_ < 2; ++part_) {
                if (AX) {
                    ax[part_] = AX[(int64_t)(2 * pole * p + part_ * p + c) * ldax + i];
                    continue;
                }
                const double* v = X + (int64_t)(2 * pole * p + part_ * p + c) * ldx;
                double s = dc * v[i];
                if (ix > 0) s += ax0.l * v[i - 1];
                if (ix < nx - 1) s += ax0.u * v[i + 1];
                if (ndim > 1) {
                    if (iy > 0) s += ax1.l * v[i - nx];
                    if (iy < ny - 1) s += ax1.u * v[i + nx];
                }
                if (ndim > 2) {
                    const int64_t st = (int64_t)nx * ny;
                    if (iz > 0) s += ax2.l * v[i - st];
                    if (iz < nz - 1) s += ax2.u * v[i + st];
                }
                ax[part_] = t * s;
            }
            const double xr = X[(int64_t)(2 * pole * p + c) * ldx + i];
            const double xi = X[(int64_t)(2 * pole * p + p + c) * ldx + i];
            // (tA - tau)(xr + i xi) = (A xr - tr xr + ti xi) + i (A xi - tr xi - ti xr)
            const double rre = B[(int64_t)c * ldb + i] - (ax[0] - tr * xr + ti * xi);
            const double rim = -(ax[1] - tr * xi - ti * xr);
            acc += rre * rre + rim * rim;
        }
    }
    red[threadIdx.x] = acc;
    __syncthreads();
    for (int st = 128; st > 0; st >>= 1) {
        if (threadIdx.x < st) red[threadIdx.x] += red[threadIdx.x + st];
        __syncthreads();
    }
    if (threadIdx.x == 0) part[(int64_t)pole * gridDim.x + blockIdx.x] = red[0];
}

__global__ void k_d2f(const double* __restrict__ in, float* __restrict__ out, int64_t n, int64_t ldin, int64_t ldout) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) out[blockIdx.y * ldout + i] = f32_rn_i(in[blockIdx.y * ldin + i]);
}

}  // namespace

cudaError_t launch_gemm(const GemmArgs& g, cudaStream_t s) {
    // FP64 work of the fullest SM per tile side: CTAs per SM times tile area; larger tiles (fewer
    // shared-memory loads per FMA) at equal work
    constexpr int64_t kSms = 152;
    int best = 4;
    int64_t cost = INT64_MAX;
    for (int tm = 4; tm >= 1; tm /= 2) {
        const int64_t b = 16 * tm, ctas = ((g.M + b - 1) / b) * ((g.N + b - 1) / b) * (int64_t)(g.nb1 * g.nb2);
        const int64_t c = (ctas + kSms - 1) / kSms * b * b;
        if (c < cost) {
            cost = c;
            best = tm;
        }
    }
    const int b = 16 * best;
    const dim3 grid((g.M + b - 1) / b, (g.N + b - 1) / b, g.nb1 * g.nb2);
    if (g.c_rs == 1) {
        if (best == 4) k_gemm<true, 4><<<grid, 256, 0, s>>>(g);
        else if (best == 2) k_gemm<true, 2><<<grid, 256, 0, s>>>(g);
        else k_gemm<true, 1><<<grid, 256, 0, s>>>(g);
    } else {
        if (best == 4) k_gemm<false, 4><<<grid, 256, 0, s>>>(g);
        else if (best == 2) k_gemm<false, 2><<<grid, 256, 0, s>>>(g);
        else k_gemm<false, 1><<<grid, 256, 0, s>>>(g);
    }
    return cudaGetLastError();
}

cudaError_t launch_tridiag_lines(const double* in, int64_t ld_in, double* out, int64_t ld_out,
                                 int p, int L, int64_t nmodes, double l_sub, const double* th_m,
                                 const double* th_c, double inv_t, cudaStream_t s) {
    if (nmodes == 1) {
        k_line_solve<<<p, kLineT, 0, s>>>(in, ld_in, out, ld_out, L, l_sub, th_m, th_c, inv_t);
        return cudaGetLastError();
    }
    const int64_t lines = nmodes * p, per_block = 128 / TSEG;
    k_tridiag_lines<<<(unsigned)((lines + per_block - 1) / per_block), 128, 0, s>>>(in, ld_in, out, ld_out, p, L,
                                                                                 nmodes, l_sub, th_m, th_c, inv_t);
    return cudaGetLastError();
}

cudaError_t launch_thomas_setup(double* th_m, double* th_c, int L, int64_t nmodes, double l,
                                double c, double u, const double* lam_y, int Ny,
                                const double* lam_z, int Nz, cudaStream_t s) {
    const int thr = 128;
    k_thomas_setup<<<(unsigned)((nmodes + thr - 1) / thr), thr, 0, s>>>(th_m, th_c, L, nmodes, l, c, u,
                                                                        lam_y, Ny, lam_z, Nz);
    return cudaGetLastError();
}

cudaError_t launch_axis_setup(double* Qf, double* Qi, double* lam, int N, double l, double c,
                              double u, cudaStream_t s) {
    const int64_t tot = (int64_t)N * N;
    k_axis_setup<<<(unsigned)((tot + 255) / 256), 256, 0, s>>>(Qf, Qi, lam, N, l, c, u);
    return cudaGetLastError();
}

static void split_host(double x, float& h, float& l) {
    h = (float)x;
    l = (float)(x - (double)h);
}

cudaError_t launch_cd_apply(const double* V, int64_t ldv, double* W, int64_t ldw, int p,
                            int ndim, int nx, int ny, int nz, const Axis* ax, double t,
                            cudaStream_t s, const double* Y, int64_t ldy, double beta, float* W32, int df) {
    const int64_t n = (int64_t)nx * ny * nz;
    if (n >= ((int64_t)1 << 31)) return cudaErrorInvalidValue;
    if (df) {
        if (Y && beta != 1.0) return cudaErrorInvalidValue;
        StencilDF k;
        split_host(t * (ax[0].c + (ndim > 1 ? ax[1].c : 0.0) + (ndim > 2 ? ax[2].c : 0.0)), k.ch, k.cl);
        for (int d = 0; d < 3; ++d) {
            split_host(t * ax[d].l, k.lh[d], k.ll[d]);
            split_host(t * ax[d].u, k.uh[d], k.ul[d]);
        }
        dim3 grid((unsigned)((n + 255) / 256), p);
        k_cd_apply_df<<<grid, 256, 0, s>>>(V, ldv, W, ldw, ndim, nx, ny, nz, k, Y, ldy, W32);
        return cudaGetLastError();
    }
    StencilT k;
    k.tc = t * (ax[0].c + (ndim > 1 ? ax[1].c : 0.0) + (ndim > 2 ? ax[2].c : 0.0));
    for (int d = 0; d < 3; ++d) {
        k.tl[d] = t * ax[d].l;
        k.tu[d] = t * ax[d].u;
    }
    dim3 grid((unsigned)((n + 255) / 256), p);
    k_cd_apply<<<grid, 256, 0, s>>>(V, ldv, W, ldw, ndim, nx, ny, nz, k, Y, ldy, beta, W32);
    return cudaGetLastError();
}

// R2 = R1 - tA D (see k_cd_next_residual)
cudaError_t launch_cd_next_residual(const double* R1, int64_t ldr, const float* D, int64_t ldd, float* R2, int64_t ld2,
                                    int p, int nx, int ny, int nz, const Axis* ax, double t, cudaStream_t s) {
    const int64_t n = (int64_t)nx * ny * nz;
    if (n >= ((int64_t)1 << 31)) return cudaErrorInvalidValue;
    StencilDF k;
    split_host(-t * (ax[0].c + ax[1].c + ax[2].c), k.ch, k.cl);
    for (int d = 0; d < 3; ++d) {
        split_host(-t * ax[d].l, k.lh[d], k.ll[d]);
        split_host(-t * ax[d].u, k.uh[d], k.ul[d]);
    }
    const dim3 grid((unsigned)((n + 255) / 256), p);
    k_cd_next_residual<<<grid, 256, 0, s>>>(R1, ldr, D, ldd, R2, ld2, nx, ny, nz, k);
    return cudaGetLastError();
}

cudaError_t launch_tridiag_lines32(float* y, int64_t ld, int p, int L, int64_t nmodes, float l_sub,
                                   const float* th_m, const float* th_c, float inv_t,
                                   cudaStream_t s) {
    if (L <= 128 && nmodes >= 1024) {
        const dim3 grid((unsigned)((nmodes + 255) / 256), (unsigned)p);
        k_tridiag_thread32<<<grid, 256, 0, s>>>(y, ld, L, nmodes, l_sub, th_m, th_c, inv_t);
        return cudaGetLastError();
    }
    const size_t shm = tridiag_tile_smem(L);
    if (shm <= kTridiagTileSmemMax) {
        const dim3 grid((unsigned)((nmodes + TK - 1) / TK), (unsigned)p);
        k_tridiag_tile32<<<grid, TK * TSG, shm, s>>>(y, ld, L, nmodes, l_sub, th_m, th_c, inv_t);
        return cudaGetLastError();
    }
    const int64_t lines = nmodes * p, per_block = 128 / TSEG;
    k_tridiag_lines32<<<(unsigned)((lines + per_block - 1) / per_block), 128, 0, s>>>(y, ld, p, L, nmodes, l_sub,
                                                                                   th_m, th_c, inv_t);
    return cudaGetLastError();
}

cudaError_t operator_set_smem_limits() {
    return cudaFuncSetAttribute(k_tridiag_tile32, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                (int)kTridiagTileSmemMax);
}

int true_resid_blocks(int64_t n) { return (int)((n + 255) / 256); }

cudaError_t launch_true_resid(const double* X, int64_t ldx, const double* B, int64_t ldb, int p, int npoles,
                              int ndim, int nx, int ny, int nz, const Axis* ax, double t, const double* tau_re,
                              const double* tau_im, double* part, cudaStream_t s, const double* AX,
                              int64_t ldax) {
    const int64_t n = (int64_t)nx * ny * nz;
    dim3 grid((unsigned)true_resid_blocks(n), npoles);
    k_true_resid<<<grid, 256, 0, s>>>(X, ldx, B, ldb, p, npoles, ndim, nx, ny, nz, ax[0], ax[1], ax[2], t,
                                      tau_re, tau_im, part, AX, ldax);
    return cudaGetLastError();
}

cudaError_t launch_d2f(const double* in, float* out, int64_t n, cudaStream_t s, int64_t ldin, int64_t ldout, int cols) {
    k_d2f<<<dim3((unsigned)((n + 255) / 256), (unsigned)cols), 256, 0, s>>>(in, out, n, ldin, ldout);
    return cudaGetLastError();
}

}  // namespace expm
