// k_poles.cu -- the projected shifted systems, one CTA or one cluster of CTAs per pole.
//
// For each pole tau_i (Im > 0) in one launch, Algorithm 2:
//   (I - tau_i H_m) Z_i = E_1 S_i                              eq. (3236)
//   S_i <- tau_i H_{m+1,m} E_m^T Z_i,  ||R_i||_F = ||S_i||_F     eq. (49) and the residual
//                                                             formula above it (collinear
//                                                             with V_{m+1}: restart factor)
//   Wc = sum_i 2 Re(omega_i H~_m Z_i) = H~_m sum_i 2 Re(omega_i Z_i)  (H~ real)
//                                          eq. (4.5): X_i - X_i^0 = (tA)^{-1} V_m Z_i = V_{m+1} H~_m Z_i
// Algorithm 1 (alg = 1): (H_m - tau_i I) Z_i = E_1 S_i (eq. (3.3)), S_i <- -H_{m+1,m} E_m^T Z_i
// (eq. (35)), Wc = [sum_i 2 Re(omega_i Z_i); 0] (X_i - X_i^0 = V_m Z_i).
// H_m is band upper Hessenberg with p sub-diagonals, so Gaussian elimination with partial
// pivoting only looks at rows j..j+p of column j (blocked by p x p blocks, see k_poles).
// After a deflated restart that keeps kk Ritz vectors (a multiple of p), the leading kk
// columns are dense down to row kk+p-1 (the projection of H~ onto the kept vectors) and the
// right-hand side E S_i sits at rows kk..kk+p-1; the elimination of those columns then looks
// at rows j..kk+p-1.  The
// matrix lives in shared memory when (mp)^2 + mp p complex numbers fit, else in a global
// workspace (L2-resident).
#include <algorithm>

#include "internal.h"

namespace expm {
namespace {

struct cplx {
    double re, im;
};
__device__ inline cplx cmul(cplx a, cplx b) { return {a.re * b.re - a.im * b.im, a.re * b.im + a.im * b.re}; }
__device__ inline double cabs2(cplx a) { return a.re * a.re + a.im * a.im; }
// x -= a * b with four fused multiply-adds
__device__ inline void cmsub(cplx& x, cplx a, cplx b) {
    x.re = fma(-a.re, b.re, fma(a.im, b.im, x.re));
    x.im = fma(-a.re, b.im, fma(-a.im, b.re, x.im));
}

constexpr size_t kSmemLimit = 200 * 1024;
constexpr int kPoleThreads = 512;   // sixteen warps per pole: four per scheduler to cover FP64 latency

// One CTA (sixteen warps) per pole.  Shared memory holds M (mp x mp complex, row-major), the
// right-hand sides / solution X (mp x p complex), the inverses of U's diagonal blocks
// (mp x p complex) and, when it fits, the real H~ ((mp+p) x mp), staged once with coalesced
// loads.  Outputs: the restart factor S_i, ||S_i||_F and Y_i = 2 Re(omega_i Z_i) (mp x p
// real).  Since H~ is real, sum_i 2 Re(omega_i H~ Z_i) = H~ sum_i Y_i, so the product with H~
// is done once for all poles by k_combine2.
//
// M is block upper Hessenberg with p x p blocks (H_m is band Hessenberg with p sub-diagonals),
// so Gaussian elimination with partial pivoting is blocked by block columns J:
//   panel   (2p x p block [M_JJ; M_J+1,J], column by column, all threads): pivot searched
//           among the panel rows only (the band) on FP32 magnitudes, full rows swapped, one
//           reciprocal per pivot, multipliers stored in place, the panel's own columns updated;
//   update  U_J,c = L_JJ^{-1} M_J,c (one column per thread), then M_J+1,c -= L_J+1,J U_J,c
//           (one (row, column) pair per thread) for every later column c of M and of X;
// then the inverses of the diagonal blocks U_JJ (one block column per thread, all blocks at
// once) and the blocked back substitution X_J = U_JJ^{-1} X_J, X_0..J-1 -= U_0..J-1,J X_J as
// parallel products.  FP64 throughout; the FP64 pipe of one SM is the bound, so the layout
// keeps every lane of every warp busy wherever the work allows.
__global__ void __launch_bounds__(kPoleThreads) k_poles(const double* __restrict__ H, int ldH, int mp, int p,
                                                        const double* __restrict__ tau_re,
                                                        const double* __restrict__ tau_im,
                                                        const double* __restrict__ om_re,
                                                        const double* __restrict__ om_im,
                                                        double* __restrict__ S, double* __restrict__ work,
                                                        double* __restrict__ Y_slots, double* res,
                                                        int* flags, int use_smem, int h_in_smem, int alg,
                                                        double* __restrict__ Zout, int kk) {
    extern __shared__ double sm[];
    __shared__ cplx rdiag[kMaxMP];
    __shared__ double red[kPoleThreads];
    __shared__ int piv_s;
    const int i = blockIdx.x, tid = threadIdx.x, nt = blockDim.x;
    const int lane = tid & 31, warp = tid >> 5;
    const cplx tau{tau_re[i], tau_im[i]};
    const cplx om{om_re[i], om_im[i]};
    const size_t per = (size_t)mp * mp + 2 * (size_t)mp * p;
    cplx* M = use_smem ? reinterpret_cast<cplx*>(sm) : reinterpret_cast<cplx*>(work) + (size_t)i * per;
    cplx* X = M + (size_t)mp * mp;
    cplx* Ui = X + (size_t)mp * p;          // Ui[J p + a][b] = (U_JJ^{-1})[a][b]
    cplx* Si = reinterpret_cast<cplx*>(S) + (size_t)i * p * p;
    const int rows = mp + p;
    // H~ (rows x mp, column-major, ld = rows) in shared memory after M, X and Ui when it fits
    double* Hs = reinterpret_cast<double*>(sm) + (use_smem ? 2 * per : 0);
    const double* Hr = h_in_smem ? Hs : H;
    const int ldr = h_in_smem ? rows : ldH;
    if (h_in_smem)
        for (int c = 0; c < mp; ++c)
            for (int r = tid; r < rows; r += nt) Hs[(int64_t)c * rows + r] = H[(int64_t)c * ldH + r];
    __syncthreads();
    // Algorithm 2: M = I - tau H_m (eq. (3236)); Algorithm 1: M = H_m - tau I (eq. (3.3)).
    // X = E_1 S_i.
    for (int r = 0; r < mp; ++r)
        for (int c = tid; c < mp; c += nt) {
            const double h = Hr[(int64_t)c * ldr + r];
            const double d = (r == c ? 1.0 : 0.0);
            M[(size_t)r * mp + c] = (alg == 2) ? cplx{d - tau.re * h, -tau.im * h} : cplx{h - d * tau.re, -d * tau.im};
        }
    // after a deflated restart the residual coordinates sit at rows kk .. kk+p-1
    for (int e = tid; e < mp * p; e += nt) {
        const int r = e / p, c = e % p;
        X[e] = (r >= kk && r < kk + p) ? Si[(r - kk) * p + c] : cplx{0.0, 0.0};
    }
    __syncthreads();
    const int nbc = mp / p;
    for (int J = 0; J < nbc; ++J) {
        const int r0 = J * p;
        // panel rows r0 .. rend-1: the band (one block below the diagonal block); the kk
        // deflated columns of a deflated restart reach down to the block row of the old
        // V_{m+1} (rows kk .. kk+p-1: H_{m+1,m} E_m^T P_k)
        const int rend = min(mp, max(r0 + 2 * p, r0 < kk ? kk + p : 0));
        for (int jj = 0; jj < p; ++jj) {
            const int c = r0 + jj;
            if (warp == 0) {
                // pivot: arg-max of |M[r][c]|^2 in FP32 over the panel rows r >= c
                float best = -1.f;
                int piv = c;
                for (int r = c + lane; r < rend; r += 32) {
                    const cplx v = M[(size_t)r * mp + c];
                    const float fr = (float)v.re, fi = (float)v.im;
                    const float m = fmaf(fr, fr, fi * fi);
                    if (m > best) { best = m; piv = r; }
                }
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) {
                    const float ob = __shfl_xor_sync(0xffffffffu, best, o);
                    const int op = __shfl_xor_sync(0xffffffffu, piv, o);
                    if (ob > best || (ob == best && op < piv)) { best = ob; piv = op; }
                }
                if (lane == 0) piv_s = piv;
            }
            __syncthreads();
            const int piv = piv_s;
            if (piv != c) {   // swap the full rows (M from column r0 on, and X)
                for (int k = r0 + tid; k < mp; k += nt) {
                    const cplx a = M[(size_t)c * mp + k];
                    M[(size_t)c * mp + k] = M[(size_t)piv * mp + k];
                    M[(size_t)piv * mp + k] = a;
                }
                for (int k = tid; k < p; k += nt) {
                    const cplx a = X[(size_t)c * p + k];
                    X[(size_t)c * p + k] = X[(size_t)piv * p + k];
                    X[(size_t)piv * p + k] = a;
                }
                __syncthreads();
            }
            if (tid == 0) {
                const cplx d = M[(size_t)c * mp + c];
                const double n2 = d.re * d.re + d.im * d.im;
                if (!(n2 > 0.0)) atomicOr(&flags[0], 2);
                const double x = 1.0 / n2;
                rdiag[c] = cplx{d.re * x, -d.im * x};
            }
            __syncthreads();
            const cplx inv = rdiag[c];
            const int nr = rend - c - 1, wc = r0 + p - c - 1;
            for (int r = c + 1 + tid; r < rend; r += nt) M[(size_t)r * mp + c] = cmul(M[(size_t)r * mp + c], inv);
            __syncthreads();
            for (int e = tid; e < nr * wc; e += nt) {
                const int r = c + 1 + e / wc, k = c + 1 + e % wc;
                cmsub(M[(size_t)r * mp + k], M[(size_t)r * mp + c], M[(size_t)c * mp + k]);
            }
            __syncthreads();
        }
        // trailing update: columns of M right of the panel, then the columns of X
        const int ncm = mp - r0 - p, ncol = ncm + p;
        for (int q = tid; q < ncol; q += nt) {      // U_J,c = L_JJ^{-1} M_J,c (unit lower)
            cplx* col;
            size_t ld;
            if (q < ncm) { col = M + r0 + p + q; ld = mp; }
            else { col = X + (q - ncm); ld = p; }
            for (int a = 1; a < p; ++a) {
                cplx s = col[(size_t)(r0 + a) * ld];
                for (int k = 0; k < a; ++k) cmsub(s, M[(size_t)(r0 + a) * mp + r0 + k], col[(size_t)(r0 + k) * ld]);
                col[(size_t)(r0 + a) * ld] = s;
            }
        }
        __syncthreads();
        const int nbelow = rend - r0 - p;              // rows below the diagonal block
        if (nbelow > 0)
            for (int e = tid; e < nbelow * ncol; e += nt) {   // M_below,c -= L_below,J U_J,c
                const int a = e / ncol, q = e % ncol;
                cplx* col;
                size_t ld;
                if (q < ncm) { col = M + r0 + p + q; ld = mp; }
                else { col = X + (q - ncm); ld = p; }
                const int r = r0 + p + a;
                cplx s = col[(size_t)r * ld];
                for (int k = 0; k < p; ++k) cmsub(s, M[(size_t)r * mp + r0 + k], col[(size_t)(r0 + k) * ld]);
                col[(size_t)r * ld] = s;
            }
        __syncthreads();
    }
    // inverses of the diagonal blocks U_JJ (upper triangular), one block column per thread
    for (int e = tid; e < nbc * p; e += nt) {
        const int J = e / p, b = e % p, r0 = J * p;
        for (int a = p - 1; a >= 0; --a) {
            cplx s{a == b ? 1.0 : 0.0, 0.0};
            for (int k = a + 1; k <= b; ++k) cmsub(s, M[(size_t)(r0 + a) * mp + r0 + k], Ui[(size_t)(r0 + k) * p + b]);
            Ui[(size_t)(r0 + a) * p + b] = (a > b) ? cplx{0.0, 0.0} : cmul(s, rdiag[r0 + a]);
        }
    }
    __syncthreads();
    // blocked back substitution
    for (int J = nbc - 1; J >= 0; --J) {
        const int r0 = J * p;
        // X_J = U_JJ^{-1} X_J: outputs (a, c); the old X_J is read before any is written
        constexpr int kXo = (kMaxP * kMaxP + kPoleThreads - 1) / kPoleThreads;
        cplx xo[kXo];
        int cnt = 0;
        for (int e = tid; e < p * p; e += nt, ++cnt) {
            const int a = e / p, c = e % p;
            cplx s{0.0, 0.0};
            for (int k = a; k < p; ++k) {
                const cplx u = Ui[(size_t)(r0 + a) * p + k], x = X[(size_t)(r0 + k) * p + c];
                s.re = fma(u.re, x.re, fma(-u.im, x.im, s.re));
                s.im = fma(u.re, x.im, fma(u.im, x.re, s.im));
            }
            xo[cnt] = s;
        }
        __syncthreads();
        cnt = 0;
        for (int e = tid; e < p * p; e += nt, ++cnt) X[(size_t)(r0 + e / p) * p + e % p] = xo[cnt];
        __syncthreads();
        for (int e = tid; e < r0 * p; e += nt) {   // X_0..J-1 -= U_0..J-1,J X_J
            const int r = e / p, c = e % p;
            cplx s = X[(size_t)r * p + c];
            for (int k = 0; k < p; ++k) cmsub(s, M[(size_t)r * mp + r0 + k], X[(size_t)(r0 + k) * p + c]);
            X[(size_t)r * p + c] = s;
        }
        __syncthreads();
    }
    // S_i and its Frobenius norm.  Algorithm 2: tau H_{m+1,m} E_m^T Z_i (eq. (49));
    // Algorithm 1: -H_{m+1,m} E_m^T Z_i (eq. (35)).
    double ss = 0.0;
    for (int e = tid; e < p * p; e += nt) {
        const int a = e / p, c = e % p;
        cplx s{0.0, 0.0};
        for (int b = 0; b < p; ++b) {
            const double h = Hr[(int64_t)(mp - p + b) * ldr + mp + a];
            const cplx x = X[(size_t)(mp - p + b) * p + c];
            s.re += h * x.re;
            s.im += h * x.im;
        }
        const cplx snew = (alg == 2) ? cmul(tau, s) : cplx{-s.re, -s.im};
        Si[e] = snew;
        ss += cabs2(snew);
    }
    red[tid] = ss;
    __syncthreads();
    for (int st = nt / 2; st > 0; st >>= 1) {
        if (tid < st) red[tid] += red[tid + st];
        __syncthreads();
    }
    if (tid == 0) {
        res[i] = sqrt(red[0]);
        if (!isfinite(red[0])) atomicOr(&flags[0], 4);
    }
    if (Zout) {   // certify mode: Z_i itself (complex, row-major [r][c])
        cplx* Zi = reinterpret_cast<cplx*>(Zout) + (size_t)i * mp * p;
        for (int e = tid; e < mp * p; e += nt) Zi[e] = X[e];
    }
    // Y_i = 2 Re(omega_i Z_i), stored r fastest (Y[c * mp + r])
    double* Yi = Y_slots + (size_t)i * mp * p;
    for (int e = tid; e < mp * p; e += nt) {
        const int r = e % mp, c = e / mp;
        const cplx x = X[(size_t)r * p + c];
        Yi[e] = 2.0 * (om.re * x.re - om.im * x.im);
    }
}

// ---------------------------------------------------------------- one cluster per pole
//
// The same blocked elimination by a cluster of kPc CTAs per pole (plans without a deflated block).
// The FP64 pipe of one SM (2 FMAs per clock) is what bounds the one-CTA kernel below, so the trailing
// columns and the right-hand sides are dealt out over the cluster's SMs; M and X live in global memory
// (L2), each column is only ever touched by its owner, and the p-wide panel is factored in shared
// memory by CTA 0 of the cluster and handed on through global memory between cluster barriers:
//
//   panel    CTA 0: rows r0 .. rend-1 of block column J, pivoted, two barriers per column; the unit
//            lower block is inverted by doubling (log2 p steps instead of p^2 / 2 dependent ones)
//   update   every CTA, its columns 32 at a time in shared memory: swaps, U = L^-1 top, below -= L U
//   back     X's columns are independent: each CTA substitutes its own
//
// Values that another CTA wrote are read past L1 (__ldcg).  Measured per launch (7 poles), one CTA per
// pole -> cluster: m = 10, p = 8 288 -> 256 us, p = 12 580 -> 412 us, p = 16 1008 -> 578 us, p = 32
// 5541 -> 2270 us; m = 30, p = 8 1196 -> 780 us, p = 16 5887 -> 2192 us.  Each block column costs ~8 us
// of barriers and L2 round trips, so narrow blocks (p = 4, m = 10: 123 -> 162 us) stay on one CTA.
constexpr int kPc = 8;            // CTAs per cluster
constexpr int kPcT = 256;

// |v|^2 for the pivot search from the operands' leading bits (truncated to FP32 with integer
// operations: a conversion occupies the FP64 pipe like an FMA)
__device__ __forceinline__ float lead32(double x) {
    const uint32_t hi = (uint32_t)__double2hiint(x), lo = (uint32_t)__double2loint(x);
    const int e = (int)((hi >> 20) & 0x7FFu) - 896;
    const uint32_t f = (e <= 0 ? 0u : e >= 255 ? 0x7F800000u : ((uint32_t)e << 23) | ((hi & 0xFFFFFu) << 3) | (lo >> 29));
    return __uint_as_float(f);
}
__device__ __forceinline__ cplx ldc(const cplx* p) {
    const double2 v = __ldcg(reinterpret_cast<const double2*>(p));
    return cplx{v.x, v.y};
}
__device__ __forceinline__ void cluster_sync() {
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}

// complex numbers of the workspace of one pole: M, X, U_JJ^{-1}, the panel in flight, |S|^2 partials
__host__ __device__ constexpr size_t poles_work(int mp, int p) {
    return (size_t)mp * mp + 2 * (size_t)mp * p + 3 * (size_t)p * p + (size_t)p + kPc;
}
constexpr size_t poles_cluster_smem(int mp, int p) {
    return sizeof(cplx) * std::max(3 * (size_t)p * p + 2 * (size_t)p * 32, (size_t)mp * ((p + kPc - 1) / kPc));
}

__global__ void __launch_bounds__(kPcT) __cluster_dims__(kPc, 1, 1)
k_poles_cluster(const double* __restrict__ H, int ldH, int mp, int p, const double* __restrict__ tau_re,
                const double* __restrict__ tau_im, const double* __restrict__ om_re, const double* __restrict__ om_im,
                double* __restrict__ S, double* work, double* __restrict__ Y_slots, double* res, int* flags, int alg,
                double* __restrict__ Zout) {
    extern __shared__ __align__(16) unsigned char smp[];
    cplx* P = reinterpret_cast<cplx*>(smp);              // 2p x p panel
    cplx* Li = P + 2 * (size_t)p * p;                    // p x p inverse of its unit lower block
    cplx* Tl = Li + (size_t)p * p;                       // 2p x 32 columns being updated (CTA 0: scratch)
    __shared__ int piv_s[kMaxP];
    __shared__ cplx inv_s;
    __shared__ double red[kPcT];
    const int rank = blockIdx.x % kPc, i = blockIdx.x / kPc, tid = threadIdx.x, lane = tid & 31;
    const cplx tau{tau_re[i], tau_im[i]}, om{om_re[i], om_im[i]};
    cplx* M = reinterpret_cast<cplx*>(work) + (size_t)i * poles_work(mp, p);
    cplx* X = M + (size_t)mp * mp;
    cplx* Ui = X + (size_t)mp * p;
    cplx* pan = Ui + (size_t)mp * p;                     // 2p x p panel, p x p inverse
    cplx* rdg = pan + 3 * (size_t)p * p;                 // pivots as integers (re)
    double* parts = reinterpret_cast<double*>(rdg + p);
    cplx* Si = reinterpret_cast<cplx*>(S) + (size_t)i * p * p;
    const int gt = rank * kPcT + tid, gn = kPc * kPcT;
    // M = I - tau H_m (eq. (3236)) or H_m - tau I (eq. (3.3)); X = E_1 S_i
    for (int e = gt; e < mp * mp; e += gn) {
        const int c = e / mp, r = e - c * mp;            // H column-major: r fastest
        const double h = H[(int64_t)c * ldH + r], d = r == c ? 1.0 : 0.0;
        M[(size_t)r * mp + c] = alg == 2 ? cplx{d - tau.re * h, -tau.im * h} : cplx{h - d * tau.re, -d * tau.im};
    }
    for (int e = gt; e < mp * p; e += gn) X[e] = e / p < p ? Si[e] : cplx{0.0, 0.0};
    cluster_sync();
    const int nbc = mp / p;
    // U_JJ^{-1} from the panel in shared memory, by doubling as for the unit lower block: run by one of
    // the CTAs that wait while CTA 0 factors the next panel
    auto invert_upper = [&](int J) {
        for (int e = tid; e < p * p; e += kPcT) {
            const int a = e / p, b = e - a * p;
            cplx v{0.0, 0.0};
            if (a == b) {
                const cplx d = P[e];
                const double x = 1.0 / (d.re * d.re + d.im * d.im);
                v = cplx{d.re * x, -d.im * x};
            }
            Li[e] = v;
        }
        __syncthreads();
        for (int s = 1; s < p; s *= 2) {
            for (int ph = 0; ph < 2; ++ph) {
                for (int e = tid; e < p * s; e += kPcT) {          // rows a of the upper block, columns c of the lower
                    const int b = e / (2 * s * s) * 2 * s, o = e % (2 * s * s), a = b + o / s, c = b + s + o % s;
                    if (o < s * s && c < p) {
                        cplx t{0.0, 0.0};
                        if (ph == 0) {                             // T = -B C^-1
                            for (int k = b + s; k <= c; ++k) cmsub(t, P[a * p + k], Li[k * p + c]);
                            Tl[a * p + c] = t;
                        } else {                                   // A^-1 T
                            for (int k = a; k < b + s; ++k) {
                                const cplx l = Li[a * p + k], x = Tl[k * p + c];
                                t.re = fma(l.re, x.re, fma(-l.im, x.im, t.re));
                                t.im = fma(l.re, x.im, fma(l.im, x.re, t.im));
                            }
                            Li[a * p + c] = t;
                        }
                    }
                }
                __syncthreads();
            }
        }
        for (int e = tid; e < p * p; e += kPcT) Ui[(size_t)J * p * p + e] = Li[e];
        __syncthreads();
    };
    for (int J = 0; J < nbc; ++J) {
        const int r0 = J * p, rows = min(2 * p, mp - r0);
        if (J > 0 && rank == 1 + (J - 1) % (kPc - 1)) invert_upper(J - 1);
        if (rank == 0) {
            for (int e = tid; e < rows * p; e += kPcT) P[e] = ldc(M + (size_t)(r0 + e / p) * mp + r0 + e % p);
            __syncthreads();
            constexpr int kEl = (2 * kMaxP * kMaxP + kPcT - 1) / kPcT;
            int er[kEl], ek[kEl];                        // this thread's panel entries
#pragma unroll
            for (int q = 0; q < kEl; ++q) {
                const int e = tid + q * kPcT;
                er[q] = e < rows * p ? e / p : -1;
                ek[q] = e - max(er[q], 0) * p;
            }
            for (int jj = 0; jj < p; ++jj) {
                // pivot: arg-max of the magnitudes in FP32, by every warp for itself
                float best = -1.f;
                int piv = jj;
                for (int r = jj + lane; r < rows; r += 32) {
                    const cplx v = P[r * p + jj];
                    const float fr = lead32(v.re), fi = lead32(v.im), m = fmaf(fr, fr, fi * fi);
                    if (m > best) {
                        best = m;
                        piv = r;
                    }
                }
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) {
                    const float ob = __shfl_xor_sync(0xffffffffu, best, o);
                    const int op = __shfl_xor_sync(0xffffffffu, piv, o);
                    if (ob > best || (ob == best && op < piv)) {
                        best = ob;
                        piv = op;
                    }
                }
                if (tid == 0) {
                    const cplx d = P[piv * p + jj];
                    const double n2 = d.re * d.re + d.im * d.im;
                    if (!(n2 > 0.0)) atomicOr(&flags[0], 2);
                    const double x = 1.0 / n2;
                    inv_s = cplx{d.re * x, -d.im * x};
                    piv_s[jj] = piv;
                }
                __syncthreads();
                const cplx inv = inv_s;
                // rows jj .. with the pivot row moved up, the others eliminated; all reads, then all
                // writes.  Columns left of jj (stored multipliers) only swap.
                cplx nv[kEl];
#pragma unroll
                for (int q = 0; q < kEl; ++q) {
                    if (q * kPcT >= rows * p) break;
                    const int r = er[q], k = ek[q];
                    if (r >= jj) {
                        const int src = r == jj ? piv : r == piv ? jj : r;
                        cplx v = P[src * p + k];
                        if (r > jj && k >= jj) {
                            const cplx mlt = cmul(P[src * p + jj], inv);
                            if (k == jj) v = mlt;
                            else cmsub(v, mlt, P[piv * p + k]);
                        }
                        nv[q] = v;
                    }
                }
                __syncthreads();
#pragma unroll
                for (int q = 0; q < kEl; ++q) {
                    if (q * kPcT >= rows * p) break;
                    if (er[q] >= jj) P[tid + q * kPcT] = nv[q];
                }
                __syncthreads();
            }
            // inverse of the unit lower block by doubling: the off-diagonal blocks of size s from the
            // inverses of the two diagonal blocks of size s
            for (int e = tid; e < p * p; e += kPcT) Li[e] = cplx{e / p == e % p ? 1.0 : 0.0, 0.0};
            __syncthreads();
            for (int s = 1; s < p; s *= 2) {
                for (int e = tid; e < p * s; e += kPcT) {          // T = B A^-1, rows of the lower blocks
                    const int b = e / (2 * s * s) * 2 * s, o = e % (2 * s * s), a = b + s + o / s, c = b + o % s;
                    if (o < s * s && a < p) {
                        cplx t{0.0, 0.0};
                        for (int k = c; k < b + s; ++k) cmsub(t, P[a * p + k], Li[k * p + c]);
                        Tl[a * p + c] = t;                         // -B A^-1
                    }
                }
                __syncthreads();
                for (int e = tid; e < p * s; e += kPcT) {
                    const int b = e / (2 * s * s) * 2 * s, o = e % (2 * s * s), a = b + s + o / s, c = b + o % s;
                    if (o < s * s && a < p) {
                        cplx t = Tl[a * p + c];                    // C^-1 (-B A^-1), C^-1 unit lower
                        for (int k = b + s; k < a; ++k) {
                            const cplx l = Li[a * p + k], x = Tl[k * p + c];
                            t.re = fma(l.re, x.re, fma(-l.im, x.im, t.re));
                            t.im = fma(l.re, x.im, fma(l.im, x.re, t.im));
                        }
                        Li[a * p + c] = t;
                    }
                }
                __syncthreads();
            }
            for (int e = tid; e < rows * p; e += kPcT) {
                pan[e] = P[e];
                M[(size_t)(r0 + e / p) * mp + r0 + e % p] = P[e];
            }
            for (int e = tid; e < p * p; e += kPcT) pan[2 * (size_t)p * p + e] = Li[e];
            if (tid < p) rdg[tid] = cplx{(double)piv_s[tid], 0.0};
        }
        cluster_sync();
        if (rank != 0) {
            for (int e = tid; e < rows * p; e += kPcT) P[e] = ldc(pan + e);
            for (int e = tid; e < p * p; e += kPcT) Li[e] = ldc(pan + 2 * (size_t)p * p + e);
            if (tid < p) piv_s[tid] = (int)ldc(rdg + tid).re;
        }
        // this CTA's columns: every kPc-th of M's trailing ones and of X's, 32 at a time
        const int ncm = mp - r0 - p, ncol = ncm + p, mine = (ncol - rank + kPc - 1) / kPc;
        for (int q0 = 0; q0 < mine; q0 += 32) {
            const int nc = min(32, mine - q0);
            auto at = [&](int r, int q) -> cplx* {       // row r0 + r of this chunk's column q
                const int c = rank + (q0 + q) * kPc;
                return c < ncm ? M + (size_t)(r0 + r) * mp + r0 + p + c : X + (size_t)(r0 + r) * p + (c - ncm);
            };
            __syncthreads();
            for (int e = tid; e < rows * nc; e += kPcT) Tl[(e / nc) * 32 + e % nc] = ldc(at(e / nc, e % nc));
            __syncthreads();
            if (tid < nc)
                for (int jj = 0; jj < p; ++jj) {
                    const int pv = piv_s[jj];
                    if (pv != jj) {
                        const cplx a = Tl[jj * 32 + tid];
                        Tl[jj * 32 + tid] = Tl[pv * 32 + tid];
                        Tl[pv * 32 + tid] = a;
                    }
                }
            __syncthreads();
            constexpr int kUo = (kMaxP * 32 + kPcT - 1) / kPcT;
            cplx u[kUo];
#pragma unroll
            for (int q = 0; q < kUo; ++q) {
                const int e = tid + q * kPcT, a = e / nc, c = e - a * nc;
                if (e < p * nc) {
                    cplx s = Tl[a * 32 + c];
                    for (int k = 0; k < a; ++k) {
                        const cplx l = Li[a * p + k], x = Tl[k * 32 + c];
                        s.re = fma(l.re, x.re, fma(-l.im, x.im, s.re));
                        s.im = fma(l.re, x.im, fma(l.im, x.re, s.im));
                    }
                    u[q] = s;
                }
            }
            __syncthreads();
#pragma unroll
            for (int q = 0; q < kUo; ++q) {
                const int e = tid + q * kPcT, a = e / nc, c = e - a * nc;
                if (e < p * nc) {
                    Tl[a * 32 + c] = u[q];
                    *at(a, c) = u[q];
                }
            }
            __syncthreads();
            for (int e = tid; e < (rows - p) * nc; e += kPcT) {
                const int a = e / nc, c = e - a * nc;
                cplx s = Tl[(p + a) * 32 + c];
                for (int k = 0; k < p; ++k) cmsub(s, P[(p + a) * p + k], Tl[k * 32 + c]);
                *at(p + a, c) = s;
            }
        }
        cluster_sync();
    }
    if (rank == 1 + (nbc - 1) % (kPc - 1)) invert_upper(nbc - 1);
    cluster_sync();
    // blocked back substitution of this CTA's columns of X (c = rank + kPc q), held in shared memory;
    // U's entries are loaded eight at a time
    const int nx = rank < p ? (p - rank + kPc - 1) / kPc : 0;
    cplx* Xl = P;                                        // mp x nx (P, Li and Tl are free now)
    for (int e = tid; e < mp * nx; e += kPcT) Xl[e] = ldc(X + (size_t)(e / nx) * p + rank + (e % nx) * kPc);
    __syncthreads();
    auto dot = [&](cplx s, const cplx* m, int k0, int k1, const cplx* x) {   // s - sum_k m[k] x[k nx]
        for (int k = k0; k < k1; k += 8) {
            cplx v[8];
#pragma unroll
            for (int u = 0; u < 8; ++u)
                if (k + u < k1) v[u] = ldc(m + k + u);
#pragma unroll
            for (int u = 0; u < 8; ++u)
                if (k + u < k1) cmsub(s, v[u], x[(size_t)(k + u) * nx]);
        }
        return s;
    };
    for (int J = nbc - 1; J >= 0; --J) {
        const int r0 = J * p;
        constexpr int kXo = (kMaxP * ((kMaxP + kPc - 1) / kPc) + kPcT - 1) / kPcT;
        cplx xn[kXo];
#pragma unroll
        for (int q = 0; q < kXo; ++q) {
            const int e = tid + q * kPcT;
            if (e < p * nx) xn[q] = dot(cplx{0.0, 0.0}, Ui + ((size_t)J * p + e / nx) * p, e / nx, p, Xl + (size_t)r0 * nx + e % nx);
        }
        __syncthreads();
#pragma unroll
        for (int q = 0; q < kXo; ++q) {
            const int e = tid + q * kPcT;
            if (e < p * nx) Xl[(size_t)r0 * nx + e] = cplx{-xn[q].re, -xn[q].im};
        }
        __syncthreads();
        for (int e = tid; e < r0 * nx; e += kPcT)
            Xl[e] = dot(Xl[e], M + (size_t)(e / nx) * mp + r0, 0, p, Xl + (size_t)r0 * nx + e % nx);
        __syncthreads();
    }
    // S_i, its norm, Y_i = 2 Re(omega_i Z_i) for this CTA's columns
    double ss = 0.0;
    for (int e = tid; e < p * nx; e += kPcT) {
        const int a = e / nx, c = rank + (e % nx) * kPc;
        cplx s{0.0, 0.0};
        for (int b = 0; b < p; ++b) {
            const double h = H[(int64_t)(mp - p + b) * ldH + mp + a];
            const cplx x = Xl[(size_t)(mp - p + b) * nx + e % nx];
            s.re += h * x.re;
            s.im += h * x.im;
        }
        const cplx snew = (alg == 2) ? cmul(tau, s) : cplx{-s.re, -s.im};
        Si[a * p + c] = snew;
        ss += cabs2(snew);
    }
    red[tid] = ss;
    __syncthreads();
    for (int st = kPcT / 2; st > 0; st >>= 1) {
        if (tid < st) red[tid] += red[tid + st];
        __syncthreads();
    }
    if (tid == 0) parts[rank] = red[0];
    double* Yi = Y_slots + (size_t)i * mp * p;
    cplx* Zi = Zout ? reinterpret_cast<cplx*>(Zout) + (size_t)i * mp * p : nullptr;
    for (int e = tid; e < mp * nx; e += kPcT) {
        const int r = e % mp, c = rank + (e / mp) * kPc;
        const cplx x = Xl[(size_t)r * nx + e / mp];
        Yi[(size_t)c * mp + r] = 2.0 * (om.re * x.re - om.im * x.im);
        if (Zi) Zi[(size_t)r * p + c] = x;
    }
    cluster_sync();
    if (rank == 0 && tid == 0) {
        double s = 0.0;
        for (int k = 0; k < kPc; ++k) s += __ldcg(parts + k);
        res[i] = sqrt(s);
        if (!isfinite(s)) atomicOr(&flags[0], 4);
    }
}

// Wc = H~ sum_i Y_i (Algorithm 2) or [sum_i Y_i; 0] (Algorithm 1), (mp+p) x p, row-major
// [r][c] as k_update_z reads it.  One thread per output, r fastest (coalesced H~ columns).
__global__ void k_combine2(const double* __restrict__ H, int ldH, int mp, int p, int npoles,
                           const double* __restrict__ Y_slots, double* __restrict__ Wc, int alg, int kk) {
    extern __shared__ double Ys[];          // mp x p, summed over poles (fixed order)
    const int rows = mp + p;
    for (int e = threadIdx.x; e < mp * p; e += blockDim.x) {
        double s = 0.0;
        for (int i = 0; i < npoles; ++i) s += Y_slots[(size_t)i * mp * p + e];
        Ys[e] = s;
    }
    __syncthreads();
    for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < rows * p; e += gridDim.x * blockDim.x) {
        const int r = e % rows, c = e / rows;
        double s = 0.0;
        if (alg == 2) {
            // band rows start p columns left of the diagonal; the rows of a deflated restart's
            // leading block (r < kk + p) are dense from column 0
            for (int k = r < kk + p ? 0 : r - p; k < mp; ++k) s = fma(H[(int64_t)k * ldH + r], Ys[c * mp + k], s);
        } else if (r < mp) {
            s = Ys[c * mp + r];
        }
        Wc[r * p + c] = s;
    }
}

// Certify mode: C[a][i 2p + c] = Re(F_i)[a][c], C[a][i 2p + p + c] = Im(F_i)[a][c] with
// F_i = H~_m Z_i (Algorithm 2: X_i - X_i^0 = V_{m+1} H~_m Z_i) or F_i = [Z_i; 0] (Algorithm 1),
// so X += V_{m+1} C updates every pole's real and imaginary parts in one tall-skinny product.
__global__ void k_certify_coeffs(const double* __restrict__ H, int ldH, int mp, int p, int npoles,
                                 const double* __restrict__ Zs, double* __restrict__ C, int alg, int kk) {
    const int rows = mp + p, w = 2 * npoles * p;
    const cplx* Z = reinterpret_cast<const cplx*>(Zs);
    for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < rows * npoles * p; e += gridDim.x * blockDim.x) {
        const int a = e % rows, ic = e / rows, i = ic / p, c = ic % p;
        const cplx* Zi = Z + (size_t)i * mp * p;
        cplx s{0.0, 0.0};
        if (alg == 2) {
            for (int k = a < kk + p ? 0 : a - p; k < mp; ++k) {   // as in k_combine2
                const double h = H[(int64_t)k * ldH + a];
                s.re = fma(h, Zi[(size_t)k * p + c].re, s.re);
                s.im = fma(h, Zi[(size_t)k * p + c].im, s.im);
            }
        } else if (a < mp) {
            s = Zi[(size_t)a * p + c];
        }
        C[(size_t)a * w + 2 * i * p + c] = s.re;
        C[(size_t)a * w + 2 * i * p + p + c] = s.im;
    }
}

}  // namespace

cudaError_t launch_certify_coeffs(const double* H, int ldH, int mp, int p, int npoles, const double* Zs,
                                  double* C, int alg, cudaStream_t s, int kk) {
    const int tot = (mp + p) * npoles * p;
    k_certify_coeffs<<<(tot + 255) / 256, 256, 0, s>>>(H, ldH, mp, p, npoles, Zs, C, alg, kk);
    return cudaGetLastError();
}

size_t poles_work_doubles(int mp, int p) {
    return 2 * std::max(poles_work(mp, p), (size_t)mp * mp + 2 * (size_t)mp * p);
}

size_t poles_smem_bytes(int mp, int p) {
    const size_t b = ((size_t)mp * mp + 2 * (size_t)mp * p) * sizeof(cplx);
    return b <= kSmemLimit ? b : 0;
}

static size_t poles_h_bytes(int mp, int p) { return (size_t)(mp + p) * mp * sizeof(double); }

cudaError_t launch_poles(const double* H, int ldH, int mp, int p, int npoles,
                         const double* tau_re, const double* tau_im, const double* om_re,
                         const double* om_im, double* S, double* work, double* Y_slots,
                         double* res, int* flags, int alg, cudaStream_t s, double* Zout, int kk) {
    // where the elimination outweighs the cluster's exchanges (p = 6: 189 against 221 us at mp = 60, 723
    // against 647 us at mp = 180; p = 8: 288 against 256 us at mp = 80)
    if (kk == 0 && p >= 6 && mp * p >= 600) {
        k_poles_cluster<<<npoles * kPc, kPcT, poles_cluster_smem(mp, p), s>>>(H, ldH, mp, p, tau_re, tau_im, om_re, om_im, S, work,
                                                                         Y_slots, res, flags, alg, Zout);
        return cudaGetLastError();
    }
    size_t shm = poles_smem_bytes(mp, p);
    int h_in = 0;
    if (shm > 0 && shm + poles_h_bytes(mp, p) <= kSmemLimit) {
        shm += poles_h_bytes(mp, p);
        h_in = 1;
    }
    k_poles<<<npoles, kPoleThreads, shm, s>>>(H, ldH, mp, p, tau_re, tau_im, om_re, om_im, S, work,
                                              Y_slots, res, flags, poles_smem_bytes(mp, p) > 0 ? 1 : 0,
                                              h_in, alg, Zout, kk);
    return cudaGetLastError();
}

cudaError_t launch_combine2(const double* H, int ldH, int mp, int p, int npoles,
                            const double* Y_slots, double* Wc, int alg, cudaStream_t s, int kk) {
    const int nout = (mp + p) * p;
    const int blocks = (nout + 255) / 256;
    k_combine2<<<blocks, 256, sizeof(double) * (size_t)mp * p, s>>>(H, ldH, mp, p, npoles, Y_slots, Wc, alg, kk);
    return cudaGetLastError();
}

cudaError_t poles_set_smem_limits() {
    // kSmemLimit (200 KB) of dynamic memory plus the kernel's few KB of static memory stays
    // below the 227 KB per-block opt-in maximum
    cudaError_t e = cudaFuncSetAttribute(k_poles, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmemLimit);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(k_poles_cluster, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)poles_cluster_smem(kMaxMP, kMaxP));
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(k_combine2, cudaFuncAttributeMaxDynamicSharedMemorySize, 140 * 1024);
    return e;
}

}  // namespace expm
