// rows_qr.cuh -- the mixed path's block step after the second projection, in two launches of one
// row width (included inside the width's namespace, after rows_chol.cuh):
//
//   k_reduce_factor   sums the second projection's and the Gram matrix's partials, adds h2 to H,
//                     and its last CTA factors G - h2^T h2 (float pairs, chol_df)
//   k_qr_apply        W <- (W - V h2) R^{-1} row by row into the next block, its FP32 copy and
//                     its column exponents
//
// The factorisation used to run in every CTA of the row pass (each waited ~10 us for its own copy
// of the serial p x p factor, so the pass was launched with few CTAs and left the memory idle);
// factored once, the row pass takes as many CTAs as fit.  Blocks that are too ill-conditioned for
// the single factor leave the done flag clear: k_qr_apply returns at once and the three-pass
// kernels that follow take over.

struct QrFac {
    float2 RT[RP * RP];               // [c][b]: R_bc as a float pair (b < c)
    float rch[RP], rcl[RP];           // 1 / R_cc
};

// x 2^k by an add to the exponent field; below the normal range it flushes to zero, above it is inf
__device__ __forceinline__ double scale_pow2(double x, int k) {
    const long long b = __double_as_longlong(x);
    const int e = (int)((b >> 52) & 0x7FF);
    long long r = b + ((long long)k << 52);
    if (e == 0 || e + k <= 0) r = b & (1LL << 63);
    if (e == 0x7FF) r = b;
    else if (e != 0 && e + k >= 0x7FF) r = (b & (1LL << 63)) | (0x7FFLL << 52);
    return __longlong_as_double(r);
}

constexpr int kRedOut = 4, kRedStripes = 64, kRedT = kRedOut * kRedStripes;

__device__ inline double red_stripe(const double* __restrict__ part, int nblk, int nout, int o, int s) {
    double a[4] = {0.0, 0.0, 0.0, 0.0};
    int b = s;
    for (; b + 3 * kRedStripes < nblk; b += 4 * kRedStripes)
#pragma unroll
        for (int k = 0; k < 4; ++k) a[k] += part[(int64_t)(b + k * kRedStripes) * nout + o];
    for (; b < nblk; b += kRedStripes) a[0] += part[(int64_t)b * nout + o];
    return (a[0] + a[1]) + (a[2] + a[3]);
}

// h[0 : cols p] = second projection, h[cols p :] = Gram matrix of W before the correction.
__global__ void __launch_bounds__(kRedT)
k_reduce_factor(const double* __restrict__ part, int nblk, const double* __restrict__ partG, int nblkG, int cols,
                int p, double* h, double* H, int ldH, int hrow, int hcol, double* R, double* Rtot, QrFac* fac,
                unsigned* ctr, int* flags, int allow) {
    constexpr int AC = 32;                        // rows of h2 staged at a time
    constexpr int PAD = RP * RP > kRedT ? RP * RP : kRedT;
    __shared__ double red[kRedStripes][kRedOut], red2[8][kRedOut];
    __shared__ float sh_[AC * RP], sl_[AC * RP];
    __shared__ float2 Gs[RP * RP], Us[RP * RP], Is[RP], comb[PAD];
    __shared__ float trd[RP];
    __shared__ float hn2[RP], combf[kRedT];
    __shared__ unsigned ticket;
    __shared__ int kexp_s, sgl_s;
    const int nh = cols * p, nout = nh + p * p, tid = threadIdx.x;
    {
        const int ol = tid % kRedOut, st = tid / kRedOut, o = blockIdx.x * kRedOut + ol;
        double v = 0.0;
        if (o < nh) v = red_stripe(part, nblk, nh, o, st);
        else if (o < nout) v = red_stripe(partG, nblkG, p * p, o - nh, st);
        red[st][ol] = v;
        __syncthreads();
        if (st < 8) {
            double g = 0.0;
#pragma unroll
            for (int k = 0; k < 8; ++k) g += red[st * 8 + k][ol];
            red2[st][ol] = g;
        }
        __syncthreads();
        if (st == 0 && o < nout) {
            const double s = ((red2[0][ol] + red2[1][ol]) + (red2[2][ol] + red2[3][ol])) +
                             ((red2[4][ol] + red2[5][ol]) + (red2[6][ol] + red2[7][ol]));
            h[o] = s;
            if (o < nh) H[(int64_t)(hcol + o % p) * ldH + o / p] += s;
            __threadfence();
        }
    }
    __syncthreads();
    if (tid == 0) ticket = atomicAdd(ctr, 1u);
    __syncthreads();
    if (ticket != gridDim.x - 1) return;
    __threadfence();
    if (tid == 0) *ctr = 0u;
    // ---- the last CTA.  Its chain is serial, so loads are issued together and the arithmetic
    // stays off the FP64 pipe where it can.
    // G is factored as G 2^-kexp (kexp even), kexp from the largest diagonal entry
    if (tid < 32) {
        int e = 0;
        if (tid < p) e = (__double2hiint(__ldcg(h + nh + tid * p + tid)) >> 20) & 0x7FF;
        e = __reduce_max_sync(0xffffffffu, e);
        if (tid == 0) kexp_s = (e - 1022) & ~1;
    }
    __syncthreads();
    const int kexp = kexp_s;
    // squared norms of the new entries of H above the block, in units of 2^kexp (the breakdown test: FP32)
    {
        const int stripes = min(8, kRedT / p), c = tid % p, st = tid / p;
        float v2 = 0.f;
        if (st < stripes)
#pragma unroll 4
            for (int a = st; a < hrow; a += stripes) {
                const float v = f32_rn_i(scale_pow2(__ldcg(H + (int64_t)(hcol + c) * ldH + a), -(kexp / 2)));
                v2 = fmaf(v, v, v2);
            }
        combf[tid] = v2;
    }
    const int ne = p * (p + 1) / 2, S = max(1, min(8, kRedT / ne));
    constexpr int KI = (RP * (RP + 1) / 2 + kRedT - 1) / kRedT + 1;
    int ii[KI], jj[KI];
    float ah[KI], al[KI];
#pragma unroll
    for (int k = 0; k < KI; ++k) {
        const int it = tid + k * kRedT;
        ii[k] = -1;
        jj[k] = 0;
        if (it < ne * S) {
            int i = 0, rem = it % ne;
            while (rem >= p - i) {
                rem -= p - i;
                ++i;
            }
            ii[k] = i;
            jj[k] = i + rem;
        }
    }
    // G - h2^T h2.  The correction is ~2^-40 of G unless the first pass cancelled almost all of W,
    // so its products are formed in FP32 first; only when a diagonal entry's correction passes
    // 2^-24 of it are they formed again in float pairs (G needs ~2^-48).
    for (int full = 0; full < 2; ++full) {
#pragma unroll
        for (int k = 0; k < KI; ++k) ah[k] = al[k] = 0.f;
        for (int a0 = 0; a0 < cols; a0 += AC) {
            const int na = min(AC, cols - a0);
            __syncthreads();
            for (int e = tid; e < na * p; e += kRedT) split_df_i(scale_pow2(__ldcg(h + (int64_t)a0 * p + e), -(kexp / 2)), sh_[e], sl_[e]);
            __syncthreads();
#pragma unroll
            for (int k = 0; k < KI; ++k)
                if (ii[k] >= 0) {
                    const int aa = (tid + k * kRedT) / ne;
                    if (full) {
                        for (int a = aa; a < na; a += S)
                            df_fma(ah[k], al[k], sh_[a * p + ii[k]], sl_[a * p + ii[k]], sh_[a * p + jj[k]], sl_[a * p + jj[k]]);
                    } else {
#pragma unroll 4
                        for (int a = aa; a < na; a += S) ah[k] = fmaf(sh_[a * p + ii[k]], sh_[a * p + jj[k]], ah[k]);
                    }
                }
        }
#pragma unroll
        for (int k = 0; k < KI; ++k)
            if (ii[k] >= 0) comb[tid + k * kRedT] = make_float2(ah[k], al[k]);
        __syncthreads();
        int big = 0;
        for (int e = tid; e < ne; e += kRedT) {
            float ch = 0.f, cl = 0.f;
            for (int k = 0; k < S; ++k) {
                df_add(ch, cl, comb[k * ne + e].x);
                cl += comb[k * ne + e].y;
            }
            int i = 0, rem = e;
            while (rem >= p - i) {
                rem -= p - i;
                ++i;
            }
            const int o = i * p + i + rem;
            float gh, gl;
            split_df_i(scale_pow2(__ldcg(h + nh + o), -kexp), gh, gl);
            if (rem == 0 && !full && ch > 0x1p-24f * gh) big = 1;
            df_add(gh, gl, -ch);
            gl -= cl;
            Gs[o] = make_float2(gh, gl);
        }
        if (!__syncthreads_or(big)) break;
    }
    if (tid < p) trd[tid] = Gs[tid * p + tid].x;
    if (tid < p) {
        const int stripes = min(8, kRedT / p);
        float s = 0.f;
        for (int k = 0; k < stripes; ++k) s += combf[k * p + tid];
        hn2[tid] = s;
    }
    // Cholesky factor by all threads, thread t holding entries t, t + kRedT, .. of the upper
    // triangle in registers: step j reads row j of the partly reduced matrix from shared memory,
    // every thread forms the pivot's root and its own two entries of row j of U and updates its
    // entries, and the owners of row j + 1 publish it.  One barrier per step and a few hundred
    // instructions of code: the same factor unrolled in one warp's registers was ~50 KB of
    // straight-line code run once, and fetching it took ~45 us at p = 16.
    __shared__ int okc_s;
    if (tid == 0) okc_s = 1;
    {
        constexpr int KE = (RP * (RP + 1) / 2 + kRedT - 1) / kRedT;
        int ei[KE], ek[KE];
        fp2 ge[KE];
        float dmax = 0.f;
        for (int c = 0; c < p; ++c) dmax = fmaxf(dmax, Gs[c * p + c].x);
#pragma unroll
        for (int q = 0; q < KE; ++q) {
            const int e = tid + q * kRedT;
            ei[q] = -1;
            ek[q] = 0;
            ge[q] = f2_make(0.f, 0.f);
            if (e < ne) {
                int i = 0, rem = e;
                while (rem >= p - i) {
                    rem -= p - i;
                    ++i;
                }
                ei[q] = i;
                ek[q] = i + rem;
                const float2 x = Gs[i * p + i + rem];
                ge[q] = f2_make(x.x, x.y);
            }
        }
        __syncthreads();
#pragma unroll 1
        for (int j = 0; j < p; ++j) {
            const float2 dd = Gs[j * p + j];
            fp2 d = f2_make(dd.x, dd.y);
            if (!(d.h > 0.f) || !isfinite(d.h) || d.h < 1e-5f * dmax) {
                if (tid == 0) okc_s = 0;
                d = f2_make(1.f, 0.f);
            }
            const fp2 rt = f2_sqrt(d), inv = f2_rcp(rt);
            if (tid == 0) Is[j] = make_float2(inv.h, inv.l);
#pragma unroll
            for (int q = 0; q < KE; ++q)
                if (ei[q] >= j) {
                    const float2 a = Gs[j * p + ei[q]], b = Gs[j * p + ek[q]];
                    const fp2 ub = f2_mul(f2_make(b.x, b.y), inv);
                    if (ei[q] == j) {
                        const fp2 u = ek[q] == j ? rt : ub;
                        Us[j * p + ek[q]] = make_float2(u.h, u.l);
                    } else {
                        const fp2 pr = f2_mul(f2_mul(f2_make(a.x, a.y), inv), ub);
                        ge[q] = f2_add(ge[q], f2_make(-pr.h, -pr.l));
                        if (ei[q] == j + 1) Gs[(j + 1) * p + ek[q]] = make_float2(ge[q].h, ge[q].l);
                    }
                }
            __syncthreads();
        }
    }
    if (tid < 32) {
        const bool ok = okc_s != 0;
        // the Gram matrix after the correction must keep most of the one before it, else its
        // relative accuracy is lost to cancellation; the scaled factor must fit in floats
        float tr = 0.f, tin = 0.f;
        if (tid < p) {
            tr = trd[tid];
            tin = f32_rn_i(scale_pow2(__ldcg(h + nh + tid * p + tid), -kexp));
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            tr += __shfl_xor_sync(0xffffffffu, tr, o);
            tin += __shfl_xor_sync(0xffffffffu, tin, o);
        }
        if (tid == 0) {
            const int sgl = allow && ok && tr >= 1e-4f * tin && kexp > -160 && kexp < 160;
            sgl_s = sgl;
            flags[3] = sgl;
            if (sgl) flags[2] = 0;
        }
    }
    __syncthreads();
    if (!sgl_s) return;
    const float sc = __int_as_float((127 + kexp / 2) << 23), isc = __int_as_float((127 - kexp / 2) << 23);
    int bad = 0;
    for (int e = tid; e < RP * RP; e += kRedT) {
        const int c = e / RP, r = e - c * RP;     // exactly the R that the substitution applies
        float2 x = make_float2(0.f, 0.f);
        if (c < p && r <= c) {
            x = Us[r * p + c];
            x.x *= sc;
            x.y *= sc;
        }
        fac->RT[e] = x;
        if (c < p && r < p) {
            const double rt = f64_of_f32_i(x.x) + f64_of_f32_i(x.y);
            R[r * p + c] = rt;
            Rtot[r * p + c] = rt;
            H[(int64_t)(hcol + c) * ldH + hrow + r] = rt;
            if (!isfinite(x.x)) bad = 1;
        }
    }
    if (tid < RP) {
        fac->rch[tid] = tid < p ? Is[tid].x * isc : 0.f;
        fac->rcl[tid] = tid < p ? Is[tid].y * isc : 0.f;
    }
    if (tid < p) {
        // breakdown: R_cc against the column's norm before orthogonalisation
        float n0 = hn2[tid];
        for (int a = 0; a <= tid; ++a) n0 = fmaf(Us[a * p + tid].x, Us[a * p + tid].x, n0);
        if (Us[tid * p + tid].x <= 1e-14f * sqrtf(n0)) atomicOr(&flags[1], 1);
    }
    if (bad) atomicOr(&flags[0], 1);
}

// W <- (W - V h2) R^{-1}.  A warp takes 32 rows.  V h2 (h2 is the O(eps_32) remainder of the first
// pass, so FP32 accuracy) runs on the tensor cores from the FP32 basis: lane group g loads rows
// 4g .. 4g + 3 of a column (one 16-byte load serves the two 16-row M tiles), both operands in
// three bf16 parts as in the projections; the result is turned through shared memory to one row
// per lane for the forward substitution with R in float pairs.
constexpr int kApplyPerSm = RP <= 8 ? 5 : RP <= 16 ? 4 : 3;
constexpr int kApNT = (RP + 7) / 8;
constexpr int kApS = 8 * kApNT + 1;               // row stride of the turned correction

__global__ void __launch_bounds__(128, kApplyPerSm)
k_qr_apply(const double* __restrict__ W, int64_t ldw, int p, int64_t n, const float* __restrict__ V32, int64_t ldv,
           int cols, const double* __restrict__ h2, const QrFac* __restrict__ fac, double* __restrict__ out,
           float* __restrict__ out32, int64_t ldo, int* __restrict__ colexp, const int* flags) {
    if (flags[3] == 0) return;
    constexpr int NT = kApNT;
    extern __shared__ __align__(16) unsigned char sma[];
    uint2* hb = reinterpret_cast<uint2*>(sma);     // [chunk][nt][split][lane]
    __shared__ QrFac f;
    __shared__ unsigned mxs[RP];
    __shared__ float turn[4][32 * kApS];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, g = lane >> 2, t = lane & 3;
    const int nk = (cols + 15) >> 4;
    const int64_t ntiles = (n + 31) >> 5, tstep = (int64_t)gridDim.x * 4;
    int64_t tile = (int64_t)blockIdx.x * 4 + warp;
    float4 v[4];
    auto load = [&](int64_t tl, int kc) {
#pragma unroll
        for (int q = 0; q < 4; ++q)
            v[q] = *reinterpret_cast<const float4*>(V32 + (int64_t)min(kc * 16 + 4 * t + q, cols - 1) * ldv + tl * 32 + 4 * g);
    };
    if (tile < ntiles) load(tile, 0);
    for (int e = tid; e < nk * NT * 32; e += 128) {
        const int ln = e & 31, j = (e >> 5) % NT, kc = (e >> 5) / NT, c = 8 * j + (ln >> 2), a = kc * 16 + 4 * (ln & 3);
        float x[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) x[q] = (c < p && a + q < cols) ? f32_rn_i(h2[(a + q) * p + c]) : 0.f;
        uint32_t s0[3], s1[3];
        split3(x[0], x[1], s0);
        split3(x[2], x[3], s1);
#pragma unroll
        for (int k = 0; k < 3; ++k) hb[((kc * NT + j) * 3 + k) * 32 + ln] = make_uint2(s0[k], s1[k]);
    }
    for (int e = tid; e < (int)(sizeof(QrFac) / sizeof(float)); e += 128)
        reinterpret_cast<float*>(&f)[e] = reinterpret_cast<const float*>(fac)[e];
    if (tid < RP) mxs[tid] = 0u;
    __syncthreads();
    unsigned mx[RP];
#pragma unroll
    for (int c = 0; c < RP; ++c) mx[c] = 0u;
    float* tw = turn[warp];
    for (; tile < ntiles; tile += tstep) {
        float cm[2][NT][4], cc[2][NT][4];
#pragma unroll
        for (int i = 0; i < 2; ++i)
#pragma unroll
            for (int j = 0; j < NT; ++j)
#pragma unroll
                for (int q = 0; q < 4; ++q) cm[i][j][q] = cc[i][j][q] = 0.f;
        for (int kc = 0; kc < nk; ++kc) {
            uint32_t a[2][3][4];                   // M tile i: MMA rows g, g + 8 are rows 4g + 2i, 4g + 2i + 1
            {
                uint32_t s[3];
#define EXPM_AF(I, R, X, Y) \
    split3(X, Y, s);        \
    a[I][0][R] = s[0];      \
    a[I][1][R] = s[1];      \
    a[I][2][R] = s[2]
                EXPM_AF(0, 0, v[0].x, v[1].x);
                EXPM_AF(0, 1, v[0].y, v[1].y);
                EXPM_AF(0, 2, v[2].x, v[3].x);
                EXPM_AF(0, 3, v[2].y, v[3].y);
                EXPM_AF(1, 0, v[0].z, v[1].z);
                EXPM_AF(1, 1, v[0].w, v[1].w);
                EXPM_AF(1, 2, v[2].z, v[3].z);
                EXPM_AF(1, 3, v[2].w, v[3].w);
#undef EXPM_AF
            }
            if (kc + 1 < nk) load(tile, kc + 1);
            else if (tile + tstep < ntiles) load(tile + tstep, 0);
            uint2 hq[NT][3];
#pragma unroll
            for (int j = 0; j < NT; ++j)
#pragma unroll
                for (int k = 0; k < 3; ++k) hq[j][k] = hb[((kc * NT + j) * 3 + k) * 32 + lane];
#pragma unroll
            for (int pr = 0; pr < 6; ++pr)
#pragma unroll
                for (int j = 0; j < NT; ++j)
#pragma unroll
                    for (int i = 0; i < 2; ++i)
                        mma_bf16(pr == 0 ? cm[i][j] : cc[i][j], a[i][kProdA[pr]], hq[j][kProdB[pr]].x, hq[j][kProdB[pr]].y);
        }
        __syncwarp();
#pragma unroll
        for (int i = 0; i < 2; ++i)
#pragma unroll
            for (int j = 0; j < NT; ++j)
#pragma unroll
                for (int q = 0; q < 4; ++q)
                    tw[(4 * g + 2 * i + (q >> 1)) * kApS + 8 * j + 2 * t + (q & 1)] = cm[i][j][q] + cc[i][j][q];
        __syncwarp();
        const int64_t r = tile * 32 + lane;
        const bool ok = r < n;
        constexpr int WB = RP <= 16 ? RP : 8;      // W's columns are loaded WB at a time
        double w[WB];
        float yh[RP], yl[RP];
#pragma unroll
        for (int c = 0; c < RP; ++c) {
            if (c % WB == 0) {
#pragma unroll
                for (int q = 0; q < WB; ++q) w[q] = W[(int64_t)min(c + q, p - 1) * ldw + r];
            }
            float sh, sl;
            split_df_i(w[c % WB], sh, sl);
            df_add(sh, sl, -tw[lane * kApS + c]);
#pragma unroll
            for (int b = 0; b < c; ++b) {          // columns past p have zero R: yh = yl = 0 there
                const float2 rr = f.RT[c * RP + b];
                const float pr = yh[b] * rr.x;
                float u = fmaf(yh[b], rr.x, -pr);
                u = fmaf(yh[b], rr.y, u);
                u = fmaf(yl[b], rr.x, u);
                df_add(sh, sl, -pr);
                sl -= u;
            }
            const float q1 = f.rch[c], q2 = f.rcl[c];
            const float pr = sh * q1;
            float u = fmaf(sh, q1, -pr);
            u = fmaf(sh, q2, u);
            u = fmaf(sl, q1, u);
            const float s2 = pr + u;
            yl[c] = u - (s2 - pr);
            yh[c] = s2;
            if (c < p && ok) {
                const double y = f64_of_f32_i(yh[c]) + f64_of_f32_i(yl[c]);
                out[(int64_t)c * ldo + r] = y;
                out32[(int64_t)c * ldo + r] = f32_rn_i(y);
                mx[c] = max(mx[c], (unsigned)__double2hiint(y) & 0x7FFFFFFFu);
            }
        }
    }
#pragma unroll
    for (int c = 0; c < RP; ++c) {
        const unsigned m = __reduce_max_sync(0xffffffffu, mx[c]);
        if (lane == 0 && c < p) atomicMax(&mxs[c], m);
    }
    __syncthreads();
    if (tid < p && mxs[tid]) atomicMax(&colexp[tid], (int)(mxs[tid] >> 20));
}

cudaError_t reduce_factor(const double* part, int nblk, const double* partG, int nblkG, int cols, int p, double* h,
                          double* H, int ldH, int hrow, int hcol, double* R, double* Rtot, float* fac, unsigned* ctr,
                          int* flags, int allow, cudaStream_t s) {
    const int nout = cols * p + p * p;
    k_reduce_factor<<<(nout + kRedOut - 1) / kRedOut, kRedT, 0, s>>>(part, nblk, partG, nblkG, cols, p, h, H, ldH, hrow,
                                                                     hcol, R, Rtot, reinterpret_cast<QrFac*>(fac), ctr,
                                                                     flags, allow);
    return cudaGetLastError();
}

cudaError_t qr_apply(const double* W, int64_t ldw, int p, int64_t n, const float* V32, int64_t ldv, int cols,
                     const double* h2, const float* fac, double* out, float* out32, int64_t ldo, int* colexp,
                     const int* flags, int sms, cudaStream_t s) {
    const int g = (int)std::min<int64_t>((n + 127) / 128, (int64_t)kApplyPerSm * sms);
    const size_t shm = (size_t)((cols + 15) / 16) * kApNT * 3 * 32 * sizeof(uint2);
    k_qr_apply<<<g, 128, shm, s>>>(W, ldw, p, n, V32, ldv, cols, h2, reinterpret_cast<const QrFac*>(fac), out, out32,
                                   ldo, colexp, flags);
    return cudaGetLastError();
}

cudaError_t qr_set_smem() {
    return cudaFuncSetAttribute(k_qr_apply, cudaFuncAttributeMaxDynamicSharedMemorySize, 128 * 1024);
}
