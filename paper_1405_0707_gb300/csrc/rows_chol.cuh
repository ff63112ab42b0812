// rows_chol.cuh -- the float-pair Cholesky factor of a block's Gram matrix (one warp), included
// per row width inside a namespace that defines RP.

// ---- float-pair (double-float) scalars for the accurate first-pass factor
struct fp2 {
    float h, l;
};
__device__ __forceinline__ fp2 f2_make(float h, float l) {
    fp2 r;
    r.h = h;
    r.l = l;
    return r;
}
__device__ __forceinline__ fp2 f2_norm(float s, float e) {
    const float h = s + e;
    return f2_make(h, e - (h - s));
}
__device__ __forceinline__ fp2 f2_add(fp2 a, fp2 b) {
    const float s = a.h + b.h, bp = s - a.h;
    const float e = ((a.h - (s - bp)) + (b.h - bp)) + (a.l + b.l);
    return f2_norm(s, e);
}
__device__ __forceinline__ fp2 f2_mul(fp2 a, fp2 b) {
    const float pr = a.h * b.h;
    float e = fmaf(a.h, b.h, -pr);
    e = fmaf(a.h, b.l, e);
    e = fmaf(a.l, b.h, e);
    return f2_norm(pr, e);
}
// sqrt(a), a > 0: s = sqrtf(a_h), corrected by one Newton step (a - s^2) / (2 s), with s^2
// formed exactly by an FMA
__device__ __forceinline__ fp2 f2_sqrt(fp2 a) {
    const float sq = sqrtf(a.h);
    const float pr = sq * sq, pe = fmaf(sq, sq, -pr);
    return f2_norm(sq, (((a.h - pr) - pe) + a.l) / (2.f * sq));
}
// 1 / a: x0 = 1 / a_h corrected by x0 (1 - a x0)
__device__ __forceinline__ fp2 f2_rcp(fp2 a) {
    const float x0 = 1.f / a.h;
    float e = fmaf(-a.h, x0, 1.f);
    e = fmaf(-a.l, x0, e);
    return f2_norm(x0, x0 * e);
}
__device__ __forceinline__ fp2 f2_shfl(fp2 a, int src) {
    return f2_make(__shfl_sync(0xffffffffu, a.h, src), __shfl_sync(0xffffffffu, a.l, src));
}

struct CholD {
    float Uh[RP * RP], Ul[RP * RP];   // the factor of G 2^-k (upper triangle) as float pairs
    float ih[RP], il[RP];             // 1 / U_cc as float pairs
    int ok;
};

// Cholesky factor of G 2^-k in float-pair arithmetic on warp 0, lane l holding column l (as
// chol32_full).  ok = every pivot is positive and at least rel_min times the largest diagonal
// entry and no column is zero: then one pass with this factor leaves the block orthonormal to
// ~kappa^2 2^-48, and the caller skips the deviation pass.  Otherwise the caller discards it.
// dep: a pivot that is zero, or below rel_min times the largest diagonal entry, marks a
// dependent column instead of a failure: R_jj = 0 and row j of R zero, so the column's
// direction is dropped (the block Krylov space loses a direction that lies in the span of
// the others to within the pivot) and the forward substitution leaves it zero.
__device__ inline void chol_df(CholD& cd, const double* G0, int p, int k, float rel_min, bool dep = false) {
    const int lane = threadIdx.x;
    const unsigned full = 0xffffffffu;
    const bool act = lane < p;
    fp2 g[RP], u[RP];
    float dg = 0.f;
#pragma unroll
    for (int a = 0; a < RP; ++a) {
        float h = 0.f, l = 0.f;
        if (act && a < p) split_df(ldexp(G0[a * p + lane], -k), h, l);
        g[a] = f2_make(h, l);
        u[a] = f2_make(0.f, 0.f);
        if (a == lane) dg = h;
    }
    float dmax = act ? dg : 0.f;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) dmax = fmaxf(dmax, __shfl_xor_sync(full, dmax, o));
    int ok_l = 1;
    fp2 myinv = f2_make(0.f, 0.f);
#pragma unroll
    for (int j = 0; j < RP; ++j) {
        if (j >= p) break;
        fp2 inv = f2_make(0.f, 0.f);
        if (lane == j) {
            fp2 d = g[j];
            if (dep && isfinite(d.h) && (G0[j * p + j] == 0.0 || !(d.h >= rel_min * dmax))) {
                u[j] = f2_make(0.f, 0.f);           // dependent column: R_jj = 0, inverse 0
            } else {
                if (G0[j * p + j] == 0.0 || !(d.h > 0.f) || !isfinite(d.h) || d.h < rel_min * dmax) {
                    ok_l = 0;
                    d = f2_make(1.f, 0.f);
                }
                u[j] = f2_sqrt(d);
                inv = f2_rcp(u[j]);
            }
            myinv = inv;
        }
        inv = f2_shfl(inv, j);
        if (act && lane > j) u[j] = f2_mul(g[j], inv);
        // trailing update G[a][l] -= U[j][a] U[j][l] for j < a <= l
#pragma unroll
        for (int a = j + 1; a < RP; ++a) {
            const fp2 uja = f2_shfl(u[j], a);
            if (act && a < p && a <= lane) {
                const fp2 pr = f2_mul(uja, u[j]);
                g[a] = f2_add(g[a], f2_make(-pr.h, -pr.l));
            }
        }
    }
    const int ok = __all_sync(full, ok_l);
    if (act) {
#pragma unroll
        for (int a = 0; a < RP; ++a)
            if (a < p) {
                cd.Uh[a * p + lane] = u[a].h;
                cd.Ul[a * p + lane] = u[a].l;
            }
        cd.ih[lane] = myinv.h;
        cd.il[lane] = myinv.l;
    }
    if (lane == 0) cd.ok = ok;
    __syncwarp();
}
