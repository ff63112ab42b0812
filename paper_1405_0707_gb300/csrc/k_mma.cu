// k_mma.cu -- the tall-skinny products of the mixed path as register-streamed tensor-core
// passes (mma.sync): the Gram-Schmidt projections h = V^T W, the update W <- W - V h, and the
// solution update Z <- Z + V Wc, for blocks of p <= 32 columns against any number of basis
// columns.
//
// What bounds these passes: each reads the n x cols basis once and does 2 n cols p useful flop
// on it, so their floor is the basis's bytes at the memory rate.  Earlier forms staged every
// element through shared memory (FP64 bytes, an integer FP64 -> FP32 conversion, a store, a
// barrier, a load per FMA) and were bound by issue slots and latency at 0.2-0.4 of that rate.
// Here the operands go from global memory straight into MMA fragments: a fragment's K (or M)
// index may be any permutation of the rows as long as both operands use the same one, so each
// lane loads 16 contiguous bytes of a column and no shared-memory pass or barrier remains.
//
//  * The projections read an FP32 copy of the basis (V32, written with every new block; the
//    FP32 rounding is the one the CUDA-core projection applied on each read), half the bytes.
//    Each FP32 value is split exactly enough into three bf16 parts, and the six products
//    v0w0 | v0w1 v1w0 v1w1 v0w2 v2w0 go to two accumulators (the second 2^-8 smaller), so the
//    product error is ~2^-25, below the FP32 rounding of the operands.  Every 16 rows the
//    main accumulator is added to a float pair, so summation error does not grow with n.
//  * The update must hold to FP64 rounding (the Arnoldi relation of eq. (4.5)).  Both operands
//    are cut into balanced base-256 digits held exactly in fp16, products of digits are summed
//    by level (digit positions i + j) in FP32 accumulators that stay below 2^24, hence exact,
//    and the level sums are combined in float pairs.  V's digits are scaled per column by the
//    exponent of its largest entry (colexp, kept with each block): seven digits then resolve
//    2^-55 of that entry.
//  * h of the first pass only seeds the second pass, so the update rounds it to four digits
//    (2^-32 of the largest scaled entry of its column, finer than the FP32 projection it came
//    from unless the columns' largest entries differ by more than 2^8, where the second pass has
//    that much more to correct), subtracts V times exactly that h and records exactly that h in H:
//    the relation does not see the rounding, and 22 digit products replace 28.  The Z update keeps
//    all seven digits of its coefficients (2^-55): beside a localised column, whose largest entry
//    is one, six left the spread ones 2^-48 / their largest entry (90 x 77, p = 32, unit vectors:
//    solution error 2.3e-14, now 1.5e-14).
//
// Measured, 96^3, p = 16, per block step averaged over a 10-step cycle: Gram-Schmidt 1.09 -> 0.66 ms
// (projection 66 us at 16 and 237 us at 160 columns, 2.9 TB/s, bound by the loads in flight; update 197 and
// 491 us, 2.8 TB/s, bound by issue slots at 12 to 16 warps per SM), 512 x 352, p = 32: 3.3 -> 0.6 ms.
#include <cuda_fp16.h>

#include <algorithm>
#include <type_traits>

#include "df.cuh"
#include "internal.h"
#include "mma.cuh"

namespace expm {
namespace {

constexpr unsigned kFull = 0xffffffffu;

// ---------------------------------------------------------------- projection
constexpr int kProjKb = 8;                       // 16-row blocks per unit: 128 rows
constexpr size_t proj_smem(int NT, int MTW) {
    return std::max((size_t)NT * MTW * 4 * 8 * 32 * sizeof(float2), (size_t)2 * kProjKb * NT * 3 * 32 * sizeof(uint2));
}

// v rounded to FP32 (nearest, ties away), below 2^-126 flushed to zero; not for inf and NaN, whose
// blocks the Gram matrix of the update flags
__device__ __forceinline__ float f32_fast(double v) {
    const uint32_t hi = (uint32_t)__double2hiint(v), lo = (uint32_t)__double2loint(v);
    const uint32_t f = __funnelshift_l(lo, hi, 3) - (384u << 23) + ((lo >> 28) & 1u);
    return ((hi & 0x7FFFFFFFu) >> 20) < 897u ? 0.f : __uint_as_float(f | (hi & 0x80000000u));
}

// partial[bx][a][c] = sum over the rows of row group bx of V[r, a] W[r, c].
// MMA: M = 16 basis columns, N = 8 block columns, K = 16 rows.  A warp owns up to MTW M tiles
// (a = 16 (cg + CG i)) and every N tile; the CTA's 8 warps are CG column groups x 8 / CG row
// groups; grid.y covers bases wider than CG MTW tiles.  Rows are taken in units of 128: W's unit
// is converted to fragments in shared memory once per CTA (its conversion from FP64 costs more
// instructions than the products it feeds when every warp repeats it), two buffers, one barrier
// per unit; V's next block is loaded while the current one is multiplied.
template <int NT, int MTW>
__global__ void __launch_bounds__(256, (NT * MTW <= 4) ? 2 : 1)
k_proj_mma(const float* __restrict__ V, int64_t ldv, int cols, const double* __restrict__ W, int64_t ldw, int p,
           int64_t n, double* __restrict__ part, int CG) {
    extern __shared__ __align__(16) unsigned char smp[];
    uint2* wf = reinterpret_cast<uint2*>(smp);             // [buf][kb][nt][split][lane]
    constexpr int WBUF = kProjKb * NT * 3 * 32;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, g = lane >> 2, t = lane & 3;
    const int cg = warp % CG, rg = warp / CG, RG = 8 / CG;
    const int mt_all = (cols + 15) >> 4, mt0 = blockIdx.y * CG * MTW + cg;
    float cm[MTW][NT][4], cc[MTW][NT][4], ch[MTW][NT][4];
#pragma unroll
    for (int i = 0; i < MTW; ++i)
#pragma unroll
        for (int j = 0; j < NT; ++j)
#pragma unroll
            for (int q = 0; q < 4; ++q) cm[i][j][q] = cc[i][j][q] = ch[i][j][q] = 0.f;
    const int nmt = mt0 < mt_all ? min(MTW, (mt_all - mt0 + CG - 1) / CG) : 0;   // tiles this warp owns
    const int64_t nblk = (n + 15) >> 4, units = (nblk + kProjKb - 1) / kProjKb;
    auto loadv = [&](float4* v, int i, int64_t blk) {
        const int a = (mt0 + i * CG) * 16 + g;
        const int64_t r0 = blk * 16 + 4 * t;
        v[0] = *reinterpret_cast<const float4*>(V + (int64_t)min(a, cols - 1) * ldv + r0);
        v[1] = *reinterpret_cast<const float4*>(V + (int64_t)min(a + 8, cols - 1) * ldv + r0);
    };
    double2 w[NT][2];
    auto loadw = [&](int64_t u) {                          // item k: block kb = warp, N tile k
        const int64_t r = (u * kProjKb + warp) * 16 + 4 * t;
#pragma unroll
        for (int j = 0; j < NT; ++j) {
            w[j][0] = w[j][1] = make_double2(0.0, 0.0);
            const double* src = W + (int64_t)min(8 * j + g, p - 1) * ldw + r;
            if (r < n) {                                   // columns are padded to 32 rows
                w[j][0] = *reinterpret_cast<const double2*>(src);
                w[j][1] = *reinterpret_cast<const double2*>(src + 2);
                if (r + 1 >= n) w[j][0].y = 0.0;           // the padding is not W's
                if (r + 2 >= n) w[j][1].x = 0.0;
                if (r + 3 >= n) w[j][1].y = 0.0;
            }
        }
    };
    auto storew = [&](int buf) {
#pragma unroll
        for (int j = 0; j < NT; ++j) {
            uint32_t s0[3], s1[3];
            split3(f32_fast(w[j][0].x), f32_fast(w[j][0].y), s0);
            split3(f32_fast(w[j][1].x), f32_fast(w[j][1].y), s1);
#pragma unroll
            for (int k = 0; k < 3; ++k) wf[buf * WBUF + ((warp * NT + j) * 3 + k) * 32 + lane] = make_uint2(s0[k], s1[k]);
        }
    };
    int64_t u = blockIdx.x;
    float4 v[MTW][2];
#pragma unroll
    for (int i = 0; i < MTW; ++i) v[i][0] = v[i][1] = make_float4(0.f, 0.f, 0.f, 0.f);   // tiles past nmt
    int buf = 0;
    if (u < units) {
        loadw(u);
        const int64_t b0 = u * kProjKb + rg;
#pragma unroll
        for (int i = 0; i < MTW; ++i)
            if (i < nmt && b0 < nblk) loadv(v[i], i, b0);
        storew(0);
    }
    __syncthreads();
    for (; u < units; u += gridDim.x) {
        const int64_t un = u + gridDim.x;
        if (un < units) loadw(un);
        const int64_t bend = min(nblk, (u + 1) * kProjKb);
        for (int64_t b = u * kProjKb + rg; b < bend; b += RG) {
            int64_t bn = b + RG;
            if (bn >= bend) bn = un * kProjKb + rg;
            const bool more = bn < nblk;
            const uint2* wq = wf + buf * WBUF + (int)(b - u * kProjKb) * NT * 3 * 32 + lane;
            uint2 wb[NT][3];
#pragma unroll
            for (int j = 0; j < NT; ++j)
#pragma unroll
                for (int k = 0; k < 3; ++k) wb[j][k] = wq[(j * 3 + k) * 32];
            // two M tiles at a time: their splits, the next block's loads, then the products
            // interleaved over the tiles and N tiles
#pragma unroll
            for (int i0 = 0; i0 < MTW; i0 += 2)
                if (i0 < nmt) {
                    uint32_t a[2][3][4];
#pragma unroll
                    for (int i = 0; i < 2; ++i) {
                        const float4 x = v[i0 + i][0], y = v[i0 + i][1];
                        uint32_t s[3];
                        split3(x.x, x.y, s);
                        a[i][0][0] = s[0]; a[i][1][0] = s[1]; a[i][2][0] = s[2];
                        split3(y.x, y.y, s);
                        a[i][0][1] = s[0]; a[i][1][1] = s[1]; a[i][2][1] = s[2];
                        split3(x.z, x.w, s);
                        a[i][0][2] = s[0]; a[i][1][2] = s[1]; a[i][2][2] = s[2];
                        split3(y.z, y.w, s);
                        a[i][0][3] = s[0]; a[i][1][3] = s[1]; a[i][2][3] = s[2];
                    }
#pragma unroll
                    for (int i = 0; i < 2; ++i)
                        if (more && i0 + i < nmt) loadv(v[i0 + i], i0 + i, bn);
#pragma unroll
                    for (int pr = 0; pr < 6; ++pr)
#pragma unroll
                        for (int i = 0; i < 2; ++i)
#pragma unroll
                            for (int j = 0; j < NT; ++j)
                                mma_bf16(pr == 0 ? cm[i0 + i][j] : cc[i0 + i][j], a[i][kProdA[pr]], wb[j][kProdB[pr]].x,
                                         wb[j][kProdB[pr]].y);
                    // the main sums go to the float pairs after every block: the MMA truncates towards zero,
                    // so a sum that one row dominates and the rest cancels drifts by 2^-24 of it per block
                    // (300 x 300, unit vectors, orthogonality: 1.0e-7 with eight blocks, 9e-9 with one; in time
                    // nothing up to p = 16, 0.4 % of a solve at p = 32)
#pragma unroll
                    for (int i = 0; i < 2; ++i)
#pragma unroll
                        for (int j = 0; j < NT; ++j)
#pragma unroll
                            for (int q = 0; q < 4; ++q) {
                                df_add(ch[i0 + i][j][q], cc[i0 + i][j][q], cm[i0 + i][j][q]);
                                cm[i0 + i][j][q] = 0.f;
                            }
                }
        }
        buf ^= 1;
        if (un < units) storew(buf);
        __syncthreads();
    }
    // the row groups' sums in float pairs (FP64 adds here cost more than the products above: one
    // FP64 warp instruction occupies its scheduler for ~64 clocks), one FP64 value per output
    float2* red = reinterpret_cast<float2*>(smp);          // [tile][q][warp][lane]
#pragma unroll
    for (int i = 0; i < MTW; ++i)
#pragma unroll
        for (int j = 0; j < NT; ++j)
#pragma unroll
            for (int q = 0; q < 4; ++q)
                red[(((i * NT + j) * 4 + q) * 8 + warp) * 32 + lane] = make_float2(ch[i][j][q], cc[i][j][q]);
    __syncthreads();
    double* out = part + (int64_t)blockIdx.x * cols * p;
    const int tiles_y = min(CG * MTW, mt_all - (int)blockIdx.y * CG * MTW);   // M tiles of this CTA
    for (int e = threadIdx.x; e < tiles_y * NT * 128; e += 256) {
        const int ln = e & 31, q = (e >> 5) & 3, mj = e >> 7, j = mj % NT, m = mj / NT;
        const int i = m / CG, w0 = m - i * CG;
        const int aa = (blockIdx.y * CG * MTW + m) * 16 + (ln >> 2) + (q >> 1) * 8, c = 8 * j + 2 * (ln & 3) + (q & 1);
        if (aa >= cols || c >= p) continue;
        const float2* src = red + ((i * NT + j) * 4 + q) * 256 + w0 * 32 + ln;
        float sh = src[0].x, sl = src[0].y;
        for (int k = 1; k < RG; ++k) {
            const float2 x = src[k * CG * 32];
            df_add(sh, sl, x.x);
            sl += x.y;
        }
        out[(int64_t)aa * p + c] = f64_of_f32_i(sh) + f64_of_f32_i(sl);
    }
}

// ---------------------------------------------------------------- digits
// The NV balanced base-256 digits of v 2^(1022 - emax) (magnitude below 1; c = digit_shift<NV>() + emax),
// as the bytes of Y = X + bias with X the two's-complement value times 2^55 (seven digits: the top 16 bits
// of Y read as fp16 are 1152 + d_0) or 2^62 (eight); 0x6400 | byte read as fp16 is 1152 + d_i.
template <int NV>
__device__ constexpr int digit_shift() { return NV == 7 ? 9 : 2; }

constexpr int kNoExp = 1 << 20;      // the shift of an all-zero column: every digit is zero

template <int NV>
__device__ __forceinline__ void digits_y(double v, int c, uint32_t& yl, uint32_t& yh) {
    const uint32_t hi = (uint32_t)__double2hiint(v), lo = (uint32_t)__double2loint(v);
    const uint32_t s = (uint32_t)(c - (int)((hi >> 20) & 0x7FFu));
    const uint32_t mh = __funnelshift_l(lo, hi, 11) | 0x80000000u, ml = lo << 11;
    unsigned long long X = ((unsigned long long)mh << 32) | ml;
    asm("shr.u64 %0, %0, %1;" : "+l"(X) : "r"(s));            // shifts of 64 and more give zero
    const int sg = (int)hi >> 31;
    const unsigned long long S = (unsigned long long)(long long)sg;
    X = (X ^ S) + ((NV == 7 ? 0x6480808080808080ull : 0x8080808080808080ull) - S);
    yl = (uint32_t)X;
    yh = (uint32_t)(X >> 32);
}

__device__ __forceinline__ uint32_t unbias(uint32_t x) {      // (1152 + d) - 1152 in both halves
    uint32_t r;
    asm("add.rn.f16x2 %0, %1, %2;" : "=r"(r) : "r"(x), "r"(0xE480E480u));
    return r;
}
// digit I of the pair (x in the low half, y in the high half): byte NV - 1 - I of Y
template <int NV, int I>
__device__ __forceinline__ uint32_t digit_pair(uint32_t xl, uint32_t xh, uint32_t yl, uint32_t yh) {
    if constexpr (NV == 7 && I == 0) return unbias(__byte_perm(xh, yh, 0x7632));
    constexpr int B = NV - 1 - I;                              // byte of Y
    const uint32_t z = B >= 6 ? __byte_perm(xh, yh, 0x7632) : B >= 4 ? __byte_perm(xh, yh, 0x5410)
                       : B >= 2 ? __byte_perm(xl, yl, 0x7632) : __byte_perm(xl, yl, 0x5410);
    if constexpr (B % 2 == 0) return unbias((z & 0x00FF00FFu) | 0x64006400u);
    return unbias(__byte_perm(z, 0x64646464u, 0x4341));
}

// x 2^k by an add to the exponent field (integer operations only); a result below the normal
// range flushes to a signed zero and one above it becomes inf
__device__ __forceinline__ double scale2_e(double x, int k) {
    const long long b = __double_as_longlong(x);
    const int e = (int)((b >> 52) & 0x7FF);
    long long r = b + ((long long)k << 52);
    if (e == 0 || e + k <= 0) r = b & (1LL << 63);
    if (e != 0 && e + k >= 0x7FF) r = (b & (1LL << 63)) | (0x7FFLL << 52);
    return __longlong_as_double(r);
}

// x 2^k as a double from the bit pattern; x finite, subnormal x and results below 2^-1022 give zero, results
// past the range inf
__device__ __forceinline__ double scaled_f32(float x, int k) {
    const uint32_t u = __float_as_uint(x), m = u & 0x7FFFFFFFu;
    const int e = (int)(m >> 23) + 896 + k;
    uint32_t hi = (m >> 3) + ((uint32_t)(896 + k) << 20), lo = m << 29;
    if (m < 0x00800000u || e <= 0) hi = lo = 0u;
    if (e >= 2047 && m >= 0x00800000u) {
        hi = 0x7FF00000u;
        lo = 0u;
    }
    return __hiloint2double((int)(hi | (u & 0x80000000u)), (int)lo);
}

// X 2^k as a double, |X| <= 2^52, built from its bit pattern (results below 2^-1022 flush to zero)
__device__ __forceinline__ double scaled_int(long long X, int k) {
    if (X == 0) return 0.0;
    const unsigned long long m = (unsigned long long)(X < 0 ? -X : X);
    const int lead = 63 - __clzll((long long)m), e = lead + k + 1023;
    if (e <= 0) return 0.0;
    const unsigned long long b = ((unsigned long long)e << 52) | ((m << (52 - lead)) & 0xFFFFFFFFFFFFFull);
    return __longlong_as_double((long long)(b | (X < 0 ? 1ull << 63 : 0ull)));
}

// L_0 + L_1 2^-8 + .. + L_8 2^-64 = x + y, the level sums exact integers below 2^24: three groups summed
// exactly in float pairs (40 bits each), joined in FP64
__device__ __forceinline__ void level_sum64(float l0, float l1, float l2, float l3, float l4, float l5, float l6, float l7,
                                            double& x, double& y, float l8 = 0.f) {
    float ah = l2 * 0x1p-16f, al = 0.f;
    df_add(ah, al, l1 * 0x1p-8f);
    df_add(ah, al, l0);
    float bh = l5 * 0x1p-40f, bl = 0.f;
    df_add(bh, bl, l4 * 0x1p-32f);
    df_add(bh, bl, l3 * 0x1p-24f);
    const float lo = bl + fmaf(l8, 0x1p-64f, fmaf(l7, 0x1p-56f, l6 * 0x1p-48f));
    x = f64_of_f32_i(ah);
    y = (f64_of_f32_i(lo) + f64_of_f32_i(bh)) + f64_of_f32_i(al);
}

constexpr int kUpdThreads = 128;
__host__ __device__ constexpr int upd_seg(int NH) { return NH == 4 ? 15 : NH == 6 ? 10 : 8; }   // 16-column chunks per exact segment
__host__ __device__ constexpr int gram_rounds(int NT) { return NT == 1 ? 5 : NT == 2 ? 5 : 17; }
__host__ __device__ constexpr int gram_split(int NT) { return NT == 1 ? 4 : 1; }   // lanes sharing one Gram entry

constexpr size_t upd_smem(int cols, int NT, int NH, bool gram) {
    const size_t nk = (size_t)((cols + 15) / 16);
    return nk * (NH / 2) * NT * 32 * 16 + nk * 16 * sizeof(int) +
           (gram ? sizeof(float2) * (size_t)std::max((kUpdThreads / 32) * 16 * (8 * NT + 1), gram_rounds(NT) * 128) : 0);
}

enum UpdMode { U_GS = 0, U_Z = 1, U_GS64 = 2, U_Z64 = 3, U_MUL64 = 4 };

// U_GS (NV = 7, NH = 4): W <- W - V h with h rounded as described at the top; CTA 0 records the rounded h
// in H (columns hcol .., rows 0 .. cols - 1) and clears the next block's colexp; the Gram matrix of the
// updated W in float pairs goes to partG[blk][p][p].
// U_Z (7, 8, seven digits used): Z <- Z + V Wc, then the restart copy V[:, 0:p] <- V[:, cols-p:cols] of this CTA's rows (and
// of V32) when asked.
// U_GS64, U_Z64 (8, 8): the same products to FP64 rounding for FP64 plans (both operands to 2^-62 of
// their column's largest entry, no Gram matrix, h not rounded).
// U_MUL64 (8, 8): out <- V h, V a p-column block (W <- W R^-1; out may be V), by pass as in TrsmPass.
// U_GS64 and U_MUL64 collect the largest exponent of each result column in oexp.
// MMA: M = 16 rows (lane group g holds rows 2g and 2g + 1, one 16-byte load per column), N = 8
// block columns, K = 16 basis columns (lane t holds columns 4t .. 4t + 3).  One warp per 16-row
// tile, the next chunk's loads in flight.  44 MMAs per 256 basis elements at p = 16 take about as
// long as the elements' 8 bytes at the memory rate.
struct UpdArgs {
    double* V;
    int64_t ldv;
    int cols;
    double* W;
    int64_t ldw;
    int p;
    int64_t n;
    const double* h;
    int* colexp;
    double* partG;
    double* H;
    int ldH, hcol;
    int* flags;
    float* V32;
    int restart;
    int* oexp;
    const int* skip;       // return at once when *skip != 0 (== 0 for skip_zero)
    int skip_zero;
    double* alt;           // U_MUL64: the destination when flags[2] is set (alternative to W)
    int64_t ldalt;
    int* altexp;
};

template <int NT, int NV, int NH, int MODE>
__global__ void __launch_bounds__(kUpdThreads, NT == 4 ? 2 : NT == 2 ? 3 : 4)
k_upd_mma(const UpdArgs A) {
    constexpr bool GS = MODE == U_GS, D64 = NV == 8;
    if (A.skip && ((*A.skip != 0) != (A.skip_zero != 0))) return;
    double* const V = A.V;
    const int64_t ldv = A.ldv, n = A.n;
    const int cols = A.cols, p = A.p;
    double* W = A.W;
    int64_t ldw = A.ldw;
    int* oexp = A.oexp;
    if (MODE == U_MUL64 && A.alt && A.flags[2]) {
        W = A.alt;
        ldw = A.ldalt;
        oexp = A.altexp;
    }
    const double* __restrict__ h = A.h;
    int* const colexp = A.colexp;
    extern __shared__ __align__(16) unsigned char smu[];
    const int nk = (cols + 15) >> 4;
    const int64_t ntiles = (n + 15) >> 4;
    const int64_t tstep = (int64_t)gridDim.x * (kUpdThreads / 32);
    int64_t tile = (int64_t)blockIdx.x * (kUpdThreads / 32) + (threadIdx.x >> 5);
    double2 v[4];
    auto load = [&](int64_t tl, int kc) {
        const int64_t r = tl * 16 + 2 * ((threadIdx.x & 31) >> 2);
#pragma unroll
        for (int q = 0; q < 4; ++q)
            v[q] = *reinterpret_cast<const double2*>(V + (int64_t)min(kc * 16 + 4 * (int)(threadIdx.x & 3) + q, cols - 1) * ldv + r);
    };
    if (tile < ntiles) load(tile, 0);            // in flight while the digits of h are formed
    __half* Bh = reinterpret_cast<__half*>(smu);
    int* c9s = reinterpret_cast<int*>(smu + (size_t)nk * (NH / 2) * NT * 512);
    float2* gbuf = reinterpret_cast<float2*>(c9s + nk * 16);
    __shared__ int fmax_s[8 * NT], bad_s;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, g = lane >> 2, t = lane & 3;
    constexpr int NCOL = 8 * NT;
    for (int a = tid; a < nk * 16; a += kUpdThreads) {
        const int em = a < cols ? colexp[a] : 0;
        c9s[a] = em > 0 ? digit_shift<NV>() + em : kNoExp;
    }
    if (tid < NCOL) fmax_s[tid] = -100000;
    if (tid == 0) bad_s = 0;
    __syncthreads();
    if (GS && blockIdx.x == 0 && tid < p) colexp[cols + tid] = 0;
    // exponent f_c of column c of the scaled h: |h[a, c]| 2^(emax_a - 1022) < 2^f_c
    for (int e = tid; e < cols * NCOL; e += kUpdThreads) {
        const int a = e / NCOL, c = e - a * NCOL;
        if (c < p) {
            const int E = (int)(((unsigned)__double2hiint(h[a * p + c]) >> 20) & 0x7FFu);
            if (E == 0x7FF) bad_s = 1;
            const int em = c9s[a] - digit_shift<NV>();
            if (E > 0 && em < 4096) atomicMax(&fmax_s[c], E - 1022 + em - 1022);
        }
    }
    __syncthreads();
    if (tid == 0 && bad_s) atomicOr(&A.flags[0], 1);
    constexpr int ND = D64 ? 8 : NH < NV ? NH : NV;       // digits of h (no product reaches past level NV - 1)
    constexpr int SC = D64 ? 62 : 8 * ND - 1;
    for (int e = tid; e < nk * 16 * NCOL; e += kUpdThreads) {
        const int a = e / NCOL, c = e - a * NCOL;
        long long X = 0;
        int sh = 0;
        if (a < cols && c < p) {
            const double hv = h[a * p + c];
            const unsigned long long b = (unsigned long long)__double_as_longlong(hv);
            const int E = (int)((b >> 52) & 0x7FF), em = c9s[a] - digit_shift<NV>(), f = fmax_s[c];
            // |h| 2^(em - 1022) 2^(SC - f) = m 2^-sh, rounded to nearest
            sh = 1075 - E + 1022 - em + f - SC;
            if (E > 0 && em < 4096 && sh <= 54) {
                const unsigned long long m = (b & 0xFFFFFFFFFFFFFull) | (1ull << 52);
                X = sh > 0 ? (long long)((m + (1ull << (sh - 1))) >> sh) : (long long)(m << -sh);
                if (b >> 63) X = -X;
            }
            if (GS && blockIdx.x == 0) {
                // the h that is applied, exactly: X 2^(f - SC) 2^(1022 - em)
                A.H[(int64_t)(A.hcol + c) * A.ldH + a] = scaled_int(X, f - SC + 1022 - em);
            }
        }
        const int kc = a >> 4, kk = a & 15;
        const int ln = (c & 7) * 4 + (kk >> 2);
#pragma unroll
        for (int j = NH - 1; j >= 0; --j) {
            int d;
            if (j >= ND) {
                d = 0;
            } else if (j > 0) {
                d = (int)((X + 128) & 255) - 128;
                X = (X - d) >> 8;
            } else {
                d = (int)X;
            }
            Bh[((((size_t)kc * (NH / 2) + (j >> 1)) * NT + (c >> 3)) * 32 + ln) * 8 + (j & 1) * 4 + (kk & 3)] =
                __int2half_rn(d);
        }
    }
    __syncthreads();

    uint32_t omax[NT][2];
#pragma unroll
    for (int j = 0; j < NT; ++j) omax[j][0] = omax[j][1] = 0u;
    constexpr int GK = GS ? gram_rounds(NT) : 1, GSP = gram_split(NT);
    const int ne = p * (p + 1) / 2;
    float gh[GK], gl[GK];
    int gi[GK];                                  // packed (row group << 16 | i << 8 | j), -1 none
    if (GS) {
#pragma unroll
        for (int k = 0; k < GK; ++k) {
            gh[k] = gl[k] = 0.f;
            const int it = lane + 32 * k;
            gi[k] = -1;
            if (it < ne * GSP) {
                int i = 0, rem = it % ne;
                while (rem >= p - i) {
                    rem -= p - i;
                    ++i;
                }
                gi[k] = ((it / ne) << 16) | (i << 8) | (i + rem);
            }
        }
    }
    float2* gw = gbuf + (size_t)warp * 16 * (NCOL + 1);
    for (; tile < ntiles; tile += tstep) {
        const int64_t r = tile * 16 + 2 * g;
        double w[NT][4];                         // [nt]: (2g, c) (2g, c + 1) (2g + 1, c) (2g + 1, c + 1)
        for (int k0 = 0; k0 < nk; k0 += upd_seg(NH)) {
            const int k1 = min(nk, k0 + upd_seg(NH));
            float acc[NV][NT][4];
#pragma unroll
            for (int l = 0; l < NV; ++l)
#pragma unroll
                for (int j = 0; j < NT; ++j)
#pragma unroll
                    for (int q = 0; q < 4; ++q) acc[l][j][q] = 0.f;
            for (int kc = k0; kc < k1; ++kc) {
                uint32_t yl[4][2], yh[4][2];
                const int4 c9 = *reinterpret_cast<const int4*>(c9s + kc * 16 + 4 * t);
                digits_y<NV>(v[0].x, c9.x, yl[0][0], yh[0][0]);
                digits_y<NV>(v[0].y, c9.x, yl[0][1], yh[0][1]);
                digits_y<NV>(v[1].x, c9.y, yl[1][0], yh[1][0]);
                digits_y<NV>(v[1].y, c9.y, yl[1][1], yh[1][1]);
                digits_y<NV>(v[2].x, c9.z, yl[2][0], yh[2][0]);
                digits_y<NV>(v[2].y, c9.z, yl[2][1], yh[2][1]);
                digits_y<NV>(v[3].x, c9.w, yl[3][0], yh[3][0]);
                digits_y<NV>(v[3].y, c9.w, yl[3][1], yh[3][1]);
                if (kc + 1 < nk) load(tile, kc + 1);
                else if (tile + tstep < ntiles) load(tile + tstep, 0);
                uint4 b[NH / 2][NT];
                const uint4* Bq = reinterpret_cast<const uint4*>(Bh) + (size_t)kc * (NH / 2) * NT * 32;
#pragma unroll
                for (int jp = 0; jp < NH / 2; ++jp)
#pragma unroll
                    for (int j = 0; j < NT; ++j) b[jp][j] = Bq[(jp * NT + j) * 32 + lane];
                auto level = [&](auto ic) {
                    constexpr int I = decltype(ic)::value;
                    uint32_t a[4];
                    a[0] = digit_pair<NV, I>(yl[0][0], yh[0][0], yl[1][0], yh[1][0]);
                    a[1] = digit_pair<NV, I>(yl[0][1], yh[0][1], yl[1][1], yh[1][1]);
                    a[2] = digit_pair<NV, I>(yl[2][0], yh[2][0], yl[3][0], yh[3][0]);
                    a[3] = digit_pair<NV, I>(yl[2][1], yh[2][1], yl[3][1], yh[3][1]);
#pragma unroll
                    for (int jj = 0; jj < NH; ++jj)
                        if (I + jj < NV) {
#pragma unroll
                            for (int j = 0; j < NT; ++j) {
                                const uint4 bq = b[jj >> 1][j];
                                mma_f16(acc[I + jj][j], a, (jj & 1) ? bq.z : bq.x, (jj & 1) ? bq.w : bq.y);
                            }
                        }
                };
                level(std::integral_constant<int, 0>{});
                level(std::integral_constant<int, 1>{});
                level(std::integral_constant<int, 2>{});
                level(std::integral_constant<int, 3>{});
                level(std::integral_constant<int, 4>{});
                level(std::integral_constant<int, 5>{});
                level(std::integral_constant<int, 6>{});
                if constexpr (NV == 8) level(std::integral_constant<int, 7>{});
            }
            if (k0 == 0) {
#pragma unroll
                for (int j = 0; j < NT; ++j)
#pragma unroll
                    for (int q = 0; q < 2; ++q) {
                        const int c = 8 * j + 2 * t + q;
                        double2 x = make_double2(0.0, 0.0);
                        if (MODE != U_MUL64 && c < p) {
                            if (r + 1 < n) x = *reinterpret_cast<const double2*>(W + (int64_t)c * ldw + r);
                            else if (r < n) x.x = W[(int64_t)c * ldw + r];
                        }
                        w[j][q] = x.x;
                        w[j][2 + q] = x.y;
                    }
            }
            // S = sum_l L_l 2^(-8 l); the product is S 2^(f - 14) (2^(f - 12) with eight digits)
#pragma unroll
            for (int j = 0; j < NT; ++j)
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    const int k = fmax_s[8 * j + 2 * t + (q & 1)] - (D64 ? 12 : 14);
                    constexpr bool SUB = MODE == U_GS || MODE == U_GS64;
                    if constexpr (!D64) {
                        // levels 0..3 in a float pair (exact but for the last bit of 49), 4..6, 2^-32 below, in
                        // FP32.  An error at 2^-48 of the largest V h counts on every row, and rows far below
                        // it (a localised block) have many: with level 3 in FP32 as well, the relation's
                        // error was 1.3e-13 in place of 4e-15 (33 x 31 x 29, unit vectors; pairs throughout, before the
                        // digits, 1e-14)
                        float sh = acc[3][j][q] * 0x1p-24f, sl = 0.f;
                        df_add(sh, sl, acc[2][j][q] * 0x1p-16f);
                        df_add(sh, sl, acc[1][j][q] * 0x1p-8f);
                        df_add(sh, sl, acc[0][j][q]);
                        float lo = fmaf(acc[6][j][q], 0x1p-48f, acc[5][j][q] * 0x1p-40f);
                        lo = fmaf(acc[4][j][q], 0x1p-32f, lo);
                        sl += lo;
                        const double x = scaled_f32(sh, k), y = scaled_f32(sl, k);
                        w[j][q] = SUB ? (w[j][q] - x) - y : (w[j][q] + x) + y;
                    } else {
                        double x, y;
                        level_sum64(acc[0][j][q], acc[1][j][q], acc[2][j][q], acc[3][j][q], acc[4][j][q], acc[5][j][q],
                                    acc[6][j][q], acc[7][j][q], x, y);
                        x = scale2_e(x, k);
                        y = scale2_e(y, k);
                        w[j][q] = SUB ? (w[j][q] - x) - y : (w[j][q] + x) + y;
                    }
                }
        }
        if constexpr (MODE == U_GS64 || MODE == U_MUL64) {
#pragma unroll
            for (int j = 0; j < NT; ++j)
#pragma unroll
                for (int q = 0; q < 4; ++q)
                    if (r + (q >> 1) < n) omax[j][q & 1] = max(omax[j][q & 1], (uint32_t)__double2hiint(w[j][q]) & 0x7FFFFFFFu);
        }
#pragma unroll
        for (int j = 0; j < NT; ++j)
#pragma unroll
            for (int q = 0; q < 2; ++q) {
                const int c = 8 * j + 2 * t + q;
                if (c < p) {
                    double* dst = W + (int64_t)c * ldw + r;
                    if (r + 1 < n) *reinterpret_cast<double2*>(dst) = make_double2(w[j][q], w[j][2 + q]);
                    else if (r < n) *dst = w[j][q];
                }
            }
        if (GS) {
            // Gram entries of the tile's 16 rows from float pairs.  Rows past n are set to zero here: V's
            // padding rows hold whatever the allocation did, and -V h of them is no part of W
            const bool in0 = r < n, in1 = r + 1 < n;
            __syncwarp();
#pragma unroll
            for (int j = 0; j < NT; ++j)
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    float wh, wl;
                    split_df_i((q < 2 ? in0 : in1) ? w[j][q] : 0.0, wh, wl);
                    gw[(2 * g + (q >> 1)) * (NCOL + 1) + 8 * j + 2 * t + (q & 1)] = make_float2(wh, wl);
                }
            __syncwarp();
#pragma unroll
            for (int k = 0; k < GK; ++k)
                if (gi[k] >= 0) {
                    const float2* rowp = gw + (gi[k] >> 16) * (16 / GSP) * (NCOL + 1);
                    const int i = (gi[k] >> 8) & 0xFF, j = gi[k] & 0xFF;
                    float sh = 0.f, sl = 0.f;
#pragma unroll 4
                    for (int rr = 0; rr < 16 / GSP; ++rr) {
                        const float2 x = rowp[rr * (NCOL + 1) + i], y = rowp[rr * (NCOL + 1) + j];
                        df_fma(sh, sl, x.x, x.y, y.x, y.y);
                    }
                    df_add(gh[k], gl[k], sh);
                    gl[k] += sl;
                }
        } else if ((MODE == U_Z || MODE == U_Z64) && A.restart) {
            __syncwarp();
            const int64_t rr = tile * 16 + 2 * (lane & 7);
            for (int c = lane >> 3; c < p; c += 4) {
                const int64_t so = (int64_t)(cols - p + c) * ldv + rr, dof = (int64_t)c * ldv + rr;
                *reinterpret_cast<double2*>(V + dof) = *reinterpret_cast<const double2*>(V + so);
                if (MODE == U_Z) *reinterpret_cast<float2*>(A.V32 + dof) = *reinterpret_cast<const float2*>(A.V32 + so);
            }
        }
    }
    if constexpr (MODE == U_GS64 || MODE == U_MUL64) {
#pragma unroll
        for (int j = 0; j < NT; ++j)
#pragma unroll
            for (int q = 0; q < 2; ++q) {
                uint32_t m = omax[j][q];
#pragma unroll
                for (int o = 4; o < 32; o <<= 1) m = max(m, __shfl_xor_sync(kFull, m, o));
                const int c = 8 * j + 2 * t + q;
                if (g == 0 && c < p && m) atomicMax(&oexp[c], (int)(m >> 20));
            }
    }
    if (GS) {
        __syncthreads();
        // the warps' pairs, then one FP64 value per entry
        float2* red = gbuf;                                  // [k][warp][lane]
#pragma unroll
        for (int k = 0; k < GK; ++k)
            if (32 * k < ne * GSP) red[(k * 4 + warp) * 32 + lane] = make_float2(gh[k], gl[k]);
        __syncthreads();
        double* out = A.partG + (int64_t)blockIdx.x * p * p;
        for (int e = tid; e < p * p; e += kUpdThreads) {
            int i = e / p, j = e % p;
            if (i > j) {
                const int x = i;
                i = j;
                j = x;
            }
            const int k = i * p - i * (i - 1) / 2 + (j - i);
            float sh = 0.f, sl = 0.f;
            for (int q = 0; q < GSP; ++q) {
                const int it = q * ne + k;
#pragma unroll
                for (int wi = 0; wi < kUpdThreads / 32; ++wi) {
                    const float2 x = red[((it >> 5) * 4 + wi) * 32 + (it & 31)];
                    df_add(sh, sl, x.x);
                    sl += x.y;
                }
            }
            out[e] = f64_of_f32_i(sh) + f64_of_f32_i(sl);
        }
    }
}

// ---------------------------------------------------------------- projection to FP64 rounding
// FP64 plans: partial[bx][a][c] = sum over the rows of row group bx of V[r, a] W[r, c], both operands in
// eight digits of their column's scale (2^-62 of its largest entry), the 36 digit products of levels 0..7
// summed exactly over 128 rows and joined in FP64: 4 FP64 adds per output and 128 rows where the FP64
// kernel spends 128 FMAs on a pipe that retires two per SM and clock.  The products left out have random
// signs but for the squares on a Gram matrix's diagonal, of which the largest, digit 4 by digit 4, is a
// 37th product: without it a localised column's norm came out short by n 2^-64 of its largest entry
// squared (300 x 300, unit vectors: |v|^2 - 1 = 6.8e-15, with it 4e-16).  MMA: M = 16 basis columns, N = 8
// block columns, K = 16 rows, lanes and units as in k_proj_mma; a warp owns one M tile.
constexpr size_t proj64_smem(int NT) { return (size_t)2 * kProjKb * NT * 8 * 32 * sizeof(uint2); }

template <int NT>
__global__ void __launch_bounds__(256, NT == 1 ? 2 : 1)
k_proj64(const double* __restrict__ V, int64_t ldv, int cols, const int* __restrict__ vexp, const double* __restrict__ W,
         int64_t ldw, int p, const int* __restrict__ wexp, int64_t n, double* __restrict__ part, int CG, const int* only) {
    if (only && *only == 0) return;
    extern __shared__ __align__(16) unsigned char smq[];
    uint2* wf = reinterpret_cast<uint2*>(smq);             // [buf][kb][nt][digit][lane]
    constexpr int WBUF = kProjKb * NT * 8 * 32;
    __shared__ double red[8][32][4];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, g = lane >> 2, t = lane & 3;
    const int RG = 8 / CG, cg = warp % CG, rg = warp / CG;
    const int mt_all = (cols + 15) >> 4, mt = blockIdx.y * CG + cg;
    const bool work = rg < RG && mt < mt_all;
    const int a0 = min(mt * 16 + g, cols - 1), a1 = min(mt * 16 + g + 8, cols - 1);
    auto shift_of = [](int em) { return em > 0 ? digit_shift<8>() + em : kNoExp; };
    const int cv0 = shift_of(vexp[a0]), cv1 = shift_of(vexp[a1]);
    const int64_t nblk = (n + 15) >> 4, units = (nblk + kProjKb - 1) / kProjKb;
    int cw[NT];
#pragma unroll
    for (int j = 0; j < NT; ++j) cw[j] = shift_of(wexp[min(8 * j + g, p - 1)]);
    double2 w[NT][2];
    auto loadw = [&](int64_t u) {                          // item k: block kb = warp, N tile k
        const int64_t r = (u * kProjKb + warp) * 16 + 4 * t;
#pragma unroll
        for (int j = 0; j < NT; ++j) {
            w[j][0] = w[j][1] = make_double2(0.0, 0.0);
            const double* src = W + (int64_t)min(8 * j + g, p - 1) * ldw + r;
            if (r < n) {                                   // columns are padded to 32 rows
                w[j][0] = *reinterpret_cast<const double2*>(src);
                w[j][1] = *reinterpret_cast<const double2*>(src + 2);
                if (r + 1 >= n) w[j][0].y = 0.0;           // the padding is not W's
                if (r + 2 >= n) w[j][1].x = 0.0;
                if (r + 3 >= n) w[j][1].y = 0.0;
            }
        }
    };
    auto storew = [&](int buf) {
#pragma unroll
        for (int j = 0; j < NT; ++j) {
            uint32_t yl[4], yh[4];
            digits_y<8>(w[j][0].x, cw[j], yl[0], yh[0]);
            digits_y<8>(w[j][0].y, cw[j], yl[1], yh[1]);
            digits_y<8>(w[j][1].x, cw[j], yl[2], yh[2]);
            digits_y<8>(w[j][1].y, cw[j], yl[3], yh[3]);
            uint2* dst = wf + buf * WBUF + (warp * NT + j) * 8 * 32 + lane;
            auto put = [&](auto ic) {
                constexpr int I = decltype(ic)::value;
                dst[I * 32] = make_uint2(digit_pair<8, I>(yl[0], yh[0], yl[1], yh[1]), digit_pair<8, I>(yl[2], yh[2], yl[3], yh[3]));
            };
            put(std::integral_constant<int, 0>{});
            put(std::integral_constant<int, 1>{});
            put(std::integral_constant<int, 2>{});
            put(std::integral_constant<int, 3>{});
            put(std::integral_constant<int, 4>{});
            put(std::integral_constant<int, 5>{});
            put(std::integral_constant<int, 6>{});
            put(std::integral_constant<int, 7>{});
        }
    };
    double2 v[2][2];                                       // columns a0, a1: rows 4t, 4t + 1 | 4t + 2, 4t + 3
    auto loadv = [&](int64_t blk) {
        const int64_t r = blk * 16 + 4 * t;                // rows past n: padding, met by W's zeros
        v[0][0] = *reinterpret_cast<const double2*>(V + (int64_t)a0 * ldv + r);
        v[0][1] = *reinterpret_cast<const double2*>(V + (int64_t)a0 * ldv + r + 2);
        v[1][0] = *reinterpret_cast<const double2*>(V + (int64_t)a1 * ldv + r);
        v[1][1] = *reinterpret_cast<const double2*>(V + (int64_t)a1 * ldv + r + 2);
    };
    float acc[9][NT][4];
    double sum[NT][4];
#pragma unroll
    for (int j = 0; j < NT; ++j)
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            sum[j][q] = 0.0;
#pragma unroll
            for (int l = 0; l < 9; ++l) acc[l][j][q] = 0.f;
        }
    int64_t u = blockIdx.x;
    int buf = 0, since = 0;
    if (u < units) {
        loadw(u);
        if (work && u * kProjKb + rg < nblk) loadv(u * kProjKb + rg);
        storew(0);
    }
    __syncthreads();
    for (; u < units; u += gridDim.x) {
        const int64_t un = u + gridDim.x;
        if (un < units) loadw(un);
        const int64_t bend = min(nblk, (u + 1) * kProjKb);
        if (work)
            for (int64_t b = u * kProjKb + rg; b < bend; b += RG) {
                int64_t bn = b + RG;
                if (bn >= bend) bn = un * kProjKb + rg;
                uint32_t yl[2][4], yh[2][4];
#pragma unroll
                for (int i = 0; i < 2; ++i) {
                    const int c = i ? cv1 : cv0;
                    digits_y<8>(v[i][0].x, c, yl[i][0], yh[i][0]);
                    digits_y<8>(v[i][0].y, c, yl[i][1], yh[i][1]);
                    digits_y<8>(v[i][1].x, c, yl[i][2], yh[i][2]);
                    digits_y<8>(v[i][1].y, c, yl[i][3], yh[i][3]);
                }
                if (bn < nblk) loadv(bn);
                const uint2* wq = wf + buf * WBUF + (int)(b - u * kProjKb) * NT * 8 * 32 + lane;
                uint2 wb[NT][8];
#pragma unroll
                for (int j = 0; j < NT; ++j)
#pragma unroll
                    for (int k = 0; k < 8; ++k) wb[j][k] = wq[(j * 8 + k) * 32];
                auto level = [&](auto ic) {
                    constexpr int I = decltype(ic)::value;
                    uint32_t a[4];
                    a[0] = digit_pair<8, I>(yl[0][0], yh[0][0], yl[0][1], yh[0][1]);
                    a[1] = digit_pair<8, I>(yl[1][0], yh[1][0], yl[1][1], yh[1][1]);
                    a[2] = digit_pair<8, I>(yl[0][2], yh[0][2], yl[0][3], yh[0][3]);
                    a[3] = digit_pair<8, I>(yl[1][2], yh[1][2], yl[1][3], yh[1][3]);
#pragma unroll
                    for (int k = 0; k + I < 8 + (I == 4); ++k)
#pragma unroll
                        for (int j = 0; j < NT; ++j) mma_f16(acc[I + k][j], a, wb[j][k].x, wb[j][k].y);
                };
                level(std::integral_constant<int, 0>{});
                level(std::integral_constant<int, 1>{});
                level(std::integral_constant<int, 2>{});
                level(std::integral_constant<int, 3>{});
                level(std::integral_constant<int, 4>{});
                level(std::integral_constant<int, 5>{});
                level(std::integral_constant<int, 6>{});
                level(std::integral_constant<int, 7>{});
                if (++since == 8) {                        // 8 pairs 2^14 128 rows = 2^24: still exact
                    since = 0;
#pragma unroll
                    for (int j = 0; j < NT; ++j)
#pragma unroll
                        for (int q = 0; q < 4; ++q) {
                            double x, y;
                            level_sum64(acc[0][j][q], acc[1][j][q], acc[2][j][q], acc[3][j][q], acc[4][j][q], acc[5][j][q],
                                        acc[6][j][q], acc[7][j][q], x, y, acc[8][j][q]);
                            sum[j][q] += x + y;
#pragma unroll
                            for (int l = 0; l < 9; ++l) acc[l][j][q] = 0.f;
                        }
                }
            }
        buf ^= 1;
        if (un < units) storew(buf);
        __syncthreads();
    }
    double* out = part + (int64_t)blockIdx.x * cols * p;
#pragma unroll
    for (int j = 0; j < NT; ++j) {
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            double x, y;
            level_sum64(acc[0][j][q], acc[1][j][q], acc[2][j][q], acc[3][j][q], acc[4][j][q], acc[5][j][q], acc[6][j][q],
                        acc[7][j][q], x, y, acc[8][j][q]);
            red[warp][lane][q] = sum[j][q] + (x + y);
        }
        __syncthreads();
        for (int e = threadIdx.x; e < CG * 128; e += 256) {
            const int q = e & 3, ln = (e >> 2) & 31, k = e >> 7;
            const int aa = (blockIdx.y * CG + k) * 16 + (ln >> 2) + (q >> 1) * 8, c = 8 * j + 2 * (ln & 3) + (q & 1);
            if (aa < cols && c < p) {
                double s = red[k][ln][q];
                for (int x = 1; x < RG; ++x) s += red[k + x * CG][ln][q];
                out[(int64_t)aa * p + c] = scale2_e(s, vexp[aa] + wexp[c] - 2044 - 12);
            }
        }
        __syncthreads();
    }
}

// wexp[c] = largest biased exponent of column c of W (zeroed by the caller); the first CTA clears two
// small arrays for the kernels that follow
__global__ void k_colmax(const double* __restrict__ W, int64_t ldw, int64_t n, int* __restrict__ wexp, int* zero0, int n0,
                         int* zero1, int n1) {
    if (blockIdx.x == 0 && blockIdx.y == 0) {
        for (int i = threadIdx.x; i < n0; i += blockDim.x) zero0[i] = 0;
        for (int i = threadIdx.x; i < n1; i += blockDim.x) zero1[i] = 0;
    }
    unsigned mx = 0;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        mx = max(mx, (unsigned)__double2hiint(W[blockIdx.y * ldw + i]) & 0x7FFFFFFFu);
    mx = __reduce_max_sync(kFull, mx);
    if ((threadIdx.x & 31) == 0 && mx) atomicMax(&wexp[blockIdx.y], (int)(mx >> 20));
}

// ---------------------------------------------------------------- the FP32 copy and colexp
// V32 and colexp of columns c0 .. c0 + p - 1 of V (blocks that no fused pass wrote: the first
// block, Ritz vectors).  skip: the fused pass wrote them (device flag).
__global__ void k_pack_block(const double* __restrict__ V, float* __restrict__ V32, int64_t ld, int64_t n,
                             int* __restrict__ colexp, const int* skip) {
    if (skip && *skip) return;
    const int c = blockIdx.y;
    unsigned mx = 0;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        const double v = V[c * ld + i];
        if (V32) V32[c * ld + i] = f32_rn_i(v);
        mx = max(mx, (unsigned)__double2hiint(v) & 0x7FFFFFFFu);
    }
    mx = __reduce_max_sync(kFull, mx);
    if ((threadIdx.x & 31) == 0 && mx) atomicMax(&colexp[c], (int)(mx >> 20));
}

__global__ void k_zero_int(int* p, int n, const int* skip) {
    if (skip && *skip) return;
    if ((int)threadIdx.x < n) p[threadIdx.x] = 0;
}

}  // namespace

// h = V^T W partials: returns the number of partials (row groups) through nb
cudaError_t launch_proj_mma(const float* V32, int64_t ldv, int cols, const double* W, int64_t ldw, int p, int64_t n,
                            double* part, int max_blocks, int sms, int* nb, cudaStream_t s) {
    const int mt = (cols + 15) / 16, NT = p <= 8 ? 1 : p <= 16 ? 2 : 4, MTW = NT == 1 ? 4 : 2;
    int CG = 1;
    while (CG < 8 && CG * MTW < mt) CG *= 2;
    const int gy = (mt + CG * MTW - 1) / (CG * MTW);
    const int64_t units = (n + 16 * kProjKb - 1) / (16 * kProjKb);
    const int ctas_sm = NT * MTW <= 4 ? 2 : 1;
    const int64_t gmax = std::max(1, std::min(max_blocks, ctas_sm * sms / gy));
    const int64_t per = (units + gmax - 1) / gmax;         // units per CTA, the CTAs evenly loaded
    const int gx = (int)((units + per - 1) / per);
    *nb = gx;
    const dim3 grid(gx, gy);
    if (NT == 1) k_proj_mma<1, 4><<<grid, 256, proj_smem(1, 4), s>>>(V32, ldv, cols, W, ldw, p, n, part, CG);
    else if (NT == 2) k_proj_mma<2, 2><<<grid, 256, proj_smem(2, 2), s>>>(V32, ldv, cols, W, ldw, p, n, part, CG);
    else k_proj_mma<4, 2><<<grid, 256, proj_smem(4, 2), s>>>(V32, ldv, cols, W, ldw, p, n, part, CG);
    return cudaGetLastError();
}

template <int NT, int NV, int NH, int MODE>
static cudaError_t upd_launch(const UpdArgs& a, int max_blocks, int sms, int* nb, cudaStream_t s) {
    const size_t shm = upd_smem(a.cols, NT, NH, MODE == U_GS);
    int per_sm = NT == 4 ? 2 : NT == 2 ? 3 : 4;
    while (per_sm > 1 && shm * per_sm > 200 * 1024) --per_sm;
    const int64_t tiles = (a.n + 15) / 16;
    const int g = (int)std::min<int64_t>({(int64_t)per_sm * sms, (tiles + 3) / 4, (int64_t)max_blocks});
    if (nb) *nb = g;
    k_upd_mma<NT, NV, NH, MODE><<<g, kUpdThreads, shm, s>>>(a);
    return cudaGetLastError();
}

#define EXPM_UPD(NV, NH, MODE, ...)                                                                            \
    (a.p <= 8 ? upd_launch<1, NV, NH, MODE>(a, __VA_ARGS__) : a.p <= 16 ? upd_launch<2, NV, NH, MODE>(a, __VA_ARGS__) \
                                                             : upd_launch<4, NV, NH, MODE>(a, __VA_ARGS__))

cudaError_t launch_upd_mma(double* V, int64_t ldv, int cols, double* W, int64_t ldw, int p, int64_t n, const double* h,
                           int* colexp, double* partG, double* H, int ldH, int hcol, int* flags, int max_blocks, int sms,
                           int* nb, cudaStream_t s) {
    UpdArgs a{V, ldv, cols, W, ldw, p, n, h, colexp, partG, H, ldH, hcol, flags};
    return EXPM_UPD(7, 4, U_GS, max_blocks, sms, nb, s);
}

cudaError_t launch_updz_mma(double* V, float* V32, int64_t ldv, int cols, double* Z, int64_t ldz, int p, int64_t n,
                            const double* Wc, int* colexp, int* flags, int restart, int sms, cudaStream_t s) {
    UpdArgs a{V, ldv, cols, Z, ldz, p, n, Wc, colexp, nullptr, nullptr, 0, 0, flags, V32, restart};
    cudaError_t e = V32 ? EXPM_UPD(7, 8, U_Z, 1 << 20, sms, nullptr, s) : EXPM_UPD(8, 8, U_Z64, 1 << 20, sms, nullptr, s);
    if (e == cudaSuccess && restart)
        e = cudaMemcpyAsync(colexp, colexp + cols - p, sizeof(int) * p, cudaMemcpyDeviceToDevice, s);
    return e;
}

// FP64 plans: W <- W - V h, the exponents of the result's columns into oexp (zeroed by the caller)
cudaError_t launch_upd64(double* V, int64_t ldv, int cols, double* W, int64_t ldw, int p, int64_t n, const double* h,
                         int* colexp, int* oexp, int* flags, int sms, cudaStream_t s) {
    UpdArgs a{V, ldv, cols, W, ldw, p, n, h, colexp, nullptr, nullptr, 0, 0, flags};
    a.oexp = oexp;
    return EXPM_UPD(8, 8, U_GS64, 1 << 20, sms, nullptr, s);
}

// out <- W Rinv (p x p), exponents into oexp; alt != null: into alt / altexp instead when flags[2] is set
// (a third pass follows); third: only when flags[2] is set
cudaError_t launch_mul64(double* W, int64_t ldw, int p, int64_t n, const double* Rinv, int* wexp, double* out, int64_t ldo,
                         int* oexp, double* alt, int64_t ldalt, int* altexp, int third, int* flags, int sms, cudaStream_t s) {
    UpdArgs a{W, ldw, p, out, ldo, p, n, Rinv, wexp, nullptr, nullptr, 0, 0, flags};
    a.oexp = oexp;
    a.alt = alt;
    a.ldalt = ldalt;
    a.altexp = altexp;
    if (third) {
        a.skip = flags + 2;
        a.skip_zero = 1;
    }
    return EXPM_UPD(8, 8, U_MUL64, 1 << 20, sms, nullptr, s);
}

// V^T W to FP64 rounding: partial[bx][a][c], nb of them; only: run only when *only != 0
cudaError_t launch_proj64(const double* V, int64_t ldv, int cols, const int* vexp, const double* W, int64_t ldw, int p,
                          const int* wexp, int64_t n, double* part, int max_blocks, int sms, int* nb, const int* only,
                          cudaStream_t s) {
    const int mt = (cols + 15) / 16, NT = p <= 8 ? 1 : p <= 16 ? 2 : 4;
    const int CG = std::min(8, mt), gy = (mt + CG - 1) / CG, RG = 8 / CG;
    const int64_t units = (n + 16 * kProjKb - 1) / (16 * kProjKb);
    const int64_t gmax = std::max(1, std::min(max_blocks, (NT == 1 ? 2 : 1) * sms / gy));
    const int64_t per = (units + gmax - 1) / gmax;
    const int gx = (int)((units + per - 1) / per);
    *nb = gx;
    const dim3 grid(gx, gy);
    (void)RG;
    if (NT == 1) k_proj64<1><<<grid, 256, proj64_smem(1), s>>>(V, ldv, cols, vexp, W, ldw, p, wexp, n, part, CG, only);
    else if (NT == 2) k_proj64<2><<<grid, 256, proj64_smem(2), s>>>(V, ldv, cols, vexp, W, ldw, p, wexp, n, part, CG, only);
    else k_proj64<4><<<grid, 256, proj64_smem(4), s>>>(V, ldv, cols, vexp, W, ldw, p, wexp, n, part, CG, only);
    return cudaGetLastError();
}

cudaError_t launch_colmax(const double* W, int64_t ldw, int p, int64_t n, int* wexp, int* zero0, int n0, int* zero1, int n1,
                          cudaStream_t s) {
    const int gx = (int)std::min<int64_t>((n + 1023) / 1024, 256);
    k_colmax<<<dim3(gx, p), 256, 0, s>>>(W, ldw, n, wexp, zero0, n0, zero1, n1);
    return cudaGetLastError();
}

bool mma_fit(int mp, int p) {
    const int NT = p <= 8 ? 1 : p <= 16 ? 2 : 4;
    return p >= 1 && p <= kMaxP && upd_smem(mp, NT, 4, true) <= 220 * 1024;
}

bool updz_mma_fit(int cols, int p) {
    const int NT = p <= 8 ? 1 : p <= 16 ? 2 : 4;
    return p >= 1 && p <= kMaxP && upd_smem(cols, NT, 8, false) <= 220 * 1024;
}

bool mma64_fit(int mp, int p) { return updz_mma_fit(mp + p, p); }

cudaError_t launch_pack_block(const double* V, float* V32, int64_t ld, int64_t n, int p, int* colexp, const int* skip,
                              cudaStream_t s) {
    for (int c = 0; c < p; c += 1024) k_zero_int<<<1, 1024, 0, s>>>(colexp + c, std::min(1024, p - c), skip);
    const int gx = (int)std::min<int64_t>((n + 255) / 256, 512);
    k_pack_block<<<dim3(gx, p), 256, 0, s>>>(V, V32, ld, n, colexp, skip);
    return cudaGetLastError();
}

cudaError_t mma_set_smem_limits() {
    cudaError_t e = cudaSuccess;
#define EXPM_SET(K) \
    if (e == cudaSuccess) e = cudaFuncSetAttribute(K, cudaFuncAttributeMaxDynamicSharedMemorySize, 224 * 1024)
    EXPM_SET((k_proj_mma<4, 2>));
    EXPM_SET((k_upd_mma<1, 7, 4, U_GS>)); EXPM_SET((k_upd_mma<2, 7, 4, U_GS>)); EXPM_SET((k_upd_mma<4, 7, 4, U_GS>));
    EXPM_SET((k_upd_mma<1, 7, 8, U_Z>)); EXPM_SET((k_upd_mma<2, 7, 8, U_Z>)); EXPM_SET((k_upd_mma<4, 7, 8, U_Z>));
    EXPM_SET((k_upd_mma<1, 8, 8, U_GS64>)); EXPM_SET((k_upd_mma<2, 8, 8, U_GS64>)); EXPM_SET((k_upd_mma<4, 8, 8, U_GS64>));
    EXPM_SET((k_upd_mma<1, 8, 8, U_Z64>)); EXPM_SET((k_upd_mma<2, 8, 8, U_Z64>)); EXPM_SET((k_upd_mma<4, 8, 8, U_Z64>));
    EXPM_SET((k_upd_mma<1, 8, 8, U_MUL64>)); EXPM_SET((k_upd_mma<2, 8, 8, U_MUL64>)); EXPM_SET((k_upd_mma<4, 8, 8, U_MUL64>));
#undef EXPM_SET
#define EXPM_SET(NT) \
    if (e == cudaSuccess) e = cudaFuncSetAttribute(k_proj64<NT>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)proj64_smem(NT))
    EXPM_SET(1);
    EXPM_SET(2);
    EXPM_SET(4);
#undef EXPM_SET
    return e;
}

}  // namespace expm
