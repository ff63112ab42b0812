// k_transform.cu -- the FP32 sine transforms of the mixed path's exact inverse on the tensor cores.
//
// Every transform is a tall product C[m, n] = sum_k A[m, k] Q[k, n], A the n p grid values (M rows of
// one block column, K along the transformed axis) and Q the K x N table shared by all.  In FP32 on
// the CUDA cores it was bound by issue slots (two shared-memory loads and address arithmetic per 8
// FMAs, ~28 TFLOP/s); its memory floor is 8 bytes per grid value.  Here both operands are split into
// three bf16 parts (24 bits together) and the six products above 2^-25 run on mma.sync; the sums of
// v0 q0 and of the five smaller products are separate accumulators, and the first is added to a third
// every 64 of K where K passes 128, so the result is at least as accurate as the FP32 FMA chain it
// replaces (relative rms against 64 bits on normal data,
// chain and this kernel: K = 31 1.0e-7 4.5e-8, 96 1.8e-7 6.9e-8, 256 2.9e-7 8.0e-8, 1300 6.5e-7 1.1e-7).
//
// A goes from global memory to fragments through a ring of shared memory that is private to each
// lane (cp.async, 16 bytes at a time, four chunks ahead across tiles; no barrier): the K index inside a
// 16-deep chunk and the row index inside a 32-row tile are permuted (lane t holds k = 4t .. 4t + 3,
// lane group g holds rows 4g .. 4g + 3), which any MMA allows as long as both operands agree.  Q is
// split once when the plan is made and stored in fragment order; a CTA keeps the slab of its 32 or 48
// columns in shared memory and its warps walk over 32-row tiles.  96^3, p = 16, all 12 transforms of a
// block step: 1.50 -> 0.92 ms (61 to 72 us each, 110 to 157 us into FP64; 8 bytes a value at 3.7 TB/s), bound now by
// dependent issue at 8 to 12 warps per SM and 48 % of the mma.sync rate.
//
//   IN_M  (rows contiguous in A)        OUT_M (rows contiguous in C): Q is the left operand (M = n)
//   IN_K  (k contiguous in A)           OUT_N (n contiguous in C):    A is the left operand (M = m)
#include <algorithm>
#include <type_traits>

#include "df.cuh"
#include "internal.h"
#include "mma.cuh"

namespace expm {
namespace {

enum { T_IN_M_OUT_M = 0, T_IN_K_OUT_M = 1, T_IN_M_OUT_N = 2 };

__device__ __forceinline__ int64_t row_off(int m, int ms, int64_t rs, int64_t ms2) {
    return ms ? (int64_t)(m % ms) * rs + (int64_t)(m / ms) * ms2 : (int64_t)m * rs;
}
__device__ __forceinline__ void cp16(uint32_t dst, const float* src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
}
__device__ __forceinline__ void cp4(uint32_t dst, const float* src) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(dst), "l"(src) : "memory");
}

constexpr int kNoFlush = 128;        // K up to which the main sums need no flush
constexpr int kRing = 4;             // chunks of A in flight per warp
constexpr int kTrThreads = 128;
constexpr size_t kRingBytes = (size_t)kRing * 4 * kTrThreads * sizeof(float4);
constexpr size_t slab_bytes(int K, int NTS) { return (size_t)((K + 15) / 16) * NTS * 1536; }

// VA / vc: A's groups of four and C's pairs are aligned and never straddle a run.  FL: the main sums
// are flushed every 64 of K (longer axes); short axes keep one accumulator less and a third CTA per SM.
// NTS: 16-column tiles of C per warp (a 16 x 32 chunk of A is split once for NTS tiles; the splitting
// and addressing take more issue slots than the MMAs).
template <int VAR, typename TC, int NTS, bool VA, bool FL>
__global__ void __launch_bounds__(kTrThreads, VA ? 3 : 2) k_transform(TransformArgs g, int batch, int qsm, int vc,
                                                                        const float* add_to, int64_t add_b) {
    extern __shared__ __align__(16) unsigned char smt[];
    const int tid = threadIdx.x, lane = tid & 31, gq = lane >> 2, t = lane & 3;
    const int nt16 = (g.N + 15) >> 4, nt0 = blockIdx.y * NTS, nts = min(NTS, nt16 - nt0);
    const int mtiles = (g.M + 31) >> 5, jobs = mtiles * batch, jstep = gridDim.x * (kTrThreads / 32);
    const int nkc = (g.K + 15) >> 4;
    uint4* Qs = reinterpret_cast<uint4*>(smt);                      // [kc][nts][part][lane]
    float4* ring = reinterpret_cast<float4*>(smt + (qsm ? (size_t)nkc * NTS * 1536 : 0)) + tid;   // [stage][4][thread]
    const uint32_t ring_s = (uint32_t)__cvta_generic_to_shared(ring);
    const float* Abase = reinterpret_cast<const float*>(g.A);

    // the next chunk to copy: job ij, chunk ik, with the offsets of this lane's rows
    int ij = blockIdx.x * (kTrThreads / 32) + (tid >> 5), ik = 0;
    int64_t off[4];
    const float* Ai = nullptr;
    auto aim = [&]() {
        const int bb = ij / mtiles, m0 = (ij - bb * mtiles) * 32;
        Ai = Abase + (int64_t)bb * g.a_b;
        if constexpr (VAR == T_IN_K_OUT_M) {
#pragma unroll
            for (int e = 0; e < 4; ++e) off[e] = row_off(min(m0 + gq + 8 * e, g.M - 1), g.ms, g.a_rs, g.a_ms2);
        } else if constexpr (VA) {
            off[0] = row_off(min(m0 + 4 * gq, (g.M - 1) & ~3), g.ms, g.a_rs, g.a_ms2);
        } else {
#pragma unroll
            for (int e = 0; e < 4; ++e) off[e] = row_off(min(m0 + 4 * gq + e, g.M - 1), g.ms, g.a_rs, g.a_ms2);
        }
    };
    auto issue = [&](int stage) {
        if (ij < jobs) {
            const uint32_t dst = ring_s + (uint32_t)(stage * 4 * kTrThreads * 16);
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const uint32_t d = dst + q * kTrThreads * 16;
                if constexpr (VAR == T_IN_K_OUT_M) {
                    if constexpr (VA) {
                        cp16(d, Ai + off[q] + min(ik * 16 + 4 * t, g.K - 4));
                    } else {
#pragma unroll
                        for (int r = 0; r < 4; ++r) cp4(d + 4 * r, Ai + off[q] + min(ik * 16 + 4 * t + r, g.K - 1));
                    }
                } else {
                    const float* src = Ai + (int64_t)min(ik * 16 + 4 * t + q, g.K - 1) * g.a_cs;
                    if constexpr (VA) {
                        cp16(d, src + off[0]);
                    } else {
#pragma unroll
                        for (int r = 0; r < 4; ++r) cp4(d + 4 * r, src + off[r]);
                    }
                }
            }
            if (++ik == nkc) {
                ik = 0;
                ij += jstep;
                if (ij < jobs) aim();
            }
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    const uint4* Qg = g.Q + (size_t)nt0 * 96;
    // the slab joins the first ring group (all of it in flight at once)
    if (qsm)
        for (int e = tid; e < nkc * nts * 96; e += kTrThreads) {
            const int kc = e / (nts * 96), r = e - kc * nts * 96;
            cp16((uint32_t)__cvta_generic_to_shared(Qs + kc * NTS * 96 + r), reinterpret_cast<const float*>(Qg + (size_t)kc * nt16 * 96 + r));
        }
    if (ij < jobs) aim();
#pragma unroll
    for (int st = 0; st < kRing - 1; ++st) issue(st);
    asm volatile("cp.async.wait_group %0;" ::"n"(kRing - 2) : "memory");
    __syncthreads();
    int stage = 0;
    for (int job = blockIdx.x * (kTrThreads / 32) + (tid >> 5); job < jobs; job += jstep) {
    const int bb = job / mtiles, m0 = (job - bb * mtiles) * 32;
    TC* C = reinterpret_cast<TC*>(g.C) + (int64_t)bb * g.c_b;
    // the extra addend, in the one variant that takes it (a kernel argument of its own: inside TransformArgs it
    // changed the code of every variant, 5 % slower at 256 x 256)
    constexpr bool kAdd = VAR == T_IN_M_OUT_M && std::is_same<TC, double>::value;
    const float* add = kAdd && add_to ? add_to + (int64_t)bb * add_b : nullptr;
    float cm[NTS][4][4], cc[NTS][4][4], cs[FL ? NTS : 1][4][4];
#pragma unroll
    for (int i = 0; i < NTS; ++i)
#pragma unroll
        for (int e = 0; e < 4; ++e)
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                cm[i][e][q] = cc[i][e][q] = 0.f;
                if (FL) cs[i][e][q] = 0.f;
            }
    for (int kc = 0; kc < nkc; ++kc) {
        asm volatile("cp.async.wait_group %0;" ::"n"(kRing - 2) : "memory");
        float4 d[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) d[q] = ring[(stage * 4 + q) * kTrThreads];
        issue((stage + kRing - 1) % kRing);
        stage = (stage + 1) % kRing;
        uint32_t s[4][2][3];              // [component e][k half][part]
        if constexpr (VAR == T_IN_K_OUT_M) {
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                split3(d[e].x, d[e].y, s[e][0]);
                split3(d[e].z, d[e].w, s[e][1]);
            }
        } else {
            split3(d[0].x, d[1].x, s[0][0]);
            split3(d[2].x, d[3].x, s[0][1]);
            split3(d[0].y, d[1].y, s[1][0]);
            split3(d[2].y, d[3].y, s[1][1]);
            split3(d[0].z, d[1].z, s[2][0]);
            split3(d[2].z, d[3].z, s[2][1]);
            split3(d[0].w, d[1].w, s[3][0]);
            split3(d[2].w, d[3].w, s[3][1]);
        }
#pragma unroll
        for (int i = 0; i < NTS; ++i)
            if (i < nts) {
                uint4 q[3];
#pragma unroll
                for (int k = 0; k < 3; ++k)
                    q[k] = qsm ? Qs[(kc * NTS + i) * 96 + k * 32 + lane] : Qg[(size_t)(kc * nt16 + i) * 96 + k * 32 + lane];
#pragma unroll
                for (int pr = 0; pr < 6; ++pr) {
                    const int pa = kProdA[pr], pb = kProdB[pr];      // parts of Q and of A
#pragma unroll
                    for (int e = 0; e < 4; ++e) {
                        float* acc = pr == 0 ? cm[i][e] : cc[i][e];
                        if constexpr (VAR != T_IN_M_OUT_N) {
                            const uint32_t a[4] = {q[pa].x, q[pa].y, q[pa].z, q[pa].w};
                            mma_bf16(acc, a, s[e][0][pb], s[e][1][pb]);
                        } else {
                            // e = 2 mi + h: M tile mi (rows 4 gq + 2 mi, + 1), columns 8 h .. of the 16
                            const int mi = e >> 1, h = e & 1;
                            const uint32_t a[4] = {s[2 * mi][0][pb], s[2 * mi + 1][0][pb], s[2 * mi][1][pb],
                                                   s[2 * mi + 1][1][pb]};
                            mma_bf16(acc, a, h ? q[pa].y : q[pa].x, h ? q[pa].w : q[pa].z);
                        }
                    }
                }
            }
        if (FL && (kc & 3) == 3) {
#pragma unroll
            for (int i = 0; i < NTS; ++i)
#pragma unroll
                for (int e = 0; e < 4; ++e)
#pragma unroll
                    for (int r = 0; r < 4; ++r) {
                        cs[i][e][r] += cm[i][e][r];
                        cm[i][e][r] = 0.f;
                    }
        }
    }
#pragma unroll
    for (int i = 0; i < NTS; ++i)
#pragma unroll
        for (int e = 0; e < 4; ++e)
#pragma unroll
            for (int r = 0; r < 4; ++r) cm[i][e][r] = (FL ? cs[i][e][r] + cm[i][e][r] : cm[i][e][r]) + cc[i][e][r];
    // pairs (x, y) to consecutive elements of C; an FP64 C that is added to is read for all pairs of a
    // tile before any is written.  Row offsets of the job's rows first.
    constexpr int NR = VAR == T_IN_M_OUT_N ? 4 : 8;
    int64_t ro[NR];
#pragma unroll
    for (int k = 0; k < NR; ++k) {
        // OUT_M: rows 8t + k (IN_M) or 8 (k / 2) + 2t + k % 2 (IN_K); OUT_N: rows 4 gq + k
        const int m = m0 + (VAR == T_IN_M_OUT_M ? 8 * t + k : VAR == T_IN_K_OUT_M ? 8 * (k >> 1) + 2 * t + (k & 1) : 4 * gq + k);
        ro[k] = m < g.M ? row_off(m, g.ms, g.c_rs, g.c_ms2) : -1;
    }
#pragma unroll
    for (int i = 0; i < NTS; ++i) {
        if (i >= nts) break;
        const int nb = (nt0 + i) * 16;
        if constexpr (VAR == T_IN_M_OUT_N) {
#pragma unroll
            for (int r = 0; r < 4; ++r)
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const int n = nb + 8 * h + 2 * t;
                    const float x = cm[i][(r >> 1) * 2 + h][2 * (r & 1)], y = cm[i][(r >> 1) * 2 + h][2 * (r & 1) + 1];
                    if (ro[r] < 0 || n >= g.N) continue;
                    TC* d = C + ro[r] + n;
                    if (vc) {
                        *reinterpret_cast<float2*>(d) = make_float2(x, y);
                    } else {
                        d[0] = x;
                        if (n + 1 < g.N) d[1] = y;
                    }
                }
        } else {
#pragma unroll
            for (int hr = 0; hr < 2; ++hr) {
                const int n = nb + gq + 8 * hr;
                if (n >= g.N) continue;
                TC* Cn = C + (int64_t)n * g.c_cs;
                // row k of the list above
                auto val = [&](int k) {
                    return VAR == T_IN_M_OUT_M ? cm[i][k & 3][2 * hr + (k >> 2)] : cm[i][k >> 1][2 * hr + (k & 1)];
                };
                if constexpr (sizeof(TC) == 8) {
                    double2 o[4];
                    float2 o32[4];
#pragma unroll
                    for (int k = 0; k < 4; ++k) {
                        o[k] = make_double2(0.0, 0.0);
                        if (g.accumulate) {
                            if (vc) {
                                if (ro[2 * k] >= 0) o[k] = *reinterpret_cast<const double2*>(Cn + ro[2 * k]);
                            } else {
                                if (ro[2 * k] >= 0) o[k].x = Cn[ro[2 * k]];
                                if (ro[2 * k + 1] >= 0) o[k].y = Cn[ro[2 * k + 1]];
                            }
                        }
                        if constexpr (kAdd) o32[k] = make_float2(0.f, 0.f);
                        if (kAdd && add) {
                            const float* an = add + (int64_t)n * g.c_cs;
                            if (vc) {
                                if (ro[2 * k] >= 0) o32[k] = *reinterpret_cast<const float2*>(an + ro[2 * k]);
                            } else {
                                if (ro[2 * k] >= 0) o32[k].x = an[ro[2 * k]];
                                if (ro[2 * k + 1] >= 0) o32[k].y = an[ro[2 * k + 1]];
                            }
                        }
                    }
#pragma unroll
                    for (int k = 0; k < 4; ++k) {
                        double2 v = make_double2(f64_of_f32_i(val(2 * k)), f64_of_f32_i(val(2 * k + 1)));
                        if (kAdd && add) {
                            v.x += f64_of_f32_i(o32[k].x);
                            v.y += f64_of_f32_i(o32[k].y);
                        }
                        if (g.accumulate) {
                            v.x += o[k].x;
                            v.y += o[k].y;
                        }
                        if (vc) {
                            if (ro[2 * k] >= 0) *reinterpret_cast<double2*>(Cn + ro[2 * k]) = v;
                        } else {
                            if (ro[2 * k] >= 0) Cn[ro[2 * k]] = v.x;
                            if (ro[2 * k + 1] >= 0) Cn[ro[2 * k + 1]] = v.y;
                        }
                    }
                } else {
#pragma unroll
                    for (int k = 0; k < 4; ++k) {
                        if (vc) {
                            if (ro[2 * k] >= 0) *reinterpret_cast<float2*>(Cn + ro[2 * k]) = make_float2(val(2 * k), val(2 * k + 1));
                        } else {
                            if (ro[2 * k] >= 0) Cn[ro[2 * k]] = val(2 * k);
                            if (ro[2 * k + 1] >= 0) Cn[ro[2 * k + 1]] = val(2 * k + 1);
                        }
                    }
                }
            }
        }
    }
    }
    asm volatile("cp.async.wait_all;" ::: "memory");
}

// Q (N x N FP64, row-major [k][n]) rounded to FP32 and split, in fragment order
// [kc][nt][part][lane]: register r of lane (g, t) holds n = 16 nt + g + 8 (r & 1), k = 16 kc + 4 t +
// 2 (r >> 1) and the next; zero past N.
__global__ void k_table_frags(const double* __restrict__ Q, int N, uint4* __restrict__ F) {
    const int nt16 = (N + 15) >> 4;
    const int e = blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= nt16 * nt16 * 32) return;
    const int lane = e & 31, nt = (e >> 5) % nt16, kc = (e >> 5) / nt16, g = lane >> 2, t = lane & 3;
    uint32_t u[4][3];
#pragma unroll
    for (int r = 0; r < 4; ++r) {
        const int n = 16 * nt + g + 8 * (r & 1), k = 16 * kc + 4 * t + 2 * (r >> 1);
        const float x = (n < N && k < N) ? (float)Q[(int64_t)k * N + n] : 0.f;
        const float y = (n < N && k + 1 < N) ? (float)Q[(int64_t)(k + 1) * N + n] : 0.f;
        split3(x, y, u[r]);
    }
#pragma unroll
    for (int k = 0; k < 3; ++k) F[((size_t)(kc * nt16 + nt) * 3 + k) * 32 + lane] = make_uint4(u[0][k], u[1][k], u[2][k], u[3][k]);
}

template <int VAR, typename TC>
cudaError_t launch_var(const TransformArgs& g, int batch, int sms, cudaStream_t s, const float* add = nullptr,
                       int64_t add_b = 0) {
    // aligned groups of four of A and aligned pairs of C: strides between them multiples of 4 (2) and
    // no group crossing a run of the split row index
    auto mult = [](int64_t x, int k) { return x % k == 0; };
    const bool am = VAR == T_IN_K_OUT_M ? mult(g.a_rs, 4) && mult(g.a_ms2, 4) && mult(g.K, 4)
                                        : mult(g.a_cs, 4) && mult(g.ms, 4) && mult(g.a_ms2, 4) && mult(g.M, 4);
    const bool va = am && mult(g.a_b, 4) && (reinterpret_cast<uintptr_t>(g.A) & 15) == 0;
    const bool cmv = VAR == T_IN_M_OUT_N ? mult(g.c_rs, 2) && mult(g.c_ms2, 2) && mult(g.N, 2)
                                         : mult(g.c_cs, 2) && mult(g.ms, 2) && mult(g.c_ms2, 2) && mult(g.M, 2);
    const bool vc = cmv && mult(g.c_b, 2) && (reinterpret_cast<uintptr_t>(g.C) & (2 * sizeof(TC) - 1)) == 0 &&
                    (!add || (mult(add_b, 2) && (reinterpret_cast<uintptr_t>(add) & 7) == 0));
    // column tiles per warp: three on short axes (no flush); two on long ones, where the flush costs an
    // accumulator and the smaller 2-D problems need the warps (256 x 256, p = 8: 14 us against 29 us
    // with four tiles, 512 x 352, p = 32: 104 us against 152 us with three)
    const int nt16 = (g.N + 15) / 16;
    const bool fl = !va || g.K > kNoFlush;
    const int NTS = fl ? 2 : 3, ngroups = (nt16 + NTS - 1) / NTS;
    const int64_t jobs = (int64_t)((g.M + 31) / 32) * batch;
    if (jobs > (1 << 30)) return cudaErrorInvalidValue;
    // CTAs walk over the tiles (the slab is staged once), as many as are resident, evenly loaded
    const int qsm = slab_bytes(g.K, NTS) + kRingBytes <= 224 * 1024 ? 1 : 0;
    const size_t shm = kRingBytes + (qsm ? slab_bytes(g.K, NTS) : 0);
    const int64_t resident = std::min<int64_t>(va ? 3 : 2, 224 * 1024 / (int64_t)shm) * sms;
    const int64_t gmax = std::max<int64_t>(1, std::min((jobs + 3) / 4, std::max<int64_t>(1, resident / ngroups)));
    const int64_t per = (jobs + 4 * gmax - 1) / (4 * gmax);
    const dim3 grid((unsigned)((jobs + 4 * per - 1) / (4 * per)), (unsigned)ngroups);
    if (!va) k_transform<VAR, TC, 2, false, true><<<grid, kTrThreads, shm, s>>>(g, batch, qsm, vc, add, add_b);
    else if (fl) k_transform<VAR, TC, 2, true, true><<<grid, kTrThreads, shm, s>>>(g, batch, qsm, vc, add, add_b);
    else k_transform<VAR, TC, 3, true, false><<<grid, kTrThreads, shm, s>>>(g, batch, qsm, vc, add, add_b);
    return cudaGetLastError();
}

template <int VAR, typename TC>
cudaError_t set_var_smem() {
    cudaError_t e = cudaSuccess;
#define EXPM_SET(...) \
    if (e == cudaSuccess) \
        e = cudaFuncSetAttribute(k_transform<VAR, TC, __VA_ARGS__>, cudaFuncAttributeMaxDynamicSharedMemorySize, 225 * 1024)
    EXPM_SET(2, false, true);
    EXPM_SET(2, true, true);
    EXPM_SET(3, true, false);
#undef EXPM_SET
    return e;
}

}  // namespace

size_t table_frag_count(int N) {
    const size_t nt = (size_t)(N + 15) / 16;
    return nt * nt * 96;
}

cudaError_t launch_table_frags(const double* Q, int N, uint4* F, cudaStream_t s) {
    const int nt = (N + 15) / 16, tot = nt * nt * 32;
    k_table_frags<<<(tot + 127) / 128, 128, 0, s>>>(Q, N, F);
    return cudaGetLastError();
}

cudaError_t launch_transform(const TransformArgs& g, int batch, int sms, cudaStream_t s, const float* add, int64_t add_b) {
    // strides of one on both sides of A (an axis of one point): either reading is right, rows contiguous is taken
    const bool in_k = g.a_cs == 1 && g.a_rs != 1;
    if (add && !(g.c_rs == 1 && !in_k && g.c_f64)) return cudaErrorInvalidValue;
    if (g.c_rs == 1) {
        if (in_k)
            return g.c_f64 ? launch_var<T_IN_K_OUT_M, double>(g, batch, sms, s) : launch_var<T_IN_K_OUT_M, float>(g, batch, sms, s);
        return g.c_f64 ? launch_var<T_IN_M_OUT_M, double>(g, batch, sms, s, add, add_b) : launch_var<T_IN_M_OUT_M, float>(g, batch, sms, s);
    }
    if (g.c_cs != 1 || g.a_rs != 1 || g.c_f64) return cudaErrorInvalidValue;
    return launch_var<T_IN_M_OUT_N, float>(g, batch, sms, s);
}

cudaError_t transform_set_smem() {
    cudaError_t e = set_var_smem<T_IN_K_OUT_M, float>();
    if (e == cudaSuccess) e = set_var_smem<T_IN_K_OUT_M, double>();
    if (e == cudaSuccess) e = set_var_smem<T_IN_M_OUT_M, float>();
    if (e == cudaSuccess) e = set_var_smem<T_IN_M_OUT_M, double>();
    if (e == cudaSuccess) e = set_var_smem<T_IN_M_OUT_N, float>();
    return e;
}

}  // namespace expm
