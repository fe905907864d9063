// Plain float32 CUDA-core kernels: the reference GPU form of the hot path, and the building
// blocks every precision shares (pair tables, energy reductions).
//
// Steps (arXiv 2401.04189, "Convolution operation"):
//   k_chain         rho = psi_a psi_b (pointwise on the nodes), then modes 3 and 2 of the
//                   projection onto the shared Tucker basis (Eq. TuckerDecompField); the same
//                   chain with every term's operators gives the gradients' transposed modes
//   simt_gemm       mode 1 of the projection; mode 1 of the expansion (Eq. final) for all t
//   k_consume       modes 2 and 3 of the expansion, summed over the Gaussian terms t (Eq. final),
//                   then W -= psi_j * phi (Eq. hadam) and the weighted energy sums
#include <cuda_runtime.h>

#include <algorithm>
#include <string>

#include "tx_internal.h"
#include "tx_packed.cuh"
#include "tx_tc_common.cuh"

namespace tx {

namespace {
// ====================================================================================
// strided batched GEMM: C[b1,b2][m][n] = alpha * sum_k A[m][k] B[k][n] (+ C)
// BM x BN tiles of 256 threads, each (BM / 16) x (BN / 16) outputs; 16-deep K slices, two
// shared-memory buffers, the next slice in registers while one is multiplied.  Bound by the
// float32 pipes where M, N >= 128 (an 8 x 8 thread tile reads four 16-byte fragments for 64
// multiply-adds); the host picks the tile with the least padding.
// ====================================================================================
constexpr int GK = 16;

// how a tile operand lies in memory: element (row, k) at row * s_row + k * s_k
enum : int { GL_SCALAR_K = 0, GL_SCALAR_R = 1, GL_VEC_K = 2, GL_VEC_R = 3 };

// one BR x GK slice into registers (zero outside R x K)
template <int BR>
__device__ __forceinline__ void gemm_fetch(const float* __restrict__ P, long s_row, long s_k, int r0, int k0, int R, int K,
                                           int mode, float (&v)[BR * GK / 256]) {
    constexpr int NE = BR * GK / 256;
    const int tid = threadIdx.x;
    if constexpr (NE >= 4) {
        if (mode == GL_VEC_R) {
#pragma unroll
            for (int i = 0; i < NE / 4; ++i) {
                const int e = i * 256 + tid, r = r0 + 4 * (e % (BR / 4)), k = k0 + e / (BR / 4);
                const float4 q = (r < R && k < K) ? *(const float4*)(P + r + k * s_k) : make_float4(0.f, 0.f, 0.f, 0.f);
                v[4 * i] = q.x; v[4 * i + 1] = q.y; v[4 * i + 2] = q.z; v[4 * i + 3] = q.w;
            }
            return;
        }
        if (mode == GL_VEC_K) {
#pragma unroll
            for (int i = 0; i < NE / 4; ++i) {
                const int e = i * 256 + tid, r = r0 + e / (GK / 4), k = k0 + 4 * (e % (GK / 4));
                const float4 q = (r < R && k < K) ? *(const float4*)(P + r * s_row + k) : make_float4(0.f, 0.f, 0.f, 0.f);
                v[4 * i] = q.x; v[4 * i + 1] = q.y; v[4 * i + 2] = q.z; v[4 * i + 3] = q.w;
            }
            return;
        }
    }
    const bool kfast = mode == GL_SCALAR_K || mode == GL_VEC_K;
#pragma unroll
    for (int i = 0; i < NE; ++i) {
        const int e = i * 256 + tid;
        const int r = r0 + (kfast ? e / GK : e % BR), k = k0 + (kfast ? e % GK : e / BR);
        v[i] = (r < R && k < K) ? P[r * s_row + k * s_k] : 0.f;
    }
}

template <int BR>
__device__ __forceinline__ void gemm_stash(float* __restrict__ S, int mode, const float (&v)[BR * GK / 256]) {
    constexpr int NE = BR * GK / 256, LD = BR + 4;
    const int tid = threadIdx.x;
    if constexpr (NE >= 4) {
        if (mode == GL_VEC_R) {
#pragma unroll
            for (int i = 0; i < NE / 4; ++i) {
                const int e = i * 256 + tid;
                *(float4*)(S + (e / (BR / 4)) * LD + 4 * (e % (BR / 4))) =
                    make_float4(v[4 * i], v[4 * i + 1], v[4 * i + 2], v[4 * i + 3]);
            }
            return;
        }
        if (mode == GL_VEC_K) {
#pragma unroll
            for (int i = 0; i < NE / 4; ++i) {
                const int e = i * 256 + tid, r = e / (GK / 4), k = 4 * (e % (GK / 4));
#pragma unroll
                for (int q = 0; q < 4; ++q) S[(k + q) * LD + r] = v[4 * i + q];
            }
            return;
        }
    }
    const bool kfast = mode == GL_SCALAR_K || mode == GL_VEC_K;
#pragma unroll
    for (int i = 0; i < NE; ++i) {
        const int e = i * 256 + tid;
        S[(kfast ? e % GK : e / BR) * LD + (kfast ? e / GK : e % BR)] = v[i];
    }
}

// element i of thread t's share of a tile side of 16 * W elements: groups of min(W, 4)
// neighbours, so that fragments are read with one instruction per group
template <int W>
__device__ __forceinline__ int gemm_index(int t, int i) {
    if constexpr (W == 8) return 4 * t + (i & 3) + 64 * (i >> 2);
    return W * t + i;
}

template <int BM, int BN>
__global__ void __launch_bounds__(256, BM * BN >= 8192 ? 2 : 3) k_gemm(GemmArgs g, int modeA, int modeB, int vecC) {
    constexpr int TM = BM / 16, TN = BN / 16;
    __shared__ __align__(16) float As[2][GK * (BM + 4)];
    __shared__ __align__(16) float Bs[2][GK * (BN + 4)];
    const int b = blockIdx.z;
    const int b1 = b % g.nb1, b2 = b / g.nb1;
    const float* A = g.A + b1 * g.a_b1 + b2 * g.a_b2;
    const float* B = g.B + b1 * g.b_b1 + b2 * g.b_b2;
    float* C = g.C + b1 * g.c_b1 + b2 * g.c_b2;
    const int m0 = blockIdx.y * BM, n0 = blockIdx.x * BN;
    const int tm = threadIdx.x >> 4, tn = threadIdx.x & 15;
    uint64_t acc[TM][TN / 2];
#pragma unroll
    for (int i = 0; i < TM; ++i)
#pragma unroll
        for (int j = 0; j < TN / 2; ++j) acc[i][j] = 0ull;
    float ra[BM * GK / 256], rb[BN * GK / 256];
    gemm_fetch<BM>(A, g.a_m, g.a_k, m0, 0, g.M, g.K, modeA, ra);
    gemm_fetch<BN>(B, g.b_n, g.b_k, n0, 0, g.N, g.K, modeB, rb);
    int buf = 0;
    for (int k0 = 0; k0 < g.K; k0 += GK, buf ^= 1) {
        gemm_stash<BM>(As[buf], modeA, ra);
        gemm_stash<BN>(Bs[buf], modeB, rb);
        __syncthreads();
        if (k0 + GK < g.K) {
            gemm_fetch<BM>(A, g.a_m, g.a_k, m0, k0 + GK, g.M, g.K, modeA, ra);
            gemm_fetch<BN>(B, g.b_n, g.b_k, n0, k0 + GK, g.N, g.K, modeB, rb);
        }
        const float* as = As[buf];
        const float* bs = Bs[buf];
#pragma unroll
        for (int kk = 0; kk < GK; ++kk) {
            float a[TM];
            uint64_t bb[TN / 2];
#pragma unroll
            for (int i = 0; i < TM; i += (TM < 4 ? TM : 4)) {
                const float* p = as + kk * (BM + 4) + gemm_index<TM>(tm, i);
                if constexpr (TM >= 4) {
                    const float4 q = *(const float4*)p;
                    a[i] = q.x; a[i + 1] = q.y; a[i + 2] = q.z; a[i + 3] = q.w;
                } else {
                    const float2 q = *(const float2*)p;
                    a[i] = q.x; a[i + 1] = q.y;
                }
            }
#pragma unroll
            for (int j = 0; j < TN; j += (TN < 4 ? TN : 4)) {
                const float* p = bs + kk * (BN + 4) + gemm_index<TN>(tn, j);
                if constexpr (TN >= 4) {
                    const ulonglong2 q = *(const ulonglong2*)p;
                    bb[j / 2] = q.x; bb[j / 2 + 1] = q.y;
                } else {
                    bb[j / 2] = *(const uint64_t*)p;
                }
            }
#pragma unroll
            for (int i = 0; i < TM; ++i) {
                const uint64_t ai = dup2(a[i]);
#pragma unroll
                for (int j = 0; j < TN / 2; ++j) fma2(acc[i][j], ai, bb[j]);
            }
        }
        // the other buffer was last read one slice ago, before this slice's barrier
    }
    if (g.split) {
        // hi + lo parts straight from the accumulators into the tiles that the converter kernel copies
        const int ke = g.split == 1 ? 8 : 16;                // elements per 32-byte K step
        const long lo = (long)g.ld_b * g.nr;                 // ld_b / ke steps of nr * ke elements
        if constexpr (TN >= 4) {
            if (g.nb % 4 == 0) {
                // four neighbouring b of one g at a time: half (TF32) or a quarter (bf16) of a K step's row
#pragma unroll
                for (int j = 0; j < TN; j += 4) {
                    const int n = n0 + gemm_index<TN>(tn, j);
                    if (n >= g.N) continue;
                    const int gg = n / g.nb, b = n - gg * g.nb, sw = ((gg >> 2) & 1) * (ke / 2);
                    const long col = b2 * g.c_b2 + (long)(b / ke) * g.nr * ke + gg * ke + ((b % ke) ^ sw);
                    const int npad = b == g.nb - 4 ? g.ld_b - g.nb : 0;      // zeros after the last b, 4 at a time
#pragma unroll
                    for (int i = 0; i < TM; ++i) {
                        const int m = m0 + gemm_index<TM>(tm, i);
                        if (m >= g.M) continue;
                        const float2 q0 = unpack2(acc[i][j / 2]), q1 = unpack2(acc[i][j / 2 + 1]);
                        const float v[4] = {g.alpha * q0.x, g.alpha * q0.y, g.alpha * q1.x, g.alpha * q1.y};
                        const long o = col + m * g.c_m;
                        if (g.split == 1) {
                            float h[4], l[4];
#pragma unroll
                            for (int k = 0; k < 4; ++k) {
                                h[k] = tc::tf32_hi(v[k]);
                                l[k] = tc::tf32_hi(v[k] - h[k]);
                            }
                            *(float4*)(g.C + o) = make_float4(h[0], h[1], h[2], h[3]);
                            *(float4*)(g.C + o + lo) = make_float4(l[0], l[1], l[2], l[3]);
                        } else {
                            __nv_bfloat16* C16 = (__nv_bfloat16*)g.C + o;
                            const __nv_bfloat162 h0 = __floats2bfloat162_rn(v[0], v[1]), h1 = __floats2bfloat162_rn(v[2], v[3]);
                            const float2 f0 = __bfloat1622float2(h0), f1 = __bfloat1622float2(h1);
                            const __nv_bfloat162 l0 = __floats2bfloat162_rn(v[0] - f0.x, v[1] - f0.y);
                            const __nv_bfloat162 l1 = __floats2bfloat162_rn(v[2] - f1.x, v[3] - f1.y);
                            *(uint2*)C16 = make_uint2(*(const uint32_t*)&h0, *(const uint32_t*)&h1);
                            *(uint2*)(C16 + lo) = make_uint2(*(const uint32_t*)&l0, *(const uint32_t*)&l1);
                        }
                        for (int k = 4; k < 4 + npad; k += 4) {
                            const int bb = b + k;
                            const long z = b2 * g.c_b2 + m * g.c_m + (long)(bb / ke) * g.nr * ke + gg * ke + ((bb % ke) ^ sw);
                            if (g.split == 1) {
                                *(float4*)(g.C + z) = *(float4*)(g.C + z + lo) = make_float4(0.f, 0.f, 0.f, 0.f);
                            } else {
                                __nv_bfloat16* C16 = (__nv_bfloat16*)g.C + z;
                                *(uint2*)C16 = *(uint2*)(C16 + lo) = make_uint2(0u, 0u);
                            }
                        }
                    }
                }
                return;
            }
        }
#pragma unroll
        for (int j = 0; j < TN; ++j) {
            const int n = n0 + gemm_index<TN>(tn, j);
            if (n >= g.N) continue;
            const int gg = n / g.nb, b = n - gg * g.nb;
            const int npad = b == g.nb - 1 ? g.ld_b - g.nb : 0;      // zeros after the last b
            const int sw = ((gg >> 2) & 1) * (ke / 2);               // rows 4-7 of 8 swap their 16-byte halves
            auto at = [&](int bb) { return (long)(bb / ke) * g.nr * ke + gg * ke + ((bb % ke) ^ sw); };
            const long col = b2 * g.c_b2 + at(b);
#pragma unroll
            for (int i = 0; i < TM; ++i) {
                const int m = m0 + gemm_index<TM>(tm, i);
                if (m >= g.M) continue;
                const float2 q = unpack2(acc[i][j / 2]);
                const float v = g.alpha * ((j & 1) ? q.y : q.x);
                const long o = col + m * g.c_m;
                if (g.split == 1) {
                    const float h = tc::tf32_hi(v);
                    g.C[o] = h;
                    g.C[o + lo] = tc::tf32_hi(v - h);
                } else {
                    const __nv_bfloat16 h = __float2bfloat16_rn(v);
                    __nv_bfloat16* C16 = (__nv_bfloat16*)g.C;
                    C16[o] = h;
                    C16[o + lo] = __float2bfloat16_rn(v - __bfloat162float(h));
                }
                for (int k = 1; k <= npad; ++k) {
                    const long z = b2 * g.c_b2 + m * g.c_m + at(b + k);
                    if (g.split == 1) g.C[z] = g.C[z + lo] = 0.f;
                    else ((__nv_bfloat16*)g.C)[z] = ((__nv_bfloat16*)g.C)[z + lo] = __float2bfloat16_rn(0.f);
                }
            }
        }
        return;
    }
#pragma unroll
    for (int i = 0; i < TM; ++i) {
        const int m = m0 + gemm_index<TM>(tm, i);
        if (m >= g.M) continue;
#pragma unroll
        for (int j = 0; j < TN; j += 2) {
            const int n = n0 + gemm_index<TN>(tn, j);
            if (n >= g.N) continue;
            const float2 q = unpack2(acc[i][j / 2]);
            float* dst = C + m * g.c_m + n * g.c_n;
            float v0 = g.alpha * q.x, v1 = g.alpha * q.y;
            if (vecC) {                       // c_n == 1, even rows and N: n + 1 is inside
                if (g.accumulate) {
                    const float2 o = *(const float2*)dst;
                    v0 += o.x;
                    v1 += o.y;
                }
                *(float2*)dst = make_float2(v0, v1);
            } else {
                *dst = g.accumulate ? *dst + v0 : v0;
                if (n + 1 < g.N) dst[g.c_n] = g.accumulate ? dst[g.c_n] + v1 : v1;
            }
        }
    }
}

struct Dims {
    int n1, n2, n3, r1, r2, r3;
};

Dims dims_of(const Shape& h) { return Dims{h.n1, h.n2, h.n3, h.r1, h.r2, h.r3}; }

// ====================================================================================
// pair tables
// ====================================================================================
__global__ void k_build_pairs(PairRec* recs, int mode, int role, int n_occ, int n_tgt, int k0) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n_tgt) return;
    long q = (mode == PAIRS_GENERAL) ? (long)i * n_occ : (long)i * n_occ - (long)i * (i - 1) / 2;
    const int g = k0 + i;
    for (int j = 0; j < n_occ; ++j) {
        if (mode == PAIRS_SUBSET && j >= k0 && j < g) continue;   // counted in an earlier row
        PairRec r;
        r.ia = (mode == PAIRS_SUBSET) ? g : i;
        r.ib = j;
        const bool partner = (mode == PAIRS_SUBSET) && j > g && j < k0 + n_tgt;
        if (role == ROLE_APPLY) {
            r.o0 = i; r.m0 = j; r.o1 = partner ? j - k0 : -1; r.m1 = g;
        } else if (role == ROLE_VJP_FWD) {
            r.o0 = j; r.m0 = i; r.o1 = -1; r.m1 = -1;
        } else {
            r.o0 = i; r.m0 = j; r.o1 = j; r.m1 = i;
        }
        r.ew = (mode == PAIRS_SUBSET) ? (j == g ? 1.f : 2.f) : 1.f;
        r.pad = 0;
        recs[q++] = r;
    }
}

// ====================================================================================
// modes 3 and 2 of a projection: out[p][t][x][(b,g)] = sum_{y,z} M2_t[y][b] M3_t[z][g] q_p[x][y][z]
// with q_p the product of two orbitals (times the quadrature weights where asked).  One term with
// M3 = U3, M2 = U2 is the projection onto the core; the Gaussian terms' A_t3, A_t2 give the
// adjoint's first two modes.  One CTA per (x, pair): the plane's product is staged z-major in
// slices of PZ columns (the next slice's orbitals are already in registers), mode 3 (8 y x up to
// 8 g per thread) leaves S1[y][g] in shared memory and mode 2 (4 b x up to 8 g) reads it there.
// Bound by shared-memory reads and the float32 pipes about equally.  Pt-shaped projection (96^3,
// rank 40): 6.6 us per pair; 8.7 with 4 rows per thread and no prefetch, 16.3 with one output per thread.
// ====================================================================================
constexpr int kRows = 8;           // rows per thread of the tall thread tiles
constexpr int PZ = 16;             // z columns per slice

// acc[c] += A[k][8 rows] * B[k][CL c], both K-major in shared memory
template <int CL, int RG, int NA>
__device__ __forceinline__ void panel8(const float* __restrict__ A, int lda, const float* __restrict__ B, int ldb, int K,
                                       uint64_t (&acc)[NA][4]) {
#pragma unroll 2
    for (int k = 0; k < K; ++k) {
        const ulonglong2 a = *(const ulonglong2*)(A + k * lda), a2 = *(const ulonglong2*)(A + k * lda + 4);
#pragma unroll
        for (int c = 0; c < RG; ++c) {
            const uint64_t b = dup2(B[k * ldb + CL * c]);
            fma2(acc[c][0], a.x, b);
            fma2(acc[c][1], a.y, b);
            fma2(acc[c][2], a2.x, b);
            fma2(acc[c][3], a2.y, b);
        }
    }
}
// the same for rg column groups, rg <= NA (a runtime value: every warp takes the same branch); seven groups run as
// eight, the last on values that lie behind the row and are not stored
template <int CL, int NA>
__device__ __forceinline__ void panel8_any(int rg, const float* A, int lda, const float* B, int ldb, int K,
                                           uint64_t (&acc)[NA][4]) {
    if (rg == 1) panel8<CL, 1>(A, lda, B, ldb, K, acc);
    else if (rg == 2) panel8<CL, 2>(A, lda, B, ldb, K, acc);
    else if (rg == 3) panel8<CL, 3>(A, lda, B, ldb, K, acc);
    else if (NA == 4 || rg == 4) panel8<CL, 4>(A, lda, B, ldb, K, acc);
    else if (NA == 5 || rg == 5) panel8<CL, NA < 5 ? 4 : 5>(A, lda, B, ldb, K, acc);
    else if (rg == 6) panel8<CL, NA < 6 ? 4 : 6>(A, lda, B, ldb, K, acc);
    else panel8<CL, NA < 8 ? 4 : 8>(A, lda, B, ldb, K, acc);
}

// s[c] += sum_k M[k][4 b] * S[k][col[c]]
template <int CB>
__device__ __forceinline__ void panel4(const float* __restrict__ M, int ldm, const float* __restrict__ S, int lds,
                                       const int (&col)[8], int K, uint64_t (&s)[8][2]) {
#pragma unroll 4
    for (int k = 0; k < K; ++k) {
        const ulonglong2 m = *(const ulonglong2*)(M + k * ldm);
#pragma unroll
        for (int c = 0; c < CB; ++c) {
            const uint64_t q = dup2(S[k * lds + col[c]]);
            fma2(s[c][0], m.x, q);
            fma2(s[c][1], m.y, q);
        }
    }
}

struct ChainArgs {
    Dims d;
    const PairRec* recs;
    int p0, nt;
    const float* SA;
    const float* SB;
    const float* M2;               // [nt][n2][r2]
    const float* M3;               // [nt][n3][r3]
    const float* w1;
    const float* w2;
    const float* w3;
    int flags;
    float* out;
    int ty, gw, bw, mh;            // y rows per tile (a multiple of 8), g (<= 64) and b (<= 256) columns per pass, M2 rows held
    int zq;                        // z columns of the product held: PZ (a slice), or n3 (the whole plane, over every term)
    int ldy, ldg, lds, ldb, vec;   // row strides of the product, M3, S1 and M2; vec: 16-byte orbital rows
    int flat3, flat2;              // M3 / M2 tiles are contiguous runs of whole 16-byte pieces
    int bg;                        // 1: out[b][g] (the float32 consumer's order), 0: out[g][b]
};

__global__ void __launch_bounds__(384) k_chain(const ChainArgs a) {
    extern __shared__ __align__(16) float sm[];
    const Dims d = a.d;
    float* qs = sm;                            // [zq][ldy]   the pair product, z-major
    float* m2s = qs + a.zq * a.ldy;            // [mh][ldb]
    float* m3s = m2s + a.mh * a.ldb;           // [zq][ldg]
    float* s1 = m3s + ((a.zq * a.ldg + 3) & ~3);   // [ty][lds]
    const int x = blockIdx.x, pl = blockIdx.y, tid = threadIdx.x, nth = blockDim.x;
    const bool plain = (a.flags & PROD_PLAIN) != 0;
    const PairRec rec = plain ? PairRec{} : a.recs[a.p0 + pl];
    const long N3 = (long)d.n1 * d.n2 * d.n3;
    const float* pa = a.SA + (plain ? pl : rec.ia) * N3 + (long)x * d.n2 * d.n3;
    const float* pb = plain ? pa : a.SB + rec.ib * N3 + (long)x * d.n2 * d.n3;
    const bool mulw = (a.flags & PROD_MULW) != 0, whole = a.zq > PZ, m2_tile = a.mh >= a.ty && d.r2 <= a.bw;
    const bool pre3 = whole && m2_tile && a.gw >= d.r3;           // the next term's M3 is loaded one stage ahead
    const float wx = mulw ? a.w1[x] : 1.f;
    const int tz = tid & 7, row0 = kRows * (tid >> 3);
    const int nbq = a.bw / 4, ngt = nth / nbq;                    // mode 2: 4 b per thread
    // the index that out has fastest runs along the lanes
    const int bq = a.bg ? tid / ngt : tid % nbq, gq = a.bg ? tid % ngt : tid / nbq;
    const bool act2 = a.bg ? bq < nbq : gq < ngt;
    const long og = a.bg ? 1 : d.r2, ob = a.bg ? d.r3 : 1;
    // this thread's (at most 4) 16-byte pieces of a slice, the same in every slice: 32 lanes are 16 rows
    // x 2 neighbouring pieces (whole sectors; with ldy = 4 (mod 8) the transposed stores hit 32 banks)
    const int ngr = (min(a.ty, d.n2) + 15) / 16, npc = ngr * (PZ / 8) * 32;
    int py[4], pz[4];                          // row in the tile and first column in the slice; py < 0: none
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const int e = i * nth + tid, grp = e >> 5, l = e & 31;
        py[i] = e < npc ? (grp % ngr) * 16 + (l & 15) : -1;
        pz[i] = 4 * (2 * (grp / ngr) + (l >> 4));
    }
    float4 fa[4], fb[4];
    auto fetch = [&](int y0, int yn, int z0) {
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            if (py[i] < 0 || py[i] >= yn || z0 + pz[i] >= d.n3) continue;
            const long o = (long)(y0 + py[i]) * d.n3 + z0 + pz[i];
            fa[i] = *(const float4*)(pa + o);
            fb[i] = plain ? make_float4(1.f, 1.f, 1.f, 1.f) : *(const float4*)(pb + o);
        }
    };
    // the slice z0 .. of the product into q rows [0, PZ)
    auto stage = [&](float* q0, int y0, int yn, int z0, int zn) {
        if (a.vec) {
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                if (py[i] < 0 || py[i] >= yn || z0 + pz[i] >= d.n3) continue;
                float q[4] = {fa[i].x * fb[i].x, fa[i].y * fb[i].y, fa[i].z * fb[i].z, fa[i].w * fb[i].w};
                if (mulw) {
                    const float wxy = wx * a.w2[y0 + py[i]];
#pragma unroll
                    for (int k = 0; k < 4; ++k) q[k] *= wxy * a.w3[z0 + pz[i] + k];
                }
                float* dst = q0 + pz[i] * a.ldy + py[i];
#pragma unroll
                for (int k = 0; k < 4; ++k) dst[k * a.ldy] = q[k];
            }
        } else {
            for (int e = tid; e < yn * zn; e += nth) {
                const int yy = e / zn, z = e - yy * zn;
                const long o = (long)(y0 + yy) * d.n3 + z0 + z;
                float q = plain ? pa[o] : pa[o] * pb[o];
                if (mulw) q *= wx * a.w2[y0 + yy] * a.w3[z0 + z];
                q0[z * a.ldy + yy] = q;
            }
        }
    };
    // M3 rows z0 .. z0 + zn - 1 (columns g0 .. of a pass) of term t
    auto load3 = [&](int t, int z0, int zn, int g0, int gn) {
        const float* M3 = a.M3 + ((long)t * d.n3 + z0) * d.r3;
        if (a.flat3) {
            for (int e = 4 * tid; e < zn * d.r3; e += 4 * nth) cp_async16(m3s + e, M3 + e);
        } else {
            for (int e = tid; e < zn * gn; e += nth) {
                const int z = e / gn, g = e - z * gn;
                cp_async4(m3s + z * a.ldg + g, M3 + (long)z * d.r3 + g0 + g);
            }
        }
    };
    // rows y0 + yb .. of M2 (columns b0 ..) of term t
    auto load2 = [&](int t, int y0, int yn, int b0, int bn) {
        const float* M2 = a.M2 + ((long)t * d.n2 + y0) * d.r2;
        if (a.flat2) {
            for (int e = 4 * tid; e < yn * d.r2; e += 4 * nth) cp_async16(m2s + e, M2 + e);
        } else {
            for (int e = tid; e < yn * bn; e += nth) {
                const int yy = e / bn, bb = e - yy * bn;
                cp_async4(m2s + yy * a.ldb + bb, M2 + (long)yy * d.r2 + b0 + bb);
            }
        }
    };
    for (int y0 = 0; y0 < d.n2; y0 += a.ty) {
        const int yn = min(a.ty, d.n2 - y0);
        if (whole) {                           // the tile's product once, for every term
            if (a.vec) fetch(y0, yn, 0);
            __syncthreads();                   // the previous tile's last readers
            for (int z0 = 0; z0 < d.n3; z0 += PZ) {
                stage(qs + z0 * a.ldy, y0, yn, z0, min(PZ, d.n3 - z0));
                if (a.vec && z0 + PZ < d.n3) fetch(y0, yn, z0 + PZ);
            }
        }
        for (int t = 0; t < a.nt; ++t) {
            float* out = a.out + (((long)pl * a.nt + t) * d.n1 + x) * d.r3 * d.r2;
            for (int g0 = 0; g0 < d.r3; g0 += a.gw) {
                const int gn = min(a.gw, d.r3 - g0), rg = (gn + 7) / 8;
                uint64_t acc[8][4];
#pragma unroll
                for (int c = 0; c < 8; ++c) acc[c][0] = acc[c][1] = acc[c][2] = acc[c][3] = 0ull;
                if (a.vec && !whole) fetch(y0, yn, 0);
                for (int z0 = 0; z0 < d.n3; z0 += a.zq) {
                    const int zn = min(a.zq, d.n3 - z0);
                    if (!pre3 || t == 0) {
                        __syncthreads();       // the previous slice (and S1, M2) has been read
                        if (!whole) stage(qs, y0, yn, z0, zn);
                        load3(t, z0, zn, g0, gn);
                    }
                    cp_async_wait_all();
                    __syncthreads();
                    if (z0 == 0 && m2_tile) load2(t, y0, yn, 0, d.r2);      // lands under mode 3
                    if (a.vec && !whole && z0 + PZ < d.n3) fetch(y0, yn, z0 + PZ);
                    if (row0 < a.ty) panel8_any<8>(rg, qs + row0, a.ldy, m3s + tz, a.ldg, zn, acc);
                }
                if (row0 < a.ty) {
#pragma unroll
                    for (int c = 0; c < 8; ++c)
                        if (c < rg) {
#pragma unroll
                            for (int i = 0; i < 4; ++i) {
                                const float2 u = unpack2(acc[c][i]);
                                float* p = s1 + (row0 + 2 * i) * a.lds + tz + 8 * c;
                                p[0] = u.x;
                                p[a.lds] = u.y;
                            }
                        }
                }
                // mode 2: S2[g][b] = sum_y S1[y][g] M2[y][b], this y tile's share added to the earlier ones'
                const int npass = (gn + 8 * ngt - 1) / (8 * ngt), cb = (gn + ngt * npass - 1) / (ngt * npass);
                for (int b0 = 0; b0 < d.r2; b0 += a.bw)
                    for (int gc = 0; gc < gn; gc += cb * ngt) {
                        const int bn = min(a.bw, d.r2 - b0);
                        uint64_t s[8][2];
                        int col[8];
#pragma unroll
                        for (int c = 0; c < 8; ++c) {
                            s[c][0] = s[c][1] = 0ull;
                            col[c] = min(gc + gq + c * ngt, a.lds - 1);      // past gn: a padding column, never stored
                        }
                        for (int yb = 0; yb < yn; yb += a.mh) {
                            const int ync = min(a.mh, yn - yb);
                            cp_async_wait_all();
                            __syncthreads();       // S1 (and the M2 tile) written; the previous M2 slice has been read
                            if (pre3 && gc == 0 && t + 1 < a.nt) load3(t + 1, 0, d.n3, 0, d.r3);    // lands under mode 2
                            if (!m2_tile) {
                                load2(t, y0 + yb, ync, b0, bn);
                                cp_async_wait_all();
                                __syncthreads();
                            }
                            if (act2) {
                                const float* sp = s1 + yb * a.lds;
                                const float* mp = m2s + 4 * bq;
                                switch (cb) {
                                    case 1: panel4<1>(mp, a.ldb, sp, a.lds, col, ync, s); break;
                                    case 2: panel4<2>(mp, a.ldb, sp, a.lds, col, ync, s); break;
                                    case 3: panel4<3>(mp, a.ldb, sp, a.lds, col, ync, s); break;
                                    case 4: panel4<4>(mp, a.ldb, sp, a.lds, col, ync, s); break;
                                    case 5: panel4<5>(mp, a.ldb, sp, a.lds, col, ync, s); break;
                                    case 6: panel4<6>(mp, a.ldb, sp, a.lds, col, ync, s); break;
                                    default: panel4<8>(mp, a.ldb, sp, a.lds, col, ync, s); break;
                                }
                            }
                        }
                        if (act2) {
#pragma unroll
                            for (int c = 0; c < 8; ++c) {
                                const int g = gc + gq + c * ngt;
                                if (c >= cb || g >= gn) continue;
                                const float2 u = unpack2(s[c][0]), v = unpack2(s[c][1]);
                                const float q[4] = {u.x, u.y, v.x, v.y};
                                float* o = out + (g0 + g) * og + (b0 + 4 * bq) * ob;
#pragma unroll
                                for (int k = 0; k < 4; ++k)
                                    if (4 * bq + k < bn) o[k * ob] = y0 ? o[k * ob] + q[k] : q[k];
                            }
                        }
                    }
            }
        }
    }
}

__device__ __forceinline__ double block_sum(double v, double* red) {
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    if (lane == 0) red[wid] = v;
    __syncthreads();
    double s = 0.0;
    if (threadIdx.x == 0)
        for (int i = 0; i < (int)(blockDim.x >> 5); ++i) s += red[i];
    return s;
}

// ====================================================================================
// expansion consumer: for each term t, Y_t = Z_t x2 M2_t (a tile of rows (x, y)), then
// phi += Y_t x3 M3_t; epilogue Hadamard-accumulate and energy sums.
//
// A CTA owns `rows` rows: px planes x ty y-rows.  A thread owns 8 neighbouring rows and
// RN = 4 RN4 + 2 H columns of phi (CL column lanes, 16-byte pieces 4 CL columns apart), kept in
// registers over every term.  Per term mode 2 leaves Y in shared memory (K-major) and mode 3 reads
// it back: 8 RN multiply-adds per 2 + RN4 16-byte fragments.  The next operator tiles arrive
// by cp.async under the arithmetic: M3 under mode 2, the next term's M2 and Z under mode 3.
// Ranks above a part (gc, bc) run in parts of K.
// Bound by the float32 pipes and, next, by the shared-memory reads: with 4 rows per thread the
// reads took 57% of their peak at 46% of the multiply-adds', so the thread tile is as tall as the
// registers allow (8 x 12 up to 96 columns; 16 column lanes above).  Pt-shaped pair (96^3, rank
// 40, 40 terms): 94 us (43 TF/s); 114 with 4 rows per
// thread, 461 with one output per thread.
// ====================================================================================
struct SimtPlan {
    int cl, rn2;               // column lanes, columns per thread / 2
    int ty, ny, px, nx, rows;  // y rows per plane (a multiple of 8), y tiles, planes per CTA, x slabs, rows per CTA
    int gc, bc;                // K parts of mode 3 and mode 2
    int threads;
    size_t smem;
};

struct ConsumeF32Args {
    Dims d;
    const PairRec* recs;
    int p0, nt;
    const float* Z;            // [np][nt][n1][r2][r3], or [r3][r2] slices (z_mode)
    const float* M2;           // [nt][r2][ld2], y fastest
    const float* M3;           // [nt][r3][NC], z fastest
    int ld2;
    long m2_ps, m3_ps;
    FieldArgs f;
    const float* w1;
    const float* w2;
    const float* w3;
    int flags;
    double* epart;
    int ty, px, ny, gc, bc, rows, vec;
    int m2_flat, z_mode;       // M2 part / Z part as one contiguous run (z_mode 2), Z rows of g (1) or of b (0)
    int tc;                    // terms per CTA: blockIdx.z takes terms z tc .. z tc + tc - 1 (EPI_STORE), nt otherwise
    long out_ps, out_cs;       // EPI_STORE: floats between the results of two pairs, of two term groups
};

// Registers: 8 RN for phi, 8 per mode-2 column; the K part of mode 3 (gc) is at most CL * consume_max_rg
// columns so that both fit the 168 registers that leave 12 warps per SM (255 above 12 columns).
__host__ __device__ constexpr int consume_max_rg(int cl, int rn) { return cl == 16 ? 4 : (rn > 8 ? 5 : (rn == 6 ? 6 : 8)); }
__host__ __device__ constexpr int consume_max_threads(int cl, int rn) { return rn <= 12 ? 384 : 256; }

template <int CL, int RN4, int H>
__global__ void __launch_bounds__(consume_max_threads(CL, 4 * RN4 + 2 * H)) k_consume(const ConsumeF32Args a) {
    constexpr int NC = CL * (4 * RN4 + 2 * H);         // columns of phi
    constexpr int MRG = consume_max_rg(CL, 4 * RN4 + 2 * H);
    constexpr int NP = 2 * RN4 + H;                    // packed column pairs per thread
    extern __shared__ __align__(16) float sm[];
    __shared__ double red[16];
    const Dims d = a.d;
    const int ldy = a.rows + 4, ldz = a.z_mode ? a.gc : (a.gc | 1), rgw = CL * ((a.gc + CL - 1) / CL);
    float* m2s = sm;                                   // [bc][ty]
    float* m3s = m2s + a.bc * a.ty;                    // [gc][NC]
    float* ys = m3s + a.gc * NC;                       // [rgw][ldy]
    float* zs = ys + rgw * ldy;                        // [px][bc][ldz]
    const int tid = threadIdx.x, nth = blockDim.x, lane = tid & 31, warp = tid >> 5, nw = nth >> 5;
    const int iy = blockIdx.x % a.ny, x0 = (blockIdx.x / a.ny) * a.px, pl = blockIdx.y;
    const int y0 = iy * a.ty;
    const PairRec rec = (a.flags & EPI_STORE) ? PairRec{} : a.recs[a.p0 + pl];
    const int tz = tid % CL, row0 = kRows * (tid / CL);
    const int pr = min(row0 / a.ty, a.px - 1);         // plane of this thread's rows
    const int yr = min(row0 - pr * a.ty, a.ty - kRows);    // rows past the last plane repeat valid ones (not stored)
    const long zslice = (long)d.r3 * d.r2;
    const int ng = (d.r3 + a.gc - 1) / a.gc, nb = (d.r2 + a.bc - 1) / a.bc;

    // Where the registers allow (grids of at most 48 columns, the coarse grids among them), each term is
    // summed by itself and then added to the total: two short float32 sums round less than one long one.
    constexpr bool FOLD = 4 * RN4 + 2 * H <= 6;
    uint64_t acc[kRows][NP], total[FOLD ? kRows : 1][FOLD ? NP : 1];
#pragma unroll
    for (int i = 0; i < kRows; ++i)
#pragma unroll
        for (int c = 0; c < NP; ++c) {
            acc[i][c] = 0ull;
            if constexpr (FOLD) total[i][c] = 0ull;
        }

    // M2 and Z of part (t, g part, b part)
    auto load2 = [&](int t, int gp, int bp) {
        const int g0 = gp * a.gc, gn = min(a.gc, d.r3 - g0), b0 = bp * a.bc, bn = min(a.bc, d.r2 - b0);
        const float* m2 = a.M2 + pl * a.m2_ps + ((long)t * d.r2 + b0) * a.ld2 + y0;
        if (a.m2_flat) {
            for (int e = 4 * tid; e < bn * a.ty; e += 4 * nth) cp_async16(m2s + e, m2 + e);
        } else {
            const int w = min(a.ty, a.ld2 - y0);       // ld2 is n2 rounded up to 8
            for (int k = warp; k < bn; k += nw)
                for (int q = 4 * lane; q < w; q += 128) cp_async16(m2s + k * a.ty + q, m2 + (long)k * a.ld2 + q);
        }
        for (int p = 0; p < a.px; ++p) {
            if (x0 + p >= d.n1) break;
            const float* zt = a.Z + (((long)pl * a.nt + t) * d.n1 + x0 + p) * zslice;
            float* zd = zs + p * a.bc * ldz;
            if (a.z_mode == 2) {
                zt += (long)b0 * d.r3;
                for (int e = 4 * tid; e < bn * d.r3; e += 4 * nth) cp_async16(zd + e, zt + e);
            } else if (a.z_mode == 1) {
                zt += (long)b0 * d.r3 + g0;
                for (int b = warp; b < bn; b += nw)
                    for (int g = lane; g < gn; g += 32) cp_async4(zd + b * ldz + g, zt + (long)b * d.r3 + g);
            } else {                                   // the odd row stride spreads the transposed stores over the banks
                zt += (long)g0 * d.r2 + b0;
                for (int g = warp; g < gn; g += nw)
                    for (int b = lane; b < bn; b += 32) cp_async4(zd + b * ldz + g, zt + (long)g * d.r2 + b);
            }
        }
        cp_async_commit();
    };
    auto load3 = [&](int t, int gp) {
        const int g0 = gp * a.gc, gn = min(a.gc, d.r3 - g0);
        const float* m3 = a.M3 + pl * a.m3_ps + ((long)t * d.r3 + g0) * NC;
        for (int e = 4 * tid; e < gn * NC; e += 4 * nth) cp_async16(m3s + e, m3 + e);
        cp_async_commit();
    };

    const int t0 = blockIdx.z * a.tc, t1 = min(a.nt, t0 + a.tc);
    load2(t0, 0, 0);
    for (int t = t0; t < t1; ++t)
        for (int gp = 0; gp < ng; ++gp) {
            const int gn = min(a.gc, d.r3 - gp * a.gc), rg = (gn + CL - 1) / CL;
            uint64_t y[MRG][4];
#pragma unroll
            for (int c = 0; c < MRG; ++c) y[c][0] = y[c][1] = y[c][2] = y[c][3] = 0ull;
            for (int bp = 0; bp < nb; ++bp) {
                cp_async_wait_all();
                __syncthreads();               // M2 and Z have landed; the previous mode 3 is done
                if (bp == 0) load3(t, gp);
                panel8_any<CL>(rg, m2s + yr, a.ty, zs + pr * a.bc * ldz + tz, ldz, min(a.bc, d.r2 - bp * a.bc), y);
                if (bp + 1 < nb) {
                    __syncthreads();
                    load2(t, gp, bp + 1);
                }
            }
#pragma unroll
            for (int c = 0; c < MRG; ++c)
                if (c < rg) {
                    float* p = ys + (tz + CL * c) * ldy + row0;
                    *(ulonglong2*)p = make_ulonglong2(y[c][0], y[c][1]);
                    *(ulonglong2*)(p + 4) = make_ulonglong2(y[c][2], y[c][3]);
                }
            cp_async_wait_all();
            __syncthreads();                   // Y and M3 are there, M2 and Z free
            if (gp + 1 < ng) load2(t, gp + 1, 0);
            else if (t + 1 < t1) load2(t + 1, 0, 0);
#pragma unroll 2
            for (int g = 0; g < gn; ++g) {
                const float4 ya = *(const float4*)(ys + g * ldy + row0), yb = *(const float4*)(ys + g * ldy + row0 + 4);
                uint64_t b[NP];
#pragma unroll
                for (int c = 0; c < RN4; ++c) {
                    const ulonglong2 q = *(const ulonglong2*)(m3s + g * NC + 4 * tz + 4 * CL * c);
                    b[2 * c] = q.x;
                    b[2 * c + 1] = q.y;
                }
                if constexpr (H) b[2 * RN4] = *(const uint64_t*)(m3s + g * NC + 4 * CL * RN4 + 2 * tz);
                const float yv[kRows] = {ya.x, ya.y, ya.z, ya.w, yb.x, yb.y, yb.z, yb.w};
#pragma unroll
                for (int i = 0; i < kRows; ++i) {
                    const uint64_t yi = dup2(yv[i]);
#pragma unroll
                    for (int c = 0; c < NP; ++c) fma2(acc[i][c], yi, b[c]);
                }
            }
            if constexpr (FOLD)
                if (gp + 1 == ng)
#pragma unroll
                    for (int i = 0; i < kRows; ++i)
#pragma unroll
                        for (int c = 0; c < NP; ++c) {
                            total[i][c] = add2(total[i][c], acc[i][c]);
                            acc[i][c] = 0ull;
                        }
        }
    // epilogue
    const long N3 = (long)d.n1 * d.n2 * d.n3;
    double e = 0.0;
    const int x = x0 + pr;
    const bool rows_ok = row0 < a.px * a.ty && x < d.n1;
    const bool o0 = (a.flags & EPI_OUT) && rec.o0 >= 0 && a.f.OUT0, o1 = (a.flags & EPI_OUT) && rec.o1 >= 0 && a.f.OUT1;
    const float* mul0 = a.f.MUL0 + rec.m0 * N3;
    const float* mul1 = a.f.MUL1 + rec.m1 * N3;
    float* out0 = a.f.OUT0 + rec.o0 * N3;
    float* out1 = a.f.OUT1 + rec.o1 * N3;
    // a coarse grid has no weights (they are null)
    const bool weighted = (a.flags & (EPI_MULW | EPI_ENERGY)) != 0;
    const float wx = weighted && x < d.n1 ? a.w1[x] : 0.f;
#pragma unroll
    for (int i = 0; i < kRows; ++i) {
        const int y = y0 + yr + i;
        if (!rows_ok || y >= d.n2) continue;
        const float wxy = weighted ? wx * a.w2[y] : 0.f;
        const long base = ((long)x * d.n2 + y) * d.n3;
#pragma unroll
        for (int c = 0; c < NP; ++c) {
            const int z = c < 2 * RN4 ? 4 * CL * (c / 2) + 4 * tz + 2 * (c & 1) : 4 * CL * RN4 + 2 * tz;
            float2 ph;
            if constexpr (FOLD) ph = unpack2(total[i][c]);
            else ph = unpack2(acc[i][c]);
            const float phi[2] = {ph.x, ph.y};
            if (a.flags & EPI_STORE) {
                float* dst = a.f.OUT0 + pl * a.out_ps + blockIdx.z * a.out_cs + base + z;
                if (z < d.n3) dst[0] = phi[0];
                if (z + 1 < d.n3) dst[1] = phi[1];
                continue;
            }
            if (a.vec && z < d.n3) {           // even n3: the pair z, z + 1 is inside and 8-byte aligned
                float f[2] = {phi[0], phi[1]};
                if (a.flags & EPI_MULW) {
                    f[0] *= wxy * a.w3[z];
                    f[1] *= wxy * a.w3[z + 1];
                }
                if (o0) {
                    const float2 m = *(const float2*)(mul0 + base + z);
                    atomicAdd((float2*)(out0 + base + z), make_float2(-m.x * f[0], -m.y * f[1]));
                }
                if (o1) {
                    const float2 m = *(const float2*)(mul1 + base + z);
                    atomicAdd((float2*)(out1 + base + z), make_float2(-m.x * f[0], -m.y * f[1]));
                }
            } else if (!a.vec) {
#pragma unroll
                for (int k = 0; k < 2; ++k) {
                    if (z + k >= d.n3) continue;
                    const float f = (a.flags & EPI_MULW) ? phi[k] * (wxy * a.w3[z + k]) : phi[k];
                    if (o0) atomicAdd(out0 + base + z + k, -mul0[base + z + k] * f);
                    if (o1) atomicAdd(out1 + base + z + k, -mul1[base + z + k] * f);
                }
            }
            if (a.flags & EPI_ENERGY) {
#pragma unroll
                for (int k = 0; k < 2; ++k) {
                    if (z + k >= d.n3) continue;
                    const long o = base + z + k;
                    e += (double)(wxy * a.w3[z + k]) * (double)a.f.SA[rec.ia * N3 + o] * (double)a.f.SB[rec.ib * N3 + o] *
                         (double)phi[k];
                }
            }
        }
    }
    if (a.flags & EPI_ENERGY) {
        const double s = block_sum(e * rec.ew, red);
        if (tid == 0) a.epart[(long)pl * gridDim.x + blockIdx.x] = s;
    }
}

// out[p][e] = sum_c part[p][c][e], the groups of terms in their order
__global__ void __launch_bounds__(256) k_sum_groups(const float* __restrict__ part, long ps, long cs, int nc, long N,
                                                    float* __restrict__ out) {
    const long e = blockIdx.x * 256L + threadIdx.x;
    if (e >= N) return;
    const float* q = part + blockIdx.y * ps + e;
    float v = q[0];
    for (int c = 1; c < nc; ++c) v += q[c * cs];
    out[blockIdx.y * N + e] = v;
}

// dst[t][k][i] (row stride ld, zero past n) = src[t][i][k]: operators with the grid index fastest
__global__ void k_kmajor(const float* __restrict__ src, int nt, int n, int r, int ld, float* __restrict__ dst) {
    const long e = (long)blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= (long)nt * r * ld) return;
    const int i = (int)(e % ld), k = (int)((e / ld) % r), t = (int)(e / ((long)ld * r));
    dst[e] = i < n ? src[((long)t * n + i) * r + k] : 0.f;
}

// ====================================================================================
// float64 energy reductions in a fixed order
// ====================================================================================
__global__ void __launch_bounds__(256) k_reduce(const double* __restrict__ src, long count, double* dst) {
    __shared__ double red[8];
    double s = 0.0;
    for (long i = threadIdx.x; i < count; i += 256) s += src[i];
    const double tot = block_sum(s, red);
    if (threadIdx.x == 0) *dst = tot;
}

__global__ void k_finalize(const double* __restrict__ batches, int nb, double scale, double* e_dev) {
    double s = 0.0;
    for (int i = 0; i < nb; ++i) s += batches[i];
    *e_dev = scale * s;
}

// partial[b] = sum over block b's share of the flat index (i, x, y, z) of w(x, y, z) a[i] b[i]:
// float32 within groups of 32 products, float64 across groups and threads
__global__ void __launch_bounds__(256) k_weighted_dot(const float* __restrict__ A, const float* __restrict__ B,
                                                      const float* __restrict__ w1, const float* __restrict__ w2,
                                                      const float* __restrict__ w3, int n1, int n2, int n3, long total,
                                                      double* partial) {
    __shared__ double red[8];
    const long N23 = (long)n2 * n3, N3 = (long)n1 * N23;
    const long stride = (long)gridDim.x * 256;
    double s = 0.0;
    float f = 0.f;
    int cnt = 0;
    for (long i = blockIdx.x * 256L + threadIdx.x; i < total; i += stride) {
        const long r = i % N3;
        const int x = (int)(r / N23), yz = (int)(r - x * N23), y = yz / n3, z = yz - y * n3;
        f += w1[x] * w2[y] * w3[z] * A[i] * B[i];
        if (++cnt == 32) {
            s += (double)f;
            f = 0.f;
            cnt = 0;
        }
    }
    s += (double)f;
    const double tot = block_sum(s, red);
    if (threadIdx.x == 0) partial[blockIdx.x] = tot;
}

int smem_attr(const void* fn, size_t bytes) {
    if (bytes > 48 * 1024) {
        cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
        if (e != cudaSuccess) return fail(TX_ERR_CUDA, std::string("cudaFuncSetAttribute: ") + cudaGetErrorString(e));
    }
    return TX_OK;
}
}  // namespace

// ====================================================================================
// host wrappers
// ====================================================================================
namespace {
// how the tile loader may read an operand (rows along `s_row`, K along `s_k`)
int gemm_load_mode(const float* p, long s_row, long s_k, long b1, long b2, int R, int K) {
    const bool al = (((uintptr_t)p & 15u) == 0) && b1 % 4 == 0 && b2 % 4 == 0;
    if (s_row == 1) return (al && s_k % 4 == 0 && R % 4 == 0) ? GL_VEC_R : GL_SCALAR_R;
    if (s_k == 1) return (al && s_row % 4 == 0 && K % 4 == 0) ? GL_VEC_K : GL_SCALAR_K;
    return GL_SCALAR_R;
}

struct GemmTile {
    int bm, bn;
    double eff;                // share of the float32 peak a full tile reaches, relative
};
constexpr GemmTile kGemmTiles[] = {{128, 128, 1.0}, {128, 64, 0.9}, {64, 128, 0.9}, {64, 64, 0.75}, {128, 32, 0.7},
                                   {32, 128, 0.7}, {32, 64, 0.5},   {64, 32, 0.5},  {32, 32, 0.35}};
}  // namespace

int simt_gemm(const GemmArgs& g, cudaStream_t s) {
    if (g.M <= 0 || g.N <= 0 || g.K <= 0) return TX_OK;
    // the tile that wastes least on padding, and leaves at least two CTAs per SM where it can
    const GemmTile* best = nullptr;
    double best_cost = 0.0;
    for (const GemmTile& t : kGemmTiles) {
        const long tm = (g.M + t.bm - 1) / t.bm, tn = (g.N + t.bn - 1) / t.bn;
        const double ctas = (double)tm * tn * g.nb1 * g.nb2;
        const double cost = (double)(tm * t.bm) * (double)(tn * t.bn) / t.eff * (ctas < 304.0 ? 304.0 / ctas : 1.0);
        if (!best || cost < best_cost) {
            best = &t;
            best_cost = cost;
        }
    }
    const int ma = gemm_load_mode(g.A, g.a_m, g.a_k, g.a_b1, g.a_b2, g.M, g.K);
    const int mb = gemm_load_mode(g.B, g.b_n, g.b_k, g.b_b1, g.b_b2, g.N, g.K);
    const int vc = g.c_n == 1 && g.c_m % 2 == 0 && g.c_b1 % 2 == 0 && g.c_b2 % 2 == 0 && g.N % 2 == 0 &&
                   ((uintptr_t)g.C & 7u) == 0;
    const dim3 grid((g.N + best->bn - 1) / best->bn, (g.M + best->bm - 1) / best->bm, g.nb1 * g.nb2);
    const int ps = prof_begin("gemm", s);
#define TX_GEMM_CASE(BM_, BN_) \
    if (best->bm == BM_ && best->bn == BN_) k_gemm<BM_, BN_><<<grid, 256, 0, s>>>(g, ma, mb, vc)
    TX_GEMM_CASE(128, 128);
    TX_GEMM_CASE(128, 64);
    TX_GEMM_CASE(64, 128);
    TX_GEMM_CASE(64, 64);
    TX_GEMM_CASE(128, 32);
    TX_GEMM_CASE(32, 128);
    TX_GEMM_CASE(32, 64);
    TX_GEMM_CASE(64, 32);
    TX_GEMM_CASE(32, 32);
#undef TX_GEMM_CASE
    prof_end(ps, s);
    TX_LAUNCHED();
    return TX_OK;
}

long pair_count(int mode, int n_occ, int n_tgt) {
    if (mode == PAIRS_GENERAL) return (long)n_occ * n_tgt;
    return (long)n_tgt * n_occ - (long)n_tgt * (n_tgt - 1) / 2;
}

int build_pairs(PairRec* d_recs, int mode, int role, int n_occ, int n_tgt, int k0, cudaStream_t s) {
    k_build_pairs<<<(n_tgt + 127) / 128, 128, 0, s>>>(d_recs, mode, role, n_occ, n_tgt, k0);
    TX_LAUNCHED();
    return TX_OK;
}

namespace {
constexpr size_t kSmemLimit = 232448;      // 227 KB per CTA

// modes 3 and 2 of a projection for nt terms of (M3 [nt][n3][r3], M2 [nt][n2][r2])
int launch_chain(const Shape& sh, const PairRec* recs, int p0, int np, const FieldArgs& f, int nt, const float* M2,
                 const float* M3, int flags, float* out, bool bg, const char* name, cudaStream_t s) {
    ChainArgs a{};
    a.d = dims_of(sh);
    a.recs = recs; a.p0 = p0; a.nt = nt;
    a.SA = f.SA; a.SB = f.SB; a.M2 = M2; a.M3 = M3;
    a.w1 = sh.w1; a.w2 = sh.w2; a.w3 = sh.w3;
    a.flags = flags; a.out = out; a.bg = bg ? 1 : 0;
    // y tiles of at most 256 rows of equal height, one thread per row
    const int ny = (a.d.n2 + 255) / 256, tyv = (a.d.n2 + ny - 1) / ny;
    a.ty = (tyv + 7) & ~7;
    const int ngp = (a.d.r3 + 63) / 64;
    a.gw = (a.d.r3 + ngp - 1) / ngp;
    a.ldy = ((a.ty + 7) & ~7) + 4;
    a.ldg = a.gw;                              // read as scalars by neighbouring lanes: no padding needed
    a.lds = 8 * ((a.gw + 7) / 8) + 2;
    a.bw = std::min(256, pad4(a.d.r2));
    a.flat2 = a.d.r2 % 4 == 0 && a.d.r2 <= a.bw && ((uintptr_t)M2 & 15u) == 0;
    a.ldb = a.flat2 ? a.d.r2 : a.bw + 4;
    // a slice starts at a multiple of 16 rows of r3 floats; a term at a multiple of n3 r3; the slice's own length counts too
    a.flat3 = ngp == 1 && ((long)a.d.n3 * a.d.r3) % 4 == 0 && ((uintptr_t)M3 & 15u) == 0;
    a.vec = a.d.n3 % 4 == 0 && (((uintptr_t)f.SA | (uintptr_t)f.SB) & 15u) == 0;
    a.mh = (size_t)a.ty * a.ldb * sizeof(float) <= 64 * 1024 ? a.ty : 32;
    // 8 more floats behind M3: the last column group of a panel may read past its last row
    auto bytes = [&](int zq) {
        return sizeof(float) * ((size_t)zq * a.ldy + (size_t)a.mh * a.ldb + (((size_t)zq * a.ldg + 3) & ~(size_t)3) +
                                (size_t)a.ty * a.lds + 8);
    };
    // several terms: hold the whole plane's product where two CTAs still share an SM
    a.zq = nt > 1 && a.d.n3 > PZ && bytes(a.d.n3) <= kSmemLimit / 2 ? a.d.n3 : PZ;
    const size_t smem = bytes(a.zq);
    // at least 64 threads; at least one per 4 b; at most 4 pieces of a slice per thread
    const int threads = std::max(std::max(64, (a.bw / 4 + 31) & ~31), (a.ty + 31) & ~31);
    TX_TRY(smem_attr((const void*)k_chain, smem));
    const int ps = prof_begin(name, s);
    k_chain<<<dim3(a.d.n1, np), threads, smem, s>>>(a);
    prof_end(ps, s);
    TX_LAUNCHED();
    return TX_OK;
}

// The split of one pair's (x, y) rows over CTAs.  Up to 96 columns of phi take 8 column lanes of at
// most 12 columns; above, 16 lanes (of at most 12 columns up to 192).  Among the row tiles that fit
// the threads and shared memory, the one with the least padding, preferring 64 rows or more and
// shared memory that lets several CTAs share an SM (one CTA's barriers hide behind another's
// arithmetic).
bool simt_plan(const Dims& d, SimtPlan* out) {
    if (d.n3 > 256) return false;
    SimtPlan p{};
    p.cl = d.n3 <= 96 ? 8 : 16;
    p.rn2 = (d.n3 + 2 * p.cl - 1) / (2 * p.cl);
    const int rn = 2 * p.rn2, ncol = p.cl * rn, wrows = kRows * (32 / p.cl);    // rows per warp
    const int max_rows = consume_max_threads(p.cl, rn) / p.cl * kRows;
    const int gmax = p.cl * consume_max_rg(p.cl, rn);
    const int ngp = (d.r3 + gmax - 1) / gmax, nbp = (d.r2 + 63) / 64;
    p.gc = (d.r3 + ngp - 1) / ngp;
    p.bc = (d.r2 + nbp - 1) / nbp;
    const int rgw = p.cl * ((p.gc + p.cl - 1) / p.cl), ldz = p.gc | 1;
    double best = -1.0;
    for (int ny = (d.n2 + max_rows - 1) / max_rows; ny <= (d.n2 + 7) / 8; ++ny) {
        p.ny = ny;
        p.ty = (((d.n2 + ny - 1) / ny) + 7) & ~7;
        for (p.px = 1; p.px <= d.n1; ++p.px) {
            p.rows = (p.px * p.ty + wrows - 1) / wrows * wrows;
            if (p.rows > max_rows) break;
            p.nx = (d.n1 + p.px - 1) / p.px;
            p.threads = p.rows / kRows * p.cl;
            // the last column group of a panel may read up to CL floats past a Z row
            p.smem = sizeof(float) * ((size_t)p.bc * p.ty + (size_t)p.gc * ncol + (size_t)rgw * (p.rows + 4) +
                                      (size_t)p.px * p.bc * ldz + 16);
            if (p.smem > kSmemLimit) continue;
            double score = (double)d.n1 * d.n2 / ((double)p.ny * p.nx * p.rows);
            if (p.rows < 64) score *= p.rows < 32 ? 0.6 : 0.85;
            if (p.smem > kSmemLimit / 2) score *= 0.8;
            else if (p.smem > kSmemLimit / 3) score *= 0.93;
            if (score > best + 1e-9) {
                best = score;
                *out = p;
            }
        }
    }
    return best > 0.0;
}

template <int CL, int RN4, int H>
int launch_consume(const ConsumeF32Args& a, const SimtPlan& p, int np, cudaStream_t s) {
    TX_TRY(smem_attr((const void*)k_consume<CL, RN4, H>, p.smem));
    const int ps = prof_begin("consume", s);
    k_consume<CL, RN4, H><<<dim3(p.nx * p.ny, np, (a.nt + a.tc - 1) / a.tc), p.threads, p.smem, s>>>(a);
    prof_end(ps, s);
    TX_LAUNCHED();
    return TX_OK;
}

int dispatch_consume(const ConsumeF32Args& a, const SimtPlan& p, int np, cudaStream_t s) {
    if (p.cl == 8) {
        switch (p.rn2) {
            case 1: return launch_consume<8, 0, 1>(a, p, np, s);
            case 2: return launch_consume<8, 1, 0>(a, p, np, s);
            case 3: return launch_consume<8, 1, 1>(a, p, np, s);
            case 4: return launch_consume<8, 2, 0>(a, p, np, s);
            case 5: return launch_consume<8, 2, 1>(a, p, np, s);
            default: return launch_consume<8, 3, 0>(a, p, np, s);
        }
    }
    switch (p.rn2) {
        case 4: return launch_consume<16, 2, 0>(a, p, np, s);
        case 5: return launch_consume<16, 2, 1>(a, p, np, s);
        case 6: return launch_consume<16, 3, 0>(a, p, np, s);
        case 7: return launch_consume<16, 3, 1>(a, p, np, s);
        default: return launch_consume<16, 4, 0>(a, p, np, s);
    }
}
}  // namespace

int simt_project_s2(const tx_ctx* c, const PairRec* recs, int p0, int np, const FieldArgs& f, int flags,
                    float* S2, cudaStream_t s, bool bg) {
    const Shape sh = fine_shape(c);
    const Dims d = dims_of(sh);
    if (sizeof(float) * ((size_t)d.n3 * d.r3 + (size_t)d.n2 * d.r3 + 8 * (size_t)d.n3) > kSmemLimit)
        return fail(TX_ERR_CUDA, "float32 projection: (n2 + n3) * r3 too large");
    return launch_chain(sh, recs, p0, np, f, 1, c->f_U[1], c->f_U[2], flags, S2, bg, "project", s);
}

int simt_expand_consume_blocks(const Shape& sh) {
    SimtPlan p{};
    return simt_plan(dims_of(sh), &p) ? p.nx * p.ny : 1;
}

bool simt_expand_fits(const Shape& sh) {
    const Dims d = dims_of(sh);
    SimtPlan p{};
    return d.n3 <= 256 && simt_plan(d, &p) &&
           sizeof(float) * ((size_t)d.r3 * (d.r2 + 1) + 32 * (size_t)(d.r3 + 1) + (size_t)d.n3 * (d.r3 | 1)) <= kSmemLimit;
}

int simt_ld2(int n2) { return (n2 + 7) & ~7; }
int simt_ld3(int n3) {
    if (n3 > 256) return pad4(n3);             // no float32 consumer: never read
    const int cl = n3 <= 96 ? 8 : 16;
    return (n3 + 2 * cl - 1) / (2 * cl) * (2 * cl);
}

int simt_kmajor(const float* src, int nt, int n, int r, int ld, float* dst, cudaStream_t s) {
    const long cnt = (long)nt * r * ld;
    k_kmajor<<<(unsigned)((cnt + 255) / 256), 256, 0, s>>>(src, nt, n, r, ld, dst);
    TX_LAUNCHED();
    return TX_OK;
}

int simt_expand_consume(const Shape& sh, const PairRec* recs, int p0, int np, const FieldArgs& f, const float* Z,
                        int nterms, const float* M2, const float* M3, int flags, double* epart, cudaStream_t s,
                        bool z_bg, long m2_ps, long m3_ps, int group) {
    const Dims d = dims_of(sh);
    if (d.n3 > 256) return fail(TX_ERR_UNSUPPORTED_SHAPE, "float32 path supports n3 <= 256");
    SimtPlan p{};
    if (!simt_plan(d, &p) || (!(flags & EPI_STORE) && !simt_expand_fits(sh)))
        return fail(TX_ERR_CUDA, "float32 expansion: (r2 + n3) * r3 too large");
    ConsumeF32Args a{};
    a.d = d;
    a.recs = recs; a.p0 = p0; a.nt = nterms;
    a.Z = Z; a.M2 = M2; a.M3 = M3;
    a.ld2 = simt_ld2(d.n2);
    a.m2_ps = m2_ps; a.m3_ps = m3_ps;
    a.f = f;
    a.w1 = sh.w1; a.w2 = sh.w2; a.w3 = sh.w3;
    a.flags = flags; a.epart = epart;
    a.tc = nterms;
    a.out_ps = (long)d.n1 * d.n2 * d.n3;
    a.ty = p.ty; a.px = p.px; a.ny = p.ny; a.gc = p.gc; a.bc = p.bc; a.rows = p.rows;
    a.m2_flat = p.ny == 1;
    if (group > 0 && group < nterms) {         // a group's sum goes where its first term was: see simt_core_consume
        a.tc = group;
        a.f.OUT0 = (float*)Z;
        a.out_ps = nterms * ((long)d.n1 * d.n2 * d.n3);
        a.out_cs = group * ((long)d.n1 * d.n2 * d.n3);
    }
    // a part of Z is one 16-byte aligned run where g is its fastest index and the part holds every g
    const long rr = (long)d.r2 * d.r3;
    a.z_mode = !z_bg ? 0
               : (p.gc == d.r3 && rr % 4 == 0 && (p.bc == d.r2 || ((long)p.bc * d.r3) % 4 == 0) &&
                  ((uintptr_t)Z & 15u) == 0) ? 2 : 1;
    // pairs of z as one access: even rows, and arrays (callers' blocks and slices) that start on 8 bytes
    a.vec = d.n3 % 2 == 0 && (((uintptr_t)f.MUL0 | (uintptr_t)f.MUL1 | (uintptr_t)f.OUT0 | (uintptr_t)f.OUT1) & 7u) == 0;
    return dispatch_consume(a, p, np, s);
}

int simt_core_consume(const Shape& sh, int np, float* Z, int nterms, const float* M2, const float* M3, float* H,
                      cudaStream_t s) {
    const Dims d = dims_of(sh);
    SimtPlan p{};
    FieldArgs f{};
    f.OUT0 = H;
    if (d.n1 != d.r1 || d.n2 != d.r2 || d.n3 != d.r3 || d.n3 > 256 || !simt_plan(d, &p) || p.ny != 1)
        return simt_expand_consume(sh, nullptr, 0, np, f, Z, nterms, M2, M3, EPI_STORE, nullptr, s);
    // Fewer CTAs than SMs: groups of at least 4 terms go to CTAs of their own, towards two per SM, and a
    // second kernel adds their sums, which lie where each group's first term of Z was (one y tile: no other
    // CTA reads that slab).  A call of 6 pairs of rank (13, 18, 23), 22 terms: 144 us; 257 with every term
    // in one CTA.  From one CTA per SM on the terms stay together and no second kernel is launched.
    const long ctas = (long)p.nx * np;
    const int groups = ctas >= 152 ? 1 : (int)std::min<long>((303 + ctas) / ctas, std::max(1, nterms / 4));
    const int tc = (nterms + groups - 1) / groups, nc = (nterms + tc - 1) / tc;
    if (nc == 1) return simt_expand_consume(sh, nullptr, 0, np, f, Z, nterms, M2, M3, EPI_STORE, nullptr, s);
    TX_TRY(simt_expand_consume(sh, nullptr, 0, np, f, Z, nterms, M2, M3, EPI_STORE, nullptr, s, true, 0, 0, tc));
    const long N = (long)d.n1 * d.n2 * d.n3;
    k_sum_groups<<<dim3((unsigned)((N + 255) / 256), np), 256, 0, s>>>(Z, nterms * N, tc * N, nc, N, H);
    TX_LAUNCHED();
    return TX_OK;
}

int simt_adjoint_r(const Shape& sh, const PairRec* recs, int p0, int np, const FieldArgs& f, int nt, const float* M2,
                   const float* M3, int flags, float* R, cudaStream_t s) {
    return launch_chain(sh, recs, p0, np, f, nt, M2, M3, flags, R, true, "adjoint", s);
}

int reduce_energy_batch(const double* epart, long count, double* dst, cudaStream_t s) {
    k_reduce<<<1, 256, 0, s>>>(epart, count, dst);
    TX_LAUNCHED();
    return TX_OK;
}

int weighted_dot(const tx_ctx* c, const float* A, const float* B, int count, double* partial, int nblocks, double scale,
                 double* e_dev, cudaStream_t s) {
    const long total = (long)count * c->n[0] * c->n[1] * c->n[2];
    k_weighted_dot<<<nblocks, 256, 0, s>>>(A, B, c->f_w[0], c->f_w[1], c->f_w[2], c->n[0], c->n[1], c->n[2], total,
                                           partial);
    TX_LAUNCHED();
    k_reduce<<<1, 256, 0, s>>>(partial, nblocks, partial + nblocks);
    TX_LAUNCHED();
    return finalize_energy(partial + nblocks, 1, scale, e_dev, s);
}

int finalize_energy(const double* batches, int nb, double scale, double* e_dev, cudaStream_t s) {
    k_finalize<<<1, 1, 0, s>>>(batches, nb, scale, e_dev);
    TX_LAUNCHED();
    return TX_OK;
}

}  // namespace tx
