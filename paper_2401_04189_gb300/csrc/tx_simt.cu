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

namespace tx {

// ====================================================================================
// packed float32 arithmetic: two fused multiply-adds per instruction (fma.rn.f32x2 rounds each
// half as fmaf does), which halves the issue slots of the inner loops and leaves the rest of
// them to the shared-memory reads
// ====================================================================================
namespace {
__device__ __forceinline__ uint64_t dup2(float v) {
    uint64_t r;
    asm("mov.b64 %0, {%1, %1};" : "=l"(r) : "f"(v));
    return r;
}
__device__ __forceinline__ void fma2(uint64_t& d, uint64_t a, uint64_t b) {
    asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(d) : "l"(a), "l"(b));
}
__device__ __forceinline__ float2 unpack2(uint64_t v) {
    float2 r;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(v));
    return r;
}
__device__ __forceinline__ uint32_t smem_addr(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ void cp_async16(float* dst, const float* src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_addr(dst)), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async4(float* dst, const float* src) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(smem_addr(dst)), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_all;" ::: "memory"); }

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
__global__ void __launch_bounds__(256) k_gemm(GemmArgs g, int modeA, int modeB, int vecC) {
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

Dims dims_of(const tx_ctx* c) {
    return Dims{c->n[0], c->n[1], c->n[2], c->r[0], c->r[1], c->r[2]};
}

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
// The two inner loops every float32 mode product is built from.  A thread owns 4 neighbouring
// rows (one 16-byte fragment, two packed pairs) and RG columns tz, tz + 8, ... of a panel:
// acc[c] += A[k][row .. row + 3] * B[k][tz + 8 c], both operands K-major in shared memory.
// The 8 column lanes x 4 row groups of a warp read one 64-byte and one 32-byte segment per
// fragment (broadcast), so the float32 pipes, not shared memory, bound it from RG = 4 on.
// ====================================================================================
constexpr int kMaxRG = 8;          // columns per thread; a panel is at most 64 columns wide

template <int RG>
__device__ __forceinline__ void panel(const float* __restrict__ A, int lda, const float* __restrict__ B, int ldb, int K,
                                      uint64_t (&acc)[kMaxRG][2]) {
#pragma unroll 4
    for (int k = 0; k < K; ++k) {
        const ulonglong2 a = *(const ulonglong2*)(A + k * lda);
#pragma unroll
        for (int c = 0; c < RG; ++c) {
            const uint64_t b = dup2(B[k * ldb + 8 * c]);
            fma2(acc[c][0], a.x, b);
            fma2(acc[c][1], a.y, b);
        }
    }
}

// B must be readable up to column 8 * rg - 1 (its row stride is at least that)
__device__ __forceinline__ void panel_any(int rg, const float* A, int lda, const float* B, int ldb, int K,
                                          uint64_t (&acc)[kMaxRG][2]) {
    switch (rg) {
        case 1: panel<1>(A, lda, B, ldb, K, acc); break;
        case 2: panel<2>(A, lda, B, ldb, K, acc); break;
        case 3: panel<3>(A, lda, B, ldb, K, acc); break;
        case 4: panel<4>(A, lda, B, ldb, K, acc); break;
        case 5: panel<5>(A, lda, B, ldb, K, acc); break;
        case 6: panel<6>(A, lda, B, ldb, K, acc); break;
        case 7: panel<7>(A, lda, B, ldb, K, acc); break;
        default: panel<8>(A, lda, B, ldb, K, acc); break;
    }
}

// ====================================================================================
// modes 3 and 2 of a projection: out[p][t][x][g][b] = sum_{y,z} M2_t[y][b] M3_t[z][g] q_p[x][y][z]
// with q_p the product of two orbitals (times the quadrature weights where asked).  One term with
// M3 = U3, M2 = U2 is the projection onto the core; the Gaussian terms' A_t3, A_t2 give the
// adjoint's first two modes.  One CTA per (x, pair): the plane's product is staged z-major in
// slices of PZ columns, mode 3 leaves S1[y][g] in shared memory and mode 2 reads it there.
// With rows of 4 y x RG g per thread instead of one output per thread, the Pt-shaped projection
// (96^3, rank 40) takes 8.7 us per pair instead of 16.3.
// ====================================================================================
constexpr int PZ = 32;             // z columns per slice

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
    int ty, gw, bw;                // y rows per tile (a multiple of 4), g (<= 64) and b (<= 256) columns per pass
    int ldy, ldg, ldb, vec;        // shared-memory row strides; vec: 16-byte orbital rows
};

__global__ void __launch_bounds__(512) k_chain(const ChainArgs a) {
    extern __shared__ __align__(16) float sm[];
    const Dims d = a.d;
    float* qs = sm;                            // [PZ][ldy]   the pair product, z-major
    float* m3s = qs + PZ * a.ldy;              // [PZ][ldg]
    float* s1 = m3s + PZ * a.ldg;              // [ty][ldg]
    float* m2s = s1 + a.ty * a.ldg;            // [PZ][ldb]
    const int x = blockIdx.x, pl = blockIdx.y, tid = threadIdx.x, nth = blockDim.x;
    const PairRec rec = a.recs[a.p0 + pl];
    const long N3 = (long)d.n1 * d.n2 * d.n3;
    const float* pa = a.SA + rec.ia * N3 + (long)x * d.n2 * d.n3;
    const float* pb = a.SB + rec.ib * N3 + (long)x * d.n2 * d.n3;
    const bool mulw = (a.flags & PROD_MULW) != 0;
    const float wx = mulw ? a.w1[x] : 1.f;
    const int tz = tid & 7, row0 = 4 * (tid >> 3);
    const int nbq = a.bw / 4, ngt = nth / nbq;                    // mode 2: 4 b per thread
    const int bq = tid % nbq, gq = tid / nbq;
    for (int t = 0; t < a.nt; ++t) {
        const float* M3 = a.M3 + (long)t * d.n3 * d.r3;
        const float* M2 = a.M2 + (long)t * d.n2 * d.r2;
        float* out = a.out + (((long)pl * a.nt + t) * d.n1 + x) * d.r3 * d.r2;
        for (int g0 = 0; g0 < d.r3; g0 += a.gw) {
            const int gn = min(a.gw, d.r3 - g0), rg = (gn + 7) / 8;
            for (int y0 = 0; y0 < d.n2; y0 += a.ty) {
                const int yn = min(a.ty, d.n2 - y0);
                uint64_t acc[kMaxRG][2];
#pragma unroll
                for (int c = 0; c < kMaxRG; ++c) acc[c][0] = acc[c][1] = 0ull;
                for (int z0 = 0; z0 < d.n3; z0 += PZ) {
                    const int zn = min(PZ, d.n3 - z0);
                    __syncthreads();           // the previous slice (and S1) has been read
                    if (a.vec) {
                        // 2 neighbouring 16-byte pieces x 16 rows per warp: whole sectors, and with
                        // ldy = 4 (mod 8) the transposed stores hit 32 different banks
                        const int ngr = (yn + 15) / 16;
                        for (int e = tid; e < ngr * (PZ / 8) * 32; e += nth) {
                            const int grp = e >> 5, l = e & 31;
                            const int yy = (grp % ngr) * 16 + (l & 15), z = 4 * (2 * (grp / ngr) + (l >> 4));
                            if (yy >= yn || z >= zn) continue;
                            const long o = (long)(y0 + yy) * d.n3 + z0 + z;
                            const float4 u = *(const float4*)(pa + o), v = *(const float4*)(pb + o);
                            float q[4] = {u.x * v.x, u.y * v.y, u.z * v.z, u.w * v.w};
                            if (mulw) {
                                const float wxy = wx * a.w2[y0 + yy];
#pragma unroll
                                for (int k = 0; k < 4; ++k) q[k] *= wxy * a.w3[z0 + z + k];
                            }
#pragma unroll
                            for (int k = 0; k < 4; ++k) qs[(z + k) * a.ldy + yy] = q[k];
                        }
                    } else {
                        for (int e = tid; e < yn * zn; e += nth) {
                            const int yy = e / zn, z = e - yy * zn;
                            const long o = (long)(y0 + yy) * d.n3 + z0 + z;
                            float q = pa[o] * pb[o];
                            if (mulw) q *= wx * a.w2[y0 + yy] * a.w3[z0 + z];
                            qs[z * a.ldy + yy] = q;
                        }
                    }
                    for (int e = tid; e < zn * gn; e += nth) {
                        const int z = e / gn, g = e - z * gn;
                        m3s[z * a.ldg + g] = M3[(long)(z0 + z) * d.r3 + g0 + g];
                    }
                    __syncthreads();
                    if (row0 < a.ty) panel_any(rg, qs + row0, a.ldy, m3s + tz, a.ldg, zn, acc);
                }
                if (row0 < a.ty) {
#pragma unroll
                    for (int c = 0; c < kMaxRG; ++c)
                        if (c < rg) {
                            const float2 u = unpack2(acc[c][0]), v = unpack2(acc[c][1]);
                            float* p = s1 + row0 * a.ldg + tz + 8 * c;
                            p[0] = u.x; p[a.ldg] = u.y; p[2 * a.ldg] = v.x; p[3 * a.ldg] = v.y;
                        }
                }
                // mode 2: S2[g][b] = sum_y S1[y][g] M2[y][b], this y tile's share added to the earlier ones'
                for (int b0 = 0; b0 < d.r2; b0 += a.bw)
                    for (int gc = 0; gc < gn; gc += 4 * ngt) {
                        const int bn = min(a.bw, d.r2 - b0);
                        uint64_t s[4][2];
#pragma unroll
                        for (int c = 0; c < 4; ++c) s[c][0] = s[c][1] = 0ull;
                        for (int yb = 0; yb < yn; yb += PZ) {
                            const int ync = min(PZ, yn - yb);
                            __syncthreads();       // S1 written; the previous M2 slice has been read
                            for (int e = tid; e < ync * bn; e += nth) {
                                const int yy = e / bn, bb = e - yy * bn;
                                m2s[yy * a.ldb + bb] = M2[(long)(y0 + yb + yy) * d.r2 + b0 + bb];
                            }
                            __syncthreads();
                            if (gq < ngt) {
                                const float* sp = s1 + yb * a.ldg;
                                const float* mp = m2s + 4 * bq;
                                // columns past gn repeat the last padding column (never stored)
                                const int cl = a.ldg - 1, c0 = gc + gq;
                                const int o0 = min(c0, cl), o1 = min(c0 + ngt, cl), o2 = min(c0 + 2 * ngt, cl),
                                          o3 = min(c0 + 3 * ngt, cl);
#pragma unroll 4
                                for (int k = 0; k < ync; ++k) {
                                    const ulonglong2 m = *(const ulonglong2*)(mp + k * a.ldb);
                                    const float* q = sp + k * a.ldg;
                                    const uint64_t b0_ = dup2(q[o0]), b1_ = dup2(q[o1]), b2_ = dup2(q[o2]), b3_ = dup2(q[o3]);
                                    fma2(s[0][0], m.x, b0_); fma2(s[0][1], m.y, b0_);
                                    fma2(s[1][0], m.x, b1_); fma2(s[1][1], m.y, b1_);
                                    fma2(s[2][0], m.x, b2_); fma2(s[2][1], m.y, b2_);
                                    fma2(s[3][0], m.x, b3_); fma2(s[3][1], m.y, b3_);
                                }
                            }
                        }
                        if (gq < ngt) {
#pragma unroll
                            for (int c = 0; c < 4; ++c) {
                                const int g = gc + gq + c * ngt;
                                if (g >= gn) continue;
                                const float2 u = unpack2(s[c][0]), v = unpack2(s[c][1]);
                                const float q[4] = {u.x, u.y, v.x, v.y};
                                float* o = out + (long)(g0 + g) * d.r2 + b0 + 4 * bq;
#pragma unroll
                                for (int k = 0; k < 4; ++k)
                                    if (4 * bq + k < bn) o[k] = y0 ? o[k] + q[k] : q[k];
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
// A CTA owns `rows` rows: px planes x ty y-rows, 2 threads per row; a thread owns 4 rows and
// 4 * RN4 + 2 * H columns of phi (8 column lanes, 16-byte pieces 32 columns apart), kept in
// registers over every term.  Per term mode 2 leaves Y in shared memory (K-major) and mode 3 reads
// it back: 4 * RN multiply-adds per 1 + RN4 16-byte fragments.  The next operator tiles arrive
// by cp.async under the arithmetic: M3 under mode 2, the next term's M2 and Z under mode 3.
// Ranks above 64 run in parts of K (the Y tile, M2 and Z slices stay at most 64 deep).
// Bound by the float32 pipes.  Pt-shaped pair (96^3, rank 40, 40 terms): 114 us (35 TF/s) instead of 461.
// ====================================================================================
struct SimtPlan {
    int rn4, h;                // columns: 32 * rn4 + 16 * h
    int ty, ny, px, nx, rows;  // y rows per plane (a multiple of 4), y tiles, planes per CTA, x slabs, rows per CTA
    int gc, bc;                // K parts of mode 3 and mode 2
    size_t smem;
};

struct ConsumeF32Args {
    Dims d;
    const PairRec* recs;
    int p0, nt;
    const float* Z;            // [np][nt][n1][r3][r2]
    const float* M2;           // [nt][r2][ld2], y fastest
    const float* M3;           // [nt][r3][ld3], z fastest
    int ld2, ld3;
    long m2_ps, m3_ps;
    FieldArgs f;
    const float* w1;
    const float* w2;
    const float* w3;
    int flags;
    double* epart;
    int ty, px, ny, gc, bc, rows, vec;
};

// threads per CTA: 2 per row, and registers for phi
__host__ __device__ constexpr int consume_max_threads(int units) { return units <= 6 ? 512 : (units <= 10 ? 384 : 256); }

template <int RN4, int H>
__global__ void __launch_bounds__(consume_max_threads(2 * RN4 + H)) k_consume(const ConsumeF32Args a) {
    constexpr int NC = 32 * RN4 + 16 * H;              // columns of phi
    extern __shared__ __align__(16) float sm[];
    __shared__ double red[16];
    const Dims d = a.d;
    const int ldy = a.rows + 4, ldz = a.gc | 1, rgw = 8 * ((a.gc + 7) / 8);
    float* m2s = sm;                                   // [bc][ty]
    float* m3s = m2s + a.bc * a.ty;                    // [gc][NC]
    float* ys = m3s + a.gc * NC;                       // [gc][ldy]
    float* zs = ys + rgw * ldy;                        // [px][bc][ldz]
    const int tid = threadIdx.x, nth = blockDim.x, lane = tid & 31, warp = tid >> 5, nw = nth >> 5;
    const int iy = blockIdx.x % a.ny, x0 = (blockIdx.x / a.ny) * a.px, pl = blockIdx.y;
    const int y0 = iy * a.ty;
    const PairRec rec = a.recs[a.p0 + pl];
    const int tz = tid & 7, row0 = 4 * (tid >> 3);
    const int pr = min(row0 / a.ty, a.px - 1);         // plane of this thread's rows
    const int yr = min(row0 - pr * a.ty, a.ty - 4);    // rows past the last plane repeat valid ones (not stored)
    const long zslice = (long)d.r3 * d.r2;
    const int ng = (d.r3 + a.gc - 1) / a.gc, nb = (d.r2 + a.bc - 1) / a.bc;

    uint64_t acc[4][2 * RN4 + H];
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int c = 0; c < 2 * RN4 + H; ++c) acc[i][c] = 0ull;

    // M2 and Z of part (t, g part, b part)
    auto load2 = [&](int t, int gp, int bp) {
        const int g0 = gp * a.gc, gn = min(a.gc, d.r3 - g0), b0 = bp * a.bc, bn = min(a.bc, d.r2 - b0);
        const float* m2 = a.M2 + pl * a.m2_ps + ((long)t * d.r2 + b0) * a.ld2 + y0;
        const int nq = min(a.ty, a.ld2 - y0) / 4;      // ld2 is n2 rounded up to 4
        for (int e = tid; e < bn * nq; e += nth) {
            const int k = e / nq, q = e - k * nq;
            cp_async16(m2s + k * a.ty + 4 * q, m2 + (long)k * a.ld2 + 4 * q);
        }
        // Z comes with b fastest and is wanted with g fastest: the odd row stride spreads the
        // transposed 4-byte stores over the banks
        for (int p = 0; p < a.px; ++p) {
            if (x0 + p >= d.n1) break;
            const float* zt = a.Z + (((long)pl * a.nt + t) * d.n1 + x0 + p) * zslice + (long)g0 * d.r2 + b0;
            float* zd = zs + p * a.bc * ldz;
            for (int g = warp; g < gn; g += nw)
                for (int b = lane; b < bn; b += 32) cp_async4(zd + b * ldz + g, zt + (long)g * d.r2 + b);
        }
        cp_async_commit();
    };
    auto load3 = [&](int t, int gp) {
        const int g0 = gp * a.gc, gn = min(a.gc, d.r3 - g0), nq = a.ld3 / 4;
        const float* m3 = a.M3 + pl * a.m3_ps + ((long)t * d.r3 + g0) * a.ld3;
        for (int e = tid; e < gn * nq; e += nth) {
            const int k = e / nq, q = e - k * nq;
            cp_async16(m3s + k * NC + 4 * q, m3 + (long)k * a.ld3 + 4 * q);
        }
        cp_async_commit();
    };

    load2(0, 0, 0);
    for (int t = 0; t < a.nt; ++t)
        for (int gp = 0; gp < ng; ++gp) {
            const int gn = min(a.gc, d.r3 - gp * a.gc), rg = (gn + 7) / 8;
            uint64_t y[kMaxRG][2];
#pragma unroll
            for (int c = 0; c < kMaxRG; ++c) y[c][0] = y[c][1] = 0ull;
            for (int bp = 0; bp < nb; ++bp) {
                cp_async_wait_all();
                __syncthreads();               // M2 and Z have landed; the previous mode 3 is done
                if (bp == 0) load3(t, gp);
                panel_any(rg, m2s + yr, a.ty, zs + pr * a.bc * ldz + tz, ldz, min(a.bc, d.r2 - bp * a.bc), y);
                if (bp + 1 < nb) {
                    __syncthreads();
                    load2(t, gp, bp + 1);
                }
            }
#pragma unroll
            for (int c = 0; c < kMaxRG; ++c)
                if (c < rg) *(ulonglong2*)(ys + (tz + 8 * c) * ldy + row0) = make_ulonglong2(y[c][0], y[c][1]);
            cp_async_wait_all();
            __syncthreads();                   // Y and M3 are there, M2 and Z free
            if (gp + 1 < ng) load2(t, gp + 1, 0);
            else if (t + 1 < a.nt) load2(t + 1, 0, 0);
#pragma unroll 4
            for (int g = 0; g < gn; ++g) {
                const float4 yv = *(const float4*)(ys + g * ldy + row0);
                uint64_t b[2 * RN4 + H];
#pragma unroll
                for (int c = 0; c < RN4; ++c) {
                    const ulonglong2 q = *(const ulonglong2*)(m3s + g * NC + 4 * tz + 32 * c);
                    b[2 * c] = q.x;
                    b[2 * c + 1] = q.y;
                }
                if constexpr (H) b[2 * RN4] = *(const uint64_t*)(m3s + g * NC + 32 * RN4 + 2 * tz);
                const uint64_t y4[4] = {dup2(yv.x), dup2(yv.y), dup2(yv.z), dup2(yv.w)};
#pragma unroll
                for (int i = 0; i < 4; ++i)
#pragma unroll
                    for (int c = 0; c < 2 * RN4 + H; ++c) fma2(acc[i][c], y4[i], b[c]);
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
    const float wx = x < d.n1 ? a.w1[x] : 0.f;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const int y = y0 + yr + i;
        if (!rows_ok || y >= d.n2) continue;
        const float wxy = wx * a.w2[y];
        const long base = ((long)x * d.n2 + y) * d.n3;
#pragma unroll
        for (int c = 0; c < 2 * RN4 + H; ++c) {
            const int z = c < 2 * RN4 ? 32 * (c / 2) + 4 * tz + 2 * (c & 1) : 32 * RN4 + 2 * tz;
            const float2 ph = unpack2(acc[i][c]);
            const float phi[2] = {ph.x, ph.y};
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
int launch_chain(const tx_ctx* c, const PairRec* recs, int p0, int np, const FieldArgs& f, int nt, const float* M2,
                 const float* M3, int flags, float* out, const char* name, cudaStream_t s) {
    ChainArgs a{};
    a.d = dims_of(c);
    a.recs = recs; a.p0 = p0; a.nt = nt;
    a.SA = f.SA; a.SB = f.SB; a.M2 = M2; a.M3 = M3;
    a.w1 = c->f_w[0]; a.w2 = c->f_w[1]; a.w3 = c->f_w[2];
    a.flags = flags; a.out = out;
    // y tiles of at most 128 rows of equal height, 2 threads per row (at least 128 threads)
    const int ny = (a.d.n2 + 127) / 128, tyv = (a.d.n2 + ny - 1) / ny;
    a.ty = (tyv + 3) & ~3;
    const int ngp = (a.d.r3 + 63) / 64;
    a.gw = (a.d.r3 + ngp - 1) / ngp;
    a.ldy = ((a.ty + 7) & ~7) + 4;
    a.ldg = 8 * ((a.gw + 7) / 8) + 2;
    a.bw = std::min(256, pad4(a.d.r2));
    a.ldb = a.bw + 4;
    a.vec = a.d.n3 % 4 == 0 && (((uintptr_t)f.SA | (uintptr_t)f.SB) & 15u) == 0;
    // qs and m3s rows are 16-byte multiples where float4 reads them (qs, m2s); s1 and m3s are read as scalars
    const size_t words = (size_t)PZ * a.ldy + (size_t)PZ * a.ldg + (size_t)a.ty * a.ldg;
    const size_t smem = sizeof(float) * (words + (size_t)PZ * a.ldb);
    const int threads = std::max(128, ((2 * a.ty + 31) / 32) * 32);
    TX_TRY(smem_attr((const void*)k_chain, smem));
    const int ps = prof_begin(name, s);
    k_chain<<<dim3(a.d.n1, np), threads, smem, s>>>(a);
    prof_end(ps, s);
    TX_LAUNCHED();
    return TX_OK;
}

// The split of one pair's (x, y) rows over CTAs.  Phi's columns per thread fix the registers and so
// the threads (512 up to 96 columns, 384 up to 160, 256 above); among the row tiles that fit, the
// one with the least padding, preferring those that let two CTAs share an SM.
bool simt_plan(const Dims& d, SimtPlan* out) {
    if (d.n3 > 256) return false;
    const int units = (d.n3 + 15) / 16;
    SimtPlan p{};
    p.rn4 = units / 2;
    p.h = units & 1;
    const int ncol = 16 * units, max_rows = consume_max_threads(units) / 2;
    const int ngp = (d.r3 + 63) / 64, nbp = (d.r2 + 63) / 64;
    p.gc = (d.r3 + ngp - 1) / ngp;
    p.bc = (d.r2 + nbp - 1) / nbp;
    const int rgw = 8 * ((p.gc + 7) / 8), ldz = p.gc | 1;
    double best = -1.0;
    for (int ny = (d.n2 + max_rows - 1) / max_rows; ny <= (d.n2 + 15) / 16; ++ny) {
        p.ny = ny;
        p.ty = (((d.n2 + ny - 1) / ny) + 3) & ~3;
        for (p.px = 1; p.px <= d.n1 && ((p.px * p.ty + 15) & ~15) <= max_rows; ++p.px) {
            p.nx = (d.n1 + p.px - 1) / p.px;
            p.rows = (p.px * p.ty + 15) & ~15;
            // 8 more floats: the last column group of a panel may read past a Z row
            p.smem = sizeof(float) * ((size_t)p.bc * p.ty + (size_t)p.gc * ncol + (size_t)rgw * (p.rows + 4) +
                                      (size_t)p.px * p.bc * ldz + 8);
            if (p.smem > kSmemLimit) continue;
            double score = (double)d.n1 * d.n2 / ((double)p.ny * p.nx * p.rows);
            if (p.rows < 96) score *= p.rows < 64 ? 0.8 : 0.9;
            if (p.smem > kSmemLimit / 2) score *= 0.85;
            if (p.rows > 192) score *= 0.95;
            if (score > best + 1e-9) {
                best = score;
                *out = p;
            }
        }
    }
    return best > 0.0;
}

template <int RN4, int H>
int launch_consume(const ConsumeF32Args& a, const SimtPlan& p, int np, cudaStream_t s) {
    TX_TRY(smem_attr((const void*)k_consume<RN4, H>, p.smem));
    const int ps = prof_begin("consume", s);
    k_consume<RN4, H><<<dim3(p.nx * p.ny, np), 2 * p.rows, p.smem, s>>>(a);
    prof_end(ps, s);
    TX_LAUNCHED();
    return TX_OK;
}
}  // namespace

int simt_project_s2(const tx_ctx* c, const PairRec* recs, int p0, int np, const FieldArgs& f, int flags,
                    float* S2, cudaStream_t s) {
    const Dims d = dims_of(c);
    if (sizeof(float) * ((size_t)d.n3 * d.r3 + (size_t)d.n2 * d.r3 + 8 * (size_t)d.n3) > kSmemLimit)
        return fail(TX_ERR_CUDA, "float32 projection: (n2 + n3) * r3 too large");
    return launch_chain(c, recs, p0, np, f, 1, c->f_U[1], c->f_U[2], flags, S2, "project", s);
}

int simt_expand_consume_blocks(const tx_ctx* c) {
    SimtPlan p{};
    return simt_plan(dims_of(c), &p) ? p.nx * p.ny : 1;
}

int simt_kmajor(const float* src, int nt, int n, int r, float* dst, cudaStream_t s) {
    const long cnt = (long)nt * r * pad4(n);
    k_kmajor<<<(unsigned)((cnt + 255) / 256), 256, 0, s>>>(src, nt, n, r, pad4(n), dst);
    TX_LAUNCHED();
    return TX_OK;
}

int simt_expand_consume(const tx_ctx* c, const PairRec* recs, int p0, int np, const FieldArgs& f, const float* Z,
                        int nterms, const float* M2, const float* M3, int flags, double* epart, cudaStream_t s,
                        long m2_ps, long m3_ps) {
    const Dims d = dims_of(c);
    if (d.n3 > 256) return fail(TX_ERR_UNSUPPORTED_SHAPE, "float32 path supports n3 <= 256");
    SimtPlan p{};
    if (!simt_plan(d, &p) || sizeof(float) * ((size_t)d.r3 * (d.r2 + 1) + 32 * (size_t)(d.r3 + 1) +
                                              (size_t)d.n3 * (d.r3 | 1)) > kSmemLimit)
        return fail(TX_ERR_CUDA, "float32 expansion: (r2 + n3) * r3 too large");
    ConsumeF32Args a{};
    a.d = d;
    a.recs = recs; a.p0 = p0; a.nt = nterms;
    a.Z = Z; a.M2 = M2; a.M3 = M3;
    a.ld2 = pad4(d.n2); a.ld3 = pad4(d.n3);
    a.m2_ps = m2_ps; a.m3_ps = m3_ps;
    a.f = f;
    a.w1 = c->f_w[0]; a.w2 = c->f_w[1]; a.w3 = c->f_w[2];
    a.flags = flags; a.epart = epart;
    a.ty = p.ty; a.px = p.px; a.ny = p.ny; a.gc = p.gc; a.bc = p.bc; a.rows = p.rows;
    // pairs of z as one access: even rows, and arrays (callers' blocks and slices) that start on 8 bytes
    a.vec = d.n3 % 2 == 0 && (((uintptr_t)f.MUL0 | (uintptr_t)f.MUL1 | (uintptr_t)f.OUT0 | (uintptr_t)f.OUT1) & 7u) == 0;
    switch (2 * p.rn4 + p.h) {
        case 1: return launch_consume<0, 1>(a, p, np, s);
        case 2: return launch_consume<1, 0>(a, p, np, s);
        case 3: return launch_consume<1, 1>(a, p, np, s);
        case 4: return launch_consume<2, 0>(a, p, np, s);
        case 5: return launch_consume<2, 1>(a, p, np, s);
        case 6: return launch_consume<3, 0>(a, p, np, s);
        case 7: return launch_consume<3, 1>(a, p, np, s);
        case 8: return launch_consume<4, 0>(a, p, np, s);
        case 9: return launch_consume<4, 1>(a, p, np, s);
        case 10: return launch_consume<5, 0>(a, p, np, s);
        case 11: return launch_consume<5, 1>(a, p, np, s);
        case 12: return launch_consume<6, 0>(a, p, np, s);
        case 13: return launch_consume<6, 1>(a, p, np, s);
        case 14: return launch_consume<7, 0>(a, p, np, s);
        case 15: return launch_consume<7, 1>(a, p, np, s);
        default: return launch_consume<8, 0>(a, p, np, s);
    }
}

int simt_adjoint_r(const tx_ctx* c, const PairRec* recs, int p0, int np, const FieldArgs& f, int flags, float* R,
                   cudaStream_t s) {
    const Dims d = dims_of(c);
    if (sizeof(float) * ((size_t)d.n2 * d.n3 + (size_t)d.n2 * d.r3) > 220 * 1024)
        return fail(TX_ERR_UNSUPPORTED_SHAPE, "float32 adjoint needs n2*(n3+r3) <= 56K");
    return launch_chain(c, recs, p0, np, f, c->T, c->f_A[1], c->f_A[2], flags, R, "adjoint", s);
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
