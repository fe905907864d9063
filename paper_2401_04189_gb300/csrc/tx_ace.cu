// Adaptively compressed exchange (the paper's "ACE implementation" section, Eqs. eta and ace1),
// built on top of the exchange potentials W_i = K psi_i of the hot path:
//
//   M_ij = <psi_i, W_j>_w                 weighted Gram matrix (float32 sums of 32, float64 beyond)
//   M_s  = (M + M^T) / 2                  (the paper is silent on the asymmetry a truncated Tucker
//                                          rank leaves; the symmetric part is factorised)
//   -M_s = L L^T                          Cholesky, float64 (M_s is negative definite)
//   xi_k = sum_i (L^-1)_ki W_i            the ACE projection vectors
//   V_ACE f = - sum_k xi_k <xi_k, f>_w    the ACE operator applied to a block
//
// The Gram matrices and the two small-by-large products cost O(N^2 n^3) flops, about 0.1% of the
// N^2 / 2 pair potentials behind W, so they run on the CUDA cores: float32 sums of 32
// products, summed in float64 across the grid (the factorisation needs M to about the accuracy of W).
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <string>

#include "tx_internal.h"
#include "tx_packed.cuh"
#include "tx_paths.h"

namespace tx {
namespace {

constexpr int kGramChunk = 64;    // grid points per shared-memory chunk
constexpr int kGramLd = kGramChunk + 4;
constexpr int kGramFold = 64;     // chunks per float64 addition

// partial[s][i][j] = sum over slice s of the grid of w(x) A_i(x) B_j(x): float32 sums of 32 products (the even and
// the odd points of a chunk of 64), added in float64 in effect.  This GPU adds float64 at 1/64 of the float32 rate,
// so the sums of up to 64 chunks are added in float32 with every rounding error caught exactly (Knuth's TwoSum) and
// summed beside, and the pair is then added to the float64 partial in memory, which only this thread touches.
// What a group loses is the rounding of its error sum, at most 2^-34 of the sum of its terms' magnitudes; the
// terms' own rounding is 2^-24 and more.  (With a Kahan sum in place of this, chunk sums of 1, 1e8, 1, -1e8 came out
// as 0.)  BI x BJ outputs per CTA
// of 128 threads (8 x 16), (BI / 8) x (BJ / 16) each.  The orbitals keep their own layout in shared
// memory (rows along the grid, stride 68: the 16-byte reads of 16 rows hit different banks) and the
// packed multiply-adds run along the grid, so nothing is transposed or duplicated; two buffers, filled
// by cp.async.  The whole apply of 64 x 64 orbitals of 96^3: 439 us; 448 with a Kahan sum, 2,024 with one output
// per thread and a float64 add per 32 points (the orbitals take 67 us of HBM time).
template <int BI, int BJ>
__global__ void __launch_bounds__(128) k_wgram(const float* __restrict__ A, int na, const float* __restrict__ B, int nb,
                                               const float* __restrict__ w1, const float* __restrict__ w2,
                                               const float* __restrict__ w3, int n1, int n2, int n3, long slice, int vec,
                                               double* __restrict__ partial) {
    constexpr int TI = BI / 8, TJ = BJ / 16;
    extern __shared__ __align__(16) float sm[];
    constexpr int kBuf = (BI + BJ) * kGramLd + kGramChunk;      // A rows, B rows, weights
    const long N3 = (long)n1 * n2 * n3, N23 = (long)n2 * n3;
    const int tid = threadIdx.x, ti = tid >> 4, tj = tid & 15;
    const int i0 = blockIdx.x * BI, j0 = blockIdx.y * BJ;
    const long x0 = (long)blockIdx.z * slice, x1 = min(N3, x0 + slice);
    auto load = [&](long xc, int buf) {
        float* As = sm + buf * kBuf;
        float* Bs = As + BI * kGramLd;
        if (vec) {
            for (int e = tid; e < BI * (kGramChunk / 4); e += 128) {
                const int r = e / (kGramChunk / 4), q = 4 * (e % (kGramChunk / 4));
                const bool ok = i0 + r < na && xc + q < x1;
                cp_async16(As + r * kGramLd + q, ok ? A + (long)(i0 + r) * N3 + xc + q : A, ok);
            }
            for (int e = tid; e < BJ * (kGramChunk / 4); e += 128) {
                const int r = e / (kGramChunk / 4), q = 4 * (e % (kGramChunk / 4));
                const bool ok = j0 + r < nb && xc + q < x1;
                cp_async16(Bs + r * kGramLd + q, ok ? B + (long)(j0 + r) * N3 + xc + q : B, ok);
            }
        } else {
            for (int e = tid; e < BI * kGramChunk; e += 128) {
                const int r = e / kGramChunk, q = e % kGramChunk;
                As[r * kGramLd + q] = (i0 + r < na && xc + q < x1) ? A[(long)(i0 + r) * N3 + xc + q] : 0.f;
            }
            for (int e = tid; e < BJ * kGramChunk; e += 128) {
                const int r = e / kGramChunk, q = e % kGramChunk;
                Bs[r * kGramLd + q] = (j0 + r < nb && xc + q < x1) ? B[(long)(j0 + r) * N3 + xc + q] : 0.f;
            }
        }
        if (tid < kGramChunk) {
            const long x = xc + tid;
            float wv = 0.f;
            if (x < x1) {
                const int a = (int)(x / N23), yz = (int)(x - a * N23), b = yz / n3, c = yz - b * n3;
                wv = w1[a] * w2[b] * w3[c];
            }
            Bs[BJ * kGramLd + tid] = wv;
        }
        cp_async_commit();
    };
    uint64_t sum[TI / 2][TJ], err[TI / 2][TJ];             // rows i and i + 1 in one register pair
    if (x0 < x1) load(x0, 0);
    int buf = 0;
    bool first = true;
    for (long xc = x0; first || xc < x1; first = false) {
#pragma unroll
        for (int i = 0; i < TI / 2; ++i)
#pragma unroll
            for (int j = 0; j < TJ; ++j) sum[i][j] = err[i][j] = 0ull;
        for (int n = 0; n < kGramFold && xc < x1; ++n, xc += kGramChunk, buf ^= 1) {
            cp_async_wait_all();
            __syncthreads();             // this chunk has landed; the other buffer has been read
            if (xc + kGramChunk < x1) load(xc + kGramChunk, buf ^ 1);
            const float* As = sm + buf * kBuf;
            const float* Bs = As + BI * kGramLd;
            const float* ws = Bs + BJ * kGramLd;
            uint64_t acc[TI][TJ];
#pragma unroll
            for (int i = 0; i < TI; ++i)
#pragma unroll
                for (int j = 0; j < TJ; ++j) acc[i][j] = 0ull;
#pragma unroll 4
            for (int k = 0; k < kGramChunk; k += 4) {
                const ulonglong2 w = *(const ulonglong2*)(ws + k);
                ulonglong2 a[TI], b[TJ];
#pragma unroll
                for (int j = 0; j < TJ; ++j) {
                    const ulonglong2 v = *(const ulonglong2*)(Bs + (tj + 16 * j) * kGramLd + k);
                    b[j] = make_ulonglong2(mul2(v.x, w.x), mul2(v.y, w.y));
                }
#pragma unroll
                for (int i = 0; i < TI; ++i) a[i] = *(const ulonglong2*)(As + (ti + 8 * i) * kGramLd + k);
#pragma unroll
                for (int i = 0; i < TI; ++i)
#pragma unroll
                    for (int j = 0; j < TJ; ++j) {
                        fma2(acc[i][j], a[i].x, b[j].x);
                        fma2(acc[i][j], a[i].y, b[j].y);
                    }
            }
#pragma unroll
            for (int i = 0; i < TI / 2; ++i)
#pragma unroll
                for (int j = 0; j < TJ; ++j) {
                    const uint64_t x = pack2(lo2(acc[2 * i][j]), lo2(acc[2 * i + 1][j]));
                    const uint64_t y = pack2(hi2(acc[2 * i][j]), hi2(acc[2 * i + 1][j]));
                    uint64_t ef, et;
                    const uint64_t f = two_sum(x, y, ef), t = two_sum(sum[i][j], f, et);
                    err[i][j] = add2(err[i][j], add2(et, ef));
                    sum[i][j] = t;
                }
        }
#pragma unroll
        for (int i = 0; i < TI; ++i)
#pragma unroll
            for (int j = 0; j < TJ; ++j) {
                const int r = i0 + ti + 8 * i, c = j0 + tj + 16 * j;
                if (r >= na || c >= nb) continue;
                const uint64_t t = sum[i / 2][j], e = err[i / 2][j];
                const float ef = i & 1 ? hi2(e) : lo2(e);
                double v = (double)(i & 1 ? hi2(t) : lo2(t));
                if (fabsf(ef) < INFINITY) v += (double)ef;       // an infinite sum stays infinite
                double* p = partial + ((long)blockIdx.z * na + r) * nb + c;
                *p = first ? v : *p + v;
            }
    }
}

// G[i][j] = sum_s partial[s][i][j] (fixed order: 8 interleaved sums, then their sum), and
// optionally its transpose in float32 scaled.  32 outputs x 8 slice groups per CTA.
__global__ void __launch_bounds__(256) k_gram_reduce(const double* __restrict__ partial, int ns, int na, int nb,
                                                     double* __restrict__ G, float* __restrict__ GTf, float scale) {
    __shared__ double red[8][33];
    const int lane = threadIdx.x & 31, grp = threadIdx.x >> 5;
    const long cnt = (long)na * nb, idx = blockIdx.x * 32L + lane;
    double s = 0.0;
    if (idx < cnt)
        for (int k = grp; k < ns; k += 8) s += partial[(long)k * cnt + idx];
    red[grp][lane] = s;
    __syncthreads();
    if (grp || idx >= cnt) return;
    for (int g = 1; g < 8; ++g) s += red[g][lane];
    if (G) G[idx] = s;
    if (GTf) {
        const int i = (int)(idx / nb), j = (int)(idx - (long)i * nb);
        GTf[(long)j * na + i] = (float)(scale * s);
    }
}

// One CTA: A = -(M + M^T) / 2 in float64, Cholesky A = L L^T in place (lower triangle), then
// Linv = L^-1 (lower triangular), written in float64 and in float32.  flag[0] = 1 + the first
// pivot that is not positive (M not negative definite), else 0.
__global__ void __launch_bounds__(1024) k_ace_factor(const double* __restrict__ M, int N, double* __restrict__ A,
                                                     double* __restrict__ Linv, float* __restrict__ Linv32, int* flag) {
    __shared__ int bad;
    if (threadIdx.x == 0) bad = 0;
    for (long e = threadIdx.x; e < (long)N * N; e += blockDim.x) {
        const int i = (int)(e / N), j = (int)(e - (long)i * N);
        A[e] = -0.5 * (M[(long)i * N + j] + M[(long)j * N + i]);
    }
    __syncthreads();
    for (int k = 0; k < N; ++k) {
        const double d = A[(long)k * N + k];
        if (!(d > 0.0)) {
            if (threadIdx.x == 0) bad = k + 1;
            __syncthreads();
            break;
        }
        const double s = sqrt(d);
        __syncthreads();
        for (int i = k + threadIdx.x; i < N; i += blockDim.x) A[(long)i * N + k] = (i == k) ? s : A[(long)i * N + k] / s;
        __syncthreads();
        // trailing update of the lower triangle: A[i][j] -= L[i][k] L[j][k], k < j <= i
        const long m = N - k - 1, cnt = m * (m + 1) / 2;
        for (long e = threadIdx.x; e < cnt; e += blockDim.x) {
            // e -> (ii, jj) with 0 <= jj <= ii < m
            long ii = (long)((sqrt(8.0 * (double)e + 1.0) - 1.0) * 0.5);
            while (ii * (ii + 1) / 2 > e) --ii;
            while ((ii + 1) * (ii + 2) / 2 <= e) ++ii;
            const long jj = e - ii * (ii + 1) / 2;
            const int i = k + 1 + (int)ii, j = k + 1 + (int)jj;
            A[(long)i * N + j] -= A[(long)i * N + k] * A[(long)j * N + k];
        }
        __syncthreads();
    }
    __syncthreads();
    if (bad) {
        if (threadIdx.x == 0) flag[0] = bad;
        return;
    }
    // Linv column by column (forward substitution), one thread per column
    for (int j = threadIdx.x; j < N; j += blockDim.x) {
        for (int i = 0; i < N; ++i) {
            double v = 0.0;
            if (i >= j) {
                double s = (i == j) ? 1.0 : 0.0;
                for (int k = j; k < i; ++k) s -= A[(long)i * N + k] * Linv[(long)k * N + j];
                v = s / A[(long)i * N + i];
            }
            Linv[(long)i * N + j] = v;
            Linv32[(long)i * N + j] = (float)v;
        }
    }
    if (threadIdx.x == 0) flag[0] = 0;
}

size_t up256(size_t v) { return (v + 255) & ~(size_t)255; }

// output tile of the Gram kernel along one side: the block size padded least
int gram_tile(int n) { return n <= 16 ? 16 : (n <= 32 ? 32 : 64); }

// grid slices of the Gram kernel: as many CTAs as the GPU holds at once, of at least 1024 points (and
// whole chunks) each
int gram_slices(long N3, int na, int nb) {
    const int bi = gram_tile(na), bj = gram_tile(nb);
    const long tiles = (long)((na + bi - 1) / bi) * ((nb + bj - 1) / bj);
    const long per_sm = bi * bj >= 64 * 64 ? 2 : 4;
    const long want = std::max<long>(1, (per_sm * 152 + tiles - 1) / tiles);
    return (int)std::min<long>(want, std::max<long>(1, N3 / 1024));
}

// weighted Gram matrix of A (na orbitals) and B (nb orbitals) into G (float64 [na][nb]) and/or
// the scaled float32 transpose GTf [nb][na]; partials in `scratch`
int wgram(const tx_ctx* c, const float* A, int na, const float* B, int nb, double* partial, int ns, double* G,
          float* GTf, float scale, cudaStream_t s) {
    const long N3 = (long)c->n[0] * c->n[1] * c->n[2];
    const long slice = ((N3 + ns - 1) / ns + kGramChunk - 1) / kGramChunk * kGramChunk;
    const int bi = gram_tile(na), bj = gram_tile(nb);
    const dim3 grid((unsigned)((na + bi - 1) / bi), (unsigned)((nb + bj - 1) / bj), (unsigned)ns);
    const int vec = c->n[2] % 4 == 0 && (((uintptr_t)A | (uintptr_t)B) & 15u) == 0;
    const size_t smem = sizeof(float) * 2 * ((bi + bj) * kGramLd + kGramChunk);
#define TX_GRAM(BI_, BJ_)                                                                                              \
    if (bi == BI_ && bj == BJ_) {                                                                                      \
        if (smem > 48 * 1024)                                                                                          \
            TX_TRY_CUDA(cudaFuncSetAttribute(k_wgram<BI_, BJ_>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem)); \
        k_wgram<BI_, BJ_><<<grid, 128, smem, s>>>(A, na, B, nb, c->f_w[0], c->f_w[1], c->f_w[2], c->n[0], c->n[1],      \
                                                  c->n[2], slice, vec, partial);                                       \
    }
    TX_GRAM(16, 16);
    TX_GRAM(16, 32);
    TX_GRAM(16, 64);
    TX_GRAM(32, 16);
    TX_GRAM(32, 32);
    TX_GRAM(32, 64);
    TX_GRAM(64, 16);
    TX_GRAM(64, 32);
    TX_GRAM(64, 64);
#undef TX_GRAM
    TX_LAUNCHED();
    const long cnt = (long)na * nb;
    k_gram_reduce<<<(unsigned)((cnt + 31) / 32), 256, 0, s>>>(partial, ns, na, nb, G, GTf, scale);
    TX_LAUNCHED();
    return TX_OK;
}

// out[k][x] = alpha * sum_i C[k][i] X[i][x]  (C float32 [nk][ni], X float32 [ni][N3])
int mix(const float* C, int nk, int ni, const float* X, long N3, float alpha, float* out, cudaStream_t s) {
    // the GEMM's column index is an int: blocks of grid points on very large grids
    const long block = 1L << 30;
    for (long x = 0; x < N3; x += block) {
        GemmArgs g{};
        g.M = nk; g.N = (int)std::min(block, N3 - x); g.K = ni;
        g.A = C; g.a_m = ni; g.a_k = 1;
        g.B = X + x; g.b_k = N3; g.b_n = 1;
        g.C = out + x; g.c_m = N3; g.c_n = 1;
        g.nb1 = g.nb2 = 1; g.alpha = alpha;
        TX_TRY(simt_gemm(g, s));
    }
    return TX_OK;
}

bool aligned16(const void* p) { return ((uintptr_t)p & 15u) == 0; }

int check_orbitals(const float* p, int n, const char* what) {
    if (n < 1 || !p) return fail(TX_ERR_INVALID_ARG, std::string(what) + " is NULL or empty");
    if (!aligned16(p)) return fail(TX_ERR_ALIGNMENT, std::string(what) + " is not 16-byte aligned");
    return TX_OK;
}

}  // namespace
}  // namespace tx

using namespace tx;

extern "C" int tx_ace_projectors(tx_ctx* c, const float* psi_occ, int n_occ, const float* W, float* xi, double* M,
                                 tx_stream_t stream) {
    if (!c || c->magic != kMagic) return fail(TX_ERR_NOT_SETUP, "context is NULL or was destroyed");
    TX_TRY(check_orbitals(psi_occ, n_occ, "psi_occ"));
    TX_TRY(check_orbitals(W, n_occ, "W"));
    TX_TRY(check_orbitals(xi, n_occ, "xi"));
    if (n_occ > 4096) return fail(TX_ERR_UNSUPPORTED_SHAPE, "ACE construction supports at most 4096 orbitals");
    const long N3 = (long)c->n[0] * c->n[1] * c->n[2];
    {
        const uintptr_t bytes = (uintptr_t)n_occ * N3 * sizeof(float);
        const uintptr_t o = (uintptr_t)xi;
        for (const float* in : {psi_occ, W}) {
            const uintptr_t a = (uintptr_t)in;
            if (o < a + bytes && a < o + bytes) return fail(TX_ERR_INVALID_ARG, "xi overlaps psi_occ or W");
        }
    }
    DeviceGuard dg;
    TX_TRY(dg.use(c->device));
    cudaStream_t s = (cudaStream_t)stream;
    c->last_stream = s;
    const int N = n_occ;
    const int ns = gram_slices(N3, N, N);
    const size_t nn = (size_t)N * N;
    const size_t off_part = 0, off_M = up256(sizeof(double) * ns * nn), off_A = off_M + up256(sizeof(double) * nn),
                 off_Li = off_A + up256(sizeof(double) * nn), off_L32 = off_Li + up256(sizeof(double) * nn),
                 off_flag = off_L32 + up256(sizeof(float) * nn), total = off_flag + 256;
    TX_TRY(ensure_workspace(c, total));
    char* ws = c->ws;
    double* partial = (double*)(ws + off_part);
    double* Mw = M ? M : (double*)(ws + off_M);
    int* flag = (int*)(ws + off_flag);
    TX_TRY_CUDA(cudaMemsetAsync(flag, 0xff, sizeof(int), s));
    TX_TRY(wgram(c, psi_occ, N, W, N, partial, ns, Mw, nullptr, 1.f, s));
    k_ace_factor<<<1, 1024, 0, s>>>(Mw, N, (double*)(ws + off_A), (double*)(ws + off_Li), (float*)(ws + off_L32), flag);
    TX_LAUNCHED();
    TX_TRY(mix((const float*)(ws + off_L32), N, N, W, N3, 1.f, xi, s));
    // the factorisation's outcome decides the status: read it back (the call synchronises)
    int h = -1;
    TX_TRY_CUDA(cudaMemcpyAsync(&h, flag, sizeof(int), cudaMemcpyDeviceToHost, s));
    TX_TRY_CUDA(cudaStreamSynchronize(s));
    if (h != 0)
        return fail(TX_ERR_NOT_DEFINITE, "the symmetric part of M = <psi_i, W_j>_w is not negative definite (pivot " +
                                             std::to_string(h - 1) + "); xi is not valid");
    return TX_OK;
}

extern "C" int tx_ace_apply(tx_ctx* c, const float* xi, int n_xi, const float* psi, int n, float* out,
                            tx_stream_t stream) {
    if (!c || c->magic != kMagic) return fail(TX_ERR_NOT_SETUP, "context is NULL or was destroyed");
    TX_TRY(check_orbitals(xi, n_xi, "xi"));
    TX_TRY(check_orbitals(psi, n, "psi"));
    TX_TRY(check_orbitals(out, n, "out"));
    const long N3 = (long)c->n[0] * c->n[1] * c->n[2];
    {
        const uintptr_t o = (uintptr_t)out, ob = (uintptr_t)n * N3 * sizeof(float);
        const uintptr_t a = (uintptr_t)psi, ab = ob;
        const uintptr_t x = (uintptr_t)xi, xb = (uintptr_t)n_xi * N3 * sizeof(float);
        if ((o < a + ab && a < o + ob) || (o < x + xb && x < o + ob))
            return fail(TX_ERR_INVALID_ARG, "out overlaps psi or xi");
    }
    DeviceGuard dg;
    TX_TRY(dg.use(c->device));
    cudaStream_t s = (cudaStream_t)stream;
    c->last_stream = s;
    const int ns = gram_slices(N3, n_xi, n);
    const size_t off_part = 0, off_C = up256(sizeof(double) * ns * (size_t)n_xi * n),
                 total = off_C + up256(sizeof(float) * (size_t)n_xi * n);
    TX_TRY(ensure_workspace(c, total));
    double* partial = (double*)c->ws;
    float* CT = (float*)(c->ws + off_C);   // CT[a][k] = <xi_k, psi_a>_w
    TX_TRY(wgram(c, xi, n_xi, psi, n, partial, ns, nullptr, CT, 1.f, s));
    // out[a] = - sum_k CT[a][k] xi_k
    return mix(CT, n, n_xi, xi, N3, -1.f, out, s);
}
