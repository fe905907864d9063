// Two-sided (Galerkin) projection of the separable convolution onto the Tucker basis.
//
// The one-sided operator of Eq. final, phi = sum_t mu_t G x_d A_td with G = rho x_d U_d^T, is
// C P with P = (x)_d U_d U_d^T.  Projecting its output as well, with P^* = D^-1 P D (the adjoint
// of P in the inner product weighted by the quadrature weights D), gives
//   phi = P^* C P rho = (sum_t mu_t G x_d B_td) x_d (D_d^-1 U_d),   B_td = U_d^T D_d A_td,
// whose form <sigma, P^* C P rho>_w is symmetric and positive semi-definite, so the exchange
// energy -1/2 sum_ij <G_ij, sum_t mu_t G_ij x_d B_td> is exactly non-positive and is evaluated
// in core space at O(T r^4) per pair.  Everything here runs in float32 on the CUDA cores; the
// projection and the single reconstruction are the float32 path's own kernels.
#include <cuda_runtime.h>

#include <algorithm>

#include "tx_paths.h"

namespace tx {
namespace {

struct OperatorArgs {
    const double* UW[3];       // U_d[a][i] w_d[a]
    const double* U[3];
    const double* w[3];
    const double* A64[3];
    float* B[3];
    float* Ut[3];
    int n[3], r[3], ldb[3], ldu[3];
    int T;
};

// B_td[i][k] = sum_a U_d[a][i] w_d[a] A_td[a][k]  (mu_t is already folded into A_t3), and
// Ut_d[a][k] = U_d[a][k] / w_d[a].  Modes 2 and 3 (ldb, ldu > 0) are stored [k][i] and [k][a] with those
// row strides, as the consumer reads them.  blockIdx.y is the mode; one thread per output element,
// float64 sums: bound by float64 multiply-adds, one per point (w_d is folded into U_d at set-up).
__global__ void k_galerkin_operators(const OperatorArgs o) {
    const int d = blockIdx.y, n = o.n[d], r = o.r[d];
    const long e = (long)blockIdx.x * blockDim.x + threadIdx.x;
    const long nb = (long)o.T * r * r;
    if (e < nb) {
        const int t = (int)(e / ((long)r * r)), i = (int)((e / r) % r), k = (int)(e % r);
        const double* At = o.A64[d] + (long)t * n * r;
        const double* UW = o.UW[d];
        double s = 0.0;
        for (int a = 0; a < n; ++a) s = fma(UW[(long)a * r + i], At[(long)a * r + k], s);
        o.B[d][o.ldb[d] ? ((long)t * r + k) * o.ldb[d] + i : e] = (float)s;
    } else if (e < nb + (long)n * r) {
        const long q = e - nb;
        const long a = q / r, k = q - a * r;
        o.Ut[d][o.ldu[d] ? k * o.ldu[d] + a : q] = (float)(o.U[d][q] / o.w[d][a]);
    }
}

// epart[p] = ew_p * <G_p, H_p> with G [(b,g)][a] and H [a][(b,g)]  (float64 sum; one block per pair)
__global__ void __launch_bounds__(256) k_core_dot(const PairRec* __restrict__ recs, int p0, const float* __restrict__ G,
                                                  const float* __restrict__ H, int r1, long rr, double* __restrict__ epart) {
    __shared__ double red[256];
    const int p = blockIdx.x;
    const long m = r1 * rr;
    const float* g = G + (long)p * m;
    const float* h = H + (long)p * m;
    double s = 0.0;
    for (long e = threadIdx.x; e < m; e += blockDim.x) {
        const long q = e / r1, a = e - q * r1;
        s += (double)g[e] * (double)h[a * rr + q];
    }
    red[threadIdx.x] = s;
    __syncthreads();
    for (int k = 128; k > 0; k >>= 1) {
        if (threadIdx.x < k) red[threadIdx.x] += red[threadIdx.x + k];
        __syncthreads();
    }
    if (threadIdx.x == 0) epart[p] = red[0] * (double)recs[p0 + p].ew;
}

int ldb_of(const tx_ctx* c, int d) { return d == 0 ? 0 : d == 1 ? simt_ld2(c->r[1]) : simt_ld3(c->r[2]); }
int ldu_of(const tx_ctx* c, int d) { return d == 0 ? 0 : d == 1 ? simt_ld2(c->n[1]) : simt_ld3(c->n[2]); }
// (sizes in 64 bits: T r_d^2 passes 2^31 for modes of many thousand points)
size_t up4(size_t v) { return (v + 3) & ~(size_t)3; }
size_t b_floats(const tx_ctx* c, int d) { return up4((size_t)c->T * c->r[d] * (d ? ldb_of(c, d) : c->r[d])); }
size_t ut_floats(const tx_ctx* c, int d) { return up4((size_t)c->r[d] * (d ? ldu_of(c, d) : c->n[d])); }

}  // namespace

size_t galerkin_operator_floats(const tx_ctx* c) {
    size_t f = 0;
    for (int d = 0; d < 3; ++d) f += b_floats(c, d) + ut_floats(c, d);
    return f;
}

int galerkin_operators(const tx_ctx* c, float* ops, GalerkinOps* g, cudaStream_t s) {
    OperatorArgs o{};
    float* q = ops;
    long most = 0;
    for (int d = 0; d < 3; ++d) {
        o.B[d] = q;
        o.Ut[d] = q + b_floats(c, d);
        q = o.Ut[d] + ut_floats(c, d);
        g->B[d] = o.B[d];
        g->Ut[d] = o.Ut[d];
        o.UW[d] = c->d_UW[d]; o.U[d] = c->d_U[d]; o.w[d] = c->d_w[d]; o.A64[d] = c->d_A64[d];
        o.n[d] = c->n[d]; o.r[d] = c->r[d]; o.ldb[d] = ldb_of(c, d); o.ldu[d] = ldu_of(c, d);
        most = std::max(most, (long)c->T * c->r[d] * c->r[d] + (long)c->n[d] * c->r[d]);
    }
    o.T = c->T;
    k_galerkin_operators<<<dim3((unsigned)((most + 255) / 256), 3), 256, 0, s>>>(o);
    TX_LAUNCHED();
    return TX_OK;
}

// H[p][a'][b'][g'] = sum_t G[p] x1 B_t1 x2 B_t2 x3 B_t3: the expansion onto a grid of r_d points whose
// operators are B_td.  Mode 1 of every term is one GEMM; the consumer runs modes 2 and 3 and the sum
// over t in registers (X1 holds [np][T][r1][(b,g)]).  Differentiation-shaped block (rank 32, 35 terms, 136
// pairs): 845 us; 1456 as three GEMM passes over every term and a sum.
int galerkin_core(const tx_ctx* c, const GalerkinOps& o, const float* G, float* X1, float* H, int np, cudaStream_t s) {
    TX_TRY(simt_expand_mode1_grid(c, G, o.B[0], c->r[0], c->T, X1, np, s));
    return simt_core_consume(coarse_shape(c), np, X1, c->T, o.B[1], o.B[2], H, s);
}

int galerkin_core_dot(const tx_ctx* c, const PairRec* recs, int p0, const float* G, const float* H, int np,
                      double* epart, cudaStream_t s) {
    k_core_dot<<<np, 256, 0, s>>>(recs, p0, G, H, c->r[0], (long)c->r[1] * c->r[2], epart);
    TX_LAUNCHED();
    return TX_OK;
}

}  // namespace tx
