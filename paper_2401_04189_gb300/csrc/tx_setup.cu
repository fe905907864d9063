// Set-up of the 1-D convolution factors, in float64 on the device.
//
// The paper precomputes the quadrature sums of the 1-D convolutions once and reuses them for
// every pair (the rearranged sum after Eq. discInteg).  With nodal quadrature on the grid the
// precomputed quantity is C_td[a][b] = w_b exp(-theta_t (x_a - x_b)^2), and applied to the
// basis it gives A_td = C_td U_d, the 1-D convolutions of the basis functions in Eq. final.
// mu_t is folded into the mode-3 factor in float64 before any rounding.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <string>
#include <vector>

#include "tx_internal.h"

namespace tx {
namespace {

// rows a of C_td at the target points xt (the grid itself, or the coarse nodes of the smooth terms)
__global__ void k_conv_factor(const double* __restrict__ xt, const double* __restrict__ x, const double* __restrict__ w,
                              const double* __restrict__ U, const double* __restrict__ theta,
                              const double* __restrict__ mu, int n, int r, int fold_mu,
                              double* __restrict__ A64, float* __restrict__ A32, float* __restrict__ C32) {
    extern __shared__ double kv[];   // [n]: row a of C_td
    const int a = blockIdx.x, t = blockIdx.y, na = gridDim.x;
    const double th = theta[t];
    for (int b = threadIdx.x; b < n; b += blockDim.x) {
        const double dx = xt[a] - x[b];
        kv[b] = w[b] * exp(-th * dx * dx);
    }
    __syncthreads();
    const double scale = fold_mu ? mu[t] : 1.0;
    if (C32)
        for (int b = threadIdx.x; b < n; b += blockDim.x) C32[((long)t * n + a) * n + b] = (float)(scale * kv[b]);
    for (int k = threadIdx.x; k < r; k += blockDim.x) {
        double s = 0.0;
        for (int b = 0; b < n; ++b) s = fma(kv[b], U[(long)b * r + k], s);
        s *= scale;
        const long o = ((long)t * na + a) * r + k;
        A64[o] = s;
        A32[o] = (float)s;
    }
}

// Finite-element quadrature (Eqs. quadVal, discInteg): the 1-D field is interpolated by Lagrange
// elements of order p (element e holds nodes p e .. p e + p) and each convolution integral is
// evaluated with q Gauss-Legendre points per element:
//   C_td[a][b] = sum_{e contains b} sum_q J_e w_q N_b(x_q) exp(-theta_t (x_a - x_q)^2)
__global__ void k_conv_factor_fe(const double* __restrict__ xt, const double* __restrict__ x, const double* __restrict__ U,
                                 const double* __restrict__ theta, const double* __restrict__ mu, int n, int r,
                                 int fold_mu, int p, int q, const double* __restrict__ gx, const double* __restrict__ gw,
                                 double* __restrict__ A64, float* __restrict__ A32, float* __restrict__ C32) {
    extern __shared__ double kv[];   // [n]: row a of C_td
    const int a = blockIdx.x, t = blockIdx.y, na = gridDim.x;
    const double th = theta[t], xa = xt[a];
    const int nel = (n - 1) / p;
    for (int b = threadIdx.x; b < n; b += blockDim.x) {
        double v = 0.0;
        // the one or two elements that hold node b
        const int e_hi = min(b / p, nel - 1);
        const int e_lo = (b % p == 0 && b > 0) ? b / p - 1 : e_hi;
        for (int e = e_lo; e <= e_hi; ++e) {
            const int k = b - p * e;                     // local node index in element e
            const double* xe = x + p * e;
            const double xl = xe[0], xr = xe[p], half = 0.5 * (xr - xl), mid = 0.5 * (xl + xr);
            for (int g = 0; g < q; ++g) {
                const double xq = mid + half * gx[g];
                double L = 1.0;
                for (int m = 0; m <= p; ++m)
                    if (m != k) L *= (xq - xe[m]) / (xe[k] - xe[m]);
                const double dx = xa - xq;
                v += half * gw[g] * L * exp(-th * dx * dx);
            }
        }
        kv[b] = v;
    }
    __syncthreads();
    const double scale = fold_mu ? mu[t] : 1.0;
    if (C32)
        for (int b = threadIdx.x; b < n; b += blockDim.x) C32[((long)t * n + a) * n + b] = (float)(scale * kv[b]);
    for (int k = threadIdx.x; k < r; k += blockDim.x) {
        double s = 0.0;
        for (int b = 0; b < n; ++b) s = fma(kv[b], U[(long)b * r + k], s);
        s *= scale;
        const long o = ((long)t * na + a) * r + k;
        A64[o] = s;
        A32[o] = (float)s;
    }
}

}  // namespace

// Gauss-Legendre nodes and weights on [-1, 1]: Newton's method on the Legendre polynomial P_q
// (three-term recurrence for P_q and its derivative), started from cos(pi (i - 1/4) / (q + 1/2)).
static void gauss_legendre(int q, double* xg, double* wg) {
    const double pi = 3.14159265358979323846;
    for (int i = 0; i < q; ++i) {
        double z = cos(pi * (i + 0.75) / (q + 0.5)), dp = 1.0;
        for (int it = 0; it < 100; ++it) {
            double p0 = 1.0, p1 = z;
            for (int k = 2; k <= q; ++k) {
                const double p2 = ((2.0 * k - 1.0) * z * p1 - (k - 1.0) * p0) / k;
                p0 = p1;
                p1 = p2;
            }
            dp = q * (z * p1 - p0) / (z * z - 1.0);
            const double dz = p1 / dp;
            z -= dz;
            if (fabs(dz) < 1e-16) break;
        }
        xg[i] = z;
        wg[i] = 2.0 / ((1.0 - z * z) * dp * dp);
    }
}

// A_td for nt terms at the target points xt (na of them), by the context's quadrature rule: FE
// elements where gx (Gauss points) is given, the nodal rule otherwise
static int conv_factors(const tx_ctx* c, int d, const double* xt, int na, const double* theta, const double* mu, int nt,
                        int order, int points, const double* gx, double* A64, float* A32, float* C32, cudaStream_t s) {
    const int n = c->n[d], r = c->r[d];
    const size_t smem = sizeof(double) * n;
    if (gx)
        k_conv_factor_fe<<<dim3(na, nt), 128, smem, s>>>(xt, c->d_x[d], c->d_U[d], theta, mu, n, r, d == 2 ? 1 : 0, order,
                                                         points, gx, gx + points, A64, A32, C32);
    else
        k_conv_factor<<<dim3(na, nt), 128, smem, s>>>(xt, c->d_x[d], c->d_w[d], c->d_U[d], theta, mu, n, r, d == 2 ? 1 : 0,
                                                      A64, A32, C32);
    TX_LAUNCHED();
    return TX_OK;
}

// the sharp terms' fine operators are some of the context's own (terms idx[0 .. ns - 1]), and the term after them
// (the interpolation, already there in float64) gets its float32 form
__global__ void __launch_bounds__(256) k_gather_terms(const double* __restrict__ A64, const float* __restrict__ A32,
                                                      const int* __restrict__ idx, int ns, long per,
                                                      double* __restrict__ F64, float* __restrict__ F32) {
    const long e = blockIdx.x * 256L + threadIdx.x, o = blockIdx.y * per + e;
    if (e >= per) return;
    if ((int)blockIdx.y < ns) {
        const long q = idx[blockIdx.y] * per + e;
        F64[o] = A64[q];
        F32[o] = A32[q];
    } else {
        F32[o] = (float)F64[o];
    }
}

static int ld_of(int d, int n) { return d == 1 ? simt_ld2(n) : simt_ld3(n); }

struct BasisArgs {
    const double* U[3];
    const double* w[3];
    double* UW[3];
    int r[3];
    long m[3];
};
__global__ void __launch_bounds__(256) k_weighted_basis(const BasisArgs a) {
    const int d = blockIdx.y;
    const long e = blockIdx.x * 256L + threadIdx.x;
    if (e < a.m[d]) a.UW[d][e] = a.U[d][e] * a.w[d][e / a.r[d]];
}

int setup_basis_forms(tx_ctx* c, cudaStream_t s) {
    BasisArgs a{};
    long most = 0;
    for (int d = 0; d < 3; ++d) {
        a.U[d] = c->d_U[d];
        a.w[d] = c->d_w[d];
        a.UW[d] = c->d_UW[d];
        a.r[d] = c->r[d];
        a.m[d] = (long)c->n[d] * c->r[d];
        most = std::max(most, a.m[d]);
    }
    k_weighted_basis<<<dim3((unsigned)((most + 255) / 256), 3), 256, 0, s>>>(a);
    TX_LAUNCHED();
    for (int d = 1; d < 3; ++d) TX_TRY(simt_kmajor(c->f_U[d], 1, c->n[d], c->r[d], ld_of(d, c->n[d]), c->f_UK[d], s));
    return TX_OK;
}

// every operator of the context for one quadrature rule
static int all_factors(tx_ctx* c, int order, int points, const double* gx, cudaStream_t s, bool with_c) {
    const TermSplit& ts = c->ts;
    for (int d = 0; d < 3; ++d) {
        const int n = c->n[d], r = c->r[d];
        TX_TRY(conv_factors(c, d, c->d_x[d], n, c->d_theta, c->d_mu, c->T, order, points, gx, c->d_A64[d], c->f_A[d],
                            with_c ? c->f_C[d] : nullptr, s));
        if (ts.nc) {
            const int ns = ts.nf - 1;
            const long per = (long)n * r;
            k_gather_terms<<<dim3((unsigned)((per + 255) / 256), (unsigned)ts.nf), 256, 0, s>>>(c->d_A64[d], c->f_A[d],
                                                                                                ts.d_idx, ns, per, ts.F64[d], ts.F[d]);
            TX_LAUNCHED();
            TX_TRY(conv_factors(c, d, ts.d_xi[d], r, ts.d_theta, ts.d_mu, ts.nc, order, points, gx, ts.Q64[d],
                                ts.Q[d], nullptr, s));
            if (d > 0) {
                TX_TRY(simt_kmajor(ts.Q[d], ts.nc, r, r, ld_of(d, r), ts.QK[d], s));
                TX_TRY(simt_kmajor(ts.Q[d], ts.nc, r, r, ld_of(3 - d, r), ts.QKs[d], s));
            }
        }
        if (d > 0) TX_TRY(simt_kmajor(ts.F[d], ts.nf, n, r, ld_of(d, n), ts.FK[d], s));
    }
    return TX_OK;
}

int setup_factor_matrices_fe(tx_ctx* c, int order, int points, cudaStream_t s, bool with_c) {
    double hx[64], hw[64];
    gauss_legendre(points, hx, hw);
    double* d = nullptr;
    if (cudaMalloc(&d, sizeof(double) * 2 * points) != cudaSuccess) {
        cudaGetLastError();
        return fail(TX_ERR_OOM, "quadrature points");
    }
    int st = TX_OK;
    if (cudaMemcpy(d, hx, sizeof(double) * points, cudaMemcpyHostToDevice) != cudaSuccess ||
        cudaMemcpy(d + points, hw, sizeof(double) * points, cudaMemcpyHostToDevice) != cudaSuccess)
        st = fail(TX_ERR_CUDA, "quadrature points copy");
    if (st == TX_OK) st = copies_done();
    if (st == TX_OK) st = all_factors(c, order, points, d, s, with_c);
    cudaStreamSynchronize(s);
    cudaFree(d);
    return st;
}

int setup_factor_matrices(tx_ctx* c, cudaStream_t s, bool with_c) { return all_factors(c, 0, 0, nullptr, s, with_c); }

// ======================================================================================
// the split of the Gaussian sum
// ======================================================================================
// Bound on the error of interpolating exp(-theta (x - c)^2), any real c, on an interval of half-length h
// at N + 1 Chebyshev nodes: 4 M rho^-N / (rho - 1) with M the largest modulus on the Bernstein ellipse of
// parameter rho = e^eta (Trefethen, Approximation Theory and Approximation Practice, Thm 8.2).  On the
// ellipse |Im z| <= h sinh(eta), so M = exp(theta h^2 sinh(eta)^2); the exponent
// theta h^2 sinh(eta)^2 - N eta is least at sinh(2 eta) = N / (theta h^2).
static double chebyshev_bound(double theta, double h, int N) {
    const double a = theta * h * h;
    const double eta = 0.5 * std::asinh((double)N / a), sh = std::sinh(eta);
    return 4.0 * std::exp(a * sh * sh - (double)N * eta) / (std::exp(eta) - 1.0);
}

// A term is smooth where every mode's r_d Chebyshev nodes interpolate its kernel to 1e-9 of its maximum:
// 60 times below the float32 rounding of the operators, so the split changes results by rounding only.
constexpr double kSmoothTol = 1e-9;

int smooth_terms(const int n[3], const int r[3], const double extent[3], int T, const double* theta, int* smooth) {
    int count = 0;
    for (int t = 0; t < T; ++t) {
        smooth[t] = 1;
        for (int d = 0; d < 3 && smooth[t]; ++d)
            smooth[t] = chebyshev_bound(theta[t], 0.5 * extent[d], r[d] - 1) <= kSmoothTol;
        count += smooth[t];
    }
    // worth it where the smooth terms' fine-grid work is more than their coarse work plus the
    // interpolation (one fine term); a tenth of a fine term stands for the extra launches
    auto mode_flops = [&](const int m[3]) {
        const double r1 = r[0], r2 = r[1], r3 = r[2];
        return m[0] * r1 * r2 * r3 + (double)m[0] * m[1] * r2 * r3 + (double)m[0] * m[1] * m[2] * r3;
    };
    const double fine = mode_flops(n), coarse = mode_flops(r), nc = (double)count;
    // (coarse grids up to 160 nodes per mode: every float32 kernel takes them)
    return nc * fine > 1.1 * fine + nc * coarse && std::max(r[1], r[2]) <= 160 ? count : 0;
}

int plan_terms(tx_ctx* c, const double* const x[3], const double* theta, const double* mu) {
    TermSplit& ts = c->ts;
    std::memset(&ts, 0, sizeof(ts));
    double lo[3], hi[3], extent[3];
    for (int d = 0; d < 3; ++d) {
        lo[d] = *std::min_element(x[d], x[d] + c->n[d]);
        hi[d] = *std::max_element(x[d], x[d] + c->n[d]);
        extent[d] = hi[d] - lo[d];
    }
    std::vector<int> smooth(c->T);
    std::vector<double> host;          // smooth exponents, weights, then the coarse nodes
    std::vector<int> idx;              // sharp terms
    ts.nc = smooth_terms(c->n, c->r, extent, c->T, theta, smooth.data());
    for (int t = 0; t < c->T; ++t)
        if (!smooth[t]) idx.push_back(t);
    const bool on = ts.nc > 0;
    ts.nf = on ? (int)idx.size() + 1 : c->T;
    // one allocation for every operator of the split
    struct Piece {
        void** p;
        size_t bytes;
    };
    std::vector<Piece> pieces;
    auto want = [&](auto** p, size_t count) { pieces.push_back(Piece{(void**)p, (sizeof(**p) * count + 255) & ~(size_t)255}); };
    for (int d = 0; d < 3; ++d) {
        const size_t n = c->n[d], r = c->r[d];
        if (d > 0) want(&ts.FK[d], (size_t)ts.nf * r * ld_of(d, (int)n));
        if (!on) {
            ts.F[d] = c->f_A[d];
            continue;
        }
        want(&ts.F64[d], (size_t)ts.nf * n * r);
        want(&ts.F[d], (size_t)ts.nf * n * r);
        want(&ts.Q64[d], (size_t)ts.nc * r * r);
        want(&ts.Q[d], (size_t)ts.nc * r * r);
        if (d > 0) want(&ts.QK[d], (size_t)ts.nc * r * ld_of(d, (int)r));
        if (d > 0) want(&ts.QKs[d], (size_t)ts.nc * r * ld_of(3 - d, (int)r));
    }
    // ... and one copy for the smooth terms' exponents and weights, the coarse nodes and the sharp terms' indices
    const size_t nodes = (size_t)c->r[0] + c->r[1] + c->r[2], small = sizeof(double) * (2 * ts.nc + nodes) + sizeof(int) * idx.size();
    if (on) want(&ts.d_theta, (small + 7) / 8);
    size_t total = 0;
    for (const Piece& q : pieces) total += q.bytes;
    if (cudaMalloc(&ts.pool, total) != cudaSuccess) {
        cudaGetLastError();
        ts.pool = nullptr;
        return fail(TX_ERR_OOM, "operators of the term split");
    }
    char* at = (char*)ts.pool;
    for (const Piece& q : pieces) {
        *q.p = at;
        at += q.bytes;
    }
    if (!on) return TX_OK;
    ts.d_mu = ts.d_theta + ts.nc;
    ts.d_xi[0] = ts.d_mu + ts.nc;
    ts.d_xi[1] = ts.d_xi[0] + c->r[0];
    ts.d_xi[2] = ts.d_xi[1] + c->r[1];
    ts.d_idx = (int*)(ts.d_xi[2] + c->r[2]);
    for (const double* v : {theta, mu})
        for (int t = 0; t < c->T; ++t)
            if (smooth[t]) host.push_back(v[t]);
    for (int d = 0; d < 3; ++d) {
        // Chebyshev nodes and the barycentric Lagrange values at the grid nodes
        const size_t n = c->n[d], r = c->r[d];
        const double pi = 3.14159265358979323846;
        std::vector<double> xi(r), bw(r), I(n * r);
        for (size_t k = 0; k < r; ++k) {
            xi[k] = 0.5 * (lo[d] + hi[d]) - 0.5 * (hi[d] - lo[d]) * std::cos(pi * (k + 0.5) / r);
            bw[k] = (k % 2 ? -1.0 : 1.0) * std::sin(pi * (k + 0.5) / r);
        }
        for (size_t a = 0; a < n; ++a) {
            double den = 0.0;
            size_t hit = r;
            for (size_t k = 0; k < r; ++k) {
                if (x[d][a] == xi[k]) hit = k;
                else den += bw[k] / (x[d][a] - xi[k]);
            }
            for (size_t k = 0; k < r; ++k)
                I[a * r + k] = hit < r ? (k == hit ? 1.0 : 0.0) : bw[k] / (x[d][a] - xi[k]) / den;
        }
        host.insert(host.end(), xi.begin(), xi.end());
        if (cudaMemcpy(ts.F64[d] + (size_t)(ts.nf - 1) * n * r, I.data(), sizeof(double) * n * r, cudaMemcpyHostToDevice) != cudaSuccess)
            return fail(TX_ERR_CUDA, "term split copy");
    }
    const size_t words = host.size();
    host.resize(words + (idx.size() + 1) / 2);
    std::memcpy(host.data() + words, idx.data(), sizeof(int) * idx.size());
    if (cudaMemcpy(ts.d_theta, host.data(), sizeof(double) * host.size(), cudaMemcpyHostToDevice) != cudaSuccess)
        return fail(TX_ERR_CUDA, "term split copy");
    return TX_OK;
}

void free_terms(tx_ctx* c) {
    cudaFree(c->ts.pool);
    std::memset(&c->ts, 0, sizeof(c->ts));
}

Shape fine_shape(const tx_ctx* c) {
    return Shape{c->n[0], c->n[1], c->n[2], c->r[0], c->r[1], c->r[2], c->f_w[0], c->f_w[1], c->f_w[2]};
}
Shape coarse_shape(const tx_ctx* c, bool swapped) {
    // the grid's own weights are not the coarse nodes', and with modes 2 and 3 exchanged n_2 of them may be
    // fewer than the r_3 rows
    const int r2 = swapped ? c->r[2] : c->r[1], r3 = swapped ? c->r[1] : c->r[2];
    return Shape{c->r[0], r2, r3, c->r[0], r2, r3, nullptr, nullptr, nullptr};
}

}  // namespace tx

namespace tx {

// float32 copies of the convolution matrices C_td (mu_t folded into mode 3), made on first use
// (the per-pair path needs them) with the context's current quadrature
int ensure_conv_matrices(tx_ctx* c, cudaStream_t s) {
    if (c->c_valid) return TX_OK;
    for (int d = 0; d < 3; ++d)
        if (!c->f_C[d]) {
            if (cudaMalloc(&c->f_C[d], sizeof(float) * (size_t)c->T * c->n[d] * c->n[d]) != cudaSuccess) {
                cudaGetLastError();
                c->f_C[d] = nullptr;
                return fail(TX_ERR_OOM, "convolution matrices");
            }
        }
    if (c->quad_order > 0) TX_TRY(setup_factor_matrices_fe(c, c->quad_order, c->quad_points, s, true));
    else TX_TRY(setup_factor_matrices(c, s, true));
    c->c_valid = true;
    return TX_OK;
}

}  // namespace tx
