// Model M2 of Sec. 2.2, second step: non-negative superposition weights of
// the dictionary Psi_q = diag(a_q) Phi_q (eq. psi_def) over all easy-axis
// angles (eq. LSfitM2), regularised by truncating the SVD of the stacked
// Sigma-weighted dictionary matrix M (eq. LSfitM2_alternative,
// eq. approx_low_rank).
//
//   fp_m2_gram (GPU)   the complex Gram matrix of [M | y]: every product the
//                      fit needs (M^H M, M^H y, y^H y), as one FP64 reduction
//                      over rows r = (angle, voxel, channel, frequency row)
//   fp_m2_solve (host) M^H M = V diag(s^2) V^H -> U_s^H M = diag(s_s) V_s^H and
//                      U_s^H y = diag(1/s_s) V_s^H M^H y; real and imaginary
//                      parts stacked (the weights are real); the quadratic
//                      program min 1/2 w^T Q w + f^T w, w >= 0 solved by a
//                      primal-dual interior-point method
#include <cuda_runtime.h>
#include <math.h>
#include <algorithm>
#include <cstring>
#include <vector>
#include "fp_internal.h"

#define M2_T 16            // output tile (M2_T x M2_T entries of the Gram matrix)
#define M2_R 16            // rows staged per step

struct GramArgs {
    const double2* phi;    // [A][J][N][C][K1]
    const double2* a;      // [A][J][C][K1]
    const double2* S;      // [A][N][C][K1]
    const double* smax;    // [A][C][K1]
    const int* ks;         // [nk]
    int A, J, N, C, K1, nk;
    long long R;           // rows = A N C nk
    long long rows_per_split;
    int ntile;             // tiles per side, ceil((J + 1) / M2_T)
    double2* G;            // [(J + 1)][(J + 1)]
};

// entry (r, col) of [M | y]: col < J -> sigma a Phi, col == J -> sigma S
__device__ __forceinline__ double2 m2_entry(const GramArgs& g, long long r, int col) {
    if (col > g.J) return make_double2(0.0, 0.0);
    const int kk = (int)(r % g.nk);
    long long t = r / g.nk;
    const int c = (int)(t % g.C);
    t /= g.C;
    const int nu = (int)(t % g.N);
    const int th = (int)(t / g.N);
    const int k = __ldg(g.ks + kk);
    const size_t ck = (size_t)c * g.K1 + k;
    const double m = __ldg(g.smax + (size_t)th * g.C * g.K1 + ck);
    const double sig = m > 0.0 ? 1.0 / m : 0.0;
    if (col == g.J) {
        const double2 s = __ldg(g.S + ((size_t)th * g.N + nu) * g.C * g.K1 + ck);
        return make_double2(sig * s.x, sig * s.y);
    }
    const double2 av = __ldg(g.a + ((size_t)th * g.J + col) * g.C * g.K1 + ck);
    const double2 p = __ldg(g.phi + (((size_t)th * g.J + col) * g.N + nu) * g.C * g.K1 + ck);
    return make_double2(sig * (av.x * p.x - av.y * p.y), sig * (av.x * p.y + av.y * p.x));
}

// blockIdx.x: upper-triangle tile (ti <= tj), blockIdx.y: row split.
// Thread (row u, column v) of the tile accumulates sum_r conj(M[r][i]) M[r][j].
__global__ void __launch_bounds__(M2_T * M2_T) fp_m2_gram_kernel(GramArgs g) {
    __shared__ double2 Mi[M2_R][M2_T], Mj[M2_R][M2_T];
    int ti = 0, rem = blockIdx.x;
    while (rem >= g.ntile - ti) { rem -= g.ntile - ti; ++ti; }
    const int tj = ti + rem;
    const int u = threadIdx.x / M2_T, v = threadIdx.x % M2_T;
    const int i = ti * M2_T + u, j = tj * M2_T + v;
    const long long r0 = (long long)blockIdx.y * g.rows_per_split;
    const long long r1 = min(g.R, r0 + g.rows_per_split);
    double re = 0.0, im = 0.0;
    // staging: thread (q, w) loads row r + q of columns ti*T + w and tj*T + w
    const int q = threadIdx.x % M2_R, w = threadIdx.x / M2_R;
    for (long long r = r0; r < r1; r += M2_R) {
        const long long rr = r + q;
        const bool ok = rr < r1;
        Mi[q][w] = ok ? m2_entry(g, rr, ti * M2_T + w) : make_double2(0.0, 0.0);
        Mj[q][w] = ok ? m2_entry(g, rr, tj * M2_T + w) : make_double2(0.0, 0.0);
        __syncthreads();
#pragma unroll
        for (int s = 0; s < M2_R; ++s) {
            const double2 x = Mi[s][u], y = Mj[s][v];
            re = fma(x.x, y.x, fma(x.y, y.y, re));      // conj(x) y
            im = fma(x.x, y.y, fma(-x.y, y.x, im));
        }
        __syncthreads();
    }
    if (i <= g.J && j <= g.J) {
        atomicAdd(&g.G[(size_t)i * (g.J + 1) + j].x, re);
        atomicAdd(&g.G[(size_t)i * (g.J + 1) + j].y, im);
    }
}

// The same for 17 to 128 columns, in one block: every entry of a row block is staged
// once for all products, and a thread keeps a 4 x 4 micro tile of complex sums in
// registers (16 products from 8 shared-memory reads).  The FP64 pipe bounds it:
// 4 operations a product at 2 a clock and SM; the tiled kernel above spends a
// third as many again on forming each staged entry once per tile of its row and
// column, and half its products on padding and on the lower halves of diagonal
// tiles.  With nt = ceil((J + 1) / 4) thread (u, v), u <= v, owns the columns
// u + a nt and v + b nt (a, b < 4): neighbouring threads read neighbouring
// entries, each unordered pair of columns falls to one thread (u = v: a <= b),
// and a pair met in the wrong order is stored conjugated.  Where the nt (nt + 1) / 2
// micro tiles fill only part of a block, further groups of threads take the
// staged rows alternately.  97 columns x 1.21 million rows: 105.1 ms -> 46.8 ms, 0.99 TFLOP/s counted over the
// upper triangle, 78 % of the measured FP64 rate (25 x 26 / 2 micro tiles hold 9 % more products than
// the triangle, 352 threads 8 % more than the tiles).
#define M2_RB 16           // rows staged per step
#define M2_MAXNT 32        // J + 1 <= 128: at most 528 threads and 33 KB of staged rows, within the 48 KB
                           // that every launch may use: a larger limit would be set per process, under
                           // the launches of other host threads
struct GramRow { long long phi, a, S; double sig; };

__global__ void __launch_bounds__(544, 1) fp_m2_gram_micro_kernel(GramArgs g, int nt, int groups) {
    extern __shared__ __align__(16) unsigned char sraw[];
    const int ld = 4 * nt + 1;                             // odd: the transposing stores hit distinct banks
    double2* M = (double2*)sraw;                           // [M2_RB][ld]
    __shared__ GramRow row[M2_RB];
    const int tiles = nt * (nt + 1) / 2;
    const int grp = threadIdx.x / tiles, t = threadIdx.x - grp * tiles;
    const bool worker = grp < groups;
    int u = 0, rem = t;                                    // t -> (u, v), u-major
    while (rem >= nt - u) { rem -= nt - u; ++u; }
    const int v = u + rem;
    double re[4][4], im[4][4];
#pragma unroll
    for (int a = 0; a < 4; ++a)
#pragma unroll
        for (int b = 0; b < 4; ++b) re[a][b] = im[a][b] = 0.0;
    const long long CK = (long long)g.C * g.K1;
    const long long r0 = (long long)blockIdx.x * g.rows_per_split;
    const long long r1 = min(g.R, r0 + g.rows_per_split);
    const int q = threadIdx.x % M2_RB, nw = blockDim.x / M2_RB, w0 = threadIdx.x / M2_RB;
    for (long long r = r0; r < r1; r += M2_RB) {
        if (threadIdx.x < M2_RB) {
            const long long rr = r + threadIdx.x;
            GramRow R{0, 0, 0, 0.0};
            if (rr < r1) {
                const int kk = (int)(rr % g.nk);
                long long x = rr / g.nk;
                const int c = (int)(x % g.C);
                x /= g.C;
                const int nu = (int)(x % g.N), th = (int)(x / g.N);
                const long long ck = (long long)c * g.K1 + __ldg(g.ks + kk);
                const double m = __ldg(g.smax + th * CK + ck);
                R.sig = m > 0.0 ? 1.0 / m : 0.0;
                R.phi = ((long long)th * g.J * g.N + nu) * CK + ck;
                R.a = (long long)th * g.J * CK + ck;
                R.S = ((long long)th * g.N + nu) * CK + ck;
            }
            row[threadIdx.x] = R;
        }
        __syncthreads();
        const GramRow R = row[q];
        const bool ok = r + q < r1;
        if (w0 < nw)
            for (int col = w0; col < 4 * nt; col += nw) {
                double2 e = make_double2(0.0, 0.0);
                if (ok && col < g.J) {
                    const double2 av = __ldg(g.a + R.a + col * CK);
                    const double2 p = __ldg(g.phi + R.phi + (long long)col * g.N * CK);
                    e = make_double2(R.sig * (av.x * p.x - av.y * p.y), R.sig * (av.x * p.y + av.y * p.x));
                } else if (ok && col == g.J) {
                    const double2 s = __ldg(g.S + R.S);
                    e = make_double2(R.sig * s.x, R.sig * s.y);
                }
                M[q * ld + col] = e;
            }
        __syncthreads();
        if (worker)
            for (int s = grp; s < M2_RB; s += groups) {
                const double2* m = M + s * ld;
                double2 x[4], y[4];
#pragma unroll
                for (int a = 0; a < 4; ++a) { x[a] = m[u + a * nt]; y[a] = m[v + a * nt]; }
#pragma unroll
                for (int a = 0; a < 4; ++a)
#pragma unroll
                    for (int b = 0; b < 4; ++b) {
                        re[a][b] = fma(x[a].x, y[b].x, fma(x[a].y, y[b].y, re[a][b]));      // conj(x) y
                        im[a][b] = fma(x[a].x, y[b].y, fma(-x[a].y, y[b].x, im[a][b]));
                    }
            }
        __syncthreads();
    }
    // the groups' sums meet in shared memory, so a block adds to G once
    double* buf = (double*)sraw;                           // [32][tiles]
    for (int h = 1; h < groups; ++h) {
        if (grp == h)
#pragma unroll
            for (int a = 0; a < 4; ++a)
#pragma unroll
                for (int b = 0; b < 4; ++b) {
                    buf[(8 * a + 2 * b) * tiles + t] = re[a][b];
                    buf[(8 * a + 2 * b + 1) * tiles + t] = im[a][b];
                }
        __syncthreads();
        if (grp == 0)
#pragma unroll
            for (int a = 0; a < 4; ++a)
#pragma unroll
                for (int b = 0; b < 4; ++b) {
                    re[a][b] += buf[(8 * a + 2 * b) * tiles + t];
                    im[a][b] += buf[(8 * a + 2 * b + 1) * tiles + t];
                }
        __syncthreads();
    }
    if (grp != 0) return;
#pragma unroll
    for (int a = 0; a < 4; ++a)
#pragma unroll
        for (int b = 0; b < 4; ++b) {
            const int i = u + a * nt, j = v + b * nt;
            if (i > g.J || j > g.J || (u == v && a > b)) continue;
            double2* o = g.G + (i <= j ? (size_t)i * (g.J + 1) + j : (size_t)j * (g.J + 1) + i);
            atomicAdd(&o->x, re[a][b]);
            atomicAdd(&o->y, i <= j ? im[a][b] : -im[a][b]);
        }
}

// --------------------------------------------------------- host algebra ----
// Cyclic Jacobi eigen-decomposition of a real symmetric n x n matrix (row
// major, destroyed): eigenvalues into ev, eigenvectors as the columns of V.
static void jacobi_eigen(int n, std::vector<double>& Am, std::vector<double>& ev, std::vector<double>& V) {
    V.assign((size_t)n * n, 0.0);
    for (int i = 0; i < n; ++i) V[(size_t)i * n + i] = 1.0;
    for (int sweep = 0; sweep < 60; ++sweep) {
        double off = 0.0, tot = 0.0;
        for (int p = 0; p < n; ++p)
            for (int q = 0; q < n; ++q) {
                const double x = Am[(size_t)p * n + q] * Am[(size_t)p * n + q];
                tot += x;
                if (p != q) off += x;
            }
        if (off <= 1e-30 * tot || off == 0.0) break;
        for (int p = 0; p < n - 1; ++p)
            for (int q = p + 1; q < n; ++q) {
                const double apq = Am[(size_t)p * n + q];
                if (apq == 0.0) continue;
                const double app = Am[(size_t)p * n + p], aqq = Am[(size_t)q * n + q];
                const double theta = (aqq - app) / (2.0 * apq);
                const double t = (theta >= 0 ? 1.0 : -1.0) / (std::fabs(theta) + std::sqrt(theta * theta + 1.0));
                const double c = 1.0 / std::sqrt(t * t + 1.0), s = t * c;
                for (int k = 0; k < n; ++k) {           // A <- A J (columns p, q)
                    const double akp = Am[(size_t)k * n + p], akq = Am[(size_t)k * n + q];
                    Am[(size_t)k * n + p] = c * akp - s * akq;
                    Am[(size_t)k * n + q] = s * akp + c * akq;
                }
                for (int k = 0; k < n; ++k) {           // A <- J^T A (rows p, q)
                    const double apk = Am[(size_t)p * n + k], aqk = Am[(size_t)q * n + k];
                    Am[(size_t)p * n + k] = c * apk - s * aqk;
                    Am[(size_t)q * n + k] = s * apk + c * aqk;
                }
                for (int k = 0; k < n; ++k) {
                    const double vkp = V[(size_t)k * n + p], vkq = V[(size_t)k * n + q];
                    V[(size_t)k * n + p] = c * vkp - s * vkq;
                    V[(size_t)k * n + q] = s * vkp + c * vkq;
                }
            }
    }
    ev.resize(n);
    for (int i = 0; i < n; ++i) ev[i] = Am[(size_t)i * n + i];
}

// Cholesky solve of the SPD n x n system K x = b (K destroyed); false if not SPD
static bool cholesky_solve(int n, std::vector<double>& K, std::vector<double>& x) {
    for (int j = 0; j < n; ++j) {
        double d = K[(size_t)j * n + j];
        for (int k = 0; k < j; ++k) d -= K[(size_t)j * n + k] * K[(size_t)j * n + k];
        if (!(d > 0.0)) return false;
        d = std::sqrt(d);
        K[(size_t)j * n + j] = d;
        for (int i = j + 1; i < n; ++i) {
            double v = K[(size_t)i * n + j];
            for (int k = 0; k < j; ++k) v -= K[(size_t)i * n + k] * K[(size_t)j * n + k];
            K[(size_t)i * n + j] = v / d;
        }
    }
    for (int i = 0; i < n; ++i) {
        double v = x[i];
        for (int k = 0; k < i; ++k) v -= K[(size_t)i * n + k] * x[k];
        x[i] = v / K[(size_t)i * n + i];
    }
    for (int i = n - 1; i >= 0; --i) {
        double v = x[i];
        for (int k = i + 1; k < n; ++k) v -= K[(size_t)k * n + i] * x[k];
        x[i] = v / K[(size_t)i * n + i];
    }
    return true;
}

static void qp_polish(int n, const std::vector<double>& Q, const std::vector<double>& f, std::vector<double>& w,
                      const std::vector<double>& z);

// min 1/2 w^T Q w + f^T w, w >= 0: primal-dual interior point (Mehrotra
// predictor-corrector) on Q w + f - z = 0, w z = mu, w, z > 0
static int qp_nonneg(int n, const std::vector<double>& Q, const std::vector<double>& f, std::vector<double>& w) {
    std::vector<double> z(n), rd(n), dw(n), dz(n), K((size_t)n * n), rhs(n), dwa(n), dza(n);
    double scale = 1.0;
    for (int i = 0; i < n; ++i) scale = std::max(scale, std::max(std::fabs(Q[(size_t)i * n + i]), std::fabs(f[i])));
    w.assign(n, 1.0);
    for (int i = 0; i < n; ++i) z[i] = scale;
    auto newton = [&](const std::vector<double>& rc, std::vector<double>& ow, std::vector<double>& oz) -> bool {
        // (Q + Z/W) dw = -rd - rc/w ;  dz = (-rc - z dw) / w
        for (size_t e = 0; e < K.size(); ++e) K[e] = Q[e];
        for (int i = 0; i < n; ++i) {
            K[(size_t)i * n + i] += z[i] / w[i];
            rhs[i] = -rd[i] - rc[i] / w[i];
        }
        if (!cholesky_solve(n, K, rhs)) return false;
        for (int i = 0; i < n; ++i) {
            ow[i] = rhs[i];
            oz[i] = (-rc[i] - z[i] * rhs[i]) / w[i];
        }
        return true;
    };
    auto step_to_boundary = [&](const std::vector<double>& a, const std::vector<double>& da) {
        double s = 1.0;
        for (int i = 0; i < n; ++i)
            if (da[i] < 0.0) s = std::min(s, -a[i] / da[i]);
        return s;
    };
    std::vector<double> rc(n);
    for (int it = 0; it < 200; ++it) {
        double mu = 0.0, rdn = 0.0;
        for (int i = 0; i < n; ++i) {
            double v = f[i] - z[i];
            for (int k = 0; k < n; ++k) v += Q[(size_t)i * n + k] * w[k];
            rd[i] = v;
            rdn = std::max(rdn, std::fabs(v));
            mu += w[i] * z[i];
        }
        mu /= n;
        if (mu <= 1e-15 * scale && rdn <= 1e-13 * scale) {
            qp_polish(n, Q, f, w, z);
            return it;
        }
        for (int i = 0; i < n; ++i) rc[i] = w[i] * z[i];                      // affine step
        if (!newton(rc, dwa, dza)) return -1;
        const double aw = step_to_boundary(w, dwa), az = step_to_boundary(z, dza);
        double mua = 0.0;
        for (int i = 0; i < n; ++i) mua += (w[i] + aw * dwa[i]) * (z[i] + az * dza[i]);
        mua /= n;
        const double sigma = std::pow(mua / mu, 3.0);
        for (int i = 0; i < n; ++i) rc[i] = w[i] * z[i] + dwa[i] * dza[i] - sigma * mu;   // corrector
        if (!newton(rc, dw, dz)) return -1;
        const double a = std::min(1.0, 0.995 * std::min(step_to_boundary(w, dw), step_to_boundary(z, dz)));
        for (int i = 0; i < n; ++i) {
            w[i] = std::max(w[i] + a * dw[i], 1e-300);
            z[i] = std::max(z[i] + a * dz[i], 1e-300);
        }
    }
    return -2;
}

static double qp_value(int n, const std::vector<double>& Q, const std::vector<double>& f, const std::vector<double>& w) {
    double v = 0.0;
    for (int i = 0; i < n; ++i) {
        double qi = 0.0;
        for (int k = 0; k < n; ++k) qi += Q[(size_t)i * n + k] * w[k];
        v += w[i] * (0.5 * qi + f[i]);
    }
    return v;
}

// Polish an interior-point solution: the components with w_i > z_i are taken
// as free, the rest as zero, and the free block solves Q_FF w_F = -f_F (no
// free component: the candidate is w = 0).  The result is kept if it is
// non-negative and does not raise the objective (interior points approach a
// degenerate optimum, where the gradient vanishes on zero weights too, only
// like sqrt(mu)).
static void qp_polish(int n, const std::vector<double>& Q, const std::vector<double>& f, std::vector<double>& w,
                      const std::vector<double>& z) {
    std::vector<int> F;
    for (int i = 0; i < n; ++i)
        if (w[i] > z[i]) F.push_back(i);
    const int m = (int)F.size();
    if (m == 0) {
        const std::vector<double> w0(n, 0.0);
        if (qp_value(n, Q, f, w0) <= qp_value(n, Q, f, w)) w = w0;
        return;
    }
    std::vector<double> K((size_t)m * m), x(m);
    for (int a = 0; a < m; ++a) {
        x[a] = -f[F[a]];
        for (int b = 0; b < m; ++b) K[(size_t)a * m + b] = Q[(size_t)F[a] * n + F[b]];
    }
    if (!cholesky_solve(m, K, x)) return;
    std::vector<double> wp(n, 0.0);
    for (int a = 0; a < m; ++a) {
        if (x[a] < 0.0) return;
        wp[F[a]] = x[a];
    }
    if (qp_value(n, Q, f, wp) <= qp_value(n, Q, f, w)) w = wp;
}

extern "C" {

long long fp_m2_gram_bytes(int J) { return (long long)(J + 1) * (J + 1) * 16; }

int fp_m2_gram(const double* d_phi, const double* d_a, const double* d_S, const double* d_smax, int A, int J, int N,
               int C, int K1, const int* d_ks, int nk, double* d_G, void* stream) {
    if (!d_phi || !d_a || !d_S || !d_smax || !d_ks || !d_G) return fp_fail(FP_EINVAL, "fp_m2_gram: NULL buffer");
    if (A < 1 || J < 1 || N < 1 || C < 1 || K1 < 1 || nk < 1) return fp_fail(FP_EINVAL, "fp_m2_gram: bad sizes");
    GramArgs g;
    g.phi = (const double2*)d_phi;
    g.a = (const double2*)d_a;
    g.S = (const double2*)d_S;
    g.smax = d_smax;
    g.ks = d_ks;
    g.A = A; g.J = J; g.N = N; g.C = C; g.K1 = K1; g.nk = nk;
    g.R = (long long)A * N * C * nk;
    g.ntile = (J + 1 + M2_T - 1) / M2_T;
    g.G = (double2*)d_G;
    const int tiles = g.ntile * (g.ntile + 1) / 2;
    int dev = 0, sms = 152;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    cudaStream_t st = (cudaStream_t)stream;
    if (cudaMemsetAsync(d_G, 0, (size_t)fp_m2_gram_bytes(J), st) != cudaSuccess)
        return fp_fail(FP_ECUDA, "fp_m2_gram: clearing the output failed");
    // row splits of the tiled kernel: four blocks an SM, whole steps of M2_R rows
    const long long max_split = (g.R + M2_R - 1) / M2_R;
    long long splits = (4LL * sms + tiles - 1) / tiles;
    if (splits > max_split) splits = max_split;
    if (splits > 65535) splits = 65535;
    const long long tiled_rows = ((g.R + splits - 1) / splits + M2_R - 1) / M2_R * M2_R;
    splits = (g.R + tiled_rows - 1) / tiled_rows;
    const int nt = (J + 1 + 3) / 4;
    if (nt >= 5 && nt <= M2_MAXNT && g.R >= 2048) {
        // 17 to 128 columns (below, the micro tiles fill less than half a warp; above, the
        // threads of one block do not suffice) and 2,048 rows or more; then the kernel that the
        // estimates name.  Both are steps of 16 rows on the busiest SM, in us, fitted to 930 times of 30
        // column counts and 31 row counts (the micro tiles within 22 %, on average 5 %, the tiled
        // kernel 13 % and 2 %): a step of the micro tiles takes 0.0165 us per row of a thread,
        // adding up the groups 1.8 us each; a step of the tiled kernel 5.8 us per block of the
        // SM and 1.4 us of latency.  Few rows leave the micro tiles' blocks with one step or
        // two and part of the SMs with twice the work of others: 17 columns x 2,304 rows 46 us
        // against 24 tiled, 8,192 rows 59 against 76; 64 x 2,720 rows 108 against 80, 4,096 rows
        // 111 against 129; 97 x 1.2 million rows 46.8 ms against 105.1
        const int mt = nt * (nt + 1) / 2;
        const int groups = mt > 128 ? 1 : (256 / mt < M2_RB ? 256 / mt : M2_RB);
        const int threads = (mt * groups + 31) / 32 * 32;
        const long long steps = (g.R + M2_RB - 1) / M2_RB;
        const long long ctas = steps < 2LL * sms ? steps : (mt * groups > 272 ? (long long)sms : 2LL * sms);
        const long long cta_steps = (steps + ctas - 1) / ctas, grid = (steps + cta_steps - 1) / cta_steps;
        const double micro_us = 12.5 + 1.8 * (groups - 1) +
                                0.0165 * (double)((grid + sms - 1) / sms * cta_steps) * threads *
                                    ((M2_RB + groups - 1) / groups);
        const double tiled_us = 6.8 + (double)(tiled_rows / M2_R) *
                                          (1.4 + 5.8 * (double)((tiles * splits + sms - 1) / sms));
        if (micro_us < 0.97 * tiled_us) {
            size_t sm = (size_t)M2_RB * (4 * nt + 1) * sizeof(double2);
            if (groups > 1 && sm < (size_t)mt * 256) sm = (size_t)mt * 256;
            g.rows_per_split = cta_steps * M2_RB;
            fp_m2_gram_micro_kernel<<<(unsigned)grid, threads, sm, st>>>(g, nt, groups);
            if (cudaGetLastError() != cudaSuccess) return fp_fail(FP_ECUDA, "fp_m2_gram: launch failed");
            return FP_OK;
        }
    }
    g.rows_per_split = tiled_rows;
    fp_m2_gram_kernel<<<dim3(tiles, (unsigned)splits), M2_T * M2_T, 0, st>>>(g);
    if (cudaGetLastError() != cudaSuccess) return fp_fail(FP_ECUDA, "fp_m2_gram: launch failed");
    return FP_OK;
}

int fp_m2_solve(const double* h_G, int J, int s_rank, double* h_w, double* h_objective, double* h_residual,
                double* h_sv) {
    if (!h_G || !h_w || J < 1) return fp_fail(FP_EINVAL, "fp_m2_solve: bad argument");
    const int J1 = J + 1;
    // Hermitian: the products are read from the upper triangle (i <= j) only
    auto G = [&](int i, int j, int part) {
        if (i <= j) return h_G[((size_t)i * J1 + j) * 2 + part];
        const double v = h_G[((size_t)j * J1 + i) * 2 + part];
        return part == 0 ? v : -v;
    };
    // Hermitian M^H M as the real symmetric [[Re, -Im], [Im, Re]] of size 2J
    const int n2 = 2 * J;
    std::vector<double> H((size_t)n2 * n2), ev, V;
    for (int i = 0; i < J; ++i)
        for (int j = 0; j < J; ++j) {
            const double re = G(i, j, 0), im = G(i, j, 1);
            H[(size_t)i * n2 + j] = re;
            H[(size_t)(i + J) * n2 + (j + J)] = re;
            H[(size_t)i * n2 + (j + J)] = -im;
            H[(size_t)(i + J) * n2 + j] = im;
        }
    jacobi_eigen(n2, H, ev, V);
    std::vector<int> order(n2);
    for (int i = 0; i < n2; ++i) order[i] = i;
    std::sort(order.begin(), order.end(), [&](int a, int b) { return ev[a] > ev[b]; });
    // complex orthonormal eigenvectors v = x + i y, one per eigenvalue pair
    std::vector<double> vr, vi, lam;
    for (int o = 0; o < n2 && (int)lam.size() < J; ++o) {
        const int col = order[o];
        std::vector<double> xr(J), xi(J);
        for (int i = 0; i < J; ++i) { xr[i] = V[(size_t)i * n2 + col]; xi[i] = V[(size_t)(i + J) * n2 + col]; }
        for (size_t q = 0; q < lam.size(); ++q) {       // remove components along chosen vectors
            double pr = 0.0, pi = 0.0;                  // <v_q, x> = sum conj(v_q) x
            for (int i = 0; i < J; ++i) {
                const double ar = vr[q * J + i], ai = vi[q * J + i];
                pr += ar * xr[i] + ai * xi[i];
                pi += ar * xi[i] - ai * xr[i];
            }
            for (int i = 0; i < J; ++i) {
                const double ar = vr[q * J + i], ai = vi[q * J + i];
                xr[i] -= pr * ar - pi * ai;
                xi[i] -= pr * ai + pi * ar;
            }
        }
        double nrm = 0.0;
        for (int i = 0; i < J; ++i) nrm += xr[i] * xr[i] + xi[i] * xi[i];
        if (nrm < 0.25) continue;                       // the partner i v of a chosen vector
        nrm = 1.0 / std::sqrt(nrm);
        for (int i = 0; i < J; ++i) { vr.push_back(xr[i] * nrm); vi.push_back(xi[i] * nrm); }
        lam.push_back(std::max(ev[col], 0.0));
    }
    const int nv = (int)lam.size();
    if (h_sv)
        for (int k = 0; k < J; ++k) h_sv[k] = k < nv ? std::sqrt(lam[k]) : 0.0;
    // reduced problem: rows diag(s) V^H (M columns) and diag(1/s) V^H M^H y (data)
    const double smax = nv > 0 ? std::sqrt(lam[0]) : 0.0;
    int s = (s_rank > 0 && s_rank < nv) ? s_rank : nv;
    while (s > 0 && !(std::sqrt(lam[s - 1]) > 1e-13 * smax)) --s;     // drop numerically zero directions
    std::vector<double> Gr((size_t)2 * s * J), hr(2 * s);
    for (int k = 0; k < s; ++k) {
        const double sk = std::sqrt(lam[k]);
        double br = 0.0, bi = 0.0;                      // (V^H M^H y)_k
        for (int i = 0; i < J; ++i) {
            const double ar = vr[k * J + i], ai = vi[k * J + i];      // conj(v_ik) (M^H y)_i
            const double yr = G(i, J, 0), yi = G(i, J, 1);
            br += ar * yr + ai * yi;
            bi += ar * yi - ai * yr;
            Gr[(size_t)k * J + i] = sk * ar;             // s_k conj(v_ik)
            Gr[(size_t)(s + k) * J + i] = -sk * ai;
        }
        hr[k] = br / sk;
        hr[s + k] = bi / sk;
    }
    std::vector<double> Q((size_t)J * J, 0.0), f(J, 0.0), w;
    for (int r = 0; r < 2 * s; ++r)
        for (int i = 0; i < J; ++i) {
            const double gi = Gr[(size_t)r * J + i];
            f[i] -= gi * hr[r];
            for (int j = 0; j < J; ++j) Q[(size_t)i * J + j] += gi * Gr[(size_t)r * J + j];
        }
    // weights of dictionary columns that are zero in the truncated problem
    // (Q_ii = |column i|^2 = 0, hence f_i = 0) leave the objective unchanged:
    // they are set to 0 and the QP runs over the others
    double qmax = 0.0;
    for (int i = 0; i < J; ++i) qmax = std::max(qmax, Q[(size_t)i * J + i]);
    std::vector<int> act;
    for (int i = 0; i < J; ++i)
        if (Q[(size_t)i * J + i] > 1e-24 * qmax) act.push_back(i);
    const int na = (int)act.size();
    w.assign(J, 0.0);
    if (na > 0) {
        std::vector<double> Qa((size_t)na * na), fa(na), wa;
        for (int a = 0; a < na; ++a) {
            fa[a] = f[act[a]];
            for (int b = 0; b < na; ++b) Qa[(size_t)a * na + b] = Q[(size_t)act[a] * J + act[b]];
        }
        const int its = qp_nonneg(na, Qa, fa, wa);
        if (its < 0)
            return fp_fail(FP_EUNSUPPORTED, "fp_m2_solve: interior-point iteration did not converge (%d)", its);
        for (int a = 0; a < na; ++a) w[act[a]] = wa[a];
    }
    double obj = 0.0;                                    // ||Gr w - hr||^2
    for (int r = 0; r < 2 * s; ++r) {
        double v = -hr[r];
        for (int i = 0; i < J; ++i) v += Gr[(size_t)r * J + i] * w[i];
        obj += v * v;
    }
    for (int i = 0; i < J; ++i) h_w[i] = w[i];
    if (h_objective) *h_objective = obj;
    if (h_residual) {                                    // ||M w - y||^2 from the Gram matrix
        double r2 = G(J, J, 0);
        for (int i = 0; i < J; ++i) {
            r2 -= 2.0 * w[i] * G(i, J, 0);
            for (int j = 0; j < J; ++j) r2 += w[i] * w[j] * G(i, j, 0);
        }
        *h_residual = r2 > 0.0 ? r2 : 0.0;
    }
    return s;
}

}  // extern "C"
