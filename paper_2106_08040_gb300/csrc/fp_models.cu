// Data-driven system-matrix models of Sec. 2.2 and the distance measures of
// Sec. 2.3 on sm_103a:
//   fp_equilibrium  -- model M0: the equilibrium mean moment m_equ/m0 =
//                      L(bT |B|) B/|B| (Eq. Langevin) and its exact time
//                      derivative at every output sample, in the layout of
//                      fp_solve_batch (so fp_signal turns it into phi_hat_D)
//   fp_m1_fit       -- model M1 (and M0): per dictionary element q, channel c
//                      and row k, a_qk = S_k conj(Phi_qk)^T / ||Phi_qk||^2 and the
//                      row error of Eq. error1 for S_model = diag(a_q) Phi_q
//   fp_nrmse        -- per-frequency and global NRMSE (eq. globalMeasure) from
//                      row errors over a frequency index set
//   fp_mixing_order / fp_freq_index_set -- Eq. mix and I_freq (host only)
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>
#include <type_traits>
#include "fp_internal.h"

// ------------------------------------------------------------- Langevin ----
// L(x) = coth x - 1/x = sum_n c_n x^(2n-1), c_n = 2^(2n) B_2n / (2n)!  (B_2n the
// Bernoulli numbers), n = 1..11; below x = 0.5 the closed form cancels
// (relative error ~ 3 eps / x^2), so g = L/x and d = L' - g come from the series
// there: g = sum c_n x^(2n-2), d = sum (2n-2) c_n x^(2n-2).
#define FP_LSER_N 11
#define FP_LSER_MAX 0.5
__constant__ double c_lser[FP_LSER_N];

static void langevin_series(double* c) {
    // reduced fractions 2^(2n) B_2n / (2n)!, divided in long double
    static const long double num[FP_LSER_N] = {1.0L, -1.0L, 2.0L, -1.0L, 2.0L, -1382.0L, 4.0L, -3617.0L, 87734.0L,
                                               -349222.0L, 310732.0L};
    static const long double den[FP_LSER_N] = {3.0L, 45.0L, 945.0L, 4725.0L, 93555.0L, 638512875.0L, 18243225.0L,
                                               162820783125.0L, 38979295480125.0L, 1531329465290625.0L,
                                               13447856940643125.0L};
    for (int i = 0; i < FP_LSER_N; ++i) c[i] = (double)(num[i] / den[i]);
}

// g = L(x)/x and d = L'(x) - L(x)/x for x >= 0; ix = 1/x (read above FP_LSER_MAX only)
__device__ __forceinline__ void langevin_gd(double x, double ix, double& g, double& d) {
    if (x < FP_LSER_MAX) {
        const double x2 = x * x;
        double gs = c_lser[FP_LSER_N - 1], ds = (2.0 * FP_LSER_N - 2.0) * c_lser[FP_LSER_N - 1];
#pragma unroll
        for (int n = FP_LSER_N - 2; n >= 0; --n) {
            gs = fma(gs, x2, c_lser[n]);
            ds = fma(ds, x2, (2.0 * n) * c_lser[n]);
        }
        g = gs;
        d = ds;
    } else {
        const double e = exp(-2.0 * x), r = 1.0 / (1.0 - e);
        const double coth = (1.0 + e) * r, csch2 = 4.0 * e * r * r;
        g = (coth - ix) * ix;
        d = (ix * ix - csch2) - g;
    }
}

struct EqArgs {
    fp_material mat;
    fp_drive drv;
    const fp_instance* inst;
    int n, S_out;
    double* m_out;
    double* dmdt_out;
};

// A thread takes one sample and FP_EQ_MAXG instances at most; a block 2^lw samples of 128 >> lw groups
// of instances (instance q of the block belongs to group q mod their number): B = off + amp sin(w t + ph),
// dB/dt = amp w cos(w t + ph); m = L(xi) B/|B| = bT g B,
// dm/dt = bT [g dB/dt + d (Bhat . dB/dt) Bhat]   (xi = bT |B|).
// The FP64 pipe bounds it: the drive's three sincos (the larger half of the
// operations) depend on the sample alone and are formed once per thread, the
// instance's bT and 1/bT once per CTA, and the quotients share one reciprocal
// square root of |B|^2 and one of 1 - e^(-2 xi).  1,024 instances x 1,632 samples
// with fp_signal (816 harmonics, 2 channels): 11.02 ms -> 0.67 ms together.
// An SM's pipe serves a warp in the same time however few of its lanes have a sample: blocks of 128
// samples throughout made 129 samples x 1,024 instances 77 us, 64 us with a thread per
// sample and instance; the launch takes 8 samples a block there, 55 us.
#define FP_EQ_BS 128
#define FP_EQ_MAXG 16
#define FP_EQ_MINLW 2                                     // 4 samples a block at least: 96 bytes of an instance
#define FP_EQ_MAXI (FP_EQ_MAXG * (FP_EQ_BS >> FP_EQ_MINLW))
__global__ void __launch_bounds__(FP_EQ_BS) fp_equilibrium_kernel(EqArgs A, int G, int lw) {
    __shared__ double si[FP_EQ_MAXI][5];                  // offset (3), bT (-1: no moment), 1 / bT
    const int j = (blockIdx.x << lw) + (threadIdx.x & ((1 << lw) - 1));
    const int group = threadIdx.x >> lw, groups = FP_EQ_BS >> lw;
    const double twopi = 6.283185307179586476925286766559;
    double Bs[3], Bd[3];
    if (j < A.S_out) {
        const double t = ((double)A.drv.warmup_periods + (double)j / (double)A.drv.samples_per_period) * A.drv.period;
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            const double w = twopi * A.drv.freq[k];
            double s, c;
            sincos(w * t + A.drv.phase[k], &s, &c);
            Bs[k] = A.drv.amp[k] * s;
            Bd[k] = A.drv.amp[k] * w * c;
        }
    }
    for (long long i0 = (long long)blockIdx.y * G; i0 < A.n; i0 += (long long)gridDim.y * G) {
        const int gn = (int)(A.n - i0 < G ? A.n - i0 : G);
        __syncthreads();
        for (int q = threadIdx.x; q < gn; q += FP_EQ_BS) {
            const fp_instance& in = A.inst[i0 + q];
            const double d = in.d;
            const bool ok = d > 0.0 && in.flags == 0;
            const double V = 3.14159265358979323846 * d * d * d / 6.0;
            const double bT = V * A.mat.Ms / (FP_KB * A.mat.T_B);
            double* s = si[q];
            for (int k = 0; k < 3; ++k) s[k] = in.h_off[k];
            s[3] = ok ? bT : -1.0;
            s[4] = 1.0 / bT;
        }
        __syncthreads();
        if (j >= A.S_out) continue;
        for (int q = group; q < gn; q += groups) {
            const double* s = si[q];
            const size_t e = ((size_t)(i0 + q) * A.S_out + j) * 3;
            const double bT = s[3];
            double m[3] = {0.0, 0.0, 0.0}, dm[3] = {0.0, 0.0, 0.0};
            if (!(bT < 0.0)) {
                const double B[3] = {s[0] + Bs[0], s[1] + Bs[1], s[2] + Bs[2]};
                const double n2 = B[0] * B[0] + B[1] * B[1] + B[2] * B[2];
                // a field whose square leaves the normal range takes the plain root
                const bool in_range = n2 > 1e-290 && n2 < 1e290;
                const double nb = in_range ? n2 * rsqrt(n2) : sqrt(n2);
                const double inb = in_range ? rsqrt(n2) : (nb > 0.0 ? 1.0 / nb : 0.0);
                double g, d;
                langevin_gd(bT * nb, inb * s[4], g, d);
                const double bh[3] = {B[0] * inb, B[1] * inb, B[2] * inb};
                const double proj = bh[0] * Bd[0] + bh[1] * Bd[1] + bh[2] * Bd[2];
#pragma unroll
                for (int k = 0; k < 3; ++k) {
                    m[k] = bT * g * B[k];
                    dm[k] = bT * fma(d * proj, bh[k], g * Bd[k]);
                }
            }
#pragma unroll
            for (int k = 0; k < 3; ++k) {
                if (A.m_out) A.m_out[e + k] = m[k];
                if (A.dmdt_out) A.dmdt_out[e + k] = dm[k];
            }
        }
    }
}

// -------------------------------------------------------------- M1 fit ----
// Columns (c, k) are contiguous in the [N][C][K1] layout, so a block takes
// COLS consecutive columns of one dictionary element and VG voxel groups
// (voxels nu = g, g + VG, ...); partial sums meet in shared memory.

// Both passes are bound by the FP64 pipe (12 operations an entry at 2 a clock
// and SM), HBM runs at a quarter of its rate: so max |S|^2 is formed by the
// first element's CTAs alone, and the residual's two products and subtraction
// are two fused operations a component.  96 elements x 1,024 voxels x 1,634
// columns with fp_nrmse: 5.41 ms -> 3.37 ms; the FP64 floor is 3.07 ms.
// pass 1: a = sum S conj(Phi) / sum |Phi|^2 and (q = 0) max |S| per column
template <int COLS, int VG>
__global__ void __launch_bounds__(COLS * VG) fp_m1_pass1(const double2* __restrict__ phi, const double2* __restrict__ S, int N, int CK,
                            double2* __restrict__ a, double* __restrict__ smax) {
    __shared__ double red[VG][COLS][4];
    const int col = blockIdx.x * COLS + (threadIdx.x % COLS);
    const int g = threadIdx.x / COLS;
    const int q = blockIdx.y;
    double sr = 0.0, si = 0.0, pp = 0.0, mx = 0.0;
    if (col < CK) {
        const double2* P = phi + (size_t)q * N * CK + col;
        const double2* Sv = S + col;
        auto sums = [&](auto with_max) {                      // one pass over the data either way
#pragma unroll 4
            for (int nu = g; nu < N; nu += VG) {
                const double2 p = __ldg(P + (size_t)nu * CK), s = __ldg(Sv + (size_t)nu * CK);
                sr = fma(s.x, p.x, fma(s.y, p.y, sr));      // S conj(Phi)
                si = fma(s.y, p.x, fma(-s.x, p.y, si));
                pp = fma(p.x, p.x, fma(p.y, p.y, pp));
                if (decltype(with_max)::value) mx = fmax(mx, s.x * s.x + s.y * s.y);
            }
        };
        if (q == 0) sums(std::true_type());
        else sums(std::false_type());
    }
    const int cl = threadIdx.x % COLS;
    red[g][cl][0] = sr; red[g][cl][1] = si; red[g][cl][2] = pp; red[g][cl][3] = mx;
    __syncthreads();
    if (g == 0 && col < CK) {
        for (int h = 1; h < VG; ++h) {
            sr += red[h][cl][0]; si += red[h][cl][1]; pp += red[h][cl][2]; mx = fmax(mx, red[h][cl][3]);
        }
        const double ip = pp > 0.0 ? 1.0 / pp : 0.0;
        a[(size_t)q * CK + col] = make_double2(sr * ip, si * ip);
        if (q == 0) smax[col] = sqrt(mx);
    }
}

// pass 2: eps = sqrt(sum |S - a Phi|^2 / N) / max |S|
template <int COLS, int VG>
__global__ void __launch_bounds__(COLS * VG) fp_m1_pass2(const double2* __restrict__ phi, const double2* __restrict__ S, int N, int CK,
                            const double2* __restrict__ a, const double* __restrict__ smax, double* __restrict__ eps) {
    __shared__ double red[VG][COLS];
    const int col = blockIdx.x * COLS + (threadIdx.x % COLS);
    const int g = threadIdx.x / COLS;
    const int q = blockIdx.y;
    double rr = 0.0;
    if (col < CK) {
        const double2 av = a[(size_t)q * CK + col];
        const double2* P = phi + (size_t)q * N * CK + col;
        const double2* Sv = S + col;
#pragma unroll 4
        for (int nu = g; nu < N; nu += VG) {
            const double2 p = __ldg(P + (size_t)nu * CK), s = __ldg(Sv + (size_t)nu * CK);
            const double dr = fma(-av.x, p.x, fma(av.y, p.y, s.x));
            const double di = fma(-av.x, p.y, fma(-av.y, p.x, s.y));
            rr = fma(dr, dr, fma(di, di, rr));
        }
    }
    const int cl = threadIdx.x % COLS;
    red[g][cl] = rr;
    __syncthreads();
    if (g == 0 && col < CK) {
        for (int h = 1; h < VG; ++h) rr += red[h][cl];
        const double m = smax[col];
        eps[(size_t)q * CK + col] = m > 0.0 ? sqrt(rr / N) / m : 0.0;
    }
}

// sums over (angle, channel) rows of eps^2 at the harmonics kof(i), i < cnt.  More than
// FP_NRMSE_NK harmonics: one to each of FP_NRMSE_BS threads, loads in flight over the rows and no
// barriers (rows x harmonics with both sums: 1 x 20,000 151 us, 16 x 817 19, 64 x 817 40; with
// the form below 355, 35 and 69).  Up to that many, where most of those threads would have
// nothing to do: warp w takes rows w, w + 32, ..., a lane four harmonics; the row groups
// meet in shared memory and thread i adds up one harmonic (64 rows x 40: 15 us, 31 by one
// thread per harmonic).  Whole warps at a time either way: an FP64 instruction holds the SM's
// pipe for 16 clocks however many lanes it serves.  part: one buffer for every instance of
// the template, within the 48 KB of static shared memory
#define FP_NRMSE_BS 512
#define FP_NRMSE_NK 128
template <class KOf, class Out>
__device__ __forceinline__ void nrmse_sums(const double* __restrict__ eps, int rows, int K1, int cnt,
                                           double (*part)[FP_NRMSE_NK], KOf kof, Out out) {
    if (cnt > FP_NRMSE_NK) {
        if (threadIdx.x < FP_NRMSE_BS)
            for (int i = threadIdx.x; i < cnt; i += FP_NRMSE_BS) {
                const double* e = eps + kof(i);
                double v = 0.0;
                int r = 0;
                if (rows >= 16) {                                 // four chains: shorter sums, smaller error
                    double u[4] = {0.0, 0.0, 0.0, 0.0};
                    for (; r + 4 <= rows; r += 4)
#pragma unroll
                        for (int c = 0; c < 4; ++c) {
                            const double x = __ldg(e + (size_t)(r + c) * K1);
                            u[c] = fma(x, x, u[c]);
                        }
                    v = (u[0] + u[1]) + (u[2] + u[3]);
                }
                for (; r < rows; ++r) {
                    const double x = __ldg(e + (size_t)r * K1);
                    v = fma(x, x, v);
                }
                out(i, v);
            }
        return;
    }
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31, nw = min(32, rows);
    double s[4] = {0.0, 0.0, 0.0, 0.0};
    int k[4];
#pragma unroll
    for (int c = 0; c < 4; ++c) k[c] = kof(min(32 * c + lane, cnt - 1));
    if (w < nw) {
        for (int r = w; r < rows; r += 32)
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                const double v = __ldg(eps + (size_t)r * K1 + k[c]);
                s[c] = fma(v, v, s[c]);
            }
#pragma unroll
        for (int c = 0; c < 4; ++c) part[w][32 * c + lane] = s[c];
    }
    __syncthreads();
    if (threadIdx.x < cnt) {
        double v = 0.0;
        for (int h = 0; h < nw; ++h) v += part[h][threadIdx.x];
        out(threadIdx.x, v);
    }
    __syncthreads();
}

// eps_freq[k] = sqrt(mean over (angle, channel) of eps^2); global = sqrt(mean over I_freq of eps_freq^2).
// One CTA of 4 to 32 warps.
__global__ void __launch_bounds__(1024) fp_nrmse_kernel(const double* __restrict__ eps, int A, int C, int K1,
                                                        const int* __restrict__ ks, int nk,
                                                        double* __restrict__ eps_freq, double* __restrict__ eps_global) {
    __shared__ double part[32][FP_NRMSE_NK], red[FP_NRMSE_BS];
    const double inv = (double)(A * C);
    if (eps_freq)
        nrmse_sums(eps, A * C, K1, K1, part, [](int i) { return i; },
                   [&](int i, double v) { eps_freq[i] = sqrt(v / inv); });
    double acc = 0.0;
    nrmse_sums(eps, A * C, K1, nk, part, [&](int i) { return __ldg(ks + i); }, [&](int, double v) { acc += v / inv; });
    const int width = nk > FP_NRMSE_NK ? FP_NRMSE_BS : FP_NRMSE_NK;     // threads that hold a part of the sum
    if (threadIdx.x < width) red[threadIdx.x] = acc;
    __syncthreads();
    for (int o = width / 2; o > 0; o >>= 1) {
        if (threadIdx.x < o) red[threadIdx.x] += red[threadIdx.x + o];
        __syncthreads();
    }
    if (threadIdx.x == 0) *eps_global = sqrt(red[0] / (double)nk);
}

// ------------------------------------------------------------- C ABI ------
static int g_lser_device = -1;

extern "C" {

int fp_equilibrium(fp_ctx* ctx, const fp_instance* d_inst, int n, double* d_m, double* d_dmdt, void* stream) {
    if (!ctx) return fp_fail(FP_EINVAL, "fp_equilibrium: NULL ctx");
    if (n < 0) return fp_fail(FP_EINVAL, "fp_equilibrium: n < 0");
    if (n == 0) return FP_OK;
    if (!d_inst || (!d_m && !d_dmdt)) return fp_fail(FP_EINVAL, "fp_equilibrium: NULL buffer");
    if (g_lser_device != ctx->device) {
        double c[FP_LSER_N];
        langevin_series(c);
        if (cudaMemcpyToSymbol(c_lser, c, sizeof(c)) != cudaSuccess)
            return fp_fail(FP_ECUDA, "fp_equilibrium: constant upload failed");
        g_lser_device = ctx->device;
    }
    EqArgs A;
    A.mat = ctx->mat;
    A.drv = ctx->drv;
    A.inst = d_inst;
    A.n = n;
    A.S_out = ctx->drv.output_periods * ctx->drv.samples_per_period;
    A.m_out = d_m;
    A.dmdt_out = d_dmdt;
    // samples a block: 128 (lw = 7), or 32 to 4 where that leaves fewer lanes without a sample.  Per
    // instance the FP64 pipe serves about as many lanes as lanes(): whole warps with 128 to a block,
    // whose idle warps count half beside the other blocks' (they hold their place on the SM), and
    // with fewer some 8 more for the drive, which is formed for fewer instances per thread.  Us by
    // 128 / by this rule / by the one thread per sample and instance before, 5,000 instances: 3
    // samples 39 / 17 / 20, 33 70 / 49 / 81, 64 70 / 70 / 140, 129 217 / 125 / 257, 300 289 / 226 / 578, 816 632 / 617 / 1,544
    int lw = 7;
    auto lanes = [&](int l) {
        const double S = A.S_out, groups = FP_EQ_BS >> l, fill = ceil(n / groups) * groups / n;
        if (l < 7) return (ceil(S / (1 << l)) * (1 << l) + 8.0) * fill;
        const double warps = ceil(S / 32.0) * 32.0, tiles = ceil(S / FP_EQ_BS);
        return tiles > 1.0 ? 0.5 * (warps + tiles * FP_EQ_BS) : warps;
    };
    for (int l = 5; l >= FP_EQ_MINLW; --l)
        if (lanes(l) < 0.97 * lanes(lw)) lw = l;
    // as many instances per thread as leave eight CTAs for every SM, four or two of those without idle warps
    const int tiles = ((A.S_out - 1) >> lw) + 1, groups = FP_EQ_BS >> lw, ctas = lw == 7 ? 8 : lw > 2 ? 4 : 2;
    long long G = (long long)n * tiles / groups / ((long long)ctas * ctx->num_sms);
    G = (G < 1 ? 1 : G > FP_EQ_MAXG ? FP_EQ_MAXG : G) * groups;
    const long long gy = (n + G - 1) / G;
    fp_equilibrium_kernel<<<dim3((unsigned)tiles, (unsigned)(gy < 65535 ? gy : 65535)), FP_EQ_BS, 0, (cudaStream_t)stream>>>(
        A, (int)G, lw);
    if (cudaGetLastError() != cudaSuccess) return fp_fail(FP_ECUDA, "fp_equilibrium: launch failed");
    return FP_OK;
}

int fp_m1_fit(const double* d_phi, int Q, const double* d_S, int N, int C, int K1, double* d_a, double* d_eps,
              double* d_smax, void* stream) {
    if (!d_phi || !d_S || !d_a || !d_eps || !d_smax) return fp_fail(FP_EINVAL, "fp_m1_fit: NULL buffer");
    if (Q < 0 || N < 0 || C < 1 || K1 < 1) return fp_fail(FP_EINVAL, "fp_m1_fit: bad sizes");
    if (Q == 0 || N == 0) return FP_OK;
    if (Q > 65535) return fp_fail(FP_EINVAL, "fp_m1_fit: Q=%d > 65535 dictionary elements per call", Q);
    const int CK = C * K1;
    cudaStream_t st = (cudaStream_t)stream;
    // Wide blocks (64 columns, four voxel groups), or narrow ones (16 columns, 32 groups: eight times
    // the parallel chains) where wide ones leave SMs idle and there are voxels enough to pay for the
    // reduction over 32 groups.  How many it takes depends on how many narrow blocks share an SM, one
    // to eight up to two wide blocks per SM; measured on both sides of each line (us, wide / narrow):
    // 16 wide blocks 17 / 17 at 32 voxels, 25 / 18 at 64; 52 blocks 19 / 21 at 40, 23 / 21 at 48; 104
    // blocks 41 / 45 at 128, 77 / 72 at 277; 140 blocks 56 / 60 at 192, 142 / 126 at 512; 200 blocks 65 / 68
    // at 128, 93 / 85 at 192; 260 blocks 133 / 138 at 277, 242 / 222 at 512.  Below 33 voxels wide ones
    // always (1 element x 16 x 40: 13 us, 17 by narrow ones)
    static const int min_voxels[9] = {0, 33, 44, 192, 272, 128, 160, 336, 640};
    int dev = 0, sms = 152;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    const long long wide = (long long)((CK + 63) / 64) * Q, per_sm = ((long long)((CK + 15) / 16) * Q + sms - 1) / sms;
    const bool narrow = wide < 2LL * sms && N >= min_voxels[per_sm < 8 ? per_sm : 8];
    auto run = [&](auto cols, auto vg) {
        constexpr int COLS = decltype(cols)::value, VG = decltype(vg)::value;
        const dim3 grid((CK + COLS - 1) / COLS, Q);
        fp_m1_pass1<COLS, VG><<<grid, COLS * VG, 0, st>>>((const double2*)d_phi, (const double2*)d_S, N, CK,
                                                          (double2*)d_a, d_smax);
        fp_m1_pass2<COLS, VG><<<grid, COLS * VG, 0, st>>>((const double2*)d_phi, (const double2*)d_S, N, CK,
                                                          (const double2*)d_a, d_smax, d_eps);
    };
    if (narrow) run(std::integral_constant<int, 16>(), std::integral_constant<int, 32>());
    else run(std::integral_constant<int, 64>(), std::integral_constant<int, 4>());
    if (cudaGetLastError() != cudaSuccess) return fp_fail(FP_ECUDA, "fp_m1_fit: launch failed");
    return FP_OK;
}

int fp_nrmse(const double* d_eps, int A, int C, int K1, const int* d_ks, int nk, double* d_eps_freq,
             double* d_eps_global, void* stream) {
    if (!d_eps || !d_ks || !d_eps_global) return fp_fail(FP_EINVAL, "fp_nrmse: NULL buffer");
    if (A < 1 || C < 1 || K1 < 1 || nk < 1) return fp_fail(FP_EINVAL, "fp_nrmse: bad sizes");
    // a warp per row, at most 32; four at least take the harmonics (1 row x 40 harmonics with the
    // fit: 25 us with 32 warps, for their barriers), FP_NRMSE_BS threads where there are more of them
    const int rows = A * C, most = d_eps_freq && K1 > nk ? K1 : nk;
    int threads = 32 * (rows < 4 ? 4 : rows > 32 ? 32 : rows);
    if (most > FP_NRMSE_NK && threads < FP_NRMSE_BS) threads = FP_NRMSE_BS;
    fp_nrmse_kernel<<<1, threads, 0, (cudaStream_t)stream>>>(d_eps, A, C, K1, d_ks, nk, d_eps_freq, d_eps_global);
    if (cudaGetLastError() != cudaSuccess) return fp_fail(FP_ECUDA, "fp_nrmse: launch failed");
    return FP_OK;
}

int fp_mixing_order(int k, int n_dens, int* mx, int* my) {
    if (n_dens < 1 || !mx || !my) return fp_fail(FP_EINVAL, "fp_mixing_order: bad argument");
    // every solution of k = m_x n + m_y (n + 1) has m_y = k (mod n): scan m_y
    // over enough periods on both sides and keep the smallest |m_x| + |m_y|
    // (then the smaller |m_x|, then m_x >= 0)
    const long long n = n_dens, kk = k;
    long long r0 = kk % n;
    if (r0 < 0) r0 += n;
    const long long span = (kk < 0 ? -kk : kk) / n + 2;
    long long best_key0 = -1, best_key1 = 0, best_key2 = 0, bx = 0, by = 0;
    for (long long j = -span; j <= span; ++j) {
        const long long yv = r0 + j * n;
        const long long rem = kk - yv * (n + 1);
        if (rem % n) continue;
        const long long xv = rem / n;
        const long long k0 = (xv < 0 ? -xv : xv) + (yv < 0 ? -yv : yv), k1 = xv < 0 ? -xv : xv, k2 = xv >= 0 ? 0 : 1;
        if (best_key0 < 0 || k0 < best_key0 || (k0 == best_key0 && (k1 < best_key1 || (k1 == best_key1 && k2 < best_key2)))) {
            best_key0 = k0; best_key1 = k1; best_key2 = k2; bx = xv; by = yv;
        }
    }
    *mx = (int)bx;
    *my = (int)by;
    return FP_OK;
}

int fp_freq_index_set(int M_x, int M_y, int n_dens, int k_limit, int* h_ks, int cap, int* count) {
    if (M_x < 0 || M_y < 0 || n_dens < 1 || !count || (cap > 0 && !h_ks))
        return fp_fail(FP_EINVAL, "fp_freq_index_set: bad argument");
    // distinct k(m_x, m_y) = m_x n + m_y (n + 1) in increasing order, without the
    // orders (0,0), (0,1), (1,0) and without k > k_limit
    int cnt = 0;
    for (int k = 0; k <= k_limit; ++k) {
        bool hit = false;
        for (int x = 0; x <= M_x && !hit; ++x) {
            const long long rem = (long long)k - (long long)x * n_dens;
            if (rem < 0 || rem % (n_dens + 1)) continue;
            const long long y = rem / (n_dens + 1);
            if (y > M_y) continue;
            if ((x == 0 && y == 0) || (x == 0 && y == 1) || (x == 1 && y == 0)) continue;
            hit = true;
        }
        if (!hit) continue;
        if (cnt < cap) h_ks[cnt] = k;
        ++cnt;
    }
    *count = cnt;
    return FP_OK;
}

}  // extern "C"
