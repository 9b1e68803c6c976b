// BF16 tensor-core MLP for the harmonic surrogate: D = A B^T on tcgen05 with
// TMEM accumulators, TMA-fed shared-memory pipeline and fused epilogues
// (bias, GELU, output de-normalisation, loss gradient, GELU derivative,
// transposed activation copies for the weight-gradient GEMM).
//
// Every GEMM here is "both operands K-major": A is [M][K] and B is [N][K]
// row-major bf16.  The backward products are brought into that form by the
// epilogues, which also store transposed copies (X^T, G^T) and by keeping W^T
// beside W, so one kernel shape serves forward, dX and dW.
//
// Tile: 128 rows (UMMA M = 128), BN columns (32..256), K blocks of 64 bf16 =
// one 128-byte swizzle row; one persistent CTA per SM walks its tiles through
// an STAGES-deep TMA ring.  Warp 0 lane 0 issues TMA, warp 1 lane 0 issues
// tcgen05.mma into a ring of TMEM accumulators (warp 1 owns the allocation),
// and the epilogue warps 2.. drain an earlier accumulator (warp w reads TMEM
// lanes 32 (w % 4) .. + 31, i.e. those tile rows, and one group of columns).
// Every wait is bounded in time; a wait that gives up sets *err and the CTA
// drains its copies and MMAs and frees TMEM before it returns.
//
// What bounds it (GB300, 262,144 queries): no unit of the chip, by its counters.  A 512 -> 512 layer takes
// 136 us with the tensor pipe busy 42 % of the time, L2 at 40 % of its sector rate (52 % of its tag rate; it
// delivers 10.7 TB/s, 48 KB per 128 x 256 x 64 block) and HBM at 44 %; both output layers together take
// 561 us with 32, 38 (45) and 30 %.  What is left is the chain of one CTA per SM: the loads in
// flight, the MMAs behind them and the epilogue's turn with the accumulators.  The first
// layer (K = 64) takes 105 us, its epilogue.  1,024,000 queries through two networks: 13.7 -> 6.32 ms.
// Small batches are a chain of launches: 257 queries 88 -> 32 us with narrow tiles and overlapped
// launches; a training step of 4096 queries 594 -> 192 us with one launch for all weight
// gradients, one for the bias gradients and one for the optimiser (25 kernels before, 13 now).
#include <cuda.h>
#include <cuda_runtime.h>
#include <cuda_bf16.h>
#include <cstdint>
#include <cstring>
#include <cstdio>
#include "../../include/fp.h"

int fp_fail(int code, const char* fmt, ...);

namespace {

constexpr int BM = 128;
constexpr int BK = 64;
constexpr int EPI_GROUPS = 4;                 // column groups of the epilogue, 4 warps each (two groups
                                              // leave latency uncovered: K = 64 layer 120 us, with four 105 us)
constexpr int NTHREADS = 64 + 128 * EPI_GROUPS;   // TMA warp, MMA warp, epilogue warps
constexpr unsigned long long WAIT_NS = 2000000000ull;   // 2 s bound on any single wait

enum Epi : int {
    EPI_HIDDEN_INFER = 0,   // out = bf16(gelu(acc + b))
    EPI_HIDDEN_TRAIN = 1,   // zf = acc + b (f32), out = bf16(gelu(zf)), outT = out^T
    EPI_OUT_INFER = 2,      // outf = (acc + b) * oscale + oshift (f32, columns < N)
    EPI_OUT_TRAIN = 3,      // g = gscale (acc + b - (y - oshift)/oscale); loss += (.)^2; out, outT = bf16(g)
    EPI_DX_GELU = 4,        // g = acc * gelu'(zin); out, outT = bf16(g)
    EPI_DW = 5,             // outf = acc (f32), several GEMMs of one K in a launch
    EPI_OUT_ENSEMBLE = 6,   // y0, y1 = both networks' (acc + b) * oscale + oshift; outf = (y0 + y1) / 2;
                            // rowacc[row] += (|y0 - y1|^2, |mean|^2)
};

constexpr int MAXG = FP_SUR_LAYERS;           // GEMMs of one grouped launch (EPI_DW)

struct EpiParams {
    int M, N;                       // valid extent of D
    const float* bias;              // [N]
    __nv_bfloat16* out; int ldo;    // [M][ldo]
    __nv_bfloat16* outT; int ldt;   // [N][ldt]
    float* outf; int ldf;           // [M][ldf]
    const float* zin; int ldz;      // [M][ldz] pre-activation (EPI_DX_GELU)
    const float* y; int ldy;        // [M][ldy] raw targets (EPI_OUT_TRAIN)
    const float* oshift;            // [N]
    const float* oscale;            // [N]
    const float *bias1, *oshift1, *oscale1;   // the second network's (EPI_OUT_ENSEMBLE)
    float* loss;                    // scalar accumulator (EPI_OUT_TRAIN)
    float* rowacc;                  // [M][2] per-row sums (EPI_OUT_ENSEMBLE)
    float gscale;
    int* err;
    int nk;                         // number of 64-wide K blocks
    int vec, vec16, vecy;           // widest aligned access of outf, out, y rows: 2 = 32 bytes, 1 = 16 bytes, 0 = scalar
    // EPI_DW: the GEMMs of the group, tiles [t0[g], t0[g + 1]) each
    int t0[MAXG + 1];
    int gM[MAXG], gN[MAXG], gld[MAXG], gvec[MAXG];
    float* gout[MAXG];
};

// ------------------------------------------------------------- PTX helpers ----
__device__ __forceinline__ uint32_t smem_u32(const void* p) {
    return (uint32_t)__cvta_generic_to_shared(p);
}

__device__ __forceinline__ unsigned long long globaltimer() {
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}

__device__ __forceinline__ void mbar_expect_tx(uint32_t bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}

__device__ __forceinline__ bool mbar_try(uint32_t bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(bar), "r"(parity)
        : "memory");
    return ok != 0;
}

// bounded wait: false if the phase did not complete within WAIT_NS
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity) {
    if (mbar_try(bar, parity)) return true;
    const unsigned long long t0 = globaltimer();
    while (true) {
        if (mbar_try(bar, parity)) return true;
        if (globaltimer() - t0 > WAIT_NS) return false;
    }
}

__device__ __forceinline__ void tma_load_2d(uint32_t dst, const CUtensorMap* map, uint32_t bar, int x, int y) {
    asm volatile(
        "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4}], [%2];"
        ::"r"(dst), "l"((unsigned long long)map), "r"(bar), "r"(x), "r"(y)
        : "memory");
}

// programmatic dependent launch: wait for the kernel before this one in the stream (its
// writes are then visible), and let the next one's CTAs start their setup
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void pdl_launch() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

// shared-memory matrix descriptor: K-major, 128-byte swizzle, 8-row groups
// 1024 bytes apart (stride byte offset), leading byte offset unused (16 B)
__device__ __forceinline__ uint64_t sw128_desc(uint32_t saddr) {
    uint64_t d = 0;
    d |= (uint64_t)((saddr >> 4) & 0x3FFF);            // start address
    d |= (uint64_t)1 << 16;                              // leading byte offset (16 B >> 4)
    d |= (uint64_t)(1024 >> 4) << 32;                    // stride byte offset
    d |= (uint64_t)1 << 46;                              // descriptor version (tcgen05)
    d |= (uint64_t)2 << 61;                              // swizzle: 128 B
    return d;
}

// instruction descriptor, kind::f16: A, B bf16, D f32, both K-major, M x N
__host__ __device__ constexpr uint32_t idesc_bf16(int M, int N) {
    return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}

__device__ __forceinline__ void mma_bf16(uint32_t tmem_d, uint64_t adesc, uint64_t bdesc, uint32_t idesc,
                                         uint32_t accumulate) {
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}"
        ::"r"(tmem_d), "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate)
        : "memory");
}

__device__ __forceinline__ void mma_commit(uint32_t bar) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar)
                 : "memory");
}

// 32 lanes x 32 bit, 16 consecutive columns per thread: issue, and wait for every load issued
// (the wait takes the registers through, so that nothing reads them before it)
__device__ __forceinline__ void tmem_ld16(uint32_t taddr, uint32_t* r) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, "
        "%14, %15}, [%16];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(taddr));
}
__device__ __forceinline__ void tmem_wait16(uint32_t* r) {
    asm volatile("tcgen05.wait::ld.sync.aligned;"
                 : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]), "+r"(r[4]), "+r"(r[5]), "+r"(r[6]), "+r"(r[7]),
                   "+r"(r[8]), "+r"(r[9]), "+r"(r[10]), "+r"(r[11]), "+r"(r[12]), "+r"(r[13]), "+r"(r[14]), "+r"(r[15])
                 :
                 : "memory");
}

// ---- two FP32 values per instruction (each rounds as the scalar one does) ----
struct f2 { unsigned long long v; };
__device__ __forceinline__ f2 pk(float lo, float hi) {
    f2 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r.v) : "f"(lo), "f"(hi));
    return r;
}
__device__ __forceinline__ f2 pk(float x) { return pk(x, x); }
__device__ __forceinline__ void upk(f2 a, float& lo, float& hi) {
    asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(a.v));
}
__device__ __forceinline__ f2 add2(f2 a, f2 b) {
    f2 r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
    return r;
}
__device__ __forceinline__ f2 mul2(f2 a, f2 b) {
    f2 r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
    return r;
}
__device__ __forceinline__ f2 fma2(f2 a, f2 b, f2 c) {
    f2 r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r.v) : "l"(a.v), "l"(b.v), "l"(c.v));
    return r;
}
__device__ __forceinline__ float rcp_approx(float x) {
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}
__device__ __forceinline__ float ex2_approx(float x) {
    float r;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}

// 1 + erf(z) by Abramowitz & Stegun 7.1.26 (|error| <= 1.5e-7, far below the BF16
// resolution of the activations): erf(x) = 1 - t (a1 + t (a2 + ... a5 t)) exp(-x^2),
// t = 1 / (1 + p x) for x >= 0, odd in x.  The epilogue's issue slots bound the hidden
// layers, so two values go through every FP32 instruction and share one reciprocal:
// 1 / d0 = d1 / (d0 d1), brought to the rounding of 1 / d0 by one
// Newton-Raphson step with an exact residual (Markstein 1990); x is cut at 10, where erf is
// 1 in FP32, so that d0 d1 stays finite, and a NaN or infinite z reaches the result
// through the caller's factor x.
__device__ __forceinline__ f2 one_plus_erf2(f2 z) {
    float z0, z1;
    upk(z, z0, z1);
    float n0, n1;
    const f2 x = pk(fminf(fabsf(z0), 10.f), fminf(fabsf(z1), 10.f));
    const f2 nd = fma2(pk(-0.3275911f), x, pk(-1.f));            // -(1 + p x)
    upk(nd, n0, n1);
    const float inv = rcp_approx(n0 * n1);
    f2 t = pk(inv * -n1, inv * -n0);
    t = fma2(t, fma2(nd, t, pk(1.f)), t);
    f2 ny = fma2(pk(-1.061405429f), t, pk(1.453152027f));        // the polynomial with its sign turned
    ny = fma2(ny, t, pk(-1.421413741f));
    ny = fma2(ny, t, pk(0.284496736f));
    ny = fma2(ny, t, pk(-0.254829592f));
    float a0, a1, e0, e1;
    upk(mul2(mul2(x, x), pk(-1.4426950408889634f)), a0, a1);     // -x^2 log2 e
    upk(fma2(mul2(ny, t), pk(ex2_approx(a0), ex2_approx(a1)), pk(1.f)), e0, e1);
    return add2(pk(copysignf(e0, z0), copysignf(e1, z1)), pk(1.f));
}

__device__ __forceinline__ f2 gelu2(f2 x) {
    return mul2(mul2(x, pk(0.5f)), one_plus_erf2(mul2(x, pk(0.70710678118654752f))));
}

// The same for one value, with the correctly rounded reciprocal: training keeps it, since the
// optimiser divides a gradient by its own size and carries any last-bit difference into the weights.
__device__ __forceinline__ float erf_as(float z) {
    const float x = fabsf(z);
    const float t = __frcp_rn(fmaf(0.3275911f, x, 1.f));
    float y = fmaf(1.061405429f, t, -1.453152027f);
    y = fmaf(y, t, 1.421413741f);
    y = fmaf(y, t, -0.284496736f);
    y = fmaf(y, t, 0.254829592f);
    const float e = 1.f - y * t * __expf(-x * x);
    return copysignf(e, z);
}

__device__ __forceinline__ float gelu(float x) { return 0.5f * x * (1.f + erf_as(x * 0.70710678118654752f)); }

__device__ __forceinline__ float gelu_grad(float x) {
    return 0.5f * (1.f + erf_as(x * 0.70710678118654752f)) + x * 0.39894228040143268f * __expf(-0.5f * x * x);
}

// one 32-byte store (a whole sector): half the store instructions of 16-byte ones, where a
// warp's 32 lanes write 32 different rows
__device__ __forceinline__ void st_v8(void* p, const uint32_t* r) {
    asm volatile("st.global.v8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(p), "r"(r[0]), "r"(r[1]), "r"(r[2]),
                 "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7])
                 : "memory");
}
__device__ __forceinline__ uint32_t bf16_pair(float lo, float hi) {
    const __nv_bfloat162 b = __floats2bfloat162_rn(lo, hi);
    return *(const uint32_t*)&b;
}

template <int BN> struct Cfg {
    static constexpr int A_BYTES = BM * BK * 2;
    static constexpr int B_BYTES = BN * BK * 2;
    static constexpr int STAGE = A_BYTES + B_BYTES;
    // one persistent CTA per SM: the ring takes most of the shared memory
    static constexpr int STAGES = (196 * 1024) / STAGE > 8 ? 8 : (196 * 1024) / STAGE;
    static constexpr int SMEM = STAGES * STAGE + 1024 /* align */ + 256 /* barriers */;
    static_assert(A_BYTES % 1024 == 0 && B_BYTES % 1024 == 0, "swizzle atoms need 1024-byte tiles");
    static_assert(BN % 16 == 0 && BN >= 16 && BN <= 256, "UMMA N for M = 128");
};

constexpr int EPI_WARPS = 4 * EPI_GROUPS;    // warps 2 ..
constexpr int MAX_EPI_COLS = 1024;           // bias / output scale staged in shared memory

// ---------------------------------------------------------------- epilogue ----
// 16 consecutive values in shared memory (a warp reads the same ones: 16-byte broadcasts)
__device__ __forceinline__ void lds16(const float* p, float* r) {
#pragma unroll
    for (int i = 0; i < 16; i += 4) {
        const float4 a = *(const float4*)(p + i);
        r[i] = a.x; r[i + 1] = a.y; r[i + 2] = a.z; r[i + 3] = a.w;
    }
}

// 16 consecutive floats of a row at o, `left` columns of them valid; vec as in EpiParams
__device__ __forceinline__ void store_row16(float* o, const float* r, int vec, int left) {
    if (left >= 16 && vec == 2) {
        st_v8(o, (const uint32_t*)r);
        st_v8(o + 8, (const uint32_t*)r + 8);
    } else if (left >= 16 && vec == 1) {
#pragma unroll
        for (int i = 0; i < 16; i += 4) *(float4*)(o + i) = make_float4(r[i], r[i + 1], r[i + 2], r[i + 3]);
    } else {
#pragma unroll
        for (int i = 0; i < 16; ++i)
            if (i < left) o[i] = r[i];
    }
}

__device__ __forceinline__ void load_row16(const float* p, float* r, int vec, int left) {
    if (left >= 16 && vec >= 1) {
#pragma unroll
        for (int i = 0; i < 16; i += 4) {
            const float4 a = __ldg((const float4*)(p + i));
            r[i] = a.x; r[i + 1] = a.y; r[i + 2] = a.z; r[i + 3] = a.w;
        }
    } else {
#pragma unroll
        for (int i = 0; i < 16; ++i) r[i] = i < left ? __ldg(p + i) : 0.f;
    }
}

// One 16-column chunk of a row: v the accumulators (v1 the second network's), sb, ssc, ssh
// bias, output scale and shift of these columns in shared memory (the second network's
// MAX_EPI_COLS further on), g the group of EPI_DW.
template <int EPI>
__device__ __forceinline__ void epilogue_chunk(const EpiParams& P, int row, int col0, float* v, const float* v1,
                                               const float* sb, const float* ssc, const float* ssh, float* racc,
                                               int grp) {
    const int M = EPI == EPI_DW ? P.gM[grp] : P.M, left = (EPI == EPI_DW ? P.gN[grp] : P.N) - col0;
    const bool rv = row < M;
    if (EPI == EPI_OUT_ENSEMBLE) {
        if (!rv) return;
        float mn[16], y1s[16], b[16], sc[16], sh[16];
        lds16(sb + MAX_EPI_COLS, b);
        lds16(ssc + MAX_EPI_COLS, sc);
        lds16(ssh + MAX_EPI_COLS, sh);
#pragma unroll
        for (int i = 0; i < 16; ++i) y1s[i] = (v1[i] + b[i]) * sc[i] + sh[i];
        lds16(sb, b);
        lds16(ssc, sc);
        lds16(ssh, sh);
#pragma unroll
        for (int i = 0; i < 16; ++i) {
            const bool cv = i < left;
            const float y0 = (v[i] + b[i]) * sc[i] + sh[i], y1 = y1s[i];
            const float d = cv ? y0 - y1 : 0.f;
            mn[i] = cv ? 0.5f * (y0 + y1) : 0.f;
            racc[0] = fmaf(d, d, racc[0]);
            racc[1] = fmaf(mn[i], mn[i], racc[1]);
        }
        store_row16(P.outf + (size_t)row * P.ldf + col0, mn, P.vec, left);
        return;
    }
    if (EPI == EPI_DW) {
        if (rv) store_row16(P.gout[grp] + (size_t)row * P.gld[grp] + col0, v, P.gvec[grp], left);
        return;
    }
    if (EPI == EPI_OUT_INFER) {
        if (!rv) return;
        float r[16], b[16], sc[16], sh[16];
        lds16(sb, b);
        lds16(ssc, sc);
        lds16(ssh, sh);
#pragma unroll
        for (int i = 0; i < 16; ++i) r[i] = (v[i] + b[i]) * sc[i] + sh[i];
        store_row16(P.outf + (size_t)row * P.ldf + col0, r, P.vec, left);
        return;
    }
    float g[16];
    if (EPI == EPI_HIDDEN_INFER || EPI == EPI_HIDDEN_TRAIN) {
        float z[16];
#pragma unroll
        for (int i = 0; i < 16; i += 4) {
            const float4 b4 = *(const float4*)(sb + i);
            const f2 za = add2(pk(v[i], v[i + 1]), pk(b4.x, b4.y));
            const f2 zb = add2(pk(v[i + 2], v[i + 3]), pk(b4.z, b4.w));
            upk(za, z[i], z[i + 1]);
            upk(zb, z[i + 2], z[i + 3]);
            if (EPI == EPI_HIDDEN_INFER) {
                upk(gelu2(za), g[i], g[i + 1]);
                upk(gelu2(zb), g[i + 2], g[i + 3]);
            }
        }
        if (EPI == EPI_HIDDEN_TRAIN)
#pragma unroll
            for (int i = 0; i < 16; ++i) g[i] = gelu(z[i]);
        if (EPI == EPI_HIDDEN_TRAIN && rv) store_row16(P.outf + (size_t)row * P.ldf + col0, z, P.vec, left);
    } else if (EPI == EPI_OUT_TRAIN) {
        float y[16], lsum = 0.f;
        if (rv) load_row16(P.y + (size_t)row * P.ldy + col0, y, P.vecy, left);
#pragma unroll
        for (int i = 0; i < 16; ++i) {
            g[i] = 0.f;
            if (rv && i < left) {
                const float d = (v[i] + sb[i]) - (y[i] - ssh[i]) / ssc[i];
                lsum += d * d;
                g[i] = P.gscale * d;
            }
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) lsum += __shfl_xor_sync(0xffffffffu, lsum, o);
        if ((threadIdx.x & 31) == 0 && lsum != 0.f) atomicAdd(P.loss, lsum);
    } else {   // EPI_DX_GELU
        float z[16];
#pragma unroll
        for (int i = 0; i < 16; ++i) z[i] = 0.f;
        if (rv) load_row16(P.zin + (size_t)row * P.ldz + col0, z, P.vec, left);
#pragma unroll
        for (int i = 0; i < 16; ++i) g[i] = v[i] * gelu_grad(z[i]);
    }
    if (!rv) return;
    __nv_bfloat16* o = P.out + (size_t)row * P.ldo + col0;
    uint32_t b[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) b[i] = bf16_pair(g[2 * i], g[2 * i + 1]);
    if (left >= 16 && P.vec16 == 2) {
        st_v8(o, b);
    } else if (left >= 16 && P.vec16 == 1) {
        *(uint4*)o = make_uint4(b[0], b[1], b[2], b[3]);
        *(uint4*)(o + 8) = make_uint4(b[4], b[5], b[6], b[7]);
    } else {
#pragma unroll
        for (int i = 0; i < 16; ++i)
            if (i < left) o[i] = __float2bfloat16_rn(g[i]);
    }
    if (EPI != EPI_HIDDEN_INFER) {
        // transposed copy: for each column, the warp's 32 rows are contiguous
#pragma unroll
        for (int i = 0; i < 16; ++i)
            if (i < left) P.outT[(size_t)(col0 + i) * P.ldt + row] = __float2bfloat16_rn(g[i]);
    }
}

// ------------------------------------------------------------------ kernel ----
// Persistent: one CTA per SM walks the output tiles (tile t -> row block
// t / ntn, column block t % ntn, so neighbouring tiles share their A rows).
// Warp 0 lane 0 streams K blocks of every tile through the TMA ring, warp 1
// lane 0 issues the MMAs into a ring of TMEM accumulators, and the epilogue
// warps drain an earlier accumulator, so the epilogue of tile u overlaps the
// main loop of tile u + 1.  A tile takes one pass (accumulator), or two for
// EPI_OUT_ENSEMBLE: both networks' output tiles are formed side by side and only
// their mean leaves the SM, where a launch per network wrote the first answer and
// read it back (9.8 GB instead of 3.3 GB at 1,024,000 queries).
template <int EPI> struct Pass {
    static constexpr int N = EPI == EPI_OUT_ENSEMBLE ? 2 : 1;          // accumulators per tile
    static constexpr int RING = EPI == EPI_OUT_ENSEMBLE ? 3 : 2;       // accumulators in TMEM
    static constexpr int MAPS = EPI == EPI_DW ? MAXG : N;
};
template <int EPI> struct Maps { CUtensorMap a[Pass<EPI>::MAPS], b[Pass<EPI>::MAPS]; };
// TMEM columns of a kernel: its ring of accumulators, a power of two from 32 to 512
template <int BN, int EPI> __host__ __device__ constexpr int tmem_cols() {
    const int n = BN * Pass<EPI>::RING;
    return n <= 32 ? 32 : n <= 64 ? 64 : n <= 128 ? 128 : n <= 256 ? 256 : 512;
}

// tile t -> its GEMM of the group, first row and first column
template <int BN, int EPI>
__device__ __forceinline__ void locate(const EpiParams& P, int t, int& g, int& m0, int& n0) {
    g = 0;
    int N = P.N;
    if (EPI == EPI_DW) {
        while (t >= P.t0[g + 1]) ++g;
        t -= P.t0[g];
        N = P.gN[g];
    }
    const int ntn = (N + BN - 1) / BN;
    m0 = (t / ntn) * BM;
    n0 = (t % ntn) * BN;
}

template <int BN, int EPI>
__global__ void __launch_bounds__(NTHREADS, 1)
mlp_gemm_kernel(const __grid_constant__ Maps<EPI> maps, const __grid_constant__ EpiParams P, int ntiles) {
    using C = Cfg<BN>;
    constexpr int ST = C::STAGES, NP = Pass<EPI>::N, RING = Pass<EPI>::RING;
    constexpr uint32_t TCOLS = (uint32_t)tmem_cols<BN, EPI>();
    static_assert(BN * RING <= 512, "the accumulators exceed TMEM");
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    unsigned char* smem = (unsigned char*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    unsigned char* tiles = smem;
    uint64_t* bars = (uint64_t*)(smem + ST * C::STAGE);   // full[ST], empty[ST], acc_full[3], acc_empty[3], drain
    uint32_t* tmem_slot = (uint32_t*)(bars + 2 * ST + 7);
    int* abort_flag = (int*)(tmem_slot + 1);
    __shared__ __align__(16) float s_bias[NP * MAX_EPI_COLS], s_osc[NP * MAX_EPI_COLS], s_osh[NP * MAX_EPI_COLS];

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int nk = P.nk;
    const uint32_t full0 = smem_u32(bars), empty0 = smem_u32(bars + ST);
    const uint32_t accf0 = smem_u32(bars + 2 * ST), acce0 = smem_u32(bars + 2 * ST + 3);
    const uint32_t drain = smem_u32(bars + 2 * ST + 6);
    if (threadIdx.x == 0) {
        for (int s = 0; s < 2 * ST + 3; ++s) mbar_init(smem_u32(bars + s), 1);
        for (int s = 0; s < 3; ++s) mbar_init(acce0 + 8 * s, EPI_WARPS);
        mbar_init(drain, 1);
        *abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)),
                     "r"(TCOLS)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    // everything above ran beside the end of the kernel before this one in the stream; from
    // here on its results are read and its inputs may be overwritten
    pdl_wait();
    pdl_launch();
    for (int j = threadIdx.x; j < MAX_EPI_COLS; j += NTHREADS) {
        const bool in = j < P.N && EPI != EPI_DW;
        s_bias[j] = (in && P.bias) ? P.bias[j] : 0.f;
        s_osc[j] = (in && P.oscale) ? P.oscale[j] : 1.f;
        s_osh[j] = (in && P.oshift) ? P.oshift[j] : 0.f;
        if (NP == 2) {
            s_bias[(NP - 1) * MAX_EPI_COLS + j] = in ? P.bias1[j] : 0.f;
            s_osc[(NP - 1) * MAX_EPI_COLS + j] = in ? P.oscale1[j] : 1.f;
            s_osh[(NP - 1) * MAX_EPI_COLS + j] = in ? P.oshift1[j] : 0.f;
        }
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tmem_slot;
    volatile int* abort_v = abort_flag;

    if (warp == 0) {
        if (lane == 0) {   // TMA producer over all tiles of this CTA
            long long g = 0;
            for (int t = blockIdx.x; t < ntiles && !*abort_v; t += gridDim.x) {
                int grp, m0, n0;
                locate<BN, EPI>(P, t, grp, m0, n0);
                for (int ps = 0; ps < NP && !*abort_v; ++ps) {
                    const int mi = EPI == EPI_DW ? grp : ps;
                    for (int kb = 0; kb < nk; ++kb, ++g) {
                        const int s = (int)(g % ST);
                        if (g >= ST && !mbar_wait(empty0 + 8 * s, (uint32_t)(((g / ST) - 1) & 1))) {
                            atomicOr(P.err, 1);
                            *abort_v = 1;
                        }
                        if (*abort_v) break;
                        const uint32_t sa = smem_u32(tiles + s * C::STAGE);
                        mbar_expect_tx(full0 + 8 * s, C::STAGE);
                        tma_load_2d(sa, &maps.a[mi], full0 + 8 * s, kb * BK, m0);
                        tma_load_2d(sa + C::A_BYTES, &maps.b[mi], full0 + 8 * s, kb * BK, n0);
                    }
                }
            }
            if (*abort_v)   // let the copies still in flight land before the CTA exits
                for (long long h = g - 1; h >= 0 && h >= g - ST; --h)
                    mbar_wait(full0 + 8 * (int)(h % ST), (uint32_t)((h / ST) & 1));
        }
    } else if (warp == 1) {
        if (lane == 0) {   // MMA issuer
            constexpr uint32_t idesc = idesc_bf16(BM, BN);
            long long g = 0;
            int u = 0;     // pass (accumulator) counter
            for (int t = blockIdx.x; t < ntiles && !*abort_v; t += gridDim.x) {
                for (int ps = 0; ps < NP && !*abort_v; ++ps, ++u) {
                    const int b = u % RING, q = u / RING;
                    if (q >= 1 && !mbar_wait(acce0 + 8 * b, (uint32_t)((q - 1) & 1))) {
                        atomicOr(P.err, 8);
                        *abort_v = 1;
                        break;
                    }
                    tc_fence_after();
                    const uint32_t acc = tmem + (uint32_t)(b * BN);
                    for (int kb = 0; kb < nk; ++kb, ++g) {
                        const int s = (int)(g % ST);
                        if (!mbar_wait(full0 + 8 * s, (uint32_t)((g / ST) & 1)) || *abort_v) {
                            atomicOr(P.err, 2);
                            *abort_v = 1;
                            break;
                        }
                        tc_fence_after();
                        const uint32_t sa = smem_u32(tiles + s * C::STAGE);
                        const uint32_t sb = sa + C::A_BYTES;
#pragma unroll
                        for (int k = 0; k < BK / 16; ++k)
                            mma_bf16(acc, sw128_desc(sa + k * 32), sw128_desc(sb + k * 32), idesc, (kb | k) != 0);
                        mma_commit(empty0 + 8 * s);        // frees the stage once these MMAs are done
                    }
                    if (*abort_v) break;
                    mma_commit(accf0 + 8 * b);             // accumulator b complete
                }
            }
            mma_commit(drain);                         // every MMA this thread issued has completed
            if (!mbar_wait(drain, 0)) atomicOr(P.err, 16);
        }
    } else {
        // epilogue warps: warp w reads TMEM lanes 32 (w % 4) .. + 31 and one column group;
        // the next chunk's accumulators are on their way while a chunk is worked on
        const int lg = warp & 3, cg = (warp - 2) >> 2;
        constexpr int NCH = BN / 16;                   // 16-column chunks of a tile
        const int c_lo = 16 * (cg * NCH / EPI_GROUPS), c_hi = 16 * ((cg + 1) * NCH / EPI_GROUPS);
        int u = 0;
        for (int t = blockIdx.x; t < ntiles; t += gridDim.x, u += NP) {
            int grp, m0, n0;
            locate<BN, EPI>(P, t, grp, m0, n0);
            const int N = EPI == EPI_DW ? P.gN[grp] : P.N;
            bool ok = !*abort_v;
#pragma unroll
            for (int ps = 0; ps < NP; ++ps)
                ok = ok && mbar_wait(accf0 + 8 * ((u + ps) % RING), (uint32_t)(((u + ps) / RING) & 1));
            __syncwarp();
            if (!__all_sync(0xffffffffu, ok)) {
                if (lane == 0) atomicOr(P.err, 4);
                *abort_v = 1;
                break;
            }
            tc_fence_after();
            const int row = m0 + lg * 32 + lane;
            const uint32_t tw = tmem + (uint32_t)((u % RING) * BN) + ((uint32_t)(lg * 32) << 16);
            const uint32_t tw1 = tmem + (uint32_t)(((u + NP - 1) % RING) * BN) + ((uint32_t)(lg * 32) << 16);
            float racc[2] = {0.f, 0.f};
            uint32_t r[2][16], r1[16];
            if (c_lo < c_hi) tmem_ld16(tw + c_lo, r[0]);
#pragma unroll 1
            for (int c = c_lo; c < c_hi; c += 32) {
#pragma unroll
                for (int hf = 0; hf < 2; ++hf) {
                    const int cc = c + 16 * hf;
                    if (cc < c_hi) {
                        tmem_wait16(r[hf]);
                        if (NP == 2) {
                            tmem_ld16(tw1 + cc, r1);
                            tmem_wait16(r1);
                        }
                        if (cc + 16 < c_hi) tmem_ld16(tw + cc + 16, r[hf ^ 1]);
                        const int co = n0 + cc;
                        if (co < N)
                            epilogue_chunk<EPI>(P, row, co, (float*)r[hf], (const float*)r1, s_bias + co, s_osc + co,
                                                s_osh + co, racc, grp);
                    }
                }
            }
            if (EPI == EPI_OUT_ENSEMBLE && row < P.M) {
                atomicAdd(P.rowacc + 2 * (size_t)row, racc[0]);
                atomicAdd(P.rowacc + 2 * (size_t)row + 1, racc[1]);
            }
            tc_fence_before();
            __syncwarp();
            if (lane == 0)
#pragma unroll
                for (int ps = 0; ps < NP; ++ps)
                    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(acce0 + 8 * ((u + ps) % RING)) : "memory");
        }
    }
    __syncwarp();
    tc_fence_before();
    __syncthreads();
    if (warp == 1) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(TCOLS) : "memory");
    }
}

// ------------------------------------------------------------ tensor maps ----
typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

EncodeTiledFn encode_fn() {
    static EncodeTiledFn fn = nullptr;
    if (!fn) {
        void* p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) ==
                cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = (EncodeTiledFn)p;
    }
    return fn;
}

int num_sms() {
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    return sms > 0 ? sms : 1;
}

// row-major bf16 [rows][cols] (cols contiguous, ld elements per row), box = box_rows x 64
int make_map(CUtensorMap* map, const void* base, long long rows, long long cols, long long ld, int box_rows) {
    EncodeTiledFn fn = encode_fn();
    if (!fn) return FP_ECUDA;
    if (((uintptr_t)base & 15) || (ld * 2) % 16 || rows < 1 || cols < 1) return FP_EINVAL;
    cuuint64_t dims[2] = {(cuuint64_t)cols, (cuuint64_t)rows};
    cuuint64_t strides[1] = {(cuuint64_t)(ld * 2)};
    cuuint32_t box[2] = {(cuuint32_t)BK, (cuuint32_t)box_rows};
    cuuint32_t es[2] = {1, 1};
    CUresult r = fn(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(base), dims, strides, box, es,
                    CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                    CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    return r == CUDA_SUCCESS ? FP_OK : FP_ECUDA;
}

template <int BN, int EPI>
int launch_t(const Maps<EPI>& maps, const EpiParams& P, int ntiles, cudaStream_t st) {
    using C = Cfg<BN>;
    if (cudaFuncSetAttribute(mlp_gemm_kernel<BN, EPI>, cudaFuncAttributeMaxDynamicSharedMemorySize, C::SMEM) !=
        cudaSuccess)
        return FP_ECUDA;
    // the setup of a launch (barriers, TMEM) overlaps the kernel before it
    cudaLaunchAttribute at;
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg;
    std::memset(&cfg, 0, sizeof(cfg));
    const int sms = num_sms();
    cfg.gridDim = dim3(ntiles < sms ? ntiles : sms);
    cfg.blockDim = dim3(NTHREADS);
    cfg.dynamicSmemBytes = C::SMEM;
    cfg.stream = st;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    if (cudaLaunchKernelEx(&cfg, mlp_gemm_kernel<BN, EPI>, maps, P, ntiles) == cudaSuccess) return FP_OK;
    cudaGetLastError();                                    // reported here: not left for the next call's check
    return FP_ECUDA;
}

int vec_of(const void* p, int ld, int size) {
    const long long row = (long long)ld * size;
    if (((uintptr_t)p & 31) == 0 && row % 32 == 0) return 2;
    return ((uintptr_t)p & 15) == 0 && row % 16 == 0 ? 1 : 0;
}

// One operand pair of a GEMM: A [M][K] and B [N][K] bf16 row-major, leading dimensions in elements.
struct Operand { const void* A; int lda; const void* B; int ldb; };

// D[M][N] = A B^T in BN-column tiles with epilogue EPI (for EPI_OUT_ENSEMBLE two operand pairs)
template <int BN, int EPI>
int gemm_bn(const Operand* op, int M, int N, int K, EpiParams P, cudaStream_t st) {
    if (M < 1 || N < 1 || K < 1) return FP_EINVAL;
    if (N > MAX_EPI_COLS) return FP_EINVAL;
    Maps<EPI> maps;
    for (int i = 0; i < Pass<EPI>::N; ++i) {
        int rc = make_map(&maps.a[i], op[i].A, M, K, op[i].lda, BM);
        if (rc != FP_OK) return rc;
        rc = make_map(&maps.b[i], op[i].B, N, K, op[i].ldb, BN);
        if (rc != FP_OK) return rc;
    }
    P.M = M;
    P.N = N;
    P.nk = (K + BK - 1) / BK;
    P.vec = EPI == EPI_DX_GELU ? vec_of(P.zin, P.ldz, 4) : vec_of(P.outf, P.ldf, 4);
    P.vec16 = vec_of(P.out, P.ldo, 2);
    P.vecy = vec_of(P.y, P.ldy, 4);
    const long long nt = (long long)((N + BN - 1) / BN) * ((M + BM - 1) / BM);
    return launch_t<BN, EPI>(maps, P, (int)nt, st);
}

// Tile width: the one with the least waves x (columns + 48).  A wave's time grows with its
// tiles' columns (epilogue and operand reads; the 48 stand for the A rows and the fill of the
// pipeline), so large batches take the widest tile, and a few hundred queries, which are
// latency-bound, a narrow one with a short epilogue (257 queries: 24 tiles of 64 columns in
// one wave).  The K order, and with it the result, is the same for all.  One inference by hidden
// tiles of 64 / 128 / 256 columns: 28.8 / 32.5 / 39.6 us at 257 queries, 32.4 / 35.9 / 43.2 at 2,432
// and 41.6 / 35.4 / 43.1 at 2,433, 49.9 / 42.6 / 51.5 at 4,800, 74 / 59 / 54 at 8,500; by output tiles of 32 /
// 80 / 160: 28.7 / 29.8 / 30.9 at 257, 31.8 / 29.8 / 30.9 at 1,200, 42.6 / 38.5 / 36.0 at 3,000.  Over 32 sizes up to
// 90,000 queries the rule is within 3 % of the best, but 9 % at 19,457 to 22,000 (112 us; 103 by 256).
long long tile_cost(int M, int N, int BN) {
    const long long tiles = (long long)((M + BM - 1) / BM) * ((N + BN - 1) / BN), sms = num_sms();
    return (tiles + sms - 1) / sms * (BN + 48);
}
template <int EPI>
int gemm_hidden(const Operand& op, int M, int N, int K, const EpiParams& P, cudaStream_t st) {
    const long long c256 = tile_cost(M, N, 256), c128 = tile_cost(M, N, 128), c64 = tile_cost(M, N, 64);
    if (c256 <= c128 && c256 <= c64) return gemm_bn<256, EPI>(&op, M, N, K, P, st);
    if (c128 <= c64) return gemm_bn<128, EPI>(&op, M, N, K, P, st);
    return gemm_bn<64, EPI>(&op, M, N, K, P, st);
}
template <int EPI>
int gemm_out(const Operand* op, int M, int N, int K, const EpiParams& P, cudaStream_t st) {
    const long long c160 = tile_cost(M, N, 160), c80 = tile_cost(M, N, 80), c32 = tile_cost(M, N, 32);
    if (c160 <= c80 && c160 <= c32) return gemm_bn<160, EPI>(op, M, N, K, P, st);
    if (c80 <= c32) return gemm_bn<80, EPI>(op, M, N, K, P, st);
    return gemm_bn<32, EPI>(op, M, N, K, P, st);
}

// The weight gradients of every layer, gW [N][K] = GT [N][q] XT [K][q]^T, in one launch.  One
// layer has 4 to 14 tiles of 128 x 256 behind a serial K loop over the batch, which leaves most
// SMs idle; the group has 137 of 128 x 80 side by side, one to an SM.
struct DwLayer { const void *GT, *XT; float* gW; int N, K; };
int gemm_dw(const DwLayer* dw, int q, int ldt, int* err, cudaStream_t st) {
    constexpr int BN = 80;
    Maps<EPI_DW> maps;
    EpiParams P;
    std::memset(&P, 0, sizeof(P));
    P.err = err;
    P.nk = (q + BK - 1) / BK;
    for (int l = 0; l < MAXG; ++l) {
        int rc = make_map(&maps.a[l], dw[l].GT, dw[l].N, q, ldt, BM);
        if (rc != FP_OK) return rc;
        rc = make_map(&maps.b[l], dw[l].XT, dw[l].K, q, ldt, BN);
        if (rc != FP_OK) return rc;
        P.gM[l] = dw[l].N;
        P.gN[l] = P.gld[l] = dw[l].K;
        P.gout[l] = dw[l].gW;
        P.gvec[l] = vec_of(dw[l].gW, dw[l].K, 4);
        P.t0[l + 1] = P.t0[l] + ((dw[l].N + BM - 1) / BM) * ((dw[l].K + BN - 1) / BN);
    }
    return launch_t<BN, EPI_DW>(maps, P, P.t0[MAXG], st);
}

// ------------------------------------------------------- small kernels ----
// x0[m][j] = bf16((x[m][j] - shift_j) * scale_j), j < 7, zero up to 64; and,
// if x0T is given, x0T[j][m] for j < 7 (leading dimension ldt).  Write-bound: a
// thread stores 16 bytes, one of the eight parts of a row (one element a thread took
// a 64-bit division each).
__global__ void prep_input_kernel(const float* __restrict__ x, int q, const float* __restrict__ shift,
                                  const float* __restrict__ scale, __nv_bfloat16* __restrict__ x0,
                                  __nv_bfloat16* __restrict__ x0T, int ldt) {
    static_assert(FP_SUR_IN <= 8 && FP_SUR_KIN == 64, "the inputs lie in the first of eight 16-byte parts");
    pdl_launch();
    const long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    const long long m = e >> 3;
    if (m >= q) return;
    uint4 w = make_uint4(0u, 0u, 0u, 0u);
    if ((e & 7) == 0) {
        __nv_bfloat16 b[8];
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            b[j] = __float2bfloat16_rn(j < FP_SUR_IN ? (x[m * FP_SUR_IN + j] - shift[j]) * scale[j] : 0.f);
            if (x0T && j < FP_SUR_IN) x0T[(size_t)j * ldt + m] = b[j];
        }
        const unsigned short* u = (const unsigned short*)b;
        w = make_uint4(u[0] | (u[1] << 16), u[2] | (u[3] << 16), u[4] | (u[5] << 16), u[6] | (u[7] << 16));
    }
    *(uint4*)(x0 + e * 8) = w;
}

// db[n] = sum_m gT[n][m] of every layer: one warp per row
struct BiasArgs {
    const __nv_bfloat16* gT[MAXG];
    float* db[MAXG];
    int row0[MAXG + 1];               // first row of each layer in the launch
    int ldt, q;
};
__global__ void bias_grad_kernel(BiasArgs a) {
    int n = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    const int lane = threadIdx.x & 31;
    if (n >= a.row0[MAXG]) return;
    int l = 0;
    while (n >= a.row0[l + 1]) ++l;
    n -= a.row0[l];
    const __nv_bfloat16* g = a.gT[l] + (size_t)n * a.ldt;
    float s = 0.f;
#pragma unroll 32                                        // latency-bound: many loads in flight, one order of summation
    for (int m = lane; m < a.q; m += 32) s += __bfloat162float(g[m]);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (lane == 0) a.db[l][n] = s;
}

struct AdamArgs {
    float lr, b1, b2, eps, c1, c2;   // c1 = 1 - b1^t, c2 = 1 - b2^t
    int step;
};

__device__ __forceinline__ float adam_update(float p, float g, float& m, float& v, const AdamArgs& a) {
    m = a.b1 * m + (1.f - a.b1) * g;
    v = a.b2 * v + (1.f - a.b2) * g * g;
    return p - a.lr * (m / a.c1) / (sqrtf(v / a.c2) + a.eps);
}

struct AdamLayer {
    float *W, *mW, *vW, *b, *mb, *vb;
    const float *gW, *gb;
    __nv_bfloat16 *Wb, *WTb;
    int N, K, t0;                     // t0: first block of the layer
};
struct AdamNet { AdamLayer l[MAXG]; AdamArgs a; };

// every layer: master W [N][K] (and b [N]) updated in place, bf16 W and W^T refreshed.  A
// block takes 32 x 32 weights and turns them in shared memory, so that both copies are
// written along their rows; the layer's last block updates the bias.
constexpr int ADAM_T = 32;
__host__ __device__ inline int adam_tiles(int N, int K) { return ((N + ADAM_T - 1) / ADAM_T) * ((K + ADAM_T - 1) / ADAM_T); }
__global__ void __launch_bounds__(256) adam_kernel(const __grid_constant__ AdamNet net) {
    __shared__ __nv_bfloat16 tile[ADAM_T][ADAM_T + 2];
    int li = 0;
    while (li + 1 < MAXG && (int)blockIdx.x >= net.l[li + 1].t0) ++li;
    const AdamLayer& L = net.l[li];
    const int t = blockIdx.x - L.t0;
    if (t == adam_tiles(L.N, L.K)) {
        if (net.a.step > 0)
            for (int n = threadIdx.x; n < L.N; n += 256) {
                float m = L.mb[n], v = L.vb[n];
                L.b[n] = adam_update(L.b[n], L.gb[n], m, v, net.a);
                L.mb[n] = m; L.vb[n] = v;
            }
        return;
    }
    const int tk = (L.K + ADAM_T - 1) / ADAM_T;
    const int n0 = (t / tk) * ADAM_T, k0 = (t % tk) * ADAM_T;
    const int c = threadIdx.x & 31, r0 = threadIdx.x >> 5;
#pragma unroll
    for (int r = r0; r < ADAM_T; r += 8) {
        const int n = n0 + r, k = k0 + c;
        if (n >= L.N || k >= L.K) continue;
        const size_t e = (size_t)n * L.K + k;
        float p = L.W[e];
        if (net.a.step > 0) {
            float m = L.mW[e], v = L.vW[e];
            p = adam_update(p, L.gW[e], m, v, net.a);
            L.mW[e] = m; L.vW[e] = v; L.W[e] = p;
        }
        const __nv_bfloat16 pb = __float2bfloat16_rn(p);
        L.Wb[e] = pb;
        tile[r][c] = pb;
    }
    if (!L.WTb) return;
    __syncthreads();
#pragma unroll
    for (int r = r0; r < ADAM_T; r += 8) {
        const int k = k0 + r, n = n0 + c;
        if (n < L.N && k < L.K) L.WTb[(size_t)k * L.N + n] = tile[c][r];
    }
}

const int KL[FP_SUR_LAYERS] = {FP_SUR_KIN, FP_SUR_HIDDEN, FP_SUR_HIDDEN, FP_SUR_HIDDEN, FP_SUR_HIDDEN};
const int NL[FP_SUR_LAYERS] = {FP_SUR_HIDDEN, FP_SUR_HIDDEN, FP_SUR_HIDDEN, FP_SUR_HIDDEN, FP_SUR_OUT};

size_t al256(size_t x) { return (x + 255) & ~(size_t)255; }

struct InferWs {
    __nv_bfloat16 *x0, *h[3];      // h[2]: the caller's output, unused until the last launch (ensemble)
    float* rowacc;                 // [q][2] (ensemble)
};

size_t infer_ws(long long q, bool ensemble, unsigned char* base, InferWs* w) {
    size_t o = 0;
    auto take = [&](size_t bytes) { unsigned char* p = base ? base + o : nullptr; o += al256(bytes); return p; };
    InferWs t;
    t.x0 = (__nv_bfloat16*)take((size_t)q * FP_SUR_KIN * 2);
    t.h[0] = (__nv_bfloat16*)take((size_t)q * FP_SUR_HIDDEN * 2);
    t.h[1] = (__nv_bfloat16*)take((size_t)q * FP_SUR_HIDDEN * 2);
    t.h[2] = nullptr;
    t.rowacc = nullptr;
    if (ensemble) t.rowacc = (float*)take((size_t)q * 2 * sizeof(float));
    if (w) *w = t;
    return o;
}

struct TrainWs {
    __nv_bfloat16 *x0, *x0T;                              // [q][64], [64][ldt]
    float* z[FP_SUR_LAYERS - 1];                          // [q][512] pre-activations
    __nv_bfloat16* h[FP_SUR_LAYERS - 1];                  // [q][512] activations (inputs of layers 1..4)
    __nv_bfloat16* hT[FP_SUR_LAYERS - 1];                 // [512][ldt]
    __nv_bfloat16 *g4, *g4T;                              // [q][800], [800][ldt]
    __nv_bfloat16* g[2];                                  // [q][512] ping-pong, in h[0] and h[1]: after the forward
                                                          // pass their transposes alone are read
    __nv_bfloat16* gT[FP_SUR_LAYERS - 1];                 // [512][ldt]: G^T of layers 0..3, kept for the dW launch
    int ldt;
};

size_t train_ws(long long q, unsigned char* base, TrainWs* w) {
    size_t o = 0;
    auto take = [&](size_t bytes) { unsigned char* p = base ? base + o : nullptr; o += al256(bytes); return p; };
    TrainWs t;
    t.ldt = (int)((q + 7) / 8 * 8);
    t.x0 = (__nv_bfloat16*)take((size_t)q * FP_SUR_KIN * 2);
    t.x0T = (__nv_bfloat16*)take((size_t)FP_SUR_KIN * t.ldt * 2);
    for (int l = 0; l < FP_SUR_LAYERS - 1; ++l) {
        t.z[l] = (float*)take((size_t)q * FP_SUR_HIDDEN * 4);
        t.h[l] = (__nv_bfloat16*)take((size_t)q * FP_SUR_HIDDEN * 2);
        t.hT[l] = (__nv_bfloat16*)take((size_t)FP_SUR_HIDDEN * t.ldt * 2);
    }
    t.g4 = (__nv_bfloat16*)take((size_t)q * FP_SUR_OUT * 2);
    t.g4T = (__nv_bfloat16*)take((size_t)FP_SUR_OUT * t.ldt * 2);
    for (int i = 0; i < 2; ++i) t.g[i] = t.h[i];
    for (int l = 0; l < FP_SUR_LAYERS - 1; ++l) t.gT[l] = (__nv_bfloat16*)take((size_t)FP_SUR_HIDDEN * t.ldt * 2);
    if (w) *w = t;
    return o;
}

EpiParams epi0(int* err) {
    EpiParams P;
    std::memset(&P, 0, sizeof(P));
    P.err = err;
    return P;
}

}  // namespace

extern "C" {

long long fp_surrogate_workspace_bytes(int q, int training) {
    if (q < 1) return fp_fail(FP_EINVAL, "fp_surrogate_workspace_bytes: q=%d", q);
    return (long long)(training && training != 2 ? train_ws(q, nullptr, nullptr)
                                                  : infer_ws(q, training == 2, nullptr, nullptr));
}

// normalised input and the four hidden layers of one network; layer l writes w.h[dst[l]]
static int hidden_layers(const fp_surrogate* net, const float* d_x, int q, const InferWs& w, const int* dst,
                         int* d_err, cudaStream_t st, const char* who) {
    for (int l = 0; l < FP_SUR_LAYERS; ++l)
        if (!net->W[l] || !net->b[l]) return fp_fail(FP_EINVAL, "%s: layer %d not set", who, l);
    if (!net->in_shift || !net->in_scale || !net->out_shift || !net->out_scale)
        return fp_fail(FP_EINVAL, "%s: normalisation not set", who);
    if ((uintptr_t)w.x0 & 15) return fp_fail(FP_EINVAL, "%s: workspace not on a 16-byte boundary", who);
    const long long tot = (long long)q * (FP_SUR_KIN / 8);
    prep_input_kernel<<<(unsigned)((tot + 255) / 256), 256, 0, st>>>(d_x, q, net->in_shift, net->in_scale, w.x0,
                                                                       nullptr, 0);
    if (cudaGetLastError() != cudaSuccess) return fp_fail(FP_ECUDA, "%s: input kernel launch", who);
    const __nv_bfloat16* x = w.x0;
    for (int l = 0; l < FP_SUR_LAYERS - 1; ++l) {
        EpiParams P = epi0(d_err);
        P.bias = net->b[l];
        P.out = w.h[dst[l]];
        P.ldo = FP_SUR_HIDDEN;
        const int rc = gemm_hidden<EPI_HIDDEN_INFER>({x, KL[l], net->W[l], KL[l]}, q, NL[l], KL[l], P, st);
        if (rc != FP_OK) return fp_fail(rc, "%s: layer %d GEMM launch failed", who, l);
        x = w.h[dst[l]];
    }
    return FP_OK;
}

int fp_surrogate_infer(const fp_surrogate* net, const float* d_x, int q, float* d_y, void* d_work,
                       unsigned long long work_bytes, int* d_err, void* stream) {
    if (!net || !d_x || !d_y || !d_work) return fp_fail(FP_EINVAL, "fp_surrogate_infer: NULL argument");
    if (q < 0) return fp_fail(FP_EINVAL, "fp_surrogate_infer: q=%d", q);
    if (q == 0) return FP_OK;
    InferWs w;
    const size_t need = infer_ws(q, false, (unsigned char*)d_work, &w);
    if (work_bytes < need)
        return fp_fail(FP_EINVAL, "fp_surrogate_infer: workspace %llu < %zu bytes", work_bytes, need);
    if (!d_err) return fp_fail(FP_EINVAL, "fp_surrogate_infer: d_err is required");
    cudaStream_t st = (cudaStream_t)stream;
    const int dst[FP_SUR_LAYERS - 1] = {0, 1, 0, 1};
    int rc = hidden_layers(net, d_x, q, w, dst, d_err, st, "fp_surrogate_infer");
    if (rc != FP_OK) return rc;
    EpiParams P = epi0(d_err);
    P.bias = net->b[4];
    P.outf = d_y;
    P.ldf = FP_SUR_OUT;
    P.oshift = net->out_shift;
    P.oscale = net->out_scale;
    const Operand op = {w.h[1], KL[4], net->W[4], KL[4]};
    rc = gemm_out<EPI_OUT_INFER>(&op, q, NL[4], KL[4], P, st);
    if (rc != FP_OK) return fp_fail(rc, "fp_surrogate_infer: layer 4 GEMM launch failed");
    return FP_OK;
}

// spread[r] = sqrt(sum |y0 - y1|^2) / (2 sqrt(sum |mean|^2))
__global__ void ensemble_spread_kernel(const float* __restrict__ rowacc, int q, float* __restrict__ spread) {
    const int r = blockIdx.x * blockDim.x + threadIdx.x;
    if (r >= q) return;
    spread[r] = sqrtf(rowacc[2 * r]) / (2.f * fmaxf(sqrtf(rowacc[2 * r + 1]), 1e-30f));
}

int fp_surrogate_infer_ensemble(const fp_surrogate* net0, const fp_surrogate* net1, const float* d_x, int q,
                                float* d_mean, float* d_spread, void* d_work, unsigned long long work_bytes,
                                int* d_err, void* stream) {
    if (!net0 || !net1 || !d_x || !d_mean || !d_spread || !d_work || !d_err)
        return fp_fail(FP_EINVAL, "fp_surrogate_infer_ensemble: NULL argument");
    if (q < 0) return fp_fail(FP_EINVAL, "fp_surrogate_infer_ensemble: q=%d", q);
    if (q == 0) return FP_OK;
    InferWs w;
    const size_t need = infer_ws(q, true, (unsigned char*)d_work, &w);
    if (work_bytes < need)
        return fp_fail(FP_EINVAL, "fp_surrogate_infer_ensemble: workspace %llu < %zu bytes", work_bytes, need);
    cudaStream_t st = (cudaStream_t)stream;
    if (cudaMemsetAsync(w.rowacc, 0, (size_t)q * 2 * sizeof(float), st) != cudaSuccess)
        return fp_fail(FP_ECUDA, "fp_surrogate_infer_ensemble: memset");
    // the first network's last activations stay in h[1], the second network's in h[0]; its own way
    // there needs a third buffer, for which the output, 3,200 bytes a query, has room until the last launch
    static_assert(FP_SUR_HIDDEN * 2 + 255 <= FP_SUR_OUT * 4, "activations of any batch fit into its output");
    w.h[2] = (__nv_bfloat16*)al256((size_t)d_mean);
    const int dst0[FP_SUR_LAYERS - 1] = {0, 1, 0, 1}, dst1[FP_SUR_LAYERS - 1] = {2, 0, 2, 0};
    int rc = hidden_layers(net0, d_x, q, w, dst0, d_err, st, "fp_surrogate_infer_ensemble");
    if (rc != FP_OK) return rc;
    rc = hidden_layers(net1, d_x, q, w, dst1, d_err, st, "fp_surrogate_infer_ensemble");
    if (rc != FP_OK) return rc;
    EpiParams P = epi0(d_err);
    P.bias = net0->b[4];
    P.oshift = net0->out_shift;
    P.oscale = net0->out_scale;
    P.bias1 = net1->b[4];
    P.oshift1 = net1->out_shift;
    P.oscale1 = net1->out_scale;
    P.outf = d_mean;
    P.ldf = FP_SUR_OUT;
    P.rowacc = w.rowacc;
    const Operand op[2] = {{w.h[1], KL[4], net0->W[4], KL[4]}, {w.h[0], KL[4], net1->W[4], KL[4]}};
    rc = gemm_out<EPI_OUT_ENSEMBLE>(op, q, NL[4], KL[4], P, st);
    if (rc != FP_OK) return fp_fail(rc, "fp_surrogate_infer_ensemble: layer 4 GEMM launch failed");
    ensemble_spread_kernel<<<(q + 255) / 256, 256, 0, st>>>(w.rowacc, q, d_spread);
    if (cudaGetLastError() != cudaSuccess) return fp_fail(FP_ECUDA, "fp_surrogate_infer_ensemble: spread kernel");
    return FP_OK;
}

int fp_surrogate_grad(const fp_surrogate_train* t, const float* d_x, const float* d_y, int q, float* d_loss,
                      float* const* d_gW, float* const* d_gb, void* d_work, unsigned long long work_bytes,
                      int* d_err, void* stream) {
    if (!t || !d_x || !d_y || !d_loss || !d_gW || !d_gb || !d_work || !d_err)
        return fp_fail(FP_EINVAL, "fp_surrogate_grad: NULL argument");
    if (q < 8 || q % 8) return fp_fail(FP_EINVAL, "fp_surrogate_grad: q=%d must be a positive multiple of 8", q);
    for (int l = 0; l < FP_SUR_LAYERS; ++l)
        if (!t->net.W[l] || !t->net.b[l] || !d_gW[l] || !d_gb[l] || (l > 0 && !t->WT[l]))
            return fp_fail(FP_EINVAL, "fp_surrogate_grad: layer %d not set", l);
    if (work_bytes < train_ws(q, nullptr, nullptr))
        return fp_fail(FP_EINVAL, "fp_surrogate_grad: workspace %llu < %zu bytes", work_bytes,
                       train_ws(q, nullptr, nullptr));
    cudaStream_t st = (cudaStream_t)stream;
    TrainWs w;
    train_ws(q, (unsigned char*)d_work, &w);
    if ((uintptr_t)w.x0 & 15) return fp_fail(FP_EINVAL, "fp_surrogate_grad: workspace not on a 16-byte boundary");
    if (cudaMemsetAsync(d_loss, 0, sizeof(float), st) != cudaSuccess ||
        cudaMemsetAsync(w.x0T, 0, (size_t)FP_SUR_KIN * w.ldt * 2, st) != cudaSuccess)
        return fp_fail(FP_ECUDA, "fp_surrogate_grad: memset");
    const long long tot = (long long)q * (FP_SUR_KIN / 8);
    prep_input_kernel<<<(unsigned)((tot + 255) / 256), 256, 0, st>>>(d_x, q, t->net.in_shift, t->net.in_scale,
                                                                       w.x0, w.x0T, w.ldt);
    if (cudaGetLastError() != cudaSuccess) return fp_fail(FP_ECUDA, "fp_surrogate_grad: input kernel launch");
    // forward, keeping pre-activations and transposed activations
    const __nv_bfloat16* x = w.x0;
    int rc;
    for (int l = 0; l < FP_SUR_LAYERS - 1; ++l) {
        EpiParams P = epi0(d_err);
        P.bias = t->net.b[l];
        P.out = w.h[l]; P.ldo = FP_SUR_HIDDEN;
        P.outT = w.hT[l]; P.ldt = w.ldt;
        P.outf = w.z[l]; P.ldf = FP_SUR_HIDDEN;
        rc = gemm_hidden<EPI_HIDDEN_TRAIN>({x, KL[l], t->net.W[l], KL[l]}, q, NL[l], KL[l], P, st);
        if (rc != FP_OK) return fp_fail(rc, "fp_surrogate_grad: forward layer %d", l);
        x = w.h[l];
    }
    {
        EpiParams P = epi0(d_err);
        P.bias = t->net.b[4];
        P.y = d_y; P.ldy = FP_SUR_OUT;
        P.oshift = t->net.out_shift; P.oscale = t->net.out_scale;
        P.loss = d_loss;
        P.gscale = 2.f / ((float)q * (float)FP_SUR_OUT);
        P.out = w.g4; P.ldo = FP_SUR_OUT;
        P.outT = w.g4T; P.ldt = w.ldt;
        const Operand op = {x, KL[4], t->net.W[4], KL[4]};
        rc = gemm_out<EPI_OUT_TRAIN>(&op, q, NL[4], KL[4], P, st);
        if (rc != FP_OK) return fp_fail(rc, "fp_surrogate_grad: output layer");
    }
    // backward: G_{l-1} = (G_l W_l) * gelu'(z_{l-1}), A = G_l [q][N_l], B = W_l^T [K_l][N_l]
    const __nv_bfloat16* G = w.g4;
    for (int l = FP_SUR_LAYERS - 1; l >= 1; --l) {
        EpiParams P = epi0(d_err);
        P.zin = w.z[l - 1]; P.ldz = FP_SUR_HIDDEN;
        P.out = w.g[l & 1]; P.ldo = FP_SUR_HIDDEN;
        P.outT = w.gT[l - 1]; P.ldt = w.ldt;
        rc = gemm_hidden<EPI_DX_GELU>({G, NL[l], t->WT[l], NL[l]}, q, KL[l], NL[l], P, st);
        if (rc != FP_OK) return fp_fail(rc, "fp_surrogate_grad: dX layer %d", l);
        G = w.g[l & 1];
    }
    // dW_l [N_l][K_l] = G_l^T X_l of all layers in one launch: A = G_l^T [N_l][q], B = X_l^T [K_l][q]
    BiasArgs ba;
    DwLayer dw[FP_SUR_LAYERS];
    ba.row0[0] = 0;
    ba.ldt = w.ldt;
    ba.q = q;
    for (int l = 0; l < FP_SUR_LAYERS; ++l) {
        const __nv_bfloat16* GT = l == FP_SUR_LAYERS - 1 ? w.g4T : w.gT[l];
        dw[l] = {GT, l == 0 ? w.x0T : w.hT[l - 1], d_gW[l], NL[l], KL[l]};
        ba.gT[l] = GT;
        ba.db[l] = d_gb[l];
        ba.row0[l + 1] = ba.row0[l] + NL[l];
    }
    rc = gemm_dw(dw, q, w.ldt, d_err, st);
    if (rc != FP_OK) return fp_fail(rc, "fp_surrogate_grad: dW");
    bias_grad_kernel<<<(ba.row0[MAXG] + 7) / 8, 256, 0, st>>>(ba);
    if (cudaGetLastError() != cudaSuccess) return fp_fail(FP_ECUDA, "fp_surrogate_grad: bias kernel");
    return FP_OK;
}

int fp_surrogate_adam(const fp_surrogate_train* t, float* const* d_gW, float* const* d_gb, float lr, float beta1,
                      float beta2, float eps, int step, void* stream) {
    if (!t || step < 0) return fp_fail(FP_EINVAL, "fp_surrogate_adam: bad argument");
    if (step > 0 && (!d_gW || !d_gb)) return fp_fail(FP_EINVAL, "fp_surrogate_adam: NULL gradients");
    AdamNet net;
    AdamArgs& a = net.a;
    a.lr = lr; a.b1 = beta1; a.b2 = beta2; a.eps = eps; a.step = step;
    a.c1 = step > 0 ? 1.f - powf(beta1, (float)step) : 1.f;
    a.c2 = step > 0 ? 1.f - powf(beta2, (float)step) : 1.f;
    int blocks = 0;
    for (int l = 0; l < FP_SUR_LAYERS; ++l) {
        if (!t->Wm[l] || !t->net.W[l] || (step > 0 && (!t->mW[l] || !t->vW[l] || !t->bm[l] || !t->mb[l] ||
                                                        !t->vb[l] || !d_gW[l] || !d_gb[l])))
            return fp_fail(FP_EINVAL, "fp_surrogate_adam: layer %d not set", l);
        net.l[l] = {t->Wm[l], t->mW[l], t->vW[l], t->bm[l], t->mb[l], t->vb[l], step > 0 ? d_gW[l] : nullptr,
                    step > 0 ? d_gb[l] : nullptr, (__nv_bfloat16*)t->net.W[l],
                    l > 0 ? (__nv_bfloat16*)t->WT[l] : nullptr, NL[l], KL[l], blocks};
        blocks += adam_tiles(NL[l], KL[l]) + 1;
    }
    adam_kernel<<<blocks, 256, 0, (cudaStream_t)stream>>>(net);
    if (cudaGetLastError() != cudaSuccess) return fp_fail(FP_ECUDA, "fp_surrogate_adam: launch");
    return FP_OK;
}

}  // extern "C"
