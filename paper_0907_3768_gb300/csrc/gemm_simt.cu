// Absorption contraction on the CUDA cores in FP32 (the plain FP32 path):
//   S[c,g] = sum_k J[c,k] W32[g,k]                          (Eq. 6, scaled)
// The paper's kernel 2 is the same matrix product with shared-memory tiles
// over wavelength intervals (Section 4.2).  Here: 128-cell x (16 TN)-grain CTA
// tiles over a work list of requests, stages of 16 wavelengths, an 8 x TN
// register tile per thread, FP32 FMA accumulation in ascending k (so a cell's
// result does not depend on the tiling or the batch).
//
// FMA-bound: at K = 200, G = 96 48 us of FMAs against 17 us of memory for 100000
// cells.  A thread's columns come in pairs, one 8-byte load and one packed FMA
// each (scalar FMAs: 112 and 251 us).  Two ways to fill the stages:
// REGS: through registers, eight wavelengths of a row per thread in two 16-byte
// loads, the next stage's while one is multiplied, two stages.  Where rows are not
// aligned that is eight words, which touch 32 lines per instruction (100003 x 201 x
// 96 took 119 us), so there
// cp.async, a word at a time with the lanes along k: rows of J may start anywhere
// (ld is the caller's), and 16 lanes read 64 consecutive bytes of one whatever its
// alignment, three stages, three CTAs per SM up to 96 columns (two: 101 us; now 98).
// Its many small copies take as long as a stage's FMAs at one CTA per SM: 612 x 6,
// 32 cells, 39 us for the whole call, 25 through registers.  launch_simt_batch chooses.
#include "dust_internal.cuh"

#include <algorithm>

namespace dust {
namespace {

constexpr int BM = 128, BK = 16, NTH = 256, NST = 3;
constexpr int AST = BM + 4;                                  // row of a stage of J: [BK][AST], 16-byte aligned
__host__ __device__ constexpr int bst(int TN) { return 16 * TN + 2; }  // and of W: [BK][bst], even
__host__ __device__ constexpr int stage_floats(int TN) { return BK * (AST + bst(TN)); }

// A word to shared memory; 0 where `on` is false (nothing is read then).
__device__ __forceinline__ void cp_word(uint32_t dst, const float *src, bool on) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(dst), "l"(src), "r"(on ? 4 : 0) : "memory");
}

template <int TN, bool REGS>
__global__ void __launch_bounds__(NTH, TN <= 6 && !REGS ? 3 : 2) k_gemm_simt(const __grid_constant__ SimtBatch B) {
    constexpr int BN = 16 * TN, NP = TN / 2, BST = bst(TN);
    extern __shared__ __align__(16) float sm[];  // stages of J, then of W: [NST], or two with REGS
    const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;

    const int64_t tile = blockIdx.x;
    let_next_kernel_start();
    if (tile == 0) clear_spans(B.zero);
    int ri = 0;
    while (ri + 1 < B.nreq && tile >= B.req[ri + 1].tile_begin) ++ri;
    const SimtReq &q = B.req[ri];
    const int64_t local = tile - q.tile_begin;
    const int64_t m0 = (local / q.ntn) * BM;
    const int n0 = (int)(local % q.ntn) * BN;
    const int K = q.K, Kw = q.Kw, Gs = q.Gs;
    const int64_t C = q.C, ld = q.ld;

    // this thread's words of a stage: wavelength tx of rows ty, ty + 16, ... of J
    // and of W.  Rows past the last are the last again (nothing of them is
    // stored), so that only wavelengths past K need a test, in the last stage.
    const int64_t jrows = min(C - m0, (int64_t)BM);
    const int wrows = min(Gs - n0, BN);
    const float *jp = q.J + m0 * ld + tx, *wp = q.W + (size_t)n0 * Kw + tx;
    const uint32_t sA = (uint32_t)__cvta_generic_to_shared(sm) + (tx * AST + ty) * 4;
    const uint32_t sB = (uint32_t)__cvta_generic_to_shared(sm) + (BK * AST + tx * BST + ty) * 4;
    auto load = [&](int t) {
        const uint32_t off = (uint32_t)(t % NST * stage_floats(TN) * 4);
        const bool on = t * BK + tx < K;
        const float *j = on ? jp + t * BK : q.J, *w = wp + t * BK;  // W's rows are padded with zeros to Kw
        if (jrows == BM) {
            const float *r = j + (on ? ty * ld : 0);
            const int64_t step = on ? 16 * ld : 0;
#pragma unroll
            for (int i = 0; i < BM / 16; ++i, r += step) cp_word(sA + off + 64 * i, r, on);
        } else {
#pragma unroll 1
            for (int i = 0; i < BM / 16; ++i) cp_word(sA + off + 64 * i, on ? j + min(ty + 16 * i, (int)jrows - 1) * ld : j, on);
        }
        if (wrows == BN) {
            const float *r = w + (size_t)ty * Kw;
#pragma unroll
            for (int i = 0; i < TN; ++i, r += 16 * Kw) cp_word(sB + off + 64 * i, r, true);
        } else {
#pragma unroll 1
            for (int i = 0; i < TN; ++i) cp_word(sB + off + 64 * i, w + (size_t)min(ty + 16 * i, wrows - 1) * Kw, true);
        }
    };

    // columns 32 p + 2 tx, 32 p + 2 tx + 1 for p < NP, and 32 NP + tx when TN is odd
    float2 acc[8][NP > 0 ? NP : 1];
    float last[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        last[i] = 0.f;
#pragma unroll
        for (int p = 0; p < NP; ++p) acc[i][p] = make_float2(0.f, 0.f);
    }

    auto multiply = [&](const float *As) {
        const float *Bs = As + BK * AST;
#pragma unroll
        for (int kk = 0; kk < BK; ++kk) {
            const float4 a0 = *reinterpret_cast<const float4 *>(As + kk * AST + ty * 8);
            const float4 a1 = *reinterpret_cast<const float4 *>(As + kk * AST + ty * 8 + 4);
            const float a[8] = {a0.x, a0.y, a0.z, a0.w, a1.x, a1.y, a1.z, a1.w};
#pragma unroll
            for (int p = 0; p < NP; ++p) {
                const float2 b = *reinterpret_cast<const float2 *>(Bs + kk * BST + 32 * p + 2 * tx);
#pragma unroll
                for (int i = 0; i < 8; ++i) acc[i][p] = __ffma2_rn(make_float2(a[i], a[i]), b, acc[i][p]);
            }
            if (TN & 1) {
                const float b = Bs[kk * BST + 32 * NP + tx];
#pragma unroll
                for (int i = 0; i < 8; ++i) last[i] = fmaf(a[i], b, last[i]);
            }
        }
    };
    const int nk = (K + BK - 1) / BK;
    if constexpr (REGS) {
        // through registers: eight wavelengths of a row of J per thread, the next
        // stage's on their way while this one is multiplied
        const int ar = tid >> 1, ak = (tid & 1) * 8;
        const float *jr = q.J + (m0 + min((int64_t)ar, jrows - 1)) * ld;
        const bool vec = ld % 4 == 0 && ((uintptr_t)q.J & 15) == 0;
        float jv[8], wv[TN];
        auto fetch = [&](int t) {
            const int k0 = t * BK + ak;
            if (vec && k0 + 8 <= K) {
                const float4 v0 = __ldg(reinterpret_cast<const float4 *>(jr + k0)), v1 = __ldg(reinterpret_cast<const float4 *>(jr + k0) + 1);
                jv[0] = v0.x; jv[1] = v0.y; jv[2] = v0.z; jv[3] = v0.w;
                jv[4] = v1.x; jv[5] = v1.y; jv[6] = v1.z; jv[7] = v1.w;
            } else {
#pragma unroll
                for (int e = 0; e < 8; ++e) jv[e] = k0 + e < K ? __ldg(jr + k0 + e) : 0.f;
            }
#pragma unroll
            for (int i = 0; i < TN; ++i) wv[i] = __ldg(wp + t * BK + (size_t)min(ty + 16 * i, wrows - 1) * Kw);
        };
        auto put = [&](int t) {
            float *As = sm + (t & 1) * stage_floats(TN), *Bs = As + BK * AST;
#pragma unroll
            for (int e = 0; e < 8; ++e) As[(ak + e) * AST + ar] = jv[e];
#pragma unroll
            for (int i = 0; i < TN; ++i) Bs[tx * BST + ty + 16 * i] = wv[i];
        };
        fetch(0);
        put(0);
        for (int t = 0; t < nk; ++t) {
            __syncthreads();  // stage t is there for all, and stage t - 1 is read by all
            if (t + 1 < nk) fetch(t + 1);
            multiply(sm + (t & 1) * stage_floats(TN));
            if (t + 1 < nk) put(t + 1);
        }
    } else {
#pragma unroll
        for (int t = 0; t < NST - 1; ++t) {
            if (t < nk) load(t);
            asm volatile("cp.async.commit_group;" ::: "memory");
        }
        for (int t = 0; t < nk; ++t) {
            asm volatile("cp.async.wait_group %0;" ::"n"(NST - 2) : "memory");
            __syncthreads();  // stage t is there for all, and stage t - 1 is read by all
            if (t + NST - 1 < nk) load(t + NST - 1);
            asm volatile("cp.async.commit_group;" ::: "memory");
            multiply(sm + t % NST * stage_floats(TN));
        }
    }
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        const int64_t row = m0 + ty * 8 + i;
        if (row >= C) break;
        float *out = q.S + row * Gs + n0;  // Gs and n0 are multiples of 16
#pragma unroll
        for (int p = 0; p < NP; ++p)
            if (n0 + 32 * p + 2 * tx < Gs) *reinterpret_cast<float2 *>(out + 32 * p + 2 * tx) = acc[i][p];
        if ((TN & 1) && n0 + 32 * NP + tx < Gs) out[32 * NP + tx] = last[i];
    }
}

template <int TN, bool REGS>
int launch_simt(const SimtBatch &B, unsigned grid, cudaStream_t st) {
    constexpr int smem = (REGS ? 2 : NST) * stage_floats(TN) * (int)sizeof(float);
    DUST_CUDA_TRY(allow_shared_memory((k_gemm_simt<TN, REGS>)));
    k_gemm_simt<TN, REGS><<<grid, NTH, smem, st>>>(B);
    DUST_CUDA_TRY(cudaGetLastError());
    return DUST_OK;
}

}  // namespace

void make_simt_req(const dust_ctx *ctx, int64_t C, const float *J, int64_t ld, float *S, SimtReq &r) {
    r.C = C;
    r.ld = ld;
    r.tile_begin = 0;
    r.J = J;
    r.W = ctx->W32;
    r.S = S;
    r.K = ctx->K;
    r.Kw = ctx->Kw;
    r.Gs = ctx->tb.Gs;
    r.ntn = 0;
}

// Picks the register tile width from the widest request, numbers the tiles
// and launches one CTA per (cell tile, grain tile).
int launch_simt_batch(SimtBatch &B, int num_sms, cudaStream_t st) {
    int gmax = 16;
    for (int i = 0; i < B.nreq; ++i) gmax = std::max(gmax, B.req[i].Gs);
    const int t16 = gmax / 16;  // 1..32
    const int ntile = (t16 + 7) / 8;
    const int TN = (t16 + ntile - 1) / ntile;
    int64_t t = 0;
    for (int i = 0; i < B.nreq; ++i) {
        SimtReq &r = B.req[i];
        r.ntn = (r.Gs + 16 * TN - 1) / (16 * TN);
        r.tile_begin = t;
        t += (r.C + BM - 1) / BM * r.ntn;
    }
    B.ntiles = t;
    if (t <= 0) return DUST_OK;
    if (t > 0x7fffffff) return set_error(DUST_EINVAL, "too many cells for one launch");
    const unsigned grid = (unsigned)t;
    // Through registers or by cp.async (see above): us, temperatures only, cp.async
    // and registers.  Aligned rows: 612 x 96, 2000 cells 69.8 / 53.4, 60000 228 / 203; 292 x
    // 96, 262144 cells 427 / 407; 200 x 96 336 / 320; with fewer than 65 columns while the
    // tiles are few, 612 x 6, 32 cells 39.0 / 24.6, 60000 110 / 103; 200 x 24, 262144 cells
    // 158 / 164.  Other rows, a word at a time: 201 x 96, 2000 cells 27.3 / 24.6, 15000 34.3 /
    // 30.8, 19456 32.8 / 32.8, 262144 337 / 346; 201 x 24 there 160 / 199.
    bool aligned = true;
    for (int i = 0; i < B.nreq; ++i) aligned = aligned && B.req[i].ld % 4 == 0 && ((uintptr_t)B.req[i].J & 15) == 0;
    const bool regs = aligned ? TN >= 5 || t <= 4 * (int64_t)num_sms : 8 * t <= 7 * (int64_t)num_sms;
    switch (TN) {
        case 1: return regs ? launch_simt<1, true>(B, grid, st) : launch_simt<1, false>(B, grid, st);
        case 2: return regs ? launch_simt<2, true>(B, grid, st) : launch_simt<2, false>(B, grid, st);
        case 3: return regs ? launch_simt<3, true>(B, grid, st) : launch_simt<3, false>(B, grid, st);
        case 4: return regs ? launch_simt<4, true>(B, grid, st) : launch_simt<4, false>(B, grid, st);
        case 5: return regs ? launch_simt<5, true>(B, grid, st) : launch_simt<5, false>(B, grid, st);
        case 6: return regs ? launch_simt<6, true>(B, grid, st) : launch_simt<6, false>(B, grid, st);
        case 7: return regs ? launch_simt<7, true>(B, grid, st) : launch_simt<7, false>(B, grid, st);
        default: return regs ? launch_simt<8, true>(B, grid, st) : launch_simt<8, false>(B, grid, st);
    }
}

int launch_gemm_simt(const dust_ctx *ctx, int64_t C, const float *J, int64_t ld, float *S, cudaStream_t st,
                     const ZeroSpans &zero) {
    if (C <= 0) return DUST_OK;
    SimtBatch B;
    B.nreq = 1;
    B.zero = zero;
    make_simt_req(ctx, C, J, ld, S, B.req[0]);
    return launch_simt_batch(B, ctx->num_sms, st);
}

}  // namespace dust
