// Self-absorption: dust that is optically thick to its own emission is heated
// by it too, so the radiation field and the temperatures have to be found
// together by iteration (Section 2; the paper's radiative-transfer code does it
// globally).  This is a local form of that iteration around the hot path:
//   J^(0) = J_ext,   J^(i) = J_ext + E (.) L^(i),   L^(i) = emission of solve(J^(i-1)),
// with a caller-supplied coupling E[c,k] >= 0 (the part of the cell's own
// emission L[c,k] that returns to its mean intensity J[c,k]).  It stops when
// the largest peak-normalised change of L between two iterations,
//   max_c max_k |L^(i)[c,k] - L^(i-1)[c,k]| / max_k L^(i)[c,k],
// falls to `tol`, or after `max_iters` solves.
#include "dust_internal.cuh"

#include <algorithm>
#include <cstring>

namespace dust {
namespace {

constexpr int CPL_TH = 128;

// One warp per cell: the change of L against the previous iterate (folded
// into *change with an integer max on the float's bits, exact for values
// >= 0), then Lprev = L and Jw = J_ext + E L.  The last CTA to finish (count)
// leaves the change in the host's word and clears both words for the next pass.
// The pass is six rows per cell, bound by memory (by L2 up to some 30000
// cells).  VEC (rows of whole, aligned 16-byte pieces): every load of a row is
// issued before the first is used, which is once for K <= 256 (CPL_V pieces a
// lane), and L stays in registers between its two uses.  16384 x 200 out of memory:
// 24 -> 19 us (79 MB: 12 us at the copy rate).
constexpr int CPL_V = 2;
constexpr unsigned int NOT_YET = 0x7f800000u;  // infinity: the host's word where no change has been measured

template <bool VEC>
__global__ void __launch_bounds__(CPL_TH) k_couple(int64_t C, int K, int64_t ld, const float *Jext,
                                                   const float *E, const float *L, float *Lprev, float *Jw,
                                                   int first, unsigned int *change, unsigned int *count,
                                                   volatile unsigned int *host) {
    const int lane = threadIdx.x & 31;
    const int64_t nw = ((int64_t)gridDim.x * CPL_TH) >> 5;
    after_previous_kernel();
    for (int64_t c = ((int64_t)blockIdx.x * CPL_TH + threadIdx.x) >> 5; c < C; c += nw) {
        const float *Lr = L + c * ld;
        float *Pr = Lprev + c * ld;
        const float *Jr = Jext + c * ld, *Er = E + c * ld;
        float *Wr = Jw + c * ld;
        float peak = 0.f, d = 0.f;
        if constexpr (VEC) {
            const int nv = K / 4;
            for (int v0 = lane; v0 < nv; v0 += 32 * CPL_V) {
                float4 l[CPL_V], q[CPL_V], j[CPL_V], e[CPL_V];
#pragma unroll
                for (int i = 0; i < CPL_V; ++i) {
                    const int v = v0 + 32 * i;
                    l[i] = q[i] = j[i] = e[i] = make_float4(0.f, 0.f, 0.f, 0.f);
                    if (v < nv) {
                        l[i] = reinterpret_cast<const float4 *>(Lr)[v];
                        if (!first) q[i] = reinterpret_cast<const float4 *>(Pr)[v];
                        j[i] = __ldg(reinterpret_cast<const float4 *>(Jr) + v);
                        e[i] = __ldg(reinterpret_cast<const float4 *>(Er) + v);
                    }
                }
#pragma unroll
                for (int i = 0; i < CPL_V; ++i) {
                    const int v = v0 + 32 * i;
                    peak = fmaxf(peak, fmaxf(fmaxf(l[i].x, l[i].y), fmaxf(l[i].z, l[i].w)));
                    if (!first)
                        d = fmaxf(d, fmaxf(fmaxf(fabsf(l[i].x - q[i].x), fabsf(l[i].y - q[i].y)),
                                           fmaxf(fabsf(l[i].z - q[i].z), fabsf(l[i].w - q[i].w))));
                    if (v < nv) {
                        reinterpret_cast<float4 *>(Pr)[v] = l[i];
                        reinterpret_cast<float4 *>(Wr)[v] =
                            make_float4(fmaf(e[i].x, l[i].x, j[i].x), fmaf(e[i].y, l[i].y, j[i].y),
                                        fmaf(e[i].z, l[i].z, j[i].z), fmaf(e[i].w, l[i].w, j[i].w));
                    }
                }
            }
        }
        for (int k = (VEC ? K / 4 * 4 : 0) + lane; k < K; k += 32) {
            const float v = Lr[k];
            peak = fmaxf(peak, v);
            if (!first) d = fmaxf(d, fabsf(v - Pr[k]));
            Pr[k] = v;
            Wr[k] = fmaf(Er[k], v, Jr[k]);
        }
        if (first) continue;
        // peak and d are >= 0 and not NaN (fmaxf drops NaN operands): they order as their bits do
        peak = __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(peak)));
        d = __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(d)));
        if (lane == 0) {
            float ch = d > 0.f ? (peak > 0.f ? d / peak : INFINITY) : 0.f;
            if (!(ch == ch)) ch = INFINITY;  // NaN counts as not converged
            atomicMax(change, __float_as_uint(ch));
        }
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();
        if (atomicAdd(count, 1u) == gridDim.x - 1) {
            __threadfence();
            const unsigned int c = atomicExch(change, 0u);
            *host = first ? NOT_YET : c;
            *count = 0u;
            __threadfence_system();
        }
    }
}

int check_dev(const void *p, int device, const char *name) {
    cudaPointerAttributes a;
    if (cudaPointerGetAttributes(&a, p) != cudaSuccess) {
        cudaGetLastError();
        return set_error(DUST_EINVAL, "%s: not a CUDA pointer", name);
    }
    if (a.type != cudaMemoryTypeDevice && a.type != cudaMemoryTypeManaged)
        return set_error(DUST_EINVAL, "%s must be device memory", name);
    if (a.type == cudaMemoryTypeDevice && a.device != device)
        return set_error(DUST_EINVAL, "%s lives on device %d, the context on device %d", name, a.device, device);
    return DUST_OK;
}

}  // namespace
}  // namespace dust

using namespace dust;

extern "C" int dust_solve_coupled(dust_ctx *ctx, int64_t n_cells, const float *J_ext, int64_t ld, const float *E,
                                  const float *n, int max_iters, double tol, float *T, float *L, double *resid,
                                  uint8_t *flags, int *iters_done, double *last_change, void *stream) {
    if (!ctx) return set_error(DUST_EINVAL, "ctx is NULL");
    if (n_cells < 0) return set_error(DUST_EINVAL, "n_cells < 0");
    if (ld < ctx->K) return set_error(DUST_EINVAL, "ld=%lld < K=%d", (long long)ld, ctx->K);
    if (max_iters < 1 || max_iters > 10000) return set_error(DUST_EINVAL, "max_iters outside [1, 10000]");
    if (!(tol >= 0.0)) return set_error(DUST_EINVAL, "tol must be >= 0");
    if (iters_done) *iters_done = 0;
    if (last_change) *last_change = 0.0;
    if (n_cells == 0) return DUST_OK;
    if (!J_ext || !E || !n || !T || !L) return set_error(DUST_EINVAL, "J_ext, E, n, T and L must be non-NULL");
    const int precision = ctx->precision;
    if (precision != DUST_PREC_FP32 && (ld % 4 != 0 || ((uintptr_t)J_ext & 15) != 0))
        return set_error(DUST_EINVAL, "tensor-core precisions need ld %% 4 == 0 and a 16-byte aligned J_ext");
    int rc;
    if ((rc = check_dev(J_ext, ctx->device, "J_ext")) || (rc = check_dev(E, ctx->device, "E")) ||
        (rc = check_dev(n, ctx->device, "n")) || (rc = check_dev(T, ctx->device, "T")) ||
        (rc = check_dev(L, ctx->device, "L")) || (resid && (rc = check_dev(resid, ctx->device, "resid"))) ||
        (flags && (rc = check_dev(flags, ctx->device, "flags"))))
        return rc;
    std::lock_guard<std::mutex> lk(ctx->mu);
    int prev = -1;
    if (cudaGetDevice(&prev) != cudaSuccess) return set_error(DUST_ECUDA, "cudaGetDevice failed");
    if (prev != ctx->device && cudaSetDevice(ctx->device) != cudaSuccess)
        return set_error(DUST_ECUDA, "cudaSetDevice(%d) failed", ctx->device);
    cudaStream_t st = (cudaStream_t)stream;
    // working J, previous L and the change word, grown on demand
    const size_t need = (size_t)2 * n_cells * ld * sizeof(float) + 256;
    rc = DUST_OK;
    if (ctx->cpl_bytes < need) {
        cudaError_t e = cudaStreamSynchronize(st);
        if (e == cudaSuccess) {
            cudaFree(ctx->cpl);
            ctx->cpl = nullptr;
            ctx->cpl_bytes = 0;
            e = cudaMalloc(&ctx->cpl, need);
        }
        // columns K..ld of the working J are read as padding by nothing, but keep them defined;
        // cleared in `st`, since nothing orders another stream's clear before the passes
        if (e == cudaSuccess) e = cudaMemsetAsync(ctx->cpl, 0, need, st);
        if (e == cudaSuccess) ctx->cpl_bytes = need;
        else rc = set_error(DUST_ENOMEM, "coupled-solve buffers: %s", cudaGetErrorString(e));
    }
    float *Jw = static_cast<float *>(ctx->cpl);
    float *Lprev = Jw + (size_t)n_cells * ld;
    unsigned int *chg = reinterpret_cast<unsigned int *>(Lprev + (size_t)n_cells * ld);
    const float *Jcur = J_ext;
    int it = 0;
    float change = INFINITY;
    if (rc == DUST_OK) rc = ensure_scratch(ctx, n_cells, st);
    const int64_t grid = std::min<int64_t>((n_cells * 32 + CPL_TH - 1) / CPL_TH, (int64_t)ctx->num_sms * 16);
    const bool vec = ld % 4 == 0 && (((uintptr_t)J_ext | (uintptr_t)E | (uintptr_t)L) & 15) == 0;
    if (rc == DUST_OK && cudaMemsetAsync(chg, 0, 2 * sizeof(unsigned int), st) != cudaSuccess) {
        cudaGetLastError();
        rc = set_error(DUST_ECUDA, "clearing the change words failed");
    }
    if (rc == DUST_OK && !ctx->cpl_host && cudaHostAlloc((void **)&ctx->cpl_host, sizeof(unsigned int), cudaHostAllocMapped) != cudaSuccess) {
        cudaGetLastError();
        ctx->cpl_host = nullptr;
        rc = set_error(DUST_ENOMEM, "the coupled solve's page-locked word: cudaHostAlloc failed");
    }
    if (rc == DUST_OK && !ctx->cpl_ev && cudaEventCreateWithFlags(&ctx->cpl_ev, cudaEventDisableTiming) != cudaSuccess) {
        cudaGetLastError();
        ctx->cpl_ev = nullptr;
        rc = set_error(DUST_ECUDA, "the coupled solve's event could not be made");
    }
    // While the host learns a pass's change, the GPU runs the next pass's
    // absorption, which writes nothing but scratch: the round trip (about 10 us)
    // would leave it idle.  Not where absorption and solve are one kernel, nor
    // while stages are timed.
    const bool ahead = !(ctx->fused && precision != DUST_PREC_FP32) && !ctx->prof_on;
    bool absorbed = false;
    auto solve = [&](int phases) {
        // the cells' classes change little from one iterate to the next, and no
        // result depends on them: the emission order is made once (16384 cells x 200 x
        // 96, 24 solves: 3.39 ms with a new order for each, 3.06 with one)
        return solve_device(ctx, precision, n_cells, Jcur, ld, n, T, L, resid, flags, ctx->S, st, false, it > 0, phases);
    };
    while (rc == DUST_OK && it < max_iters) {
        rc = solve(absorbed ? SOLVE_REST : SOLVE_ALL);
        absorbed = false;
        if (rc != DUST_OK) break;
        ++it;
        // a pass that left no change must not pass for one that left a small one
        // (the first one's word, not waited for, says the same)
        *(volatile unsigned int *)ctx->cpl_host = NOT_YET;
        cudaError_t e = launch_early(true, vec ? k_couple<true> : k_couple<false>, (unsigned)grid, CPL_TH, 0, st, n_cells, ctx->K, ld,
                                     J_ext, E, (const float *)L, Lprev, Jw, (int)(it == 1), chg, chg + 1,
                                     (volatile unsigned int *)ctx->cpl_host);
        Jcur = Jw;
        if (it == 1 && it < max_iters && e == cudaSuccess) continue;  // nothing to compare with yet: the next solve follows at once
        if (e == cudaSuccess) e = cudaEventRecord(ctx->cpl_ev, st);
        if (e == cudaSuccess && ahead && it < max_iters) {
            rc = solve(SOLVE_ABSORB);
            absorbed = rc == DUST_OK;
        }
        if (e == cudaSuccess) e = cudaEventSynchronize(ctx->cpl_ev);
        if (e != cudaSuccess && rc == DUST_OK) rc = set_error(DUST_ECUDA, "coupled iteration: %s", cudaGetErrorString(e));
        if (rc != DUST_OK) break;
        if (it > 1) {
            const unsigned int bits = *(volatile unsigned int *)ctx->cpl_host;
            std::memcpy(&change, &bits, sizeof(change));
            if (change <= tol) break;
        }
    }
    if (absorbed && cudaStreamSynchronize(st) != cudaSuccess && rc == DUST_OK) {
        cudaGetLastError();
        rc = set_error(DUST_ECUDA, "coupled iteration: waiting for the last absorption failed");
    }
    if (prev >= 0 && prev != ctx->device) cudaSetDevice(prev);
    if (iters_done) *iters_done = it;
    if (last_change) *last_change = (double)change;
    return rc;
}
