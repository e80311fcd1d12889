// vq_stream.cu -- sparse local field fused with the ballistic-SB update, one
// launch per step, state in HBM (variable-major [n][R]: the R replicas of a
// variable are contiguous, so a neighbour's state is one coalesced vector
// load shared by all lanes of the row), plus the exact readout energy.
//
// Step (App. B, ballistic form):  F_i = sum_{j != i} Qs_ij s_j  over the CSR
// row of i, then phi, y, s, walls. Couplings come as FP32 Qs or, for integer
// instances with |2 Qs| <= 127, as int8 2Qs (F = acc / 2, exact scaling).
#include <algorithm>
#include <cstdio>
#include <cstdlib>
#include <vector>

#include "vq_internal.cuh"

namespace vq {

namespace {

using vqd::vload;
using vqd::vload_plain;
using vqd::vload_stream;
using vqd::vstore_stream;
using vqd::vstore;
using vqd::wval;

// One thread per (variable i, vector v of V replicas). Y_in and Y_out may be
// the same buffer (in-place update). SIGN: the field is of PA's binarised
// spins; method selects the update (veloxq_method).
template <int V, typename WT, bool FIELD_ONLY, int UNROLL, bool SIGN, bool DEP>
__global__ void __launch_bounds__(256) k_stream_step(int64_t n, int32_t R, int32_t nvec, const int64_t* __restrict__ rp,
                                                     const int32_t* __restrict__ col, const WT* __restrict__ w,
                                                     float wscale, const float* __restrict__ S_cur,
                                                     float* __restrict__ S_nxt, const float* Y_in, float* Y_out,
                                                     const float* __restrict__ bf, const float* __restrict__ a_table,
                                                     int k, float dt, float a0, float c0, float* __restrict__ F_out,
                                                     int udeg, int method, float alpha, int32_t cvec) {
    // threads in chunk-major order: all rows of replica vectors [c cvec,
    // (c+1) cvec) before the next chunk (cvec = nvec: one chunk), so that
    // the neighbours' states a wave gathers span one chunk of every row
    const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= n * nvec) return;
    int64_t i;
    int32_t v;
    if (cvec == nvec) {
        vqd::split_index(t, n, nvec, i, v);
    } else {
        // chunk c = t / (n cvec), then row and vector within the chunk
        int64_t c, rem;
        if (n * nvec < (int64_t(1) << 32)) {
            const uint32_t per_chunk = (uint32_t)n * (uint32_t)cvec;
            c = (uint32_t)t / per_chunk;
            rem = t - c * per_chunk;
        } else {
            c = t / (n * cvec);
            rem = t - c * n * cvec;
        }
        int32_t w;
        vqd::split_index(rem, n, cvec, i, w);
        v = (int32_t)(c * cvec) + w;
    }
    const int64_t off = (int64_t)v * V;
    const int64_t me = i * R + off;
    // DEP: launched dependently; only the index arithmetic above overlaps the previous step
    if constexpr (DEP) {
        asm volatile("griddepcontrol.wait;" ::: "memory");
        asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    }
    // the variable's own state first: independent of the couplings, in flight during the gathers
    float s[V], y[V], b = 0.0f, a_k = 0.0f;
    if constexpr (!FIELD_ONLY) {
        vload<V, DEP>(S_cur + me, s);
        vload_stream<V>(Y_in + me, y);
        b = __ldg(bf + i);
        a_k = __ldg(a_table + k);
    }
    float acc[V];
    vqd::csr_row_dot<V, WT, UNROLL, SIGN, false, DEP>(rp, col, w, S_cur, R, off, i, acc, udeg);
    float F[V];
#pragma unroll
    for (int l = 0; l < V; ++l) F[l] = acc[l] * wscale;     // wscale is 1 or 1/2: exact
    if (F_out) vstore<V>(F_out + me, F);
    if constexpr (FIELD_ONLY) return;
    if (method == vqd::METHOD_BSB) {
#pragma unroll
        for (int l = 0; l < V; ++l) vqd::bsb_update(F[l], b, a_k, dt, a0, c0, s[l], y[l]);
    } else {
        const float lam = vqd::pa_lambda(a_k, a0);
#pragma unroll
        for (int l = 0; l < V; ++l) vqd::step_update(method, F[l], b, a_k, lam, dt, a0, c0, alpha, s[l], y[l]);
    }
    vstore_stream<V>(S_nxt + me, s);
    vstore_stream<V>(Y_out + me, y);
}

__device__ __forceinline__ int64_t ewval(int8_t w) { return (int64_t)w; }
__device__ __forceinline__ int64_t ewval(int64_t w) { return w; }

// Exact readout energy, fixed point: parts[g][r] = sum over the rows of group
// g of x_ri (dfix_i + sum_j wE_ij x_rj), x = [s > 0]. Block (TX, TY): TX
// vectors of replicas, TY rows; rows of a group are grid-strided.
template <int V, typename EW>
__global__ void __launch_bounds__(256) k_stream_energy(int64_t n, int32_t R, int32_t nvec, const int64_t* __restrict__ rp,
                                                       const int32_t* __restrict__ col, const EW* __restrict__ we,
                                                       const int64_t* __restrict__ dfix, const float* __restrict__ S,
                                                       int64_t* __restrict__ parts) {
    extern __shared__ int64_t sh[];
    const int TX = blockDim.x, TY = blockDim.y;
    const int32_t v = blockIdx.x * TX + threadIdx.x;
    int64_t part[V];
#pragma unroll
    for (int l = 0; l < V; ++l) part[l] = 0;
    if (v < nvec) {
        const int64_t off = (int64_t)v * V;
        for (int64_t i = (int64_t)blockIdx.y * TY + threadIdx.y; i < n; i += (int64_t)gridDim.y * TY) {
            float si[V];
            vload<V>(S + i * R + off, si);
            bool any = false;
#pragma unroll
            for (int l = 0; l < V; ++l) any |= si[l] > 0.0f;
            if (!any) continue;
            int64_t row[V];
#pragma unroll
            for (int l = 0; l < V; ++l) row[l] = 0;
            const int64_t p1 = __ldg(rp + i + 1);
            for (int64_t p = __ldg(rp + i); p < p1; ++p) {
                const int64_t j = __ldg(col + p);
                const int64_t wq = ewval(__ldg(we + p));
                float sj[V];
                vload<V>(S + j * R + off, sj);
#pragma unroll
                for (int l = 0; l < V; ++l) row[l] += sj[l] > 0.0f ? wq : 0;
            }
            const int64_t d = __ldg(dfix + i);
#pragma unroll
            for (int l = 0; l < V; ++l) part[l] += si[l] > 0.0f ? d + row[l] : 0;
        }
    }
    // reduce over TY in a fixed order
#pragma unroll
    for (int l = 0; l < V; ++l) sh[((int64_t)threadIdx.y * TX + threadIdx.x) * V + l] = part[l];
    __syncthreads();
    if (threadIdx.y == 0 && v < nvec) {
#pragma unroll
        for (int l = 0; l < V; ++l) {
            int64_t tot = 0;
            for (int y = 0; y < TY; ++y) tot += sh[((int64_t)y * TX + threadIdx.x) * V + l];
            const int32_t r = v * V + l;
            if (r < R) parts[(int64_t)blockIdx.y * R + r] = tot;
        }
    }
}

// Energy of a caller batch X [B][n] (uint8): parts[g][b].
template <typename EW>
__global__ void __launch_bounds__(256) k_sparse_energy_x(int64_t n, int64_t B, const int64_t* __restrict__ rp,
                                                         const int32_t* __restrict__ col, const EW* __restrict__ we,
                                                         const int64_t* __restrict__ dfix, const uint8_t* __restrict__ X,
                                                         int64_t* __restrict__ parts) {
    __shared__ int64_t sh[256];
    const int64_t b = blockIdx.y;
    const uint8_t* x = X + b * n;
    int64_t part = 0;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        if (!x[i]) continue;
        int64_t row = __ldg(dfix + i);
        const int64_t p1 = __ldg(rp + i + 1);
        for (int64_t p = __ldg(rp + i); p < p1; ++p)
            if (x[__ldg(col + p)]) row += ewval(__ldg(we + p));
        part += row;
    }
    sh[threadIdx.x] = part;
    __syncthreads();
    for (int s = blockDim.x / 2; s > 0; s >>= 1) {
        if (threadIdx.x < s) sh[threadIdx.x] += sh[threadIdx.x + s];
        __syncthreads();
    }
    if (threadIdx.x == 0) parts[(int64_t)blockIdx.x * B + b] = sh[0];
}

// The same for 32 vectors per block, a lane each: the block first packs the
// vectors' bits of variable j into word j in shared memory, then every warp
// takes rows, reads a coupling once for all 32 vectors and tests the
// neighbour's word. Bound by instruction issue (about five per coupling for
// 32 vectors); the form above reads every coupling and a byte per vector, with
// 64 groups of rows whatever n is.
constexpr int kPackVectors = 32;
template <typename EW>
__global__ void __launch_bounds__(256) k_sparse_energy_packed(int64_t n, int64_t B, const int64_t* __restrict__ rp,
                                                              const int32_t* __restrict__ col,
                                                              const EW* __restrict__ we,
                                                              const int64_t* __restrict__ dfix,
                                                              const uint8_t* __restrict__ X,
                                                              int64_t* __restrict__ parts) {
    extern __shared__ __align__(16) uint32_t words[];   // [n]
    __shared__ int64_t red[8][kPackVectors];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t b0 = (int64_t)blockIdx.y * kPackVectors;
    const int nb = (int)min((int64_t)kPackVectors, B - b0);
    const uint8_t* x0 = X + b0 * n;
    if (nb == kPackVectors && (n & 3) == 0 && (reinterpret_cast<uintptr_t>(x0) & 3) == 0) {
        // four variables per thread, the 32 vectors' loads in flight together
        for (int64_t j = 4 * threadIdx.x; j < n; j += 4 * 256) {
            uint32_t q[kPackVectors], w[4] = {0, 0, 0, 0};
#pragma unroll
            for (int v = 0; v < kPackVectors; ++v) q[v] = __ldg(reinterpret_cast<const uint32_t*>(x0 + (int64_t)v * n + j));
#pragma unroll
            for (int v = 0; v < kPackVectors; ++v)
#pragma unroll
                for (int u = 0; u < 4; ++u) w[u] |= (uint32_t)((q[v] & (0xffu << (8 * u))) != 0) << v;
            *reinterpret_cast<uint4*>(words + j) = make_uint4(w[0], w[1], w[2], w[3]);
        }
    } else {
        for (int64_t j = threadIdx.x; j < n; j += 256) {
            uint32_t w = 0;
            for (int v = 0; v < nb; ++v) w |= (uint32_t)(__ldg(x0 + (int64_t)v * n + j) != 0) << v;
            words[j] = w;
        }
    }
    __syncthreads();
    int64_t part = 0;
    for (int64_t i = (int64_t)blockIdx.x * 8 + warp; i < n; i += (int64_t)gridDim.x * 8) {
        const uint32_t wi = words[i];
        if (wi == 0) continue;
        int64_t row = __ldg(dfix + i);
        const int64_t p1 = __ldg(rp + i + 1);
        int64_t p = __ldg(rp + i);
        for (; p + 4 <= p1; p += 4) {
            int32_t c[4];
            EW w[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                c[u] = __ldg(col + p + u);
                w[u] = __ldg(we + p + u);
            }
#pragma unroll
            for (int u = 0; u < 4; ++u) row += ((words[c[u]] >> lane) & 1u) ? ewval(w[u]) : 0;
        }
        for (; p < p1; ++p) row += ((words[__ldg(col + p)] >> lane) & 1u) ? ewval(__ldg(we + p)) : 0;
        part += ((wi >> lane) & 1u) ? row : 0;
    }
    red[warp][lane] = part;
    __syncthreads();
    if (warp == 0 && lane < nb) {
        int64_t tot = 0;
#pragma unroll
        for (int w = 0; w < 8; ++w) tot += red[w][lane];
        parts[(int64_t)blockIdx.x * B + b0 + lane] = tot;
    }
}

template <bool FIELD_ONLY, bool SIGN>
int launch_step(veloxq_ctx* ctx, int32_t R, const float* S_cur, float* S_nxt, const float* Y_in, float* Y_out,
                const float* a_table, int k, float dt, float a0, float c0, float* F_out, const Rule& rule,
                int32_t r0 = 0, int32_t rn = 0) {
    const int V = vec_width(R);
    const int32_t nvec = (rn ? rn : R) / V;
    // a window of replicas: the same rows, from its first replica on
    S_cur += r0;
    if (S_nxt) S_nxt += r0;
    if (Y_in) Y_in += r0;
    if (Y_out) Y_out += r0;
    if (F_out) F_out += r0;
    const int32_t cvec = (!rn && ctx->stream_cvec > 0 && nvec % ctx->stream_cvec == 0) ? ctx->stream_cvec : nvec;
    const int64_t total = ctx->n * (int64_t)nvec;
    const unsigned g = (unsigned)div_up(total, 256);
    // Short steps are launched dependently, so that a step's launch and first
    // blocks overlap the last ones of the step before. Plain -> dependent, us
    // per step, by threads per step: tile planting L = 100 0.16 / 1.28 M 3.3 ->
    // 2.6 / 12.6 -> 12.1; lattice L = 40 0.26 / 1.28 / 1.54 / 3.1 M 4.0 -> 3.8 /
    // 12.0 -> 11.5 / 14.0 -> 14.2 / 36.4 -> 37.1; 3R3X (2e4 variables) 0.64 /
    // 1.28 / 2.6 M 9.3 -> 8.9 / 16.5 -> 16.6 / 40.0 -> 42.8; Pegasus P_16 1.44 /
    // 2.9 M 27.7 -> 27.2 / 63.4 -> 60.7; the longest steps lose (3R3X at 256
    // replicas 237 -> 248, lattice L = 100 677 -> 715: blocks of two steps
    // share L2), most from 1.5 M threads on.
    // Rows of unequal length of many variables with few replicas lose at any
    // size: 3-body chain (2e5 variables) at 1 / 16 replicas 3.3 -> 3.7 / 10.9
    // -> 11.4, 3R3X (2e5) at 4 8.3 -> 9.4, Zephyr Z_40 (51840) at 16 8.9 -> 9.4;
    // with 2e4 variables or 64 replicas they gain (chain 4.3 -> 3.6, Pegasus
    // P_30 at 16 4.6 -> 4.1, Z_40 at 64 20.7 -> 19.9).
    // A field alone has no step before it to overlap.
    const bool scattered = ctx->uniform_deg < 0 && ctx->n > 40000 && nvec <= 4;
    const bool dependent = !FIELD_ONLY && total <= 1500000 && !scattered;
    const int64_t* rp = ctx->rowptr.as<int64_t>();
    const int32_t* cl = ctx->col.as<int32_t>();
    const float* bf = ctx->bf.as<float>();
    cudaStream_t st = ctx->stream;
#define VQ_STEP_D(VV, WT, WPTR, SC, U, D)                                                                             \
    VQ_CUDA(launch_dependent(D, k_stream_step<VV, WT, FIELD_ONLY, U, SIGN, D>, dim3(g), dim3(256), 0, st, ctx->n, R, nvec, \
                             rp, cl, WPTR, SC, S_cur, S_nxt, Y_in, Y_out, bf, a_table, k, dt, a0, c0, F_out,           \
                             ctx->uniform_deg, rule.method, rule.alpha, cvec))
#define VQ_STEP_U(VV, WT, WPTR, SC, U)                                       \
    do {                                                                     \
        if constexpr (!FIELD_ONLY) {                                         \
            if (dependent) { VQ_STEP_D(VV, WT, WPTR, SC, U, true); break; }  \
        }                                                                    \
        VQ_STEP_D(VV, WT, WPTR, SC, U, false);                               \
    } while (0)
#define VQ_STEP(VV, WT, WPTR, SC)                                   \
    do {                                                            \
        if (unroll == 6) VQ_STEP_U(VV, WT, WPTR, SC, 6);            \
        else if (unroll == 4) VQ_STEP_U(VV, WT, WPTR, SC, 4);       \
        else VQ_STEP_U(VV, WT, WPTR, SC, 1);                        \
    } while (0)
    // without a timing trial (single steps and fields): six at once on rows of exactly six couplings, where it is
    // the form every trial picks (cubic lattice L = 100, 256 replicas: 0.70 ms against 0.80 one at a time)
    const int form = rn ? ctx->stream_wunroll : ctx->stream_unroll;
    const bool six = ctx->uniform_deg == 6 && (form == 6 || form == 0);
    const int unroll = six ? 6 : form == 4 ? 4 : 1;
    if (ctx->w8.p) {
        const int8_t* w = ctx->w8.as<int8_t>();
        if (V == 4) VQ_STEP(4, int8_t, w, 0.5f); else if (V == 2) VQ_STEP(2, int8_t, w, 0.5f); else VQ_STEP(1, int8_t, w, 0.5f);
    } else {
        const float* w = ctx->wf.as<float>();
        if (V == 4) VQ_STEP(4, float, w, 1.0f); else if (V == 2) VQ_STEP(2, float, w, 1.0f); else VQ_STEP(1, float, w, 1.0f);
    }
#undef VQ_STEP
#undef VQ_STEP_U
#undef VQ_STEP_D
    VQ_LAUNCH_CHECK("stream_step");
    return VELOXQ_OK;
}

}  // namespace

int vec_width(int32_t R) { return (R % 4 == 0) ? 4 : (R % 2 == 0) ? 2 : 1; }

int stream_step(veloxq_ctx* ctx, int32_t R, const float* S_cur, float* S_nxt, float* Y, const float* a_table, int k,
                float dt, float a0, float c0, float* F_out, const Rule& rule, int32_t r0, int32_t rn) {
    if (rule.method == VELOXQ_METHOD_PA)
        return launch_step<false, true>(ctx, R, S_cur, S_nxt, Y, Y, a_table, k, dt, a0, c0, F_out, rule, r0, rn);
    return launch_step<false, false>(ctx, R, S_cur, S_nxt, Y, Y, a_table, k, dt, a0, c0, F_out, rule, r0, rn);
}

// Replicas per window of a run of steps (0: all at once). Replicas are
// independent, so the steps between two readouts may run for one window of
// replicas after the other. When the state of all replicas lies well beyond
// L2 but a window's two state arrays and momenta stay in it with the
// couplings, every step after a window's first reads and writes L2 instead
// of HBM. The widest window of at most 96 MB is taken (L2 holds 126 MB; tile
// planting L = 300 at 256 replicas, 65.6 us all at once: windows of 35 / 69 /
// 138 MB 63.2 / 59.2 / 72.2 us; 3R3X of 3e5 variables, window 127 MB: 377
// either way), of at least 32 replicas (one 128-byte line per row) and 2.5 M
// variable-replicas (shorter steps cost more in launches than they save:
// lattices of 1.6 / 2.4 / 3.1 M per window 51.5 -> 56.7, 72.5 -> 73.6, 61.6 ->
// 56.8 us; random graphs would gain below too, 3R3X 1.9 M 95 -> 83).
int32_t stream_window(const veloxq_ctx* ctx, int32_t R, int steps) {
    const double l2 = 126e6, room = 96e6;
    const double couplings = (double)ctx->nnz * (ctx->w8.p ? 5.0 : 8.0) + 12.0 * (double)ctx->n;
    if (steps < 4 || 12.0 * (double)ctx->n * R + couplings <= 1.5 * l2) return 0;
    for (int32_t parts = 2; R / parts >= 32; ++parts) {
        const int32_t w = R / parts;
        if (R % parts != 0 || w % 32 != 0) continue;
        if (12.0 * (double)ctx->n * w + couplings > room) continue;
        return (double)ctx->n * w >= 2.5e6 ? w : 0;
    }
    return 0;
}

int stream_step_y(veloxq_ctx* ctx, int32_t R, const float* S_cur, float* S_nxt, const float* Y_in, float* Y_out,
                  const float* a_table, int k, float dt, float a0, float c0, float* F_out, const Rule& rule) {
    if (rule.method == VELOXQ_METHOD_PA)
        return launch_step<false, true>(ctx, R, S_cur, S_nxt, Y_in, Y_out, a_table, k, dt, a0, c0, F_out, rule);
    return launch_step<false, false>(ctx, R, S_cur, S_nxt, Y_in, Y_out, a_table, k, dt, a0, c0, F_out, rule);
}

int stream_field(veloxq_ctx* ctx, int32_t R, const float* S, float* F) {
    return launch_step<true, false>(ctx, R, S, nullptr, nullptr, nullptr, nullptr, 0, 0.f, 0.f, 0.f, F, Rule());
}

// Chunk widths (replica vectors) worth trying for R replicas: when one state
// array is larger than about half of L2, the widths whose chunk of every row
// (n x width x V floats) fits in 64 MB, at least 32 replicas (one 128-byte
// line per row) and dividing the vectors of a row; 0 (no chunking) always.
static std::vector<int32_t> chunk_candidates(int64_t n, int32_t R) {
    const int V = vec_width(R);
    const int32_t nvec = R / V;
    const int64_t budget = int64_t(64) << 20;
    std::vector<int32_t> out = {0};
    if (n * (int64_t)R * 4 <= budget) return out;
    int32_t widest = 0;
    for (int32_t cv = nvec / 2; cv * V >= 32; --cv)
        if (nvec % cv == 0 && n * (int64_t)cv * V * 4 <= budget) {
            widest = cv;
            break;
        }
    if (widest) {
        out.push_back(widest);
        for (int32_t cv = widest / 2; cv * V >= 32; --cv)
            if (nvec % cv == 0) {
                out.push_back(cv);
                break;
            }
    }
    return out;
}

// Pick the gather variant (one, four or six couplings at a time) and the
// replica chunk width of the streaming kernels for R replicas by timing steps
// of each pair on the caller's buffers (contents are overwritten);
// VELOXQ_STREAM_FORM fixes them instead. windows: for runs by windows of
// replicas, whose gather is picked on steps of one window; steps over all
// replicas (the caller's own steps on this context) then keep this gather with
// the chunk width that suits them, until a call that runs such steps itself
// tries every pair.
// Runs eagerly on ctx->stream; must not be called during stream capture.
int stream_autotune(veloxq_ctx* ctx, int32_t R, float* S_a, float* S_b, float* Y, bool windows) {
    if ((windows ? ctx->stream_wtuned_R : ctx->stream_tuned_R) == R) return VELOXQ_OK;
    if (const char* form = std::getenv("VELOXQ_STREAM_FORM")) {
        // a form fixed by the caller: "gather chunk", the chunk in replicas (0: all at once)
        const int V = vec_width(R);
        const int32_t nvec = R / V;
        int u = 0, cr = -1;
        const bool parsed = std::sscanf(form, "%d %d", &u, &cr) == 2 && cr >= 0 && cr % V == 0;
        const int32_t cv = parsed ? cr / V : -1;
        const bool ok = parsed && (u == 1 || u == 4 || (u == 6 && ctx->uniform_deg == 6)) &&
                        (cv == 0 || nvec % cv == 0);
        if (!ok)
            return fail(VELOXQ_EINVAL, "VELOXQ_STREAM_FORM must be \"gather chunk\": gather 1, 4 or 6 (rows of exactly "
                                       "6 couplings) and a chunk of replicas (0: all) that the replica count splits "
                                       "into");
        ctx->stream_unroll = ctx->stream_wunroll = u;
        ctx->stream_cvec = cv;
        ctx->stream_tuned_R = ctx->stream_wtuned_R = R;
        return VELOXQ_OK;
    }
    cudaEvent_t e0, e1;
    VQ_CUDA(cudaEventCreate(&e0));
    VQ_CUDA(cudaEventCreate(&e1));
    VQ_TRY(launch_init_state(ctx, R, 1, 0.1f, LAYOUT_NR, S_a, Y));
    const float* at = ctx->a_table.as<float>();
    const int32_t win = windows ? stream_window(ctx, R, 50) : 0;
    auto timed = [&](int reps, int32_t rn, float* ms) -> int {
        VQ_CUDA(cudaEventRecord(e0, ctx->stream));
        for (int k = 0; k < reps; ++k)
            VQ_TRY((launch_step<false, false>(ctx, R, (k & 1) ? S_b : S_a, (k & 1) ? S_a : S_b, Y, Y, at, 0, 0.5f,
                                              1.0f, 0.1f, nullptr, Rule(), 0, rn)));
        VQ_CUDA(cudaEventRecord(e1, ctx->stream));
        VQ_CUDA(cudaEventSynchronize(e1));
        VQ_CUDA(cudaEventElapsedTime(ms, e0, e1));
        return VELOXQ_OK;
    };
    // Two rounds over all candidates (gather, chunk), each timing `reps` steps of one form
    // (`most`, 10 for the call's own steps, when a step is shorter than 0.3 ms, else at most 3); a form's time is its
    // faster round, so a round disturbed by the previous form's state in L2
    // or by a clock change does not decide the pick.
    auto pick = [&](const std::vector<std::pair<int, int32_t>>& cands, int32_t rn, int most, size_t* best) -> int {
        std::vector<float> per_step(cands.size(), 1e30f);
        int reps = std::min(3, most);
        for (int round = 0; round < 2; ++round)
            for (size_t c = 0; c < cands.size(); ++c) {
                ctx->stream_unroll = ctx->stream_wunroll = cands[c].first;
                ctx->stream_cvec = cands[c].second;
                float ms = 0.f;
                if (round == 0) {
                    VQ_TRY(timed(1, rn, &ms));             // warm; the first form's step sets the step count
                    if (c == 0 && ms < 0.3f) reps = most;
                }
                VQ_TRY(timed(reps, rn, &ms));
                per_step[c] = std::min(per_step[c], ms / (float)reps);
            }
        *best = 0;
        for (size_t c = 1; c < cands.size(); ++c)
            if (per_step[c] < per_step[*best]) *best = c;
        return VELOXQ_OK;
    };
    const int keep_u = ctx->stream_unroll, keep_w = ctx->stream_wunroll;
    const int32_t keep_cv = ctx->stream_cvec;
    std::vector<std::pair<int, int32_t>> cands;
    for (int32_t cv : win ? std::vector<int32_t>{0} : chunk_candidates(ctx->n, R))
        for (int u : {1, 4, 6})
            if (u != 6 || ctx->uniform_deg == 6) cands.emplace_back(u, cv);
    size_t bi = 0;
    VQ_TRY(pick(cands, win, 10, &bi));
    const int u = cands[bi].first;
    if (!windows) {
        ctx->stream_unroll = u;
        ctx->stream_cvec = cands[bi].second;
        ctx->stream_tuned_R = R;
        ctx->stream_wunroll = keep_w;
    } else if (ctx->stream_tuned_R == R) {
        ctx->stream_unroll = keep_u;
        ctx->stream_cvec = keep_cv;
    } else {
        const std::vector<int32_t> chunks = chunk_candidates(ctx->n, R);
        std::vector<std::pair<int, int32_t>> whole;
        for (int32_t cv : chunks) whole.emplace_back(u, cv);
        bi = 0;
        if (whole.size() > 1) VQ_TRY(pick(whole, 0, 1, &bi));   // no steps of this call: one each
        ctx->stream_unroll = u;
        ctx->stream_cvec = whole[bi].second;
        ctx->stream_tuned_R = -1;
    }
    if (windows) {
        ctx->stream_wunroll = u;
        ctx->stream_wtuned_R = R;
    }
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    return VELOXQ_OK;
}

// number of row groups (partial sums) used by stream_energy
static int energy_groups(int32_t gx) { return std::max(1, 608 / std::max(1, gx)); }

int stream_energy(veloxq_ctx* ctx, int32_t R, const float* S, int64_t* parts, int* nparts) {
    const int V = vec_width(R);
    const int32_t nvec = R / V;
    int TX = 1;
    while (TX < nvec && TX < 32) TX <<= 1;
    const int TY = 256 / TX;
    const int32_t gx = (int32_t)div_up(nvec, TX);
    const int gy = energy_groups(gx);
    *nparts = gy;
    dim3 blk(TX, TY), grd(gx, gy);
    const size_t sm = sizeof(int64_t) * 256 * V;
    cudaStream_t st = ctx->stream;
    const int64_t* rp = ctx->rowptr.as<int64_t>();
    const int32_t* cl = ctx->col.as<int32_t>();
    const int64_t* df = ctx->dfix.as<int64_t>();
#define VQ_EN(VV, EW, WPTR) k_stream_energy<VV, EW><<<grd, blk, sm, st>>>(ctx->n, R, nvec, rp, cl, WPTR, df, S, parts)
    if (ctx->w8.p) {
        const int8_t* w = ctx->w8.as<int8_t>();
        if (V == 4) VQ_EN(4, int8_t, w); else if (V == 2) VQ_EN(2, int8_t, w); else VQ_EN(1, int8_t, w);
    } else {
        const int64_t* w = ctx->wfix.as<int64_t>();
        if (V == 4) VQ_EN(4, int64_t, w); else if (V == 2) VQ_EN(2, int64_t, w); else VQ_EN(1, int64_t, w);
    }
#undef VQ_EN
    VQ_LAUNCH_CHECK("stream_energy");
    return VELOXQ_OK;
}

int stream_energy_parts(int32_t R) {
    const int V = vec_width(R);
    const int32_t nvec = R / V;
    int TX = 1;
    while (TX < nvec && TX < 32) TX <<= 1;
    return energy_groups((int32_t)div_up(nvec, TX));
}

int sparse_energy_x(veloxq_ctx* ctx, int64_t B, const uint8_t* X, int64_t* parts, int* nparts) {
    *nparts = 64;
    if (B == 0) return VELOXQ_OK;
    // Packed words where their packing pays (about 4.5 ns per variable) and they fit the 48 KB a block has without
    // asking. Measured, bytes -> words, us: Chimera C_16, 64 / 1024 / 4096 vectors 20 -> 18, 83 -> 32, 288 -> 70;
    // Pegasus P_16, 16 / 256 / 4096 vectors 22 -> 42, 58 -> 52, 671 -> 286.
    if (B >= 64 && 24 * B >= ctx->n && ctx->n <= 11264) {
        const int64_t batches = div_up(B, kPackVectors);
        // row groups: four blocks per SM in all, at least 64 rows each, at most the 64 groups the scratch holds
        const int G = (int)std::max<int64_t>(
            1, std::min<int64_t>({64, div_up(ctx->n, 64), div_up(4 * (int64_t)device_sms(ctx->device), batches)}));
        *nparts = G;
        const size_t sm = sizeof(uint32_t) * (size_t)ctx->n;
        const dim3 g((unsigned)G, (unsigned)batches);
        if (ctx->w8.p)
            k_sparse_energy_packed<int8_t><<<g, 256, sm, ctx->stream>>>(
                ctx->n, B, ctx->rowptr.as<int64_t>(), ctx->col.as<int32_t>(), ctx->w8.as<int8_t>(),
                ctx->dfix.as<int64_t>(), X, parts);
        else
            k_sparse_energy_packed<int64_t><<<g, 256, sm, ctx->stream>>>(
                ctx->n, B, ctx->rowptr.as<int64_t>(), ctx->col.as<int32_t>(), ctx->wfix.as<int64_t>(),
                ctx->dfix.as<int64_t>(), X, parts);
        VQ_LAUNCH_CHECK("sparse_energy_x");
        return VELOXQ_OK;
    }
    const int G = 64;
    dim3 grd(G, (unsigned)B);
    if (ctx->w8.p)
        k_sparse_energy_x<int8_t><<<grd, 256, 0, ctx->stream>>>(ctx->n, B, ctx->rowptr.as<int64_t>(), ctx->col.as<int32_t>(),
                                                                ctx->w8.as<int8_t>(), ctx->dfix.as<int64_t>(), X, parts);
    else
        k_sparse_energy_x<int64_t><<<grd, 256, 0, ctx->stream>>>(ctx->n, B, ctx->rowptr.as<int64_t>(), ctx->col.as<int32_t>(),
                                                                 ctx->wfix.as<int64_t>(), ctx->dfix.as<int64_t>(), X, parts);
    VQ_LAUNCH_CHECK("sparse_energy_x");
    return VELOXQ_OK;
}

}  // namespace vq
