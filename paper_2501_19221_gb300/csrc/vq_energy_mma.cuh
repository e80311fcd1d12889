// vq_energy_mma.cuh -- one 64-row tile of the exact energy of a
// dense instance, x^T q x + d^T x in 64-bit fixed point, as tensor-core
// products of exact digits (the block body of k_dense_energy and
// k_batch_energy).
//
// The fixed-point couplings q_ij = round(Q_ij 2^S) are written in balanced
// base-4096 digits, q = sum_k 4096^k t_k with t_k in [-2048, 2048], which FP16
// holds exactly. A block stages 64 rows x 64 columns of Q at a time, extracts
// one digit plane after the other into shared memory (only as many as the
// tile's largest |q| needs: one for small integers, four for Gaussian FP32
// couplings) and multiplies it with the 0/1 matrix of its replicas
// (m16n8k16, FP32 accumulation). Every product is an integer and every
// partial sum is at most 2048 * 64 = 2^17 in magnitude per stage (the lowest
// digit's accumulators are kept over 32 stages, 2^22), so FP32 accumulation is
// exact. The accumulators are then masked by x_ri, taken as integers and
// added, shifted by 12 k, into 64-bit totals modulo 2^64, which is exact
// because the finished energy lies in range.
//
// What bounds it: latency, not memory and not a pipe. One block of 16 warps
// fits per SM (124 registers for 512 threads): four warps per scheduler, which
// issue in 44 % of the cycles (n = 2048, 1024 vectors, int32 couplings; the
// tensor pipe 10 %) and otherwise wait on fixed latencies, the loads of the
// next stage, the fragments from shared memory and the barrier behind every
// digit plane; the 256 blocks are 1.7 waves on 152 SMs. Every block of 128
// vectors cuts its tile of Q into digits anew. The previous form selected and
// added int64 couplings on the CUDA cores, four instructions per coupling and
// replica; here a coupling costs a few per digit for all replicas of the
// tile. Measured at n = 2048, 1024 vectors: int32 and int8 couplings (one
// digit) 957 -> 136 us, FP32 couplings 279 us; the readout of 256 Wishart instances (n 100 to 2000, 64 replicas, FP32
// couplings, four digits): 12.3 -> 2.3 ms. The products go through mma.sync
// because a tile's digits are cut in registers and go to shared memory at
// once: tcgen05 would take 256 x 128 tiles, hence planes kept in memory, and
// this kernel serves calls that must not allocate (veloxq_energy_dev and its
// no-allocation form).
#pragma once

#include <cuda_fp16.h>

#include <type_traits>

#include "vq_internal.cuh"

namespace vq {
namespace emma {

constexpr int TI = 64;             // rows of Q per tile (one parts entry per tile)
constexpr int TK = 64;             // columns of Q per stage
constexpr int LD = TK + 8;         // halves per shared row: 144 bytes, conflict-free for ldmatrix
constexpr int FLUSH = 32;          // stages whose lowest digit sums stay below 2^22 in FP32

// Replicas per tile: 128 (the staged couplings serve twice the replicas),
// or 64 when there are no more; four threads per replica either way.
constexpr int TR_WIDE = 128, TR_NARROW = 64;
inline int tile_replicas(int64_t R) { return R > TR_NARROW ? TR_WIDE : TR_NARROW; }

template <int TR> struct Smem {
    __align__(16) __half a[2][TI][LD];       // digit planes (two, used in turn)
    __align__(16) __half b[TR][LD];          // x of the replicas
    __align__(16) uint32_t digits[2][TR / 8];   // digits each warp's couplings need (two stages, used in turn)
    unsigned long long red[4][TR];
};

__device__ __forceinline__ void ldsm4(uint32_t (&r)[4], const void* p) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0, %1, %2, %3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                 : "r"((uint32_t)__cvta_generic_to_shared(p)));
}
__device__ __forceinline__ void mma16816(float (&d)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, "
        "{%0, %1, %2, %3};"
        : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

// Two adjacent elements; `pair`: they may be loaded as one vector.
template <typename T> struct Pair {
    T v[2];
};
template <typename T>
__device__ __forceinline__ Pair<T> load_pair(const T* p, bool pair) {
    Pair<T> o;
    if (pair) {
        using V = std::conditional_t<sizeof(T) == 1, uint16_t, std::conditional_t<sizeof(T) == 4, uint2, uint4>>;
        const V w = __ldg(reinterpret_cast<const V*>(p));
        memcpy(&o, &w, sizeof(o));
    } else {
        o.v[0] = __ldg(p);
        o.v[1] = __ldg(p + 1);
    }
    return o;
}

// x of an element: [S > 0] or [X != 0]
__device__ __forceinline__ bool is_on(float s) { return s > 0.0f; }
__device__ __forceinline__ bool is_on(uint8_t x) { return x != 0; }

// A word that grows with |q| (sums by max over elements), and from its
// maximum m a bound b with |round(q 2^shift)| < 2^b.
__device__ __forceinline__ uint32_t mag(int8_t q) { return (uint32_t)abs((int)q); }
__device__ __forceinline__ uint32_t mag(int32_t q) { return q < 0 ? 0u - (uint32_t)q : (uint32_t)q; }
__device__ __forceinline__ uint32_t mag(float q) { return __float_as_uint(q) & 0x7fffffffu; }
__device__ __forceinline__ uint32_t mag(double q) { return (uint32_t)__double2hiint(q) & 0x7fffffffu; }
template <typename QT> __device__ __forceinline__ int bits_of(uint32_t m, int shift) {
    if constexpr (std::is_same<QT, float>::value) return m ? (int)(m >> 23) - 126 + shift + 1 : 0;
    else if constexpr (std::is_same<QT, double>::value) return m ? (int)(m >> 20) - 1022 + shift + 1 : 0;
    else return m ? 32 - __clz((int)m) + shift : 0;
}

// parts_row[r] for the TR replicas from r0 on: sum over the rows i of the
// tile [i0, i0 + 64) of x_ri (dfix_i + sum_{j != i} q_ij x_rj). XT: float
// (state) or uint8_t (vectors), replica-major [R][n]. Called by all 4 TR
// threads of the block.
template <int TR, typename QT, typename XT>
__device__ __forceinline__ void energy_tile(Smem<TR>& sm, int64_t R, int32_t n, const QT* __restrict__ Q, int shift,
                                            const int64_t* __restrict__ dfix, const XT* __restrict__ x, int64_t i0,
                                            int64_t r0, int64_t* __restrict__ parts_row) {
    constexpr int WARPS = TR / 8, EQ = TI / WARPS, EX = TR / WARPS;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int wm = warp & 3, wn = warp >> 2;          // warp tile: 16 rows x 32 replicas
    const int gq = lane >> 2, tq = lane & 3;
    // vector loads of two elements need even rows and aligned bases
    const bool qpair = (n & 1) == 0 && (reinterpret_cast<uintptr_t>(Q) & (2 * sizeof(QT) - 1)) == 0;
    const bool xpair = (n & 1) == 0 && (reinterpret_cast<uintptr_t>(x) & (2 * sizeof(XT) - 1)) == 0;
    const bool rows_in = i0 + TI <= n, reps_in = r0 + TR <= R;

    // staging: a warp takes row (or replica) warp + WARPS e, a lane two adjacent columns
    Pair<QT> raw[EQ];
    Pair<XT> xr[EX];
    auto load = [&](int32_t j0) {
        const int32_t j = j0 + 2 * lane;
        const QT* qp = Q + (i0 + warp) * n + j;
        const XT* xp = x + (r0 + warp) * n + j;
        const bool cols_in = j0 + TK <= n;
        if (cols_in && rows_in) {
#pragma unroll
            for (int e = 0; e < EQ; ++e) raw[e] = load_pair(qp + (int64_t)e * WARPS * n, qpair);
        } else {
#pragma unroll
            for (int e = 0; e < EQ; ++e)
#pragma unroll
                for (int h = 0; h < 2; ++h)
                    raw[e].v[h] = (i0 + warp + WARPS * e < n && j + h < n) ? __ldg(qp + (int64_t)e * WARPS * n + h)
                                                                           : QT(0);
        }
        if (cols_in && reps_in) {
#pragma unroll
            for (int e = 0; e < EX; ++e) xr[e] = load_pair(xp + (int64_t)e * WARPS * n, xpair);
        } else {
#pragma unroll
            for (int e = 0; e < EX; ++e)
#pragma unroll
                for (int h = 0; h < 2; ++h)
                    xr[e].v[h] = (r0 + warp + WARPS * e < R && j + h < n) ? __ldg(xp + (int64_t)e * WARPS * n + h)
                                                                          : XT(0);
        }
        if (j0 == i0) {                                // the tile's own columns: no diagonal
#pragma unroll
            for (int e = 0; e < EQ; ++e)
#pragma unroll
                for (int h = 0; h < 2; ++h)
                    if (warp + WARPS * e == 2 * lane + h) raw[e].v[h] = QT(0);
        }
    };

    load(0);
    // this thread's accumulator elements: rows gq, gq + 8 of the warp's 16,
    // replicas 2 tq, 2 tq + 1 of each of the four groups of 8
    uint32_t mask = 0;
    unsigned long long tot[4][2];
#pragma unroll
    for (int c = 0; c < 4; ++c)
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int64_t r = r0 + wn * 32 + c * 8 + 2 * tq + h;
            unsigned long long t = 0;
#pragma unroll
            for (int v = 0; v < 2; ++v) {
                const int64_t i = i0 + wm * 16 + gq + 8 * v;
                const bool on = i < n && r < R && is_on(__ldg(x + r * n + i));
                mask |= (uint32_t)on << (c * 4 + v * 2 + h);
                if (on) t += (unsigned long long)__ldg(dfix + i);
            }
            tot[c][h] = t;
        }
    // the kept elements of an accumulator, as integers, into the totals:
    // acc + 1.5 * 2^23 holds the integer in its low bits
    auto add = [&](const float (&acc)[4][4], int sh) {
#pragma unroll
        for (int c = 0; c < 4; ++c)
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                int s = 0;
#pragma unroll
                for (int v = 0; v < 2; ++v) {
                    const int g = __float_as_int(acc[c][v * 2 + h] + 12582912.0f) - 0x4B400000;
                    s += ((mask >> (c * 4 + v * 2 + h)) & 1u) ? g : 0;
                }
                tot[c][h] += (unsigned long long)(long long)s << sh;
            }
    };
    auto zero = [](float (&acc)[4][4]) {
#pragma unroll
        for (int c = 0; c < 4; ++c)
#pragma unroll
            for (int v = 0; v < 4; ++v) acc[c][v] = 0.0f;
    };
    auto product = [&](int buf, float (&acc)[4][4]) {
#pragma unroll
        for (int kk = 0; kk < TK / 16; ++kk) {
            uint32_t af[4], b0[4], b1[4];
            ldsm4(af, &sm.a[buf][wm * 16 + (lane & 15)][kk * 16 + (lane >> 4) * 8]);
            // replicas 0-7, 8-15 (and 16-23, 24-31) of the warp's 32, both halves of the 16 columns
            ldsm4(b0, &sm.b[wn * 32 + (lane & 7) + ((lane >> 4) << 3)][kk * 16 + ((lane >> 3) & 1) * 8]);
            ldsm4(b1, &sm.b[wn * 32 + 16 + (lane & 7) + ((lane >> 4) << 3)][kk * 16 + ((lane >> 3) & 1) * 8]);
            mma16816(acc[0], af, b0[0], b0[1]);
            mma16816(acc[1], af, b0[2], b0[3]);
            mma16816(acc[2], af, b1[0], b1[1]);
            mma16816(acc[3], af, b1[2], b1[3]);
        }
    };

    // The couplings of a stage as their fixed-point values: FP32 and int8
    // couplings times 2^shift are exact in FP32, and their digits come from
    // the top down by rounding (the last one is the rounding to an integer,
    // ties to even). The other types take int64 values with
    // C = sum_{k < 5} 2048 4096^k added, so that digit k < 5 is the k-th
    // 12-bit field less 2048 and digit 5 what is left above.
    constexpr bool kFloat = std::is_same<QT, float>::value || std::is_same<QT, int8_t>::value;
    using Val = std::conditional_t<kFloat, float, long long>;
    constexpr long long kOffset = 2048ll * (1ll + (1ll << 12) + (1ll << 24) + (1ll << 36) + (1ll << 48));
    const float f1 = ldexpf(1.0f, min(shift, 100)), f2 = ldexpf(1.0f, max(0, shift - 100));
    float low[4][4];                                   // the lowest digit's sums, over up to FLUSH stages
    zero(low);
    int buf = 0, stage = 0, since = 0;
    for (int32_t j0 = 0; j0 < n; j0 += TK, ++stage) {
        Val q[EQ][2];
        uint32_t m = 0;
#pragma unroll
        for (int e = 0; e < EQ; ++e)
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                if constexpr (kFloat) q[e][h] = (float)raw[e].v[h] * f1 * f2;
                else q[e][h] = vqd::qfix<QT>(raw[e].v[h], shift) + kOffset;
                m = max(m, mag(raw[e].v[h]));
            }
        m = __reduce_max_sync(0xffffffffu, m);
        // L digits hold every |q| < 2^(12 L - 2)
        if (lane == 0) sm.digits[stage & 1][warp] = (uint32_t)max(1, min(6, (bits_of<QT>(m, shift) + 13) / 12));
        __syncthreads();                               // digit counts; the previous stage's products have read sm.b
        uint32_t digits = 1;
#pragma unroll
        for (int w = 0; w < WARPS / 4; ++w) {
            const uint4 d = reinterpret_cast<const uint4*>(sm.digits[stage & 1])[w];
            digits = max(digits, max(max(d.x, d.y), max(d.z, d.w)));
        }
#pragma unroll
        for (int e = 0; e < EX; ++e)
            *reinterpret_cast<uint32_t*>(&sm.b[warp + WARPS * e][2 * lane]) =
                (is_on(xr[e].v[0]) ? 0x3C00u : 0u) | (is_on(xr[e].v[1]) ? 0x3C000000u : 0u);
        if (j0 + TK < n) load(j0 + TK);
        // The plane before last is overwritten: every warp read it before the barrier that published the last one
        for (int k = (int)digits - 1; k >= 0; --k) {
            const float down = __int_as_float((127 - 12 * k) << 23), up = __int_as_float((127 + 12 * k) << 23);
#pragma unroll
            for (int e = 0; e < EQ; ++e) {
                float f[2];
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    if constexpr (kFloat) {
                        f[h] = __fsub_rn(fmaf(q[e][h], down, 12582912.0f), 12582912.0f);   // rounded: |.| <= 2048
                        q[e][h] = fmaf(-f[h], up, q[e][h]);                                // exact
                    } else {
                        f[h] = k < 5 ? __uint_as_float(((uint32_t)((unsigned long long)q[e][h] >> (12 * k)) & 4095u) |
                                                       0x4B000000u) - 8390656.0f           // 2^23 + 2048
                                     : (float)(int)(q[e][h] >> 60);
                    }
                }
                *reinterpret_cast<__half2*>(&sm.a[buf][warp + WARPS * e][2 * lane]) = __floats2half2_rn(f[0], f[1]);
            }
            __syncthreads();
            if (k == 0) {
                product(buf, low);
            } else {
                float acc[4][4];
                zero(acc);
                product(buf, acc);
                add(acc, 12 * k);
            }
            buf ^= 1;
        }
        if (++since == FLUSH) {
            add(low, 0);
            zero(low);
            since = 0;
        }
    }
    add(low, 0);
    // over the 8 rows a column's lanes hold, then over the four row warps
#pragma unroll
    for (int c = 0; c < 4; ++c)
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            unsigned long long t = tot[c][h];
            t += __shfl_xor_sync(0xffffffffu, t, 4);
            t += __shfl_xor_sync(0xffffffffu, t, 8);
            t += __shfl_xor_sync(0xffffffffu, t, 16);
            if (gq == 0) sm.red[wm][wn * 32 + c * 8 + 2 * tq + h] = t;
        }
    __syncthreads();
    if (threadIdx.x < TR && r0 + threadIdx.x < R)
        parts_row[r0 + threadIdx.x] = (int64_t)(sm.red[0][threadIdx.x] + sm.red[1][threadIdx.x] +
                                                sm.red[2][threadIdx.x] + sm.red[3][threadIdx.x]);
}

}  // namespace emma
}  // namespace vq
