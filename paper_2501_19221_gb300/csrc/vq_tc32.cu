// vq_tc32.cu -- dense local field F = Qoff S in FP32 accuracy on the
// 5th-generation tensor cores, with the update fused into the epilogue: the
// form dense contexts run in VELOXQ_PREC_FP32.
//
// Every FP32 operand is written as the exact sum of three BF16 terms
// (x = x1 + x2 + x3: 6, 8 and up to 9 significant bits), and the product is the
// sum of eight of the nine term products,
//     q s ~ q1 s1 + (q1 s2 + q2 s1) + (q2 s2 + q1 s3 + q3 s1) + (q2 s3 + q3 s2);
// the one that is left out, q3 s3, is below 2^-29 of q s (x2 is at most 2^-6
// of x, x3 at most 2^-14). The last two reach 2^-20 of q s together: without
// them a row of one coupling had 3.4 times the error of an FP32 product, one
// of six twice that of an FP32 sum, and rows of fewer than about 100
// couplings were less exact than such a sum. For Parallel Annealing the
// operand is +-1, one exact term, and three products are the whole of q s.
//
// Accuracy: the products of BF16 terms are exact in FP32, but the tensor
// cores' accumulation cuts its sums off toward zero, a relative shrinking that
// adds up over the steps of a run. Four things keep it small: the leading
// term has 6 bits only, so that a sum of leading products is mostly exact in
// 24 bits (with 8-bit leading terms the field shrank by 5.8e-8, with 6 bits by
// 3e-9 at 32 variables); the seven small products go to an accumulator of their
// own (sharing one: 8.3e-8); both are drained after every 64 or 128
// variables into FP32 registers with rounded additions; and the two parts
// stay apart in these until the last drain, so that few couplings, whose
// leading sums are exact, are rounded once. Error against FP64 (normwise, S
// uniform in [-1, 1]), the FP32 SGEMM of vq_dense.cu -> here, N(0, 1/n)
// couplings: n = 600: 2.2e-7 -> 6.0e-8, 2048: 3.1e-7 -> 7.0e-8, 4096:
// 5.8e-7 -> 9.2e-8, 8192: 1.6e-6 -> 1.6e-7. Rows of few couplings, n = 700 /
// 2600: one 2.6e-8 -> 2.6e-8 / the same, two 3.6e-8 -> 3.5e-8 / 3.5e-8 ->
// 2.5e-8, six 5.0e-8 -> 4.5e-8 / 4.8e-8 -> 2.5e-8, 64 8.1e-8 -> 5.0e-8 /
// 9.2e-8 -> 3.1e-8. Log-normal couplings (sigma 3): 2.0e-7 -> 1.4e-7 / 4.7e-7
// -> 2.1e-7. States of about four variables on full rows: 4.5e-8 -> 4.1e-8 /
// 4.4e-8 -> 2.5e-8.
//
// Time per step, SGEMM -> here: n = 8192, R = 1024: 4060 -> 625 us (0.92 of
// the measured BF16 rate at 16 n^2 R FLOP; with six products 548); n = 8192,
// R = 64: 650 -> 100 us; n = 3000, R = 1000: 690 -> 99 us; n = 1001, R = 100:
// 41 -> 11.8 us.
//
// CTA pairs (clusters of 2, cta_group::2) compute 256 x 128 tiles (rows x
// replicas), M = 256 MMAs issued by the even CTA, operands staged by TMA in
// blocks of 64 variables: the three terms of a CTA's 128 rows (48 KB) and of
// its 64 replicas (24 KB) in one 3-D copy each, 3 stages (blocks of 32, whose
// rows are half as long, took 631 instead of 585 us at n = 8192, with six
// products). Tiles of 128 replicas rather than 256 keep a thread's two parts of
// the drained field in 128 registers, and give twice the tiles to spread over
// the SMs.
//   * Enough tiles (more than half of the pairs): one launch runs every step
//     up to a readout, tiles of consecutive steps overlapping as in vq_tc.cu
//     (and one behind it that only works where SMs were held by others).
//   * Fewer: the k-loop is split over the idle pairs (at least two blocks each; with one, 14 against 13 us per
//     step at n = 1001, R = 100), the partial fields go to a workspace, and
//     k_t32_finish adds them in order, updates, and writes the next operand.
//     The two launches of a step follow each other by programmatic dependent
//     launch. The choice depends on n and R alone, so a run gives the same
//     bits however it is cut into calls.
// What bounds it: the tensor cores at large n (16 n^2 R FLOP per step);
// with few replicas the 6 bytes per coupling of the three term planes.
#include <cuda.h>
#include <cudaTypedefs.h>
#include <cuda_bf16.h>

#include <algorithm>
#include <atomic>

#include "vq_internal.cuh"
#include "vq_tc.cuh"

namespace vq {

namespace {

using namespace tc;

constexpr int BM = 128;                           // rows per CTA (2 BM per pair)
constexpr int BN_WIDE = 128, BN_NARROW = 64;      // replicas per pair (half of them staged per CTA)
constexpr int BK = 64, BKB = 2 * BK;              // variables per block: 128-byte rows
constexpr uint32_t A_TERM = BM * BKB;
template <int BN> constexpr uint32_t b_term() { return (BN / 2) * BKB; }
template <int NB, int BN> constexpr uint32_t stage_bytes() { return 3 * A_TERM + NB * b_term<BN>(); }
constexpr int STAGES = 3;
constexpr size_t T32_SMEM = (size_t)STAGES * stage_bytes<3, BN_WIDE>() + 1024 /*align*/ + 256 /*barriers, slot*/;
constexpr int EPI_WARPS = 8;
constexpr int THREADS = 32 * (2 + EPI_WARPS);
constexpr int MIN_BLOCKS = 2;                     // k-blocks per split at least

// x = t0 + t1 + t2 exactly: t0 is x rounded to 6 significant bits, t1 the rest
// rounded to 8, t2 what is left (at most 2^8 units of x's last place). A value
// that is not finite is its own first term.
__device__ __forceinline__ void split3(float x, __nv_bfloat16 (&t)[3]) {
    const uint32_t u = __float_as_uint(x);
    if ((u & 0x7f800000u) == 0x7f800000u) {
        t[0] = __float2bfloat16_rn(x);
        t[1] = t[2] = __float2bfloat16_rn(0.0f);
        return;
    }
    // (cut instead of rounded from 2^127 on, where rounding may reach infinity; adiabatic SB's states have no bound)
    const uint32_t up = (u & 0x7f800000u) < (254u << 23) ? 0x0001ffffu + ((u >> 18) & 1u) : 0u;
    const float a = __uint_as_float((u + up) & 0xfffc0000u);
    const float r = __fsub_rn(x, a);
    t[0] = __float2bfloat16_rn(a);
    t[1] = __float2bfloat16_rn(r);
    t[2] = __float2bfloat16_rn(__fsub_rn(r, __bfloat162float(t[1])));
}
// Values whose three terms may reach BF16's subnormals or round past its
// largest value, or that are not finite: these calls take the SGEMM.
__device__ __forceinline__ bool out_of_range(float x) {
    const uint32_t e = __float_as_uint(x) & 0x7f800000u;
    return e >= (254u << 23) || (e < (27u << 23) && x != 0.0f);    // |x| >= 2^127 or < 2^-100
}

template <int NB>
__device__ __forceinline__ void store_terms(__nv_bfloat16* o, int64_t plane, float s) {
    if constexpr (NB == 1) {
        o[0] = __float2bfloat16_rn(s);       // +-1
    } else {
        __nv_bfloat16 t[3];
        split3(s, t);
        o[0] = t[0];
        o[plane] = t[1];
        o[2 * plane] = t[2];
    }
}

// 128-byte-swizzled K-major operand: 8-row core groups 1024 bytes apart
__device__ __forceinline__ uint64_t desc128(uint32_t addr) {
    return (uint64_t)((addr & 0x3FFFFu) >> 4) | (uint64_t)1 << 16 | (uint64_t)(1024 >> 4) << 32 | (uint64_t)1 << 46 |
           (uint64_t)2 << 61;
}
// FP32 accumulator, BF16 operands, K-major, N = BN, M = 2 BM
template <int BN> constexpr uint32_t IDESC = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(BN >> 3) << 17) |
                           ((uint32_t)((2 * BM) >> 4) << 24);
template <int BN> __device__ __forceinline__ void mma_pair(uint32_t d, uint64_t a, uint64_t b, uint32_t accum) {
    asm volatile(
        "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p;\n\t}\n"
        ::"r"(d), "l"(a), "l"(b), "r"(IDESC<BN>), "r"(accum)
        : "memory");
}
// box of {64 variables, rows, terms} into this CTA's shared memory
__device__ __forceinline__ void tma_load_3d_pair(void* dst, const CUtensorMap* map, int x, int y, uint32_t bar_cl) {
    asm volatile(
        "cp.async.bulk.tensor.3d.shared::cluster.global.tile.mbarrier::complete_tx::bytes.cta_group::2 "
        "[%0], [%1, {%2, %3, %4}], [%5];"
        ::"r"(smem_u32(dst)), "l"((uint64_t)map), "r"(x), "r"(y), "r"(0), "r"(bar_cl)
        : "memory");
}
// 8 columns of each of two accumulators
__device__ __forceinline__ void tmem_ld8x2(uint32_t ta, uint32_t tb, uint32_t (&v)[8], uint32_t (&w)[8]) {
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                 : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7])
                 : "r"(ta));
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                 : "=r"(w[0]), "=r"(w[1]), "=r"(w[2]), "=r"(w[3]), "=r"(w[4]), "=r"(w[5]), "=r"(w[6]), "=r"(w[7])
                 : "r"(tb));
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
}

struct T32Args {
    int32_t n, R, n_pad;
    int32_t k, k_end;            // steps k .. k_end - 1 of the schedule (one launch)
    float dt, a0, c0, alpha;
    const float* S_a;            // [R][n] state of the first step (even steps of the run read it)
    float* S_b;                  // [R][n] the other state buffer
    float* Y;                    // [R][n]
    __nv_bfloat16* sop[2];       // [terms][R][n_pad] operand buffers; the first step reads sop[cur]
    int32_t cur;
    int32_t group;               // replica column blocks per group of a step's tile order
    int64_t plane;               // elements of one operand term
    const float* bf;             // [n]
    const float* a_table;
    float* F_out;                // [R][n] field of the last step, or null
    float* part;                 // [ksplit][R][n] partial fields (split form)
    int32_t kper;                // k-blocks per split (split form)
    int32_t ksplit;
    int32_t drain;               // k-blocks accumulated in tensor memory between two drains
    int* err;                    // device error word of the bounded waits
    int* err_host;               // the same, in mapped host memory
    uint32_t* done;              // [replica column blocks] finished epilogue warps, then the lists of the pairs that take
                                 // part in the run and in its shared form (zeroed per run; null for one step)
    const uint32_t* skip;        // do nothing if *skip == skip_seq (null: always run)
    uint32_t skip_seq;
};

// Which pairs take part in a run of several steps. Tiles wait for those of
// the step before, so every pair that owns tiles has to be resident; another
// kernel may hold SMs for longer than a wait lasts. Pairs therefore put
// themselves on a list (its count in the low 16 bits) before they begin. Where
// all of the grid are there, the tiles go to the pairs by their place in the
// grid. Where one has waited `patience` cycles it closes the list (top bit, the
// count so far in bits 16 to 30), all leave without having done anything, and
// the launch behind this one (SHARED, which leaves at once in the ordinary
// case) makes a list of its own and deals the tiles to the pairs on it. Which
// pair computes a tile does not change a bit. Two launches, because a kernel
// that takes its share of the tiles from a list at run time is 7 % slower (676
// against 630 us per step at n = 8192, R = 1024).
// Returns this pair's number on the list and the pairs that take part (0: it came too late).
constexpr uint32_t LIST_CLOSED = 0x80000000u;
constexpr long long kListPatience = kWaitCycles / 4, kListPatienceShared = kWaitCycles / 1000;   // ~0.5 s, ~2 ms
__device__ __forceinline__ void join_list(uint32_t* list, uint32_t grid_pairs, long long patience, uint32_t& me,
                                          uint32_t& pairs) {
    me = atomicAdd(list, 1u);
    pairs = 0;
    if (me & LIST_CLOSED) {
        me = 0;
        return;
    }
    const long long t0 = clock64();
    while (true) {
        const uint32_t w = ld_acquire_u32(list);
        if ((w & LIST_CLOSED) || w == grid_pairs) {
            pairs = w & LIST_CLOSED ? (w >> 16) & 0x7fffu : w;
            return;
        }
        if (clock64() - t0 > patience) atomicCAS(list, w, w | LIST_CLOSED | (w << 16));
    }
}

// form of the kernel: what the epilogue does with the field
enum { FORM_BSB = 0, FORM_ASB = 1, FORM_PA = 2, FORM_FIELD = 3, FORM_SPLIT = 4 };

// One launch runs steps k .. k_end - 1 (or, FORM_SPLIT, one split of one
// step's field per work item). Tile order and the dependency counters between
// steps are those of k_tc_step (vq_tc.cu): tile g = j * tiles + t of step
// k + j starts only after every epilogue warp of its replica column block has
// finished step j - 1, a pair only waits for tiles with a lower g, all pairs
// that own tiles are resident (join_list), and every wait is bounded.
template <int NB, int FORM, int BN = BN_WIDE, bool SHARED = false>
__global__ void __launch_bounds__(THREADS, 1) k_t32(const __grid_constant__ CUtensorMap tmA,
                                                    const __grid_constant__ CUtensorMap tmB0,
                                                    const __grid_constant__ CUtensorMap tmB1, const T32Args a) {
    constexpr int BNH = BN / 2;
    constexpr uint32_t B_TERM = b_term<BN>();
    constexpr uint32_t STAGE_BYTES = stage_bytes<NB, BN>();
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    uint64_t* full = reinterpret_cast<uint64_t*>(smem + STAGES * STAGE_BYTES);   // even CTA: both stages landed
    uint64_t* empty = full + STAGES;      // both CTAs: stage consumed by the MMAs
    uint64_t* accf = empty + STAGES;      // [2] both CTAs: accumulator buffer holds a block's products
    uint64_t* acce = accf + 2;            // [2] even CTA: buffer drained by both CTAs' epilogues
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(acce + 2);
    uint32_t* listed = tmem_slot + 2;     // [2], 8-byte aligned: this pair's number, the pairs that take part

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t rank = cluster_rank();
    const bool leader = rank == 0;
    int pair = blockIdx.x >> 1, pairs = gridDim.x >> 1;
    const int num_kb = (a.n_pad + BK - 1) / BK;
    const int MT = (a.n + 2 * BM - 1) / (2 * BM), NT = (a.R + BN - 1) / BN;
    const int tiles = MT * NT;
    const int steps = a.k_end - a.k;
    const uint32_t per_col = (uint32_t)(2 * EPI_WARPS) * (uint32_t)MT;   // epilogue warps of one column block and step

    if (threadIdx.x == 0) {
        for (int s = 0; s < STAGES; ++s) {
            mbar_init(&full[s], 1);
            mbar_init(&empty[s], 1);
        }
        for (int b = 0; b < 2; ++b) {
            mbar_init(&accf[b], 1);
            mbar_init(&acce[b], 2 * EPI_WARPS);
        }
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    if (warp == 1) tmem_alloc(tmem_slot, 4 * BN);
    tc_fence_before();
    cluster_sync();                              // both CTAs' barriers exist before any remote arrive
    tc_fence_after();
    const uint32_t tmem = *tmem_slot;
    // as in k_tc_step: set-up overlaps the previous kernel, nothing it wrote is read before this wait
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    const bool skip = a.skip && *a.skip == a.skip_seq;
    if constexpr (SHARED) {
        if (leader && threadIdx.x == 0) {
            uint32_t me = 0, all = 0;
            if (ld_acquire_u32(a.done + NT) & LIST_CLOSED)
                join_list(a.done + NT + 1, gridDim.x >> 1, kListPatienceShared, me, all);
            asm volatile("st.shared.v2.u32 [%0], {%1, %2};" ::"r"(smem_u32(listed)), "r"(me), "r"(all) : "memory");
            asm volatile("st.shared::cluster.v2.u32 [%0], {%1, %2};" ::"r"(mapa(smem_u32(listed), 1)), "r"(me), "r"(all)
                         : "memory");
        }
        __syncwarp();
        cluster_sync();
        pair = (int)*(volatile uint32_t*)listed;
        pairs = (int)*(volatile uint32_t*)(listed + 1);
    } else if (a.done) {
        if (leader && threadIdx.x == 0) {
            uint32_t me, all;
            join_list(a.done + NT, gridDim.x >> 1, kListPatience, me, all);
        }
        __syncwarp();
        cluster_sync();
        if (ld_acquire_u32(a.done + NT) & LIST_CLOSED) {       // final by now: closed, or all are there
            tc_fence_before();
            __syncthreads();
            cluster_sync();
            tc_fence_after();
            if (warp == 1) tmem_dealloc(tmem, 4 * BN);
            return;
        }
    }
    const int64_t work = skip || (SHARED && pairs == 0) ? 0 : FORM == FORM_SPLIT ? (int64_t)tiles * a.ksplit : (int64_t)steps * tiles;
    // work item g: step j, row block r, column block c, k-blocks [kb0, kb1)
    auto item = [&](int64_t g, int& j, int& r, int& c, int& kb0, int& kb1) {
        const int z = (int)(g / tiles), t = (int)(g - (int64_t)z * tiles);
        j = FORM == FORM_SPLIT ? 0 : z;
        kb0 = FORM == FORM_SPLIT ? z * a.kper : 0;
        kb1 = FORM == FORM_SPLIT ? min(num_kb, kb0 + a.kper) : num_kb;
        const int G = a.group;
        const int c0 = (t / (G * MT)) * G;
        const int gc = min(G, NT - c0);
        const int u = t - c0 * MT;
        r = u / gc;
        c = c0 + (u - r * gc);
    };

    if (warp == 0) {
        if (lane == 0) {
            uint32_t it = 0;
            bool ok = true;
            for (int64_t g = pair; g < work && ok; g += pairs) {
                int j, r, c, kb0, kb1;
                item(g, j, r, c, kb0, kb1);
                const int m0 = r * (2 * BM) + (int)rank * BM, n0 = c * BN + (int)rank * BNH;
                if (j > 0) {
                    if (!count_wait(a.done + c, per_col * (uint32_t)j, a.err, TC_ERR_DEPEND)) break;
                    fence_proxy_async_global();
                }
                const CUtensorMap* mb = ((a.cur + j) & 1) ? &tmB1 : &tmB0;
                for (int kb = kb0; kb < kb1; ++kb) {
                    const uint32_t s = it % STAGES, u = it / STAGES;
                    if (u > 0 && !mbar_wait<true>(&empty[s], (u - 1) & 1, a.err, TC_ERR_PRODUCER)) { ok = false; break; }
                    uint8_t* sa = smem + s * STAGE_BYTES;
                    if (leader) mbar_expect_tx(&full[s], 2 * STAGE_BYTES);
                    const uint32_t fb = mapa(smem_u32(&full[s]), 0);
                    tma_load_3d_pair(sa, &tmA, kb * BK, m0, fb);
                    tma_load_3d_pair(sa + 3 * A_TERM, mb, kb * BK, n0, fb);
                    ++it;
                }
            }
        }
    } else if (warp == 1) {
        if (lane == 0 && leader) {
            uint32_t it = 0, dr = 0;
            bool ok = true;
            for (int64_t g = pair; g < work && ok; g += pairs) {
                int j, r, c, kb0, kb1;
                item(g, j, r, c, kb0, kb1);
                for (int kb = kb0; kb < kb1; ++kb, ++it) {
                    const uint32_t s = it % STAGES, u = it / STAGES, b = dr & 1u;
                    const bool first = (kb - kb0) % a.drain == 0, last = (kb - kb0) % a.drain == a.drain - 1 || kb == kb1 - 1;
                    if (first && dr >= 2 && !mbar_wait<true>(&acce[b], ((dr >> 1) - 1) & 1u, a.err, TC_ERR_MMA)) { ok = false; break; }
                    if (!mbar_wait<true>(&full[s], u & 1, a.err, TC_ERR_MMA)) { ok = false; break; }
                    tc_fence_after();
                    const uint32_t d = tmem + b * 2 * BN, dx = d + BN;
                    const uint32_t sa = smem_u32(smem + s * STAGE_BYTES), sb = sa + 3 * A_TERM;
                    // the leading products into one accumulator, the small ones into another
#pragma unroll
                    for (int kk = 0; kk < BK / 16; ++kk) {
                        const uint32_t o = kk * 32, acc = (kk != 0 || !first) ? 1u : 0u;
                        const uint64_t a0 = desc128(sa + o), a1 = desc128(sa + A_TERM + o), a2 = desc128(sa + 2 * A_TERM + o);
                        const uint64_t b0 = desc128(sb + o);
                        if constexpr (NB == 3) {
                            const uint64_t b1 = desc128(sb + B_TERM + o), b2 = desc128(sb + 2 * B_TERM + o);
                            mma_pair<BN>(d, a0, b0, acc);
                            mma_pair<BN>(dx, a1, b2, acc);
                            mma_pair<BN>(dx, a2, b1, 1u);
                            mma_pair<BN>(dx, a0, b2, 1u);
                            mma_pair<BN>(dx, a0, b1, 1u);
                            mma_pair<BN>(dx, a1, b1, 1u);
                            mma_pair<BN>(dx, a1, b0, 1u);
                            mma_pair<BN>(dx, a2, b0, 1u);
                        } else {
                            mma_pair<BN>(d, a0, b0, acc);
                            mma_pair<BN>(dx, a2, b0, acc);
                            mma_pair<BN>(dx, a1, b0, 1u);
                        }
                    }
                    umma_commit_pair(&empty[s]);
                    if (last) {
                        umma_commit_pair(&accf[b]);
                        ++dr;
                    }
                }
            }
        }
    } else {
        // epilogue: warp w reads tensor-memory lanes 32 (w % 4) .. +31 (this CTA's rows); the first four warps
        // take the first half of the tile's replica columns, the next four the rest
        const int q = warp & 3;
        const int half = (warp - 2) >> 2;
        const uint32_t acce_cl = mapa(smem_u32(&acce[0]), 0);
        constexpr int NC = BN / 2, CW = 16;
        const uint32_t tcol = tmem + ((uint32_t)(q * 32) << 16) + (uint32_t)(half * NC);
        uint32_t it = 0;
        bool ok = true;
        for (int64_t g = pair; g < work && ok; g += pairs) {
            int j, r, c, kb0, kb1;
            item(g, j, r, c, kb0, kb1);
            float F[NC], L[NC];
#pragma unroll
            for (int v = 0; v < NC; ++v) F[v] = L[v] = 0.0f;
            for (int kb = kb0; kb < kb1; kb += a.drain, ++it) {
                const uint32_t b = it & 1u;
                if (!mbar_wait<true>(&accf[b], (it >> 1) & 1u, a.err, TC_ERR_EPILOGUE)) { ok = false; break; }
                tc_fence_after();
#pragma unroll
                for (int h = 0; h < NC / 8; ++h) {
                    uint32_t v[8], x[8];
                    tmem_ld8x2(tcol + b * 2 * BN + h * 8, tcol + b * 2 * BN + BN + h * 8, v, x);
#pragma unroll
                    for (int l = 0; l < 8; ++l) {
                        F[h * 8 + l] = __fadd_rn(F[h * 8 + l], __uint_as_float(v[l]));
                        L[h * 8 + l] = __fadd_rn(L[h * 8 + l], __uint_as_float(x[l]));
                    }
                }
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive_remote(acce_cl + b * 8);
            }
            if (!ok) break;
#pragma unroll
            for (int v = 0; v < NC; ++v) {
                // An infinite state is its own first term: the leading products are then the whole of F, and the small
                // ones may be infinite with the other sign, or 0 times infinity.
                const float t = __fadd_rn(F[v], L[v]);
                F[v] = fabsf(F[v]) == __int_as_float(0x7f800000) ? F[v] : t;
            }
            const int row = r * (2 * BM) + (int)rank * BM + q * 32 + lane;
            const int r0 = c * BN + half * NC;
            const bool row_ok = row < a.n;
            const int64_t p0 = (int64_t)r0 * a.n + row;
            if constexpr (FORM == FORM_SPLIT || FORM == FORM_FIELD) {
                float* out = FORM == FORM_SPLIT ? a.part + (g / tiles) * (int64_t)a.R * a.n : a.F_out;
#pragma unroll
                for (int v = 0; v < NC; ++v)
                    if (row_ok && r0 + v < a.R) out[p0 + (int64_t)v * a.n] = F[v];
            } else {
                const int k = a.k + j;
                const float a_k = __ldg(a.a_table + k);
                const float lam = FORM == FORM_PA ? vqd::pa_lambda(a_k, a.a0) : 0.0f;
                const float* S_cur = (j & 1) ? a.S_b : a.S_a;
                float* S_nxt = (j & 1) ? const_cast<float*>(a.S_a) : a.S_b;
                __nv_bfloat16* op = a.sop[(a.cur + j + 1) & 1];
                float* F_out = j == steps - 1 ? a.F_out : nullptr;
                const float bi = row_ok ? __ldg(a.bf + row) : 0.0f;
                // the state of these rows was written by the previous step's tile
                if (j > 0) {
                    bool got = false;
                    if (lane == 0) got = count_wait(a.done + c, per_col * (uint32_t)j, a.err, TC_ERR_DEPEND);
                    if (__shfl_sync(0xffffffffu, got ? 1 : 0, 0) == 0) break;
                    (void)ld_acquire_u32(a.done + c);
                }
#pragma unroll
                for (int cc = 0; cc < NC; cc += CW) {
                    float sv[CW], yv[CW];
#pragma unroll
                    for (int v = 0; v < CW; ++v) {
                        const bool in = row_ok && r0 + cc + v < a.R;
                        const int64_t p = p0 + (int64_t)(cc + v) * a.n;
                        sv[v] = in ? __ldcs(S_cur + p) : 0.0f;
                        yv[v] = in ? __ldcs(a.Y + p) : 0.0f;
                    }
#pragma unroll
                    for (int v = 0; v < CW; ++v) {
                        const bool in = row_ok && r0 + cc + v < a.R;
                        const int64_t p = p0 + (int64_t)(cc + v) * a.n;
                        float s = sv[v], y = yv[v];
                        const float Fv = F[cc + v];
                        if constexpr (FORM == FORM_PA) vqd::pa_update(Fv, bi, lam, a.dt, a.alpha, a.c0, s, y);
                        else if constexpr (FORM == FORM_ASB) vqd::asb_update(Fv, bi, a_k, a.dt, a.a0, a.c0, s, y);
                        else vqd::bsb_update(Fv, bi, a_k, a.dt, a.a0, a.c0, s, y);
                        if (in) {
                            if (F_out) F_out[p] = Fv;
                            __stcs(S_nxt + p, s);
                            __stcs(a.Y + p, y);
                            store_terms<NB>(op + (int64_t)(r0 + cc + v) * a.n_pad + row, a.plane,
                                            FORM == FORM_PA ? vqd::pa_sign(s) : s);
                        }
                    }
                }
                if (steps > 1) {
                    fence_proxy_async_global();
                    __threadfence();
                    __syncwarp();
                    if (lane == 0) red_release_add(a.done + c, 1u);
                }
            }
        }
    }
    // neither CTA leaves while the other may still read its shared memory or
    // arrive on its barriers
    tc_fence_before();
    __syncthreads();
    cluster_sync();
    tc_fence_after();
    if (warp == 1) tmem_dealloc(tmem, 4 * BN);
    if (threadIdx.x == 0) {
        const int e = *(volatile int*)a.err;
        if (e && a.err_host) atomicOr_system(a.err_host, e);
    }
}

// F = sum over the k splits (in order), the update of the step, and the next
// step's operand. FIELD: the field alone.
template <int NB, int FORM>
__global__ void __launch_bounds__(256) k_t32_finish(const T32Args a) {
    const int nb = (a.n + 255) / 256;
    const int64_t r = blockIdx.x / nb;
    const int i = (int)(blockIdx.x - r * nb) * 256 + threadIdx.x;
    const int64_t p = r * a.n + i, total = (int64_t)a.R * a.n;
    // This kernel starts when every CTA of the field kernel has passed its own
    // wait, so the state (written by the previous step's k_t32_finish) may be
    // read before this one; the partial fields only after it.
    float s = 0.0f, y = 0.0f;
    if constexpr (FORM != FORM_FIELD) {
        if (i < a.n) {
            s = __ldcg(a.S_a + p);
            y = __ldcg(a.Y + p);
        }
    }
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    if (i >= a.n || (a.skip && *a.skip == a.skip_seq)) return;
    // eight partial fields in flight, added in order
    float F = 0.0f;
    for (int z0 = 0; z0 < a.ksplit; z0 += 8) {
        float v[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) v[u] = z0 + u < a.ksplit ? __ldcs(a.part + (int64_t)(z0 + u) * total + p) : 0.0f;
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            if (z0 + u == 0) F = v[0];
            else if (z0 + u < a.ksplit) F = __fadd_rn(F, v[u]);
        }
    }
    if (a.F_out) a.F_out[p] = F;
    if constexpr (FORM != FORM_FIELD) {
        const float bi = __ldg(a.bf + i), a_k = __ldg(a.a_table + a.k);
        if constexpr (FORM == FORM_PA) vqd::pa_update(F, bi, vqd::pa_lambda(a_k, a.a0), a.dt, a.alpha, a.c0, s, y);
        else if constexpr (FORM == FORM_ASB) vqd::asb_update(F, bi, a_k, a.dt, a.a0, a.c0, s, y);
        else vqd::bsb_update(F, bi, a_k, a.dt, a.a0, a.c0, s, y);
        a.S_b[p] = s;
        a.Y[p] = y;
        store_terms<NB>(a.sop[0] + r * a.n_pad + i, a.plane, FORM == FORM_PA ? vqd::pa_sign(s) : s);
    }
}

// the three term planes of Qoff [3][n][n_pad] (zero in the K padding); *bad
// is set where a value's terms would leave BF16's normal range
__global__ void __launch_bounds__(256) k_t32_split_q(int64_t n, int64_t n_pad, const float* __restrict__ q,
                                                     __nv_bfloat16* __restrict__ out, int* bad) {
    const int64_t i = blockIdx.x;
    bool b = false;
    for (int64_t j = threadIdx.x; j < n_pad; j += 256) {
        const float x = j < n ? q[i * n + j] : 0.0f;
        b |= out_of_range(x);
        __nv_bfloat16 t[3];
        split3(x, t);
#pragma unroll
        for (int v = 0; v < 3; ++v) out[((int64_t)v * n + i) * n_pad + j] = t[v];
    }
    if (b) *bad = 1;
}

// the operand of S in its terms [NB][R][n_pad] (zero in the K padding);
// *bad (and *bad_host) = seq where a value's terms would leave the range
template <int NB>
__global__ void __launch_bounds__(256) k_t32_split_s(int64_t R, int64_t n, int64_t n_pad, const float* __restrict__ S,
                                                     __nv_bfloat16* __restrict__ out, int method, uint32_t* bad,
                                                     uint32_t* bad_host, uint32_t seq) {
    const int64_t nb = (n_pad + 255) / 256;
    const int64_t r = blockIdx.x / nb, j = (blockIdx.x - r * nb) * 256 + threadIdx.x;
    if (j >= n_pad) return;
    const float s = j < n ? S[r * n + j] : 0.0f;
    const float x = j < n ? vqd::field_operand(method, s) : 0.0f;
    store_terms<NB>(out + r * n_pad + j, R * n_pad, x);
    if (out_of_range(NB == 1 ? 1.0f : x) && bad) {
        *bad = seq;
        if (bad_host) {
            *(volatile uint32_t*)bad_host = seq;
            __threadfence_system();
        }
    }
}

PFN_cuTensorMapEncodeTiled_v12000 encode_fn() {
    static PFN_cuTensorMapEncodeTiled_v12000 fn = [] {
        cudaDriverEntryPointQueryResult q;
        void* p = nullptr;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) != cudaSuccess ||
            q != cudaDriverEntryPointSuccess) {
            cudaGetLastError();
            p = nullptr;
        }
        return reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(p);
    }();
    return fn;
}

// 3-D K-major operand [terms][rows][n_pad], box {64, box_rows, terms}
int make_map3(CUtensorMap* m, void* base, int64_t rows, int64_t n_pad, int box_rows, int terms) {
    auto fn = encode_fn();
    if (!fn) return fail(VELOXQ_EUNSUPPORTED, "cuTensorMapEncodeTiled is not available from the driver");
    cuuint64_t dims[3] = {(cuuint64_t)n_pad, (cuuint64_t)rows, (cuuint64_t)terms};
    cuuint64_t strides[2] = {(cuuint64_t)(n_pad * 2), (cuuint64_t)(rows * n_pad * 2)};
    cuuint32_t box[3] = {BK, (cuuint32_t)box_rows, (cuuint32_t)terms};
    cuuint32_t estr[3] = {1, 1, 1};
    CUresult r = fn(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, base, dims, strides, box, estr,
                    CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                    CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (r != CUDA_SUCCESS) return fail(VELOXQ_ECUDA, "cuTensorMapEncodeTiled failed (" + std::to_string((int)r) + ")");
    return VELOXQ_OK;
}

using T32Kernel = void (*)(const CUtensorMap, const CUtensorMap, const CUtensorMap, const T32Args);
T32Kernel pick_split(bool exact_operand, int bn) {
    if (bn == BN_NARROW)
        return exact_operand ? k_t32<1, FORM_SPLIT, BN_NARROW> : k_t32<3, FORM_SPLIT, BN_NARROW>;
    return exact_operand ? k_t32<1, FORM_SPLIT> : k_t32<3, FORM_SPLIT>;
}
template <bool SHARED> T32Kernel pick(int form) {
    switch (form) {
        case FORM_BSB: return k_t32<3, FORM_BSB, BN_WIDE, SHARED>;
        case FORM_ASB: return k_t32<3, FORM_ASB, BN_WIDE, SHARED>;
        case FORM_PA: return k_t32<1, FORM_PA, BN_WIDE, SHARED>;
        default: return k_t32<3, FORM_FIELD>;
    }
}
using FinishKernel = void (*)(const T32Args);
FinishKernel pick_finish(int form) {
    switch (form) {
        case FORM_BSB: return k_t32_finish<3, FORM_BSB>;
        case FORM_ASB: return k_t32_finish<3, FORM_ASB>;
        case FORM_PA: return k_t32_finish<1, FORM_PA>;
        default: return k_t32_finish<3, FORM_FIELD>;
    }
}

// co-resident CTA pairs of k_t32, per device (every form has the same block
// size and shared memory)
int max_pairs(int device) {
    static std::atomic<int> cache[64];
    if (device < 0 || device >= 64) return 1;
    int v = cache[device].load(std::memory_order_relaxed);
    if (v) return v;
    const int sms = device_sms(device);
    T32Kernel fn = k_t32<3, FORM_BSB>;
    int c = 0;
    cudaLaunchConfig_t cfg = {};
    cfg.blockDim = dim3(THREADS);
    cfg.gridDim = dim3((unsigned)(sms & ~1));
    cfg.dynamicSmemBytes = T32_SMEM;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = 2;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    if (cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)T32_SMEM) != cudaSuccess ||
        cudaOccupancyMaxActiveClusters(&c, fn, &cfg) != cudaSuccess || c < 1) {
        cudaGetLastError();
        c = sms / 2;
    }
    v = std::max(1, std::min(c, sms / 2));
    cache[device].store(v, std::memory_order_relaxed);
    return v;
}

struct Plan {
    int64_t MT, NT, tiles;
    int bn, pairs, ksplit, kper;
};
Plan plan(const veloxq_ctx* ctx, int32_t R) {
    Plan p;
    p.MT = div_up(ctx->n, 2 * BM);
    p.pairs = max_pairs(ctx->device);
    const int nkb = (int)div_up(tc_pad(ctx->n), BK);
    auto split = [&](int bn) {
        p.bn = bn;
        p.NT = div_up(R, bn);
        p.tiles = p.MT * p.NT;
        const int ks = (int)std::max<int64_t>(1, std::min<int64_t>(p.pairs / p.tiles, nkb / MIN_BLOCKS));
        p.kper = (int)div_up(nkb, ks);
        p.ksplit = (int)div_up(nkb, p.kper);
    };
    split(BN_WIDE);
    // Narrow tiles in the split form: half the MMA work of a tile where there
    // are no more than 64 replicas, and more pairs at work where the splits of
    // wide tiles cannot fill them (a step of n = 1001: R = 64 11.2 -> 9.6 us,
    // R = 100 11.7 -> 10.5; n = 600, R = 200 11.8 -> 10.5; n = 3000, R = 64
    // 19.1 -> 17.7; n = 8192, R = 64 91.0 -> 90.2, bound by its terms' bytes).
    if (p.ksplit > 1 && (R <= BN_NARROW || 2 * p.tiles * p.ksplit <= p.pairs)) {
        split(BN_NARROW);
        if (p.ksplit == 1) split(BN_WIDE);
    }
    return p;
}

// Steps per launch at most: the completion counters stay far below 2^32.
constexpr int kMaxRunSteps = 4096;
constexpr int64_t kMinN = 192;       // below, the SGEMM's two launches are as fast

int launch(veloxq_ctx* ctx, T32Kernel fn, int64_t pairs, const CUtensorMap& mq, const CUtensorMap* ms,
           const T32Args& a) {
    cudaLaunchConfig_t cfg = {};
    cfg.blockDim = dim3(THREADS);
    cfg.gridDim = dim3((unsigned)(2 * pairs));
    cfg.dynamicSmemBytes = T32_SMEM;
    cfg.stream = ctx->stream;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = 2;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 2;
    VQ_CUDA(cudaLaunchKernelEx(&cfg, fn, mq, ms[0], ms[1], a));
    return VELOXQ_OK;
}
int launch_finish(veloxq_ctx* ctx, FinishKernel fn, const T32Args& a) {
    cudaLaunchConfig_t cfg = {};
    cfg.blockDim = dim3(256);
    cfg.gridDim = dim3((unsigned)(div_up(a.n, 256) * a.R));
    cfg.stream = ctx->stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    VQ_CUDA(cudaLaunchKernelEx(&cfg, fn, a));
    return VELOXQ_OK;
}

}  // namespace

int async_words(veloxq_ctx* ctx) {
    if (ctx->t32h.p && ctx->t32w.p) return VELOXQ_OK;
    if (!ctx->t32h.p) VQ_TRY(ctx->t32h.make());
    VQ_TRY(ctx->t32w.ensure(sizeof(int) * 8));
    VQ_CUDA(cudaMemsetAsync(ctx->t32w.p, 0, sizeof(int) * 8, ctx->stream));
    return VELOXQ_OK;
}

// Prepares the form for R replicas: the term planes of Qoff (once per
// context), operand and counter buffers. *ready = false (and no error) where
// the SGEMM has to serve: small n, values whose terms leave BF16's range, or
// no room (for this call: the next one tries again). Allocates; with the stream in capture, *ready tells
// whether everything was there already.
int t32_prepare(veloxq_ctx* ctx, int32_t R, bool* ready) {
    *ready = false;
    if (!ctx->dense || ctx->n < kMinN || ctx->device < 0 || ctx->device >= 64 || ctx->q3_state < 0) return VELOXQ_OK;
    const int64_t n = ctx->n, np = tc_pad(n);
    const Plan p = plan(ctx, R);
    if (div_up(n, 256) * (int64_t)R > INT32_MAX || p.tiles > INT32_MAX / 2) return VELOXQ_OK;
    const size_t ob = sizeof(__nv_bfloat16) * 3 * (size_t)R * (size_t)np;
    const size_t pb = p.ksplit > 1 ? sizeof(float) * (size_t)p.ksplit * (size_t)R * (size_t)n : 0;
    const size_t db = sizeof(uint32_t) * (size_t)(p.NT + 2);
    const bool fused = p.ksplit == 1;
    if (ctx->q3_state > 0 && ctx->s3[0].bytes >= ob && (!fused || ctx->s3[1].bytes >= ob) && ctx->dpart.bytes >= pb &&
        ctx->tcdone.bytes >= db) {
        *ready = true;
    } else {
        cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
        VQ_CUDA(cudaStreamIsCapturing(ctx->stream, &cs));
        if (cs != cudaStreamCaptureStatusNone) return VELOXQ_OK;
        int st = VELOXQ_OK;
        auto room = [&](DevBuf& b, size_t need) {
            if (st == VELOXQ_OK && need) st = b.ensure(need);
        };
        if (ctx->q3_state == 0) {
            // the planes take at most half of the memory that is free
            size_t free_b = 0, total_b = 0;
            VQ_CUDA(cudaMemGetInfo(&free_b, &total_b));
            if (sizeof(__nv_bfloat16) * 3 * (size_t)n * (size_t)np + 2 * ob + pb > free_b / 2) return VELOXQ_OK;
            room(ctx->q3, sizeof(__nv_bfloat16) * 3 * (size_t)n * (size_t)np);
            if (st == VELOXQ_OK) st = async_words(ctx);
        }
        room(ctx->s3[0], ob);
        if (fused) room(ctx->s3[1], ob);
        room(ctx->dpart, pb);
        room(ctx->tcdone, db);
        if (st == VELOXQ_ENOMEM) {        // no room: the SGEMM serves this call, and has what these would hold
            ctx->q3.release();
            ctx->s3[0].release();
            ctx->s3[1].release();
            ctx->q3_state = 0;
            return VELOXQ_OK;
        }
        VQ_TRY(st);
        if (ctx->q3_state == 0) {
            int* bad = ctx->t32w.as<int>() + 2;
            k_t32_split_q<<<(unsigned)n, 256, 0, ctx->stream>>>(n, np, ctx->qoff32.as<float>(),
                                                                ctx->q3.as<__nv_bfloat16>(), bad);
            VQ_LAUNCH_CHECK("t32 split Q");
            int h = 0;
            VQ_CUDA(cudaMemcpyAsync(&h, bad, sizeof(int), cudaMemcpyDeviceToHost, ctx->stream));
            VQ_CUDA(cudaStreamSynchronize(ctx->stream));
            if (h) {
                ctx->q3.release();
                ctx->q3_state = -1;
                return VELOXQ_OK;
            }
            ctx->q3_state = 1;
        }
        *ready = true;
    }
    return VELOXQ_OK;
}

// The first step's operand from S. check: values out of range set the
// context's flag to the returned sequence number (t32_bad, T32Args::skip).
int t32_split(veloxq_ctx* ctx, int32_t R, const float* S, const Rule& rule, bool check, T32Run* t) {
    const int64_t n = ctx->n, np = tc_pad(n);
    t->cur = 0;
    t->seq = 0;
    uint32_t *bad = nullptr, *bad_h = nullptr;
    if (check) {
        if (++ctx->t32_seq == 0) ++ctx->t32_seq;
        t->seq = ctx->t32_seq;
        bad = ctx->t32w.as<uint32_t>() + 1;
        bad_h = reinterpret_cast<uint32_t*>(ctx->t32h.dev) + 1;
        // a captured call is replayed with its number: what an earlier replay found must not stay
        cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
        VQ_CUDA(cudaStreamIsCapturing(ctx->stream, &cs));
        if (cs != cudaStreamCaptureStatusNone) VQ_CUDA(cudaMemsetAsync(bad, 0, sizeof(uint32_t), ctx->stream));
    }
    t->terms = rule.method == VELOXQ_METHOD_PA ? 1 : 3;
    // the other operand buffer, which the epilogue writes first: its K padding must be zero too
    if (np != n && plan(ctx, R).ksplit == 1)
        VQ_CUDA(cudaMemsetAsync(ctx->s3[1].p, 0, sizeof(__nv_bfloat16) * (size_t)t->terms * R * np, ctx->stream));
    const unsigned g = (unsigned)(div_up(np, 256) * R);
    __nv_bfloat16* o = ctx->s3[0].as<__nv_bfloat16>();
    if (t->terms == 1)
        k_t32_split_s<1><<<g, 256, 0, ctx->stream>>>(R, n, np, S, o, rule.method, bad, bad_h, t->seq);
    else
        k_t32_split_s<3><<<g, 256, 0, ctx->stream>>>(R, n, np, S, o, rule.method, bad, bad_h, t->seq);
    VQ_LAUNCH_CHECK("t32 split S");
    return VELOXQ_OK;
}

// after a stream synchronisation: whether the operand of `t` was out of range
bool t32_bad(const veloxq_ctx* ctx, const T32Run& t) {
    return t.seq != 0 && reinterpret_cast<volatile uint32_t*>(ctx->t32h.p)[1] == t.seq;
}

// launches of `steps` steps up to a readout
int t32_launches(const veloxq_ctx* ctx, int32_t R, int steps) {
    if (plan(ctx, R).ksplit > 1) return 2 * steps;
    const int runs = (int)div_up(steps, kMaxRunSteps);
    return 2 * runs - (steps % kMaxRunSteps == 1 ? 1 : 0);       // a run of more than one step takes two
}

// Steps k_begin .. k_end - 1 from the operand t32_split (or the last call)
// left; *cur and *nxt are exchanged when the state ends in the other buffer.
// guard: run only if the operand was in range (field alone).
int t32_run(veloxq_ctx* ctx, int32_t R, T32Run* t, float** cur, float** nxt, float* Y, const float* a_table,
            int k_begin, int k_end, float dt, float a0, float c0, float* F_out, const Rule& rule, bool field_only,
            bool guard) {
    if (k_end <= k_begin) return VELOXQ_OK;
    const Plan p = plan(ctx, R);
    const int64_t n = ctx->n, np = tc_pad(n);
    const int terms = t->terms;
    CUtensorMap mq, ms[2];
    VQ_TRY(make_map3(&mq, ctx->q3.p, n, np, BM, 3));
    VQ_TRY(make_map3(&ms[0], ctx->s3[0].p, R, np, p.bn / 2, terms));
    ms[1] = ms[0];
    if (ctx->s3[1].p && p.ksplit == 1) VQ_TRY(make_map3(&ms[1], ctx->s3[1].p, R, np, p.bn / 2, terms));
    const int form = field_only ? FORM_FIELD
                     : rule.method == VELOXQ_METHOD_PA ? FORM_PA
                     : rule.method == VELOXQ_METHOD_ASB ? FORM_ASB : FORM_BSB;
    T32Args a = {};
    a.n = (int32_t)n;
    a.R = R;
    a.n_pad = (int32_t)np;
    a.dt = dt;
    a.a0 = a0;
    a.c0 = c0;
    a.alpha = rule.alpha;
    a.Y = Y;
    a.sop[0] = ctx->s3[0].as<__nv_bfloat16>();
    a.sop[1] = ctx->s3[1].as<__nv_bfloat16>();
    a.plane = (int64_t)R * np;
    a.bf = ctx->bf.as<float>();
    a.a_table = a_table;
    a.part = ctx->dpart.as<float>();
    a.kper = p.kper;
    a.ksplit = p.ksplit;
    // Tensor-core accumulation cuts its sums off toward zero, so F shrinks by a part that grows with the variables
    // between two drains: 3e-9 at 32, 7e-9 at 64, 1.9e-8 at 128. It is kept below about 3 % of the error the FP32
    // SGEMM has at that size (2e-7 to 3e-7 up to n = 2048, 6e-7 at 4096, 1.6e-6 at 8192).
    // (Parallel Annealing's products with +-1 have 6 and 8 bits and lose nothing at 256.)
    a.drain = terms == 1 ? 4 : n < 2560 ? 1 : 2;
    a.err = ctx->t32w.as<int>();
    a.err_host = static_cast<int*>(ctx->t32h.dev);
    a.skip = guard ? ctx->t32w.as<uint32_t>() + 1 : nullptr;
    a.skip_seq = t->seq;
    if (p.ksplit > 1) {
        T32Kernel fn = pick_split(terms == 1, p.bn);
        VQ_CUDA(cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)T32_SMEM));
        FinishKernel fin = pick_finish(form);
        a.group = 1;
        for (int k = k_begin; k < k_end; ++k) {
            a.k = k;
            a.k_end = k + 1;
            a.S_a = field_only ? nullptr : *cur;
            a.S_b = field_only ? nullptr : *cur;      // in place
            a.F_out = k == k_end - 1 ? F_out : nullptr;
            VQ_TRY(launch(ctx, fn, p.tiles * p.ksplit, mq, ms, a));
            VQ_TRY(launch_finish(ctx, fin, a));
        }
        return VELOXQ_OK;
    }
    // Column blocks per group: four share each block of Qoff rows in L2, as
    // long as the other groups' tiles keep every pair busy while a step's
    // last group finishes; else one, so that steps overlap.
    a.group = 1;
    for (int G : {4, 2})
        if (p.MT * (p.NT - G) >= p.pairs) {
            a.group = G;
            break;
        }
    T32Kernel fn = pick<false>(form), fn_shared = pick<true>(form);
    for (T32Kernel f : {fn, fn_shared})
        VQ_CUDA(cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)T32_SMEM));
    for (int k0 = k_begin; k0 < k_end; k0 += kMaxRunSteps) {
        const int k1 = std::min(k_end, k0 + kMaxRunSteps), steps = k1 - k0;
        a.k = k0;
        a.k_end = k1;
        a.S_a = field_only ? nullptr : *cur;
        a.S_b = field_only ? nullptr : *nxt;
        a.cur = t->cur;
        a.F_out = k1 == k_end ? F_out : nullptr;
        a.done = nullptr;
        if (steps > 1) {
            VQ_CUDA(cudaMemsetAsync(ctx->tcdone.p, 0, sizeof(uint32_t) * (size_t)(p.NT + 2), ctx->stream));
            a.done = ctx->tcdone.as<uint32_t>();
        }
        VQ_TRY(launch(ctx, fn, std::min<int64_t>(p.tiles * steps, p.pairs), mq, ms, a));
        if (steps > 1) VQ_TRY(launch(ctx, fn_shared, std::min<int64_t>(p.tiles * steps, p.pairs), mq, ms, a));
        if ((steps & 1) && !field_only) {
            std::swap(*cur, *nxt);
            t->cur ^= 1;
        }
    }
    return VELOXQ_OK;
}

// Whether a wait of an earlier call on ctx gave up (reported once, and to a
// call in capture without ending the report, which takes a synchronisation).
int t32_check(veloxq_ctx* ctx) {
    if (!ctx->t32h.p) return VELOXQ_OK;
    volatile int* h = static_cast<volatile int*>(ctx->t32h.p);
    const int code = h[0];
    if (!code) return VELOXQ_OK;
    cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
    VQ_CUDA(cudaStreamIsCapturing(ctx->stream, &cs));
    if (cs == cudaStreamCaptureStatusNone) {
        VQ_CUDA(cudaStreamSynchronize(ctx->stream));
        h[0] = 0;
        VQ_CUDA(cudaMemsetAsync(ctx->t32w.p, 0, sizeof(int), ctx->stream));
    }
    return fail(VELOXQ_ETIMEDOUT, "a bounded device wait in an earlier call on this context gave up (code " +
                                      std::to_string(code) + "); its results, and those of the calls issued since, "
                                      "are not valid");
}

}  // namespace vq
