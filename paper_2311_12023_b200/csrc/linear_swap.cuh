// Tensor-core linear with the weights as the row operand of tcgen05.mma and the tokens as its N side (cta_group::2).
//
// A pair of CTAs computes 256 output columns (128 each) for up to 512 tokens, over a slice of the contraction; the
// accumulator is the transposed output tile.  Every weight is dequantized once per chunk of tokens, whatever their number,
// the tensor core does no work for rows past the next multiple of 16, and each CTA loads half of the tokens.
// Roles: warps 0 and 1 load this CTA's half of the (one or two) token boxes by TMA, warp 2 the packed codes (bulk
// copies, a ring of their own), warp 3 of the leader issues the MMAs, sixteen warps dequantize.  Four of those share a
// step of 64 contraction elements (one thread = one row of 64 weights, so a block of 64 or more costs one table), four
// steps are in work at a time.  The slices of the contraction are further
// pairs of the same cluster: each CTA lays its fp32 accumulators down in its own (idle) shared memory and adds up and stores its share of the
// tokens (rank order: the same bits on every run).
// Forward reads the weight tile as a K-major operand, the input gradient the same bytes as an MN-major operand.
// A ring stage is one step: its token rows and its weight tile in shared memory.
// Forward with one token box (at most 256 tokens per pair): the weights go from the registers into tensor memory instead (32 columns per step), which a
// row operand may be read from, and a stage is two steps, with one wait and one commit for both.  Accumulators take at most 256 of the 512
// columns there, four stages the rest; with two boxes the accumulators need them all.  The row operand in tensor memory is K-major only, so the input
// gradient stays in shared memory.
// Every wait is bounded (see linear_tc.cuh).
//
// Two steps per stage: without loads and dequantization a step took 370 clocks, of which the issuing warp spent 140 in a wait that was satisfied and 170 to
// 210 issuing.  The input gradient has little use for it: over 1900 plans of drawn calls one step per stage takes up to 2 % less time (8 to 10 % with 8-bit codes
// and more than 128 tokens, whose two-step stages are too few), but 2.5 % more with 2-bit codes and up to 64 tokens (4944 x 11968, 18 rows 27.3 / 25.7 us), which
// therefore keep two.
// What every step needs is requested before tensor memory, the code book and the cluster barrier are set up, and arrivals on that barrier are relaxed
// (the initialisation of the mbarriers has a fence of its own): a releasing arrival waited for the scale loads in front of it.
// us as a graph, one step per stage and a set-up in front of the loads / this: 8192 x 8192 NF3, 128 rows 27.6 / 24.6, without a rank-r term (a
// memset in front of the kernel before) 30.9 / 23.2, 28672 x 8192 83.5 / 73.4.
// What bounds it: dequantization, about 450 clocks per step of an SM, of which the pipe of byte permutes and logic is busy 275 (warps started
// out of step, 24 of them with 72 registers, changed nothing or cost time).  A weight tile in shared memory costs its bandwidth twice, when written and when
// read by the tensor core, and with wide codes or many tokens it takes the room of ring stages: when the weights went to tensor memory, 8192 x 8192
// NF3 took 28.0 / 26.7 us at 128 rows and 52.9 / 50.2 at 512, 28672 x 8192 NF3 95.2 / 90.8 at 128 rows (one step per stage; shapes whose grid leaves many
// SMs idle were even).
#pragma once

#include <atomic>
#include <cmath>
#include <type_traits>

namespace lq {
namespace tc {

constexpr int kSwDeqWarps = 16;
constexpr int kSwFirstDeq = 4;                                  // warps 0..3: token boxes, packed codes, MMA
constexpr int kSwThreads = (kSwFirstDeq + kSwDeqWarps) * 32;
constexpr int kSwWBytes = 128 * 128;                            // this CTA's bf16 weight tile of one step
constexpr int kSwMaxStages = 8;
constexpr uint32_t kSwTmemA = 256;                              // first column of the weights in tensor memory (32 per stage)
constexpr int kSwTail = 512;                                    // barriers, tensor-memory slot, abort flag

struct SwapParams {
    QView q;
    __nv_bfloat16* out;
    int* status;
    int M;
    int clear_status;        // without a rank-r term: 1 = this kernel is the first of its call and clears the status word
    int out_cols;            // N (forward) or K (backward)
    int steps_q, steps_d;    // contraction steps with dequantized weights / of the rank-r term
    int c_base;              // first output column of this launch
    const __nv_bfloat16* L1; // forward with the weights in tensor memory: [N][r], read directly
    int r;
    int nbox, box;           // token boxes (1 or 2) and tokens per box (a multiple of 16, at most 256; half of them per CTA)
    int ss, sp;              // stages (of one or two steps) of the token + weight ring and of the packed-code ring
    uint32_t tail_off;       // of the barriers, behind the rings
    uint32_t tmem_cols;
};

// Ring position with a stage count known at run time; advances by up to a few passes.
struct RingAt {
    int s; uint32_t ph;
    __device__ __forceinline__ RingAt(int step, int S) : s(step % S), ph((step / S) & 1) {}
    __device__ __forceinline__ void advance(int n, int S) { s += n; while (s >= S) { s -= S; ph ^= 1u; } }
};

// Shared-memory matrix descriptor as two words: the low one (address, leading offset) advances with the operand, the high
// one (stride offset 1024 bytes, descriptor version, 128-byte swizzle) is constant.
constexpr uint32_t kDescHi = (1024u >> 4) | (1u << 14) | (2u << 29);
__device__ __forceinline__ uint32_t desc_lo(uint32_t saddr, uint32_t lbo_bytes) { return ((saddr & 0x3FFFFu) >> 4) | ((lbo_bytes >> 4) << 16); }
// Commit to the barrier at the same offset in the CTAs of `mask` (cluster ranks).
__device__ __forceinline__ void tc_commit_pair(uint32_t bar, uint16_t mask) {
    asm volatile("tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;"
                 ::"r"(bar), "h"(mask) : "memory");
}
__device__ __forceinline__ void tc_mma2_lo(uint32_t d_tmem, uint32_t a_lo, uint32_t b_lo, uint32_t idesc, uint32_t accumulate) {
    asm volatile(
        "{\n\t.reg .pred p;\n\t.reg .b64 da, db;\n\t"
        "mov.b64 da, {%1, %4};\n\tmov.b64 db, {%2, %4};\n\t"
        "setp.ne.b32 p, %5, 0;\n\t"
        "tcgen05.mma.cta_group::2.kind::f16 [%0], da, db, %3, p;\n\t}"
        ::"r"(d_tmem), "r"(a_lo), "r"(b_lo), "r"(idesc), "r"(kDescHi), "r"(accumulate) : "memory");
}

// The same with the weights in tensor memory (a lane per row, two contraction elements per column).
__device__ __forceinline__ void tc_mma2_ta(uint32_t d_tmem, uint32_t a_tmem, uint32_t b_lo, uint32_t idesc, uint32_t accumulate) {
    asm volatile(
        "{\n\t.reg .pred p;\n\t.reg .b64 db;\n\t"
        "mov.b64 db, {%2, %4};\n\t"
        "setp.ne.b32 p, %5, 0;\n\t"
        "tcgen05.mma.cta_group::2.kind::f16 [%0], [%1], db, %3, p;\n\t}"
        ::"r"(d_tmem), "r"(a_tmem), "r"(b_lo), "r"(idesc), "r"(kDescHi), "r"(accumulate) : "memory");
}
__device__ __forceinline__ void tmem_st16(uint32_t taddr, const uint32_t (&v)[16]) {
    asm volatile(
        "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, %16};"
        ::"r"(taddr), "r"(v[0]), "r"(v[1]), "r"(v[2]), "r"(v[3]), "r"(v[4]), "r"(v[5]), "r"(v[6]), "r"(v[7]),
          "r"(v[8]), "r"(v[9]), "r"(v[10]), "r"(v[11]), "r"(v[12]), "r"(v[13]), "r"(v[14]), "r"(v[15]) : "memory");
}
__device__ __forceinline__ void tmem_st_wait() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }

// The 64 weights of one row of a step.  words0 / words1: shared-memory addresses of the first word of the two 32-column
// groups (the others 128 bytes apart); s[h] = scale of the columns 16 h .. 16 h + 15; nsc = distinct scales (1, 2, 4).
// Chunk o (16 bytes) of the row lives at dst + (16 o ^ xr).
template <int B>
__device__ __forceinline__ void dequant_row64(uint32_t words0, uint32_t words1, const float (&s)[4], int nsc, uint32_t dst, uint32_t xr,
                                              const float* __restrict__ lut8) {
    BlockTable<B == 8 ? 2 : B> tab;
#pragma unroll
    for (int g = 0; g < 2; ++g) {
        uint32_t w[B];
#pragma unroll
        for (int i = 0; i < B; ++i) w[i] = lds_u32((g ? words1 : words0) + i * 128);
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            const int h = 2 * g + (c >> 1);
            const uint32_t x = dst + ((g * 64 + c * 16) ^ xr);
            if constexpr (B == 8) {
                uint32_t packed[4];
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    const uint32_t ww = w[2 * c + (e >> 1)] >> (16 * (e & 1));
                    const float q0 = lut8[(ww & 255u) << 5], q1 = lut8[((ww >> 8) & 255u) << 5];
                    const __nv_bfloat162 hh = __floats2bfloat162_rn(__fmul_rn(q0, s[h]), __fmul_rn(q1, s[h]));
                    packed[e] = *reinterpret_cast<const uint32_t*>(&hh);
                }
                sts_v4(x, packed[0], packed[1], packed[2], packed[3]);
            } else {
                if ((c & 1) == 0 && (h == 0 || nsc == 4 || (nsc == 2 && h == 2))) tab.build(s[h]);
                const uint32_t sel = chunk_selector<B>(w, c);
                uint32_t selA = sel, selB = 0u;
                if constexpr (B == 4) { selA = sel & 0x77777777u; selB = ((sel >> 1) & 0x44444444u) | 0x32103210u; }
                uint32_t o[4];
                tab.lookup4(selA, selB, o[0], o[1]);
                tab.lookup4(selA >> 16, selB >> 16, o[2], o[3]);
                sts_v4(x, o[0], o[1], o[2], o[3]);
            }
        }
    }
}

// The same into 32 columns of tensor memory from `taddr` on (this warp's lanes).
template <int B>
__device__ __forceinline__ void dequant_row64_tmem(uint32_t words0, uint32_t words1, const float (&s)[4], int nsc, uint32_t taddr,
                                                   const float* __restrict__ lut8) {
    BlockTable<B == 8 ? 2 : B> tab;
#pragma unroll
    for (int g = 0; g < 2; ++g) {
        uint32_t w[B], o[16];
#pragma unroll
        for (int i = 0; i < B; ++i) w[i] = lds_u32((g ? words1 : words0) + i * 128);
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            const int h = 2 * g + (c >> 1);
            if constexpr (B == 8) {
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    const uint32_t ww = w[2 * c + (e >> 1)] >> (16 * (e & 1));
                    const __nv_bfloat162 hh = __floats2bfloat162_rn(__fmul_rn(lut8[(ww & 255u) << 5], s[h]), __fmul_rn(lut8[((ww >> 8) & 255u) << 5], s[h]));
                    o[4 * c + e] = *reinterpret_cast<const uint32_t*>(&hh);
                }
            } else {
                if ((c & 1) == 0 && (h == 0 || nsc == 4 || (nsc == 2 && h == 2))) tab.build(s[h]);
                const uint32_t sel = chunk_selector<B>(w, c);
                uint32_t selA = sel, selB = 0u;
                if constexpr (B == 4) { selA = sel & 0x77777777u; selB = ((sel >> 1) & 0x44444444u) | 0x32103210u; }
                tab.lookup4(selA, selB, o[4 * c], o[4 * c + 1]);
                tab.lookup4(selA >> 16, selB >> 16, o[4 * c + 2], o[4 * c + 3]);
            }
        }
        tmem_st16(taddr + 16 * g, o);
    }
}

// The scales of a lane's row of 64 weights for the steps of its warp (every fourth one), requested ahead.
// Input gradient: the row changes with the step, so each step loads its own, two steps ahead.
// Forward: the codes of a row are consecutive bytes.  The lane keeps the aligned 16 bytes that hold its current ones, and the 16 behind them; 16 aligned
// blocks share their second-level scale (B1 >= 16).  (A load per step and lane touches 32 lines each time: without any scale loads 8192 x 8192
// NF3 at 128 rows took 1.4 us less.)
template <bool BWD> struct SwapScales {
    const QView& q;
    uint32_t blk, nblk;              // current block, blocks of the matrix
    int st, st_end;                  // BWD: next step to be requested
    int row;
    bool live;
    RawScale slot[2];                // BWD
    uint4 w0, w1;                    // forward
    float v0, v1;
    __device__ __forceinline__ SwapScales(const QView& q_, int row_, int col, int st_, int st_end_) : q(q_), st(st_), st_end(st_end_), row(row_) {
        live = BWD ? col < q.K : row < q.N;
        nblk = static_cast<uint32_t>(q.N) * q.KB;
        blk = BWD ? static_cast<uint32_t>(col >> q.logB0) : static_cast<uint32_t>(row) * q.KB + (col >> q.logB0);
    }
    __device__ __forceinline__ RawScale fetch() {
        RawScale r{0u, 0.0f};
        const int n = st * BK + row;
        if (live && st < st_end && n < q.N) {
            const uint32_t b = static_cast<uint32_t>(n) * q.KB + blk;
            if (q.logB0 == 4) r.sc = __ldg(reinterpret_cast<const uint32_t*>(q.sc + b));
            else if (q.logB0 == 5) r.sc = __ldg(reinterpret_cast<const uint16_t*>(q.sc + b));
            else r.sc = __ldg(q.sc + b);
            r.v = __ldg(q.v + (b >> q.logB1));
        }
        st += 4;
        return r;
    }
    __device__ __forceinline__ void window(uint32_t b, uint4& w, float& v) {
        w = make_uint4(0u, 0u, 0u, 0u); v = 0.0f;
        b &= ~15u;
        if (!live || b >= nblk) return;
        v = __ldg(q.v + (b >> q.logB1));
        if (b + 16 <= nblk) { w = __ldg(reinterpret_cast<const uint4*>(q.sc + b)); return; }
        uint32_t t[4] = {0u, 0u, 0u, 0u};                // the last blocks of the matrix
#pragma unroll
        for (int i = 0; i < 15; ++i)
            if (b + i < nblk) t[i >> 2] |= static_cast<uint32_t>(__ldg(q.sc + b + i)) << (8 * (i & 3));
        w = make_uint4(t[0], t[1], t[2], t[3]);
    }
    __device__ __forceinline__ void start() {
        if constexpr (BWD) { slot[0] = fetch(); slot[1] = fetch(); }
        else { window(blk, w0, v0); window(blk + 16, w1, v1); }
    }
    // The scale codes of the current step (a byte each, from the lowest on), and on to the next one; u = parity of the step's number.
    __device__ __forceinline__ RawScale next(int u) {
        if constexpr (BWD) {
            const RawScale r = slot[u];
            slot[u] = fetch();
            return r;
        } else {
            const uint32_t word = (blk & 8u) ? ((blk & 4u) ? w0.w : w0.z) : ((blk & 4u) ? w0.y : w0.x);
            const RawScale r{word >> (8 * (blk & 3u)), v0};
            const uint32_t to = blk + (256u >> q.logB0);
            if ((to ^ blk) & ~15u) { w0 = w1; v0 = v1; window(to + 16, w1, v1); }
            blk = to;
            return r;
        }
    }
};

__device__ __forceinline__ void cluster_wait_acquire() { asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory"); }

__device__ __forceinline__ float4 ld_dsmem_f32x4(uint32_t local_addr, uint32_t rank) {
    uint32_t ra;
    float4 v;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(ra) : "r"(local_addr), "r"(rank));
    asm volatile("ld.shared::cluster.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "r"(ra) : "memory");
    return v;
}
__device__ __forceinline__ uint32_t pack_bf16(float a, float b) {
    const __nv_bfloat162 h = __floats2bfloat162_rn(a, b);
    return *reinterpret_cast<const uint32_t*>(&h);
}

template <int B, bool BWD, bool TA, int NBOX, int PS>
__global__ void __launch_bounds__(kSwThreads, 1)
tc_swap_linear_kernel(const __grid_constant__ CUtensorMap tmX, const __grid_constant__ CUtensorMap tmT,
                      const __grid_constant__ CUtensorMap tmF, const SwapParams p) {
    // PS: steps of 64 contraction elements per stage, i.e. per round of waits and commits
    static_assert(PS * NBOX <= 2, "two warps request the boxes of a stage");
    constexpr int P_BYTES = 1024 * B;
    extern __shared__ uint8_t smem_raw[];
    uint8_t* base = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~static_cast<uintptr_t>(1023));
    const int half_box = p.box >> 1, half_bytes = half_box * 128;
    constexpr int kBoxWarps = PS * NBOX;                                 // a warp per token box of a stage (one or two)
    const int x_bytes = NBOX * half_bytes;
    constexpr int W_BYTES = TA ? 0 : kSwWBytes;
    const int step_bytes = W_BYTES + x_bytes;                            // [weight tile][token boxes] of a step; a stage is PS of them
    uint8_t* p_ring = base + p.ss * PS * step_bytes;
    uint8_t* tail = base + p.tail_off;
    uint64_t* bars = reinterpret_cast<uint64_t*>(tail);     // full[8], empty[8], full_p[8], empty_p[8], fbar[2], acc_full, drain
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(tail + 36 * 8);
    volatile int* abort_s = reinterpret_cast<volatile int*>(tmem_slot + 1);
    int* reached = reinterpret_cast<int*>(tmem_slot + 2);    // [20] per warp: the first stage (from 0 on, ring passes counted) that it has not (issued or) arrived at
    float* lut8 = reinterpret_cast<float*>(tail + kSwTail);

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t rank = cluster_rank() & 1u;                           // CTA of the pair; 0 = leader
    const int c0 = p.c_base + blockIdx.x * 128;                          // first output column of this CTA
    const int m0 = blockIdx.y * (NBOX * p.box);                          // first token
    const int nsplit = gridDim.z, split = blockIdx.z;
    const int q_lo = static_cast<int>(static_cast<long long>(p.steps_q) * split / nsplit);
    const int nq = static_cast<int>(static_cast<long long>(p.steps_q) * (split + 1) / nsplit) - q_lo;
    const int total = nq + (split == 0 ? p.steps_d : 0);                 // the rank-r steps go to the first slice
    const int rounds = (total + PS - 1) / PS;                            // stages of the slice; the last one may hold one step of two
    const int have = min(2, max(0, (p.out_cols - c0 + 63) >> 6));        // 64-column tiles of this CTA that exist
    const Ctl ctl{abort_s, p.status};

    const uint32_t ring = smem_u32(base), bar0 = smem_u32(bars);
    auto full = [&](int s) { return bar0 + 8 * s; };                     // the step's operands (leader: of both CTAs)
    auto empty = [&](int s) { return bar0 + 64 + 8 * s; };
    auto full_p = [&](int s) { return bar0 + 128 + 8 * s; };
    auto empty_p = [&](int s) { return bar0 + 192 + 8 * s; };
    auto fbar = [&](int d) { return bar0 + 256 + 8 * d; };
    const uint32_t acc_full = bar0 + 272, drain = bar0 + 280;

    // This CTA's half of token box w of a stage (PS = 1), or of the token box of its step w.  By one lane.
    auto issue_box = [&](int w, int round, int stage) {
        const int step = PS == 1 ? round : 2 * round + w;
        const int row = m0 + (PS == 1 ? w * p.box : 0) + static_cast<int>(rank) * half_box;
        const uint32_t dst = ring + W_BYTES + w * (PS == 1 ? half_bytes : step_bytes) + stage * (PS * step_bytes);
        if (step >= total) {
            mbar_arrive(full(stage));                     // the second step of the last stage does not exist
        } else {
            mbar_expect_tx(full(stage), half_bytes);
            if (step < nq) tma_load_2d(dst, &tmX, (q_lo + step) * BK, row, full(stage));
            else tma_load_2d(dst, &tmT, (step - nq) * BK, row, full(stage));
        }
    };
    // The packed codes of a stage.
    auto issue_codes = [&](int round, int stage) {
        const uint8_t* codes = reinterpret_cast<const uint8_t*>(p.q.codes);
        const uint32_t dst = smem_u32(p_ring) + stage * (PS * P_BYTES), bar = full_p(stage);
        const int qs = q_lo + round * PS;
        const bool two = PS == 2 && round * PS + 1 < nq;
        if (have == 0) {
            mbar_arrive(bar);                             // nothing behind the last column: the scales are zero
        } else if (!BWD) {
            // one tile, or two neighbouring ones
            const uint32_t bytes = two ? 2 * P_BYTES : P_BYTES;
            mbar_expect_tx(bar, bytes);
            bulk_load(dst, codes + (static_cast<size_t>(c0 >> 7) * p.q.ktiles + qs) * P_BYTES, bytes, bar);
        } else {
            // 64 rows (half a tile) of the two 64-column tiles of this CTA, for each step
            mbar_expect_tx(bar, (two ? 2 : 1) * have * (P_BYTES / 2));
#pragma unroll
            for (int h = 0; h < PS; ++h) {
                if (h == 1 && !two) break;
                const uint8_t* src = codes + (static_cast<size_t>((qs + h) >> 1) * p.q.ktiles + (c0 >> 6)) * P_BYTES + ((qs + h) & 1) * (P_BYTES / 2);
                for (int t = 0; t < have; ++t) bulk_load(dst + h * P_BYTES + t * (P_BYTES / 2), src + t * P_BYTES, P_BYTES / 2, bar);
            }
        }
    };

    // Dequantization warps: four per step, warp = steps grp, grp + 4, ...  Forward: row c0 + 32 wi + lane of the tile; backward: contraction row
    // 32 (wi & 1) + lane, 64-column tile wi >> 1.
    const int dw = warp - kSwFirstDeq, grp = (dw >> 2) & 3, wi = dw & 3;
    const int half = PS == 2 ? grp & 1 : 0;               // which step of its stage
    const int row_local = BWD ? (wi & 1) * 32 + lane : wi * 32 + lane;
    SwapScales<BWD> scales(p.q, BWD ? row_local : c0 + row_local, BWD ? c0 + (wi >> 1) * 64 : (q_lo + grp) * BK, BWD ? q_lo + grp : 0, q_lo + nq);

    // Everything that a step needs is requested first; what follows (tensor memory, the code book, the barrier of the cluster) takes about
    // as long as those requests.  Only arrivals on the other CTA's barriers have to wait for the cluster.
    // (Without a rank-r term this is the first kernel of its call, launched while the one in front ends: it waits for that one before it reads.  With one, the
    // pre-product has waited, fence included, before it let this kernel start.)
    const bool lead = p.steps_d == 0;
    const int early_x = min(p.ss, nq / PS), early_p = min(p.sp, (nq + PS - 1) / PS);
    if (warp < 2) {
        if (warp == 0 && elect_one()) {
            for (int s = 0; s < kSwMaxStages; ++s) {
                // the token boxes and four dequantization warps per step; leader: also the word of the second
                // CTA that its stage is complete
                mbar_init(full(s), kBoxWarps + 4 * PS + (rank == 0 ? 1 : 0));
                mbar_init(empty(s), 1);
            }
            mbar_init(fbar(0), 1);
            mbar_init(fbar(1), 1);
            mbar_init(acc_full, 1);
            mbar_init(drain, 1);
            *abort_s = 0;
            fence_barrier_init();
            fence_proxy_async();
        }
        __syncwarp();
        asm volatile("bar.sync 1, 64;" ::: "memory");
        if (lead) pdl_wait_for_copies();
        if (warp < kBoxWarps && elect_one()) {
            for (int i = 0; i < early_x; ++i) issue_box(warp, i, i);
        }
        __syncwarp();
    } else if (warp == 2) {
        if (elect_one()) {
            for (int s = 0; s < kSwMaxStages; ++s) {
                mbar_init(full_p(s), 1);
                mbar_init(empty_p(s), 4 * PS);
            }
            fence_barrier_init();
            fence_proxy_async();
            if (lead) pdl_wait_for_copies();
            for (int i = 0; i < early_p; ++i) issue_codes(i, i);
        }
        __syncwarp();
    } else if (warp == 3) {
        tmem_alloc2(smem_u32(tmem_slot), p.tmem_cols);
        tmem_relinquish2();
    } else if (warp >= kSwFirstDeq) {
        if (lead) {
            pdl_wait();
            if (p.clear_status && dw == 0 && lane == 0 && blockIdx.x == 0 && blockIdx.y == 0 && blockIdx.z == 0) *p.status = 0;
        }
        scales.start();
        if constexpr (B == 8) {
            for (int i = threadIdx.x - kSwFirstDeq * 32; i < 256 * 32; i += kSwDeqWarps * 32) lut8[i] = c_codebook[3][i >> 5];     // one copy per bank
        }
    }
    tc_fence_before();
    __syncthreads();
    // The barriers and tensor memory of this CTA are ready.  The threads that initialised the barriers have passed fence.mbarrier_init; a
    // releasing arrival would make every warp wait for its scales here first (1700 clocks when they come from DRAM).
    dec::cluster_arrive_relaxed();
    if (warp == 3) cluster_wait_acquire();                // (the others wait behind their loops)
    tc_fence_after();
    const uint32_t tmem = *tmem_slot;
    bool acc_ok = false;
    int issued = early_p;         // stages whose codes have been requested (warp 2)

    if (warp < kBoxWarps) {
        // ------------------------------------------------------------------ token boxes
        RingAt r(early_x, p.ss);
        int round = early_x;
        for (; round < rounds; ++round, r.advance(1, p.ss)) {
            if (!wait(empty(r.s), r.ph ^ 1, ctl, 51)) break;
            const int step = PS == 1 ? round : 2 * round + warp;
            if (step >= nq && step < nq + PS && step < total) {
                // the rank-r intermediate comes from the kernel in front (programmatic dependent launch)
                pdl_wait_for_copies();
            }
            __syncwarp();
            if (elect_one()) issue_box(warp, round, r.s);
            __syncwarp();
        }
        if (lane == 0) reached[warp] = round;
    } else if (warp == 2) {
        // ------------------------------------------------------------------ packed codes
        RingAt r(early_p, p.sp);
        for (int round = early_p; round * PS < nq; ++round, r.advance(1, p.sp)) {
            if (!wait(empty_p(r.s), r.ph ^ 1, ctl, 52)) break;
            __syncwarp();
            if (elect_one()) issue_codes(round, r.s);
            __syncwarp();
            issued = round + 1;
        }
    } else if (warp == 3) {
        // ------------------------------------------------------------------ MMA issuer (leader), messenger (second CTA)
        if (rank == 1) {
            // tells the leader that this CTA's half of a stage is complete
            RingAt r(0, p.ss);
            int round = 0;
            for (; round < rounds; ++round, r.advance(1, p.ss)) {
                if (!wait(full(r.s), r.ph, ctl, 60)) break;
                __syncwarp();
                if (elect_one()) mbar_arrive_cluster(full(r.s), cluster_rank() & ~1u);
            }
            if (lane == 0) dec::st_dsmem_f32(smem_u32(reached + 3), cluster_rank() & ~1u, __int_as_float(round));    // to the leader
        } else {
            const uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((BWD ? 1u : 0u) << 15) |
                                   (static_cast<uint32_t>(p.box >> 3) << 17) | (static_cast<uint32_t>(256 >> 4) << 24);
            const uint32_t a0 = desc_lo(ring, BWD ? 8192 : 16), b0 = desc_lo(ring + W_BYTES, 16);
            const uint32_t step16 = step_bytes >> 4, box16 = half_bytes >> 4;
            constexpr uint32_t ka = (BWD ? 2048 : 32) >> 4;            // 16 contraction elements further: rows down, or columns along
            const uint16_t pair_mask = static_cast<uint16_t>(3u << (cluster_rank() & ~1u));
            bool ok = true;
            uint32_t acc = 0;
            RingAt r(0, p.ss);
            for (int round = 0; round < rounds; ++round, r.advance(1, p.ss)) {
                ok = wait_cluster(full(r.s), r.ph, ctl, 53);
                if (!ok) break;
                __syncwarp();
                tc_fence_after();
                const bool two = PS == 2 && 2 * round + 1 < total;
                if (elect_one()) {
#pragma unroll
                    for (int h = 0; h < PS; ++h) {
                        if (h == 1 && !two) break;
                        const uint32_t slot = r.s * PS + h, b = b0 + slot * step16, keep = h == 0 ? acc : 1u;
                        if (TA) {
                            const uint32_t at = tmem + kSwTmemA + slot * 32;
                            tc_mma2_ta(tmem, at, b, idesc, keep);
                            tc_mma2_ta(tmem, at + 8, b + 2, idesc, 1u);
                            tc_mma2_ta(tmem, at + 16, b + 4, idesc, 1u);
                            tc_mma2_ta(tmem, at + 24, b + 6, idesc, 1u);
                        } else {
                            const uint32_t a = a0 + slot * step16;
                            tc_mma2_lo(tmem, a, b, idesc, keep);
                            tc_mma2_lo(tmem, a + ka, b + 2, idesc, 1u);
                            tc_mma2_lo(tmem, a + 2 * ka, b + 4, idesc, 1u);
                            tc_mma2_lo(tmem, a + 3 * ka, b + 6, idesc, 1u);
                            if (NBOX == 2) {
                                const uint32_t b2 = b + box16;
                                tc_mma2_lo(tmem + 256, a, b2, idesc, keep);
                                tc_mma2_lo(tmem + 256, a + ka, b2 + 2, idesc, 1u);
                                tc_mma2_lo(tmem + 256, a + 2 * ka, b2 + 4, idesc, 1u);
                                tc_mma2_lo(tmem + 256, a + 3 * ka, b2 + 6, idesc, 1u);
                            }
                        }
                    }
                    tc_commit_pair(round + 1 < rounds ? empty(r.s) : acc_full, pair_mask);
                }
                acc = 1u;
                __syncwarp();
            }
            if (!ok) {
                __syncwarp();
                if (elect_one()) tc_commit_pair(drain, pair_mask);      // wait (bounded) for issued MMAs before tensor memory is freed
                const long long t0 = clock64();
                while (!mbar_try_wait(drain, 0) && clock64() - t0 < 20000000LL) {}
            }
        }
        __syncwarp();
    } else if (warp >= kSwFirstDeq) {
        // ------------------------------------------------------------------ dequantization
        const QView& q = p.q;
        const int my_col = BWD ? c0 + (wi >> 1) * 64 : 0;
        const uint32_t dst0 = ring + half * step_bytes + (BWD ? (wi >> 1) * 8192 : 0) + row_local * 128;
        const uint32_t xr = (row_local & 7) << 4;
        const uint32_t wsrc = smem_u32(p_ring) + half * P_BYTES + (BWD ? (wi >> 1) * (128 * B) + (wi & 1) * (64 * B) : wi * (64 * B)) * 4;
        const int nsc = q.B0 == 16 ? 4 : q.B0 == 32 ? 2 : 1;
        float v_cached = -1.0f, sigma = 0.0f;
        RingAt rw(grp / PS, p.ss), rp(grp / PS, p.sp);
        bool ok = true;
        int next = grp / PS;
        for (int step8 = grp; step8 < rounds * PS && ok; step8 += 8) {
#pragma unroll
            for (int u = 0; u < 2; ++u) {
                const int step = step8 + 4 * u;
                if (step >= rounds * PS || !ok) break;
                const uint32_t stage = rw.s * (PS * step_bytes);
                if (step < nq) {
                    const RawScale rs = scales.next(u);
                    if (rs.v != v_cached) { v_cached = rs.v; sigma = __fdiv_rn(rs.v, q.levels); }
                    float s[4];
                    s[0] = __fmul_rn(static_cast<float>(rs.sc & 255u), sigma);
                    s[1] = s[0]; s[2] = s[0]; s[3] = s[0];
                    if (nsc == 2) { s[2] = __fmul_rn(static_cast<float>((rs.sc >> 8) & 255u), sigma); s[3] = s[2]; }
                    if (nsc == 4) {
                        s[1] = __fmul_rn(static_cast<float>((rs.sc >> 8) & 255u), sigma);
                        s[2] = __fmul_rn(static_cast<float>((rs.sc >> 16) & 255u), sigma);
                        s[3] = __fmul_rn(static_cast<float>(rs.sc >> 24), sigma);
                    }
                    const int kt = BWD ? (my_col >> 6) : q_lo + step;
                    const uint32_t src = wsrc + rp.s * (PS * P_BYTES);
                    ok = wait2(empty(rw.s), rw.ph ^ 1, full_p(rp.s), rp.ph, ctl, 55, 56);
                    if (!ok) break;
                    if constexpr (TA) {
                        tc_fence_after();               // the tensor core is done with this stage's columns
                        dequant_row64_tmem<B>(src + slab_row_slot(lane, 0, kt) * 4, src + (B * 32 + slab_row_slot(lane, 1, kt)) * 4, s, nsc,
                                              tmem + (static_cast<uint32_t>(wi * 32) << 16) + kSwTmemA + (rw.s * PS + half) * 32, lut8 + lane);
                        tmem_st_wait();
                        tc_fence_before();
                    } else {
                        dequant_row64<B>(src + slab_row_slot(lane, 0, kt) * 4, src + (B * 32 + slab_row_slot(lane, 1, kt)) * 4, s, nsc,
                                         dst0 + stage, xr, lut8 + lane);
                        fence_proxy_async();            // make the generic-proxy stores visible to the tensor core
                    }
                    __syncwarp();
                    if (lane == 0) mbar_arrive(empty_p(rp.s));
                    rp.advance(4 / PS, p.sp);
                } else if (step >= total) {
                    ok = wait(empty(rw.s), rw.ph ^ 1, ctl, 57);      // the second step of the last stage does not exist
                    if (!ok) break;
                } else {
                    // rank-r step: the weight-side operand is rows of L1 (forward) or L2; by TMA where it goes to shared memory
                    ok = wait(empty(rw.s), rw.ph ^ 1, ctl, 57);
                    if (!ok) break;
                    if constexpr (TA) {
                        // this lane's row of L1, straight from global memory (r is a multiple of 16)
                        tc_fence_after();
                        const int n = c0 + row_local, j0 = (step - nq) * BK;
#pragma unroll
                        for (int g = 0; g < 2; ++g) {
                            uint32_t o[16];
#pragma unroll
                            for (int c = 0; c < 4; ++c) {
                                const int j = j0 + g * 32 + c * 8;
                                uint4 v = make_uint4(0u, 0u, 0u, 0u);
                                if (n < q.N && j < p.r) v = __ldg(reinterpret_cast<const uint4*>(p.L1 + static_cast<size_t>(n) * p.r + j));
                                o[4 * c] = v.x; o[4 * c + 1] = v.y; o[4 * c + 2] = v.z; o[4 * c + 3] = v.w;
                            }
                            tmem_st16(tmem + (static_cast<uint32_t>(wi * 32) << 16) + kSwTmemA + (rw.s * PS + half) * 32 + 16 * g, o);
                        }
                        tmem_st_wait();
                        tc_fence_before();
                    } else if (wi == 0) {
                        const int d = step - nq;
                        if (lane == 0) {
                            if (!BWD) {
                                mbar_expect_tx(fbar(d), kSwWBytes);
                                tma_load_2d(ring + half * step_bytes + stage, &tmF, d * BK, c0, fbar(d));
                            } else {
                                mbar_expect_tx(fbar(d), have * 8192);
                                for (int t = 0; t < have; ++t) tma_load_2d(ring + half * step_bytes + stage + t * 8192, &tmF, c0 + t * 64, d * BK, fbar(d));
                            }
                        }
                        ok = wait(fbar(d), 0, ctl, 59);
                        if (!ok) { let_land(fbar(d), 0); break; }
                    }
                    __syncwarp();
                }
                if (lane == 0) mbar_arrive(full(rw.s));
                next = step / PS + 4 / PS;
                rw.advance(4 / PS, p.ss);
            }
        }
        if (lane == 0) reached[warp] = next;
        // ------------------------------------------------------------------ epilogue: warp = 32 output columns x every fourth chunk of 32 tokens
        pdl_launch_dependents();      // the next call's pre-product may take its place on the SMs (it waits for this kernel)
        acc_ok = ok && wait(acc_full, 0, ctl, 58);
        if (acc_ok) {
            tc_fence_after();
            const int quarter = warp & 3, chunks = (p.box + 31) >> 5;
            float* accbuf = reinterpret_cast<float*>(base);           // [token][128 columns], over the idle rings
            for (int ch = dw >> 2; ch < NBOX * chunks; ch += 4) {
                const int h = ch / chunks, t0 = (ch - h * chunks) * 32;
                uint32_t v[32];
                tmem_ld32(tmem + (static_cast<uint32_t>(quarter * 32) << 16) + h * 256 + t0, v);
                tmem_ld_wait();
                if (nsplit > 1) {
                    float* dst = accbuf + static_cast<size_t>(h * p.box + t0) * 128 + quarter * 32 + lane;
#pragma unroll
                    for (int i = 0; i < 32; ++i)
                        if (t0 + i < p.box) dst[i * 128] = __uint_as_float(v[i]);
                } else {
                    // even lanes store columns (n, n + 1) of the even tokens, odd lanes those of the odd tokens
                    const int n = c0 + quarter * 32 + (lane & ~1);
                    const int odd = lane & 1;
#pragma unroll
                    for (int i = 0; i < 16; ++i) {
                        const float a = __uint_as_float(v[2 * i]), b = __uint_as_float(v[2 * i + 1]);
                        const float other = __shfl_xor_sync(0xffffffffu, odd ? a : b, 1);
                        const uint32_t w = odd ? pack_bf16(other, b) : pack_bf16(a, other);
                        const int t = t0 + 2 * i + odd, m = m0 + h * p.box + t;
                        if (t < p.box && m < p.M && n < p.out_cols)
                            *reinterpret_cast<uint32_t*>(p.out + static_cast<size_t>(m) * p.out_cols + n) = w;
                    }
                }
            }
        }
    }
    if (warp != 3) { __syncwarp(); cluster_wait_acquire(); }
    if (nsplit > 1) {
        // every CTA adds up and stores its share of the tokens from the CTAs with the same columns; the barriers are executed
        // by all threads of all CTAs, whatever happened before
        const uint32_t acc_addr = ring;
        const int tokens = NBOX * p.box;
        const int t_lo = tokens * split / nsplit, t_hi = tokens * (split + 1) / nsplit;
        __syncthreads();
        cluster_barrier();
        // four items of four columns at a time: one round trip through the cluster for most calls
        const int items = (min(t_hi, p.M - m0) - t_lo) * 32;
        for (int item0 = threadIdx.x; item0 < items; item0 += 4 * kSwThreads) {
            float4 part[4][4];
#pragma unroll
            for (int u = 0; u < 4; ++u)
#pragma unroll
                for (int z = 0; z < 4; ++z) {
                    const int item = item0 + u * kSwThreads;
                    if (z < nsplit && item < items)
                        part[u][z] = ld_dsmem_f32x4(acc_addr + static_cast<uint32_t>((t_lo + (item >> 5)) * 128 + (item & 31) * 4) * 4u, rank + 2 * z);
                }
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int item = item0 + u * kSwThreads, cg = (item & 31) * 4;
                if (item >= items || c0 + cg >= p.out_cols) continue;
                float4 sum = part[u][0];
#pragma unroll
                for (int z = 1; z < 4; ++z)
                    if (z < nsplit) { sum.x += part[u][z].x; sum.y += part[u][z].y; sum.z += part[u][z].z; sum.w += part[u][z].w; }
                *reinterpret_cast<uint2*>(p.out + static_cast<size_t>(m0 + t_lo + (item >> 5)) * p.out_cols + c0 + cg) = make_uint2(pack_bf16(sum.x, sum.y), pack_bf16(sum.z, sum.w));
            }
        }
    }
    tc_fence_before();
    __syncthreads();
    cluster_barrier();            // tensor and shared memory are released only when no CTA of the cluster uses them any more
    if (*abort_s) {
        // copies in flight land before the CTA exits.  The barrier of a stage counts its token boxes, the warps of its weights and
        // the second CTA's word: those that have not come will not (everybody has left the loops), so they are made up for here, and
        // the phase then waits for the boxes alone.  A box of stage j is issued behind the end of stage j - ss, so the last ss stages
        // that any box was issued for are the ones that can be open, each in the phase j / ss of its place in the ring.
        if (warp == 0) {
            const int top = kBoxWarps == 2 ? max(reached[0], reached[1]) : reached[0];
            for (int j = max(0, top - p.ss); j < top; ++j) {
                int missing = (j >= reached[0] ? 1 : 0) + (kBoxWarps == 2 && j >= reached[1] ? 1 : 0) + (rank == 0 && j >= reached[3] ? 1 : 0);
                for (int w = 0; w < 4 * PS; ++w) missing += (j >= reached[kSwFirstDeq + 4 * PS * (j & (4 / PS - 1)) + w] ? 1 : 0);
                if (lane < missing) mbar_arrive(full(j % p.ss));
                let_land(full(j % p.ss), (j / p.ss) & 1);
            }
        } else if (warp == 2) {
            drain_ring(full_p(0), issued, p.sp);
        }
    }
    if (warp == 3) tmem_dealloc2(tmem, p.tmem_cols);
}

// ------------------------------------------------------------------------------------ host side
// Clusters of `n` CTAs (one CTA per SM, all of its shared memory) that can be resident at the same time.  A cluster lives
// inside one GPC, so fewer fit than SMs / n: 15 clusters of eight on a B200, not 18.  Asked once per cluster size; what the
// driver answered on a B200 (74, 33, 22, 15) stands in when there is no device to ask.
inline int tc_max_clusters(int n) {
    static std::atomic<int> cached[4] = {-1, -1, -1, -1};       // n = 2, 4, 6, 8 (threads that ask at the same time get the same answer)
    const int idx = n / 2 - 1;
    const int known = cached[idx].load(std::memory_order_relaxed);
    if (known >= 0) return known;
    const int fallback[4] = {74, 33, 22, 15};
    int got = 0;
    auto kern = tc_swap_linear_kernel<3, false, false, 2, 1>;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(2, 1, n / 2);
    cfg.blockDim = dim3(kSwThreads);
    cfg.dynamicSmemBytes = kSmemLimit;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = 2; attr[0].val.clusterDim.y = 1; attr[0].val.clusterDim.z = n / 2;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemLimit) != cudaSuccess ||
        cudaOccupancyMaxActiveClusters(&got, kern, &cfg) != cudaSuccess || got <= 0) {
        cudaGetLastError();
        got = fallback[idx];
    }
    cached[idx].store(got, std::memory_order_relaxed);
    return got;
}

struct SwapPlan {
    int chunks, nbox, box, ks;       // token chunks, boxes and tokens per box, slices of the contraction
    int ps;                          // steps per stage
    int ss, sp, smem;
    uint32_t tmem_cols;
    long long ctas;
    double us;                       // estimated time
};

// Steps per stage: two where the weights go to tensor memory, and in 2-bit input gradients of few tokens (see the top of the file).
inline int swap_stage_steps(int b0, bool backward, int nbox, int box) { return nbox == 1 && (!backward || (b0 == 2 && box <= 64)) ? 2 : 1; }

// Ring depths of a plan in stages; false when they do not fit.  A barrier tells only the parity of its phase, so nobody may wait for a phase while the
// one before it can be incomplete.  A dequantization warp works on every fourth step, i.e. on every g-th stage, g = 4 (one step per stage) or 2:
//   - it may wait for stage j % ss to be free (the tensor core is done with stage j - ss) once stage j - 2 ss is known to be
//     done; its own stage j - g waited for j - g - ss, hence ss >= g;
//   - it may wait for the codes of stage j once those of stage j - sp are known to have landed: they have where its own
//     group used them (sp a multiple of g) or where the tensor core is done with that stage (sp >= ss).
// (With the weights in tensor memory the kernel takes depths of its own, see run_swap; what fits here with one step per stage fits there.)
// As many stages of weights as fit beside g of codes, then codes.  Fewer stages of weights for as many of codes took more shared memory, which the
// scales miss in L1: 10112 x 15616 input gradient, 8-bit codes in blocks of 16, 17 rows, 95 us with 8 and 4 stages, 113 with 7 and 8.
inline bool swap_rings(int b0, bool backward, int ks, SwapPlan& pl) {
    const int steps = backward ? pl.ps : 1, g = 4 / steps;
    const int stage = steps * (kSwWBytes + pl.nbox * pl.box * 64), pk = steps * 1024 * b0;
    const int fixed = 1024 + kSwTail + (b0 == 8 ? 32768 : 0);
    const int room = kSmemLimit - fixed;
    pl.ss = (room - g * pk) / stage;
    if (pl.ss > kSwMaxStages / steps) pl.ss = kSwMaxStages / steps;
    if (pl.ss < g) return false;
    pl.sp = (room - pl.ss * stage) / pk;
    if (pl.sp > kSwMaxStages) pl.sp = kSwMaxStages;
    if (pl.sp < pl.ss) pl.sp = g;
    const int bytes = pl.ss * stage + pl.sp * pk;
    if (ks > 1 && pl.nbox * pl.box * 512 > bytes) return false;      // the accumulators are laid over the rings
    pl.smem = fixed + bytes;
    return true;
}

// Tokens of the largest chunk whose rings fit: 512, and 384 for 8-bit codes (their code book takes 32 KB of shared memory).
inline int swap_max_tokens(int b0) {
    SwapPlan pl{};
    pl.nbox = 2; pl.ps = 1;
    for (pl.box = 256; pl.box > 16 && !swap_rings(b0, true, 1, pl); pl.box -= 16) {}
    return 2 * pl.box;
}

// Splits of the contraction of a rank-r pre-product with `mtiles` row tiles and `steps` steps of 64 that runs beside a linear kernel of
// `main_ctas` CTAs (programmatic dependent launch): it gets the SMs that the last wave of that kernel leaves idle, and at least one CTA per row
// tile.  A power of two: it divides the 64 columns of the accumulator.
inline int pre_splits(int mtiles, int steps, long long main_ctas) {
    const int sms = dec::sm_count_cached(), idle = static_cast<int>((sms - main_ctas % sms) % sms);
    int want = idle / mtiles;
    if (main_ctas < sms) want = idle / 2 / mtiles;      // beside a single wave of clusters: half of what it leaves (clusters need room)
    if (want > steps / 4) want = steps / 4;
    if (want > 8) want = 8;          // splits of a tile form a cluster (and more than eight made the sum the critical path)
    if (idle < 48) {
        // beside a nearly full linear kernel (itself made of clusters) large pre-product clusters took a cluster's place from it
        const int cap = (idle / mtiles < 4) ? (idle / mtiles > 1 ? idle / mtiles : 1) : 4;
        if (want > cap) want = cap;
    }
    if (want < 1) want = 1;
    while (want & (want - 1)) want &= want - 1;
    // Not two splits of more than 37 row tiles: a graph of calls with 65 of them (130 CTAs in clusters of two) before 40 clusters of four of the linear kernel
    // ended in a launch failure, and neither reading nor checks of ring positions, copies, loads and accumulator addresses in the kernels showed why.
    if (want == 2 && mtiles > 37) want = 1;
    return want;
}

// Clusters of a linear kernel (`ks` pairs each) that a rank-r pre-product beside it, `mtiles` row tiles of `w` CTAs, keeps out of their GPCs while
// it runs.  Read off from the timings (the number of free clusters below which a call takes a second wave): single CTAs fill TPCs together, but an
// odd number of up to 13 holds a TPC each; beside larger clusters a GPC has a few SMs to spare, which small ones take first.
inline int clusters_kept_out(int ks, int mtiles, int w) {
    const bool odd = mtiles & 1;
    const int tpcs = w > 1 ? mtiles * w / 2 : odd ? mtiles : mtiles / 2;
    if (ks == 1) return w == 1 && mtiles >= 15 ? mtiles / 2 + (odd ? 2 : 0) : tpcs;
    if (ks == 2) return w >= 4 ? tpcs / 2 : w == 1 && odd && mtiles < 17 ? (mtiles < 11 ? 0 : 2) : tpcs > 8 ? (tpcs - 7) / 2 : 0;
    if (ks == 3) return w == 8 ? 0 : w == 4 ? mtiles - 1 : w == 2 ? (mtiles > 4 ? mtiles - 4 : 0) : mtiles < 7 ? 0 : odd ? (mtiles - 5) / 2 : mtiles < 14 ? 0 : mtiles < 18 ? 3 : tpcs - 5;
    return w == 4 ? mtiles : w == 8 ? 0 : tpcs > 10 ? 7 : 0;          // (a cluster of eight per GPC in place of two)
}
// Time until `n` clusters of `first` us have run in `slots` places, `late` of which are free only after `at` us; clusters that follow another one in
// its place take `next` us.
inline double makespan(long long n, double first, double next, long long slots, long long late, double at) {
    long long rounds = n / slots - 2 - static_cast<long long>(at / next);      // that all places have behind them in any case
    if (rounds < 0) rounds = 0;
    double t_early = first + static_cast<double>(rounds) * next, t_late = t_early + at;
    for (long long done = rounds * slots;;) {
        const bool early = late == 0 || t_early <= t_late;
        double& t = early ? t_early : t_late;
        done += early ? slots - late : late;
        if (done >= n) return t;
        t += next;
    }
}

// The split of a call that costs least by a simple model: places for clusters, each cluster with a fixed cost, its steps (the slower of
// dequantization and tensor core, softened; slower with more SMs at work) and its reduction; the pre-product, which keeps places occupied at first and is
// waited for at the end.  Fitted to the timings of all plausible chunk counts and slices of 2400 drawn calls (2 to 8 bits, 9 to 2000 rows, with and
// without a rank-r term); on 1200 others the plan that it picks takes 0.4 % longer than the best one on average, and more than a tenth longer in 12 of
// them.  (The model before counted whole waves and took one slice 15 % dearer than estimated: 1.5 %, and 62.  us as a graph, its plan / this one: 13848 x 4224
// NF4, 601 rows 99.8 / 68; 4784 x 21120 NF8, 445 rows 182 / 142; 9216 x 16896 NF4 input gradient, 19 rows 84 / 63; 2688 x 2304 NF2, 283 rows 17.4 / 14.1.)
inline SwapPlan make_swap_plan(int b0, int B0, bool backward, int64_t M, int64_t out_cols, int steps_q, int steps_d, bool beside_pre) {
    SwapPlan best{};
    best.us = -1.0;
    double best_score = 0.0;
    // us per step of 128 x 64 weights: through tensor memory; input gradient, one box; two boxes forward, input gradient.  Small blocks cost more tables.
    static const double dq_us[4][4] = {{0.212, 0.23, 0.329, 0.478}, {0.242, 0.258, 0.338, 0.497}, {0.233, 0.256, 0.32, 0.511}, {0.25, 0.271, 0.317, 0.507}};
    static const double red_us[3] = {0.021, 0.0235, 0.025};          // sum over two, three, four slices, per token
    const long long pairs = (out_cols + 255) / 256;
    const int mtiles = static_cast<int>((M + 127) / 128);
    int first = static_cast<int>((M + 511) / 512);
    // The search covers eight numbers of chunks.  Where the chunks of all of them are too large for the rings (8-bit codes
    // above 11136 rows), it starts at the fewest that are not: a plan exists for every number of rows.
    const int tokens_max = swap_max_tokens(b0), fit = static_cast<int>((M + tokens_max - 1) / tokens_max);
    if (fit > first + 7) first = fit;
    for (int ch = first; ch <= first + 7; ++ch) {
        SwapPlan pl{};
        const int per = static_cast<int>((M + ch - 1) / ch);
        if (ch > first && per < 32) break;
        pl.nbox = per > 256 ? 2 : 1;
        pl.box = ((per + pl.nbox - 1) / pl.nbox + 15) / 16 * 16;
        pl.ps = swap_stage_steps(b0, backward, pl.nbox, pl.box);
        const int tokens = pl.nbox * pl.box;
        pl.chunks = static_cast<int>((M + tokens - 1) / tokens);
        pl.tmem_cols = 32;
        while (static_cast<int>(pl.tmem_cols) < (pl.nbox == 2 ? 512 : pl.box)) pl.tmem_cols *= 2;
        const bool ta = !backward && pl.nbox == 1;
        const double block = B0 == 16 ? (ta ? 1.17 : 1.12) : B0 == 32 ? (ta ? 1.05 : 1.04) : 1.0;
        const double dq = block * dq_us[2 * (pl.nbox - 1) + (backward ? 1 : 0)][bits_index(b0)], mma = (pl.nbox == 1 ? 0.00085 : 0.00097) * tokens;
        for (int ks = 1; ks <= 4 && ks <= steps_q; ++ks) {
            if (!swap_rings(b0, backward, ks, pl)) continue;
            pl.ks = ks;
            const long long n = pairs * pl.chunks, slots = tc_max_clusters(2 * ks);
            pl.ctas = 2 * n * ks;
            const double busy = static_cast<double>(2 * ks * (n < slots ? n : slots)) / dec::sm_count_cached();
            const double step = std::sqrt(std::sqrt(dq * dq * dq * dq + mma * mma * mma * mma)) * (1.0 + (beside_pre ? 0.155 : 0.22) * busy);
            const double sum = ks == 1 ? 0.013 * tokens : 0.6 + red_us[ks - 2] * tokens;
            const double body = (beside_pre ? 5.6 : 4.2) + ((steps_q + ks - 1) / ks + steps_d) * step + sum;
            double pre = 0.0, tail = 0.0;
            long long late = 0;
            if (beside_pre) {
                const int w = pre_splits(mtiles, steps_q, pl.ctas);
                late = clusters_kept_out(ks, mtiles, w);
                if (late > slots - 1) late = slots - 1;
                pre = 0.245 * ((steps_q + w - 1) / w) + 0.12 * mtiles - (w > 1 ? 0.5 : 2.0);
                tail = pre + steps_d * step + sum + 7.3;
                if (pre < 0.0) pre = 0.0;
            }
            pl.us = makespan(n, body, (ks == 1 ? 0.86 : 0.92) * body, slots, late, pre);
            if (pl.us < tail) pl.us = tail;
            // Where one slice leaves more than half of the places empty, slices are taken up to an eighth dearer: the estimates of one slice are
            // low there (640 x 1280 NF3, 591 rows, one slice / two: estimated 11.9 / 11.4, measured 12.7 / 12.1), even on average over the drawn calls.
            const double score = pl.us * (ks == 1 && steps_q > 16 && 2 * n < slots ? 1.125 : 1.0);
            if (best.us < 0 || score < best_score) { best = pl; best_score = score; }
        }
    }
    return best;
}

// The same, with the plans of the last few shapes kept by the calling thread (pure arithmetic, some microseconds).  beside_pre: the rank-r pre-product of the
// call runs beside the launch (not where it covers the columns that the pair kernel leaves).
inline const SwapPlan& swap_plan(int b0, int B0, bool backward, int64_t M, int64_t out_cols, int steps_q, int steps_d, bool beside_pre) {
    struct Entry { int b0 = 0, B0 = 0, steps_q = 0, steps_d = 0; bool backward = false, beside_pre = false; int64_t M = 0, out_cols = 0; SwapPlan plan; };
    constexpr int kEntries = 32;
    thread_local Entry cache[kEntries];
    const uint64_t h = (static_cast<uint64_t>(M) * 0x9E3779B97F4A7C15ull) ^ (static_cast<uint64_t>(out_cols) * 0xC2B2AE3D27D4EB4Full) ^
                       (static_cast<uint64_t>(steps_q * 8 + steps_d * 64 + b0 + B0 * 4096 + (backward ? 16 : 0) + (beside_pre ? 32 : 0)) * 0x165667B19E3779F9ull);
    Entry& e = cache[(h >> 40) % kEntries];
    if (e.b0 != b0 || e.B0 != B0 || e.backward != backward || e.beside_pre != beside_pre || e.M != M || e.out_cols != out_cols || e.steps_q != steps_q || e.steps_d != steps_d) {
        e.plan = make_swap_plan(b0, B0, backward, M, out_cols, steps_q, steps_d, beside_pre);
        e.b0 = b0; e.B0 = B0; e.backward = backward; e.beside_pre = beside_pre; e.M = M; e.out_cols = out_cols; e.steps_q = steps_q; e.steps_d = steps_d;
    }
    return e.plan;
}

template <int B, bool BWD, bool TA, int NBOX, int PS>
inline int launch_swap(const CUtensorMap& tX, const CUtensorMap& tT, const CUtensorMap& tF, const SwapParams& p, const SwapPlan& pl,
                       int smem, int pairs, cudaStream_t st, bool first) {
    auto kern = tc_swap_linear_kernel<B, BWD, TA, NBOX, PS>;
    static bool attr_done = false;
    if (!attr_done) {
        if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemLimit) != cudaSuccess) {
            cudaGetLastError();
            return LQLORA_ERR_CUDA;
        }
        attr_done = true;
    }
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(2 * pairs, pl.chunks, pl.ks);
    cfg.blockDim = dim3(kSwThreads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeClusterDimension;      // a pair, and the slices of its contraction
    attr[0].val.clusterDim.x = 2; attr[0].val.clusterDim.y = 1; attr[0].val.clusterDim.z = pl.ks;
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = first ? 2 : 1;      // overlap with the rank-r pre-product, or with the call in front
    const cudaError_t e = cudaLaunchKernelEx(&cfg, kern, tX, tT, tF, p);
    count_launch(1);
    if (e != cudaSuccess) { cudaGetLastError(); return LQLORA_ERR_CUDA; }
    return LQLORA_OK;
}

// Output columns [c_base, c_base + cols) of a call with the plan `pl`; T: the rank-r intermediate [M][r] (r > 0).  first: nothing but the
// pre-product of the call runs in front of it.
inline int run_swap(const QView& q, const void* L1, const void* L2, int r, const void* A, int M, void* out, const void* T, int* status,
                    bool backward, const SwapPlan& pl, int c_base, int cols, cudaStream_t st, bool first) {
    const int C = backward ? q.N : q.K;
    SwapParams p;
    p.q = q;
    p.out = static_cast<__nv_bfloat16*>(out);
    p.status = status;
    p.M = M;
    p.out_cols = backward ? q.K : q.N;
    p.steps_q = (C + BK - 1) / BK;
    p.steps_d = (r + BK - 1) / BK;
    p.c_base = c_base;
    p.nbox = pl.nbox; p.box = pl.box; p.ss = pl.ss; p.sp = pl.sp; p.tmem_cols = pl.tmem_cols;
    p.L1 = static_cast<const __nv_bfloat16*>(L1); p.r = r;
    p.clear_status = first ? 1 : 0;
    int smem = pl.smem;
    p.tail_off = pl.ps * (pl.ss * (kSwWBytes + pl.nbox * pl.box * 64) + pl.sp * 1024 * q.b0);
    const bool ta = !backward && pl.nbox == 1;      // (256 columns of accumulators and eight stages of 32 columns fill tensor memory)
    if (ta) {
        // Without weight tiles four stages of two steps of both rings always fit (256 tokens, 8-bit codes: 230,912 of 232,448 bytes, code
        // book included), so the tensor core is done with the codes of stage j - sp (see swap_rings); the token stages alone hold the
        // accumulators that a sliced contraction lays over them (8 x 64 = 512 bytes per token).
        const int fixed = 1024 + kSwTail + (q.b0 == 8 ? 32768 : 0), x = 2 * pl.box * 64, pk = 2 * 1024 * q.b0;
        p.ss = kSwMaxStages / 2;
        p.sp = (kSmemLimit - fixed - p.ss * x) / pk;
        if (p.sp > kSwMaxStages) p.sp = kSwMaxStages;
        p.tail_off = p.ss * x + p.sp * pk;
        smem = fixed + p.tail_off;
        if (smem < 120 * 1024) smem = 120 * 1024;      // no second user of tensor memory on the SM
        p.tmem_cols = 512;
    }
    CUtensorMap tX, tT, tF;
    if (!make_map(&tX, A, M, C, pl.box / 2)) return LQLORA_ERR_CUDA;
    if (r > 0) {                          // (tF is not read where the weights go to tensor memory; its map comes from the cache)
        if (!make_map(&tT, T, M, r, pl.box / 2)) return LQLORA_ERR_CUDA;
        const bool ok = backward ? make_map(&tF, L2, r, q.K, 64) : make_map(&tF, L1, q.N, r, 128);
        if (!ok) return LQLORA_ERR_CUDA;
    } else {
        tT = tX; tF = tX;
    }
    const int pairs = (cols + 255) / 256;
    auto go = [&](auto bits) {
        constexpr int B = decltype(bits)::value;
        if (ta) return launch_swap<B, false, true, 1, 2>(tX, tT, tF, p, pl, smem, pairs, st, first);
        if (!backward) return launch_swap<B, false, false, 2, 1>(tX, tT, tF, p, pl, smem, pairs, st, first);
        if constexpr (B == 2)
            if (pl.ps == 2) return launch_swap<B, true, false, 1, 2>(tX, tT, tF, p, pl, smem, pairs, st, first);
        if (pl.nbox == 1) return launch_swap<B, true, false, 1, 1>(tX, tT, tF, p, pl, smem, pairs, st, first);
        return launch_swap<B, true, false, 2, 1>(tX, tT, tF, p, pl, smem, pairs, st, first);
    };
    switch (q.b0) {
        case 2: return go(std::integral_constant<int, 2>());
        case 3: return go(std::integral_constant<int, 3>());
        case 4: return go(std::integral_constant<int, 4>());
        default: return go(std::integral_constant<int, 8>());
    }
}

}  // namespace tc
}  // namespace lq
