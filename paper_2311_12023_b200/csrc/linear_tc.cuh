// Tensor-core path (tcgen05) for more rows of X than the weight-streaming kernels take: what its two linear kernels share
// (linear_tc2.cuh: [512, 256] output tiles on CTA pairs; linear_swap.cuh: transposed tiles with the contraction split over a
// cluster), the rank-r pre-product, and the dispatch between them.
//
// Both linear kernels run the same pipeline over steps of 64 contraction elements: copies bring the bf16 activations (TMA,
// 128-byte swizzle) and the packed codes into shared memory; sixteen dequantization warps unpack the codes, multiply by
// the block scale in fp32, round to bf16 and write the weight tile in the 128-byte-swizzled layout that the tensor core
// reads; one warp issues tcgen05.mma with fp32 accumulators in tensor memory and commits the stage back.
// The rank-r term is folded in as extra contraction steps whose two operands come by TMA
// (forward: [X L2^T | L1]; backward: [dY L1 | L2]).
//
// The same shared-memory weight tile ([rows of Q] x 64 columns, 128 bytes per row, swizzled)
// serves both passes: the forward reads it as a K-major operand (contraction along the row),
// the input gradient as an MN-major operand (contraction across rows).
//
// Every wait on an mbarrier is bounded; when a wait expires the kernel records it in the status
// word of the workspace, stops issuing work, lets its copies land, frees its tensor memory and
// returns (lqlora_workspace_status then reports LQLORA_ERR_TIMEOUT).
#pragma once

#include <cuda.h>   // CUtensorMap and enums only; cuTensorMapEncodeTiled is resolved at run time

#include "common.cuh"
#include "device_util.cuh"
#include "linear_small.cuh"

namespace lq {
namespace tc {
using namespace dev;

constexpr int BK = 64;
constexpr int BN = 256;
constexpr int kDeqWarps = 16;
constexpr int kThreads = (2 + kDeqWarps) * 32;

struct Params {
    QView q;
    __nv_bfloat16* out;
    int* status;
    int M;
    int out_cols;      // N (forward) or K (backward)
    int steps_q;       // steps whose weights are dequantized
    int steps_d;       // steps of the rank-r term
    int c_base;        // first output column of this launch (a call may be split over two launches by output columns)
    int c_tiles;       // number of 256-column output tiles of this launch
};

// ------------------------------------------------------------------------------------ PTX (tensor memory, tcgen05)
__device__ __forceinline__ void tmem_alloc(uint32_t slot_smem, uint32_t cols) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(slot_smem), "r"(cols) : "memory");
}
__device__ __forceinline__ void tmem_relinquish() { asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory"); }
__device__ __forceinline__ void tmem_dealloc(uint32_t addr, uint32_t cols) {
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(addr), "r"(cols) : "memory");
}
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_commit(uint32_t bar) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void tc_mma(uint32_t d_tmem, uint64_t adesc, uint64_t bdesc, uint32_t idesc, uint32_t accumulate) {
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}"
        ::"r"(d_tmem), "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate) : "memory");
}
__device__ __forceinline__ void tmem_ld32(uint32_t taddr, uint32_t (&v)[32]) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
        "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
        "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
        : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]),
          "=r"(v[8]), "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15]),
          "=r"(v[16]), "=r"(v[17]), "=r"(v[18]), "=r"(v[19]), "=r"(v[20]), "=r"(v[21]), "=r"(v[22]), "=r"(v[23]),
          "=r"(v[24]), "=r"(v[25]), "=r"(v[26]), "=r"(v[27]), "=r"(v[28]), "=r"(v[29]), "=r"(v[30]), "=r"(v[31])
        : "r"(taddr) : "memory");
}
__device__ __forceinline__ void tmem_ld_wait() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }

// Shared-memory matrix descriptor, 128-byte swizzle (layout type 2), descriptor version 1.
__device__ __forceinline__ uint64_t make_desc(uint32_t saddr, uint32_t lbo_bytes, uint32_t sbo_bytes) {
    uint64_t d = 0;
    d |= static_cast<uint64_t>((saddr & 0x3FFFFu) >> 4);
    d |= static_cast<uint64_t>((lbo_bytes >> 4) & 0x3FFFu) << 16;
    d |= static_cast<uint64_t>((sbo_bytes >> 4) & 0x3FFFu) << 32;
    d |= static_cast<uint64_t>(1) << 46;
    d |= static_cast<uint64_t>(2) << 61;
    return d;
}

// ------------------------------------------------------------------------------------ dequantization
__device__ __forceinline__ uint32_t lds_u32(uint32_t addr) {
    uint32_t v;
    asm volatile("ld.shared.u32 %0, [%1];" : "=r"(v) : "r"(addr));
    return v;
}
__device__ __forceinline__ void sts_v4(uint32_t addr, uint32_t a, uint32_t b, uint32_t c, uint32_t d) {
    asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(addr), "r"(a), "r"(b), "r"(c), "r"(d) : "memory");
}
// One thread dequantizes the 32 consecutive weights of one (row, group) -- b0 words of the slab,
// `words` pointing at the thread's first word, the others 32 words apart -- and writes them as four
// 16-byte chunks of the row's 128 bytes; `dst` is the row start, `goff` the byte offset of the group
// in the row (0 or 64), `xr` is (row % 8) * 16; a chunk at byte offset o of the row lives at o ^ xr.
// 8-bit codes read the code book from shared memory, where it is stored once per bank: entry c of the copy
// of lane l at lut8[c * 32 + l], and `lut8` already points at the lane's copy, so no look-up meets a bank conflict.
template <int B>
__device__ __forceinline__ void dequant_group(uint32_t words, float s_lo, float s_hi, bool two_scales,
                                              uint32_t dst, uint32_t goff, uint32_t xr, const float* __restrict__ lut8) {
    // `words` and `dst` are 32-bit shared-memory addresses (explicit shared-space loads and stores)
    uint32_t w[B];
#pragma unroll
    for (int i = 0; i < B; ++i) w[i] = lds_u32(words + i * 128);
    const uint32_t x = dst + (goff ^ xr);    // chunk c sits at this address with bits 4, 5 flipped by c
    if constexpr (B == 8) {
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            const float s = (c < 2) ? s_lo : s_hi;
            uint32_t packed[4];
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const uint32_t ww = w[2 * c + (e >> 1)] >> (16 * (e & 1));
                const float q0 = lut8[(ww & 255u) << 5];
                const float q1 = lut8[((ww >> 8) & 255u) << 5];
                const __nv_bfloat162 h = __floats2bfloat162_rn(__fmul_rn(q0, s), __fmul_rn(q1, s));
                packed[e] = *reinterpret_cast<const uint32_t*>(&h);
            }
            sts_v4(x ^ (c << 4), packed[0], packed[1], packed[2], packed[3]);
        }
    } else {
        BlockTable<B> tab;
        tab.build(s_lo);
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            if (c == 2 && two_scales) tab.build(s_hi);
            const uint32_t sel = chunk_selector<B>(w, c);
            uint32_t selA = sel, selB = 0u;
            if constexpr (B == 4) { selA = sel & 0x77777777u; selB = ((sel >> 1) & 0x44444444u) | 0x32103210u; }
            uint32_t o[4];
            tab.lookup4(selA, selB, o[0], o[1]);
            tab.lookup4(selA >> 16, selB >> 16, o[2], o[3]);
            sts_v4(x ^ (c << 4), o[0], o[1], o[2], o[3]);
        }
    }
}

// Raw scale data of the 32 weights (row, k .. k+31): the one or two 8-bit scale codes and the
// second-level scale of their group (B1 >= 16 blocks, so both codes share it).
struct RawScale { uint32_t sc; float v; };
// s~ = fl32(float(s^) * fl32(v / 127)); the quotient is recomputed only when v changes.
__device__ __forceinline__ void make_scales(const QView& q, const RawScale& r, float& v_cached, float& sigma, float& s_lo, float& s_hi) {
    if (r.v != v_cached) { v_cached = r.v; sigma = __fdiv_rn(r.v, q.levels); }
    s_lo = __fmul_rn(static_cast<float>(r.sc & 0xFFu), sigma);
    s_hi = (q.B0 == 16) ? __fmul_rn(static_cast<float>(r.sc >> 8), sigma) : s_lo;
}

// Forward pass: the scale codes a thread needs in consecutive steps are consecutive bytes of its row, so it keeps a
// window of 16 of them (one 128-bit load, with the second-level scale of the window: 16 aligned blocks share their
// group since B1 >= 16) and the next window, requested one window period ahead.  `base` = block offset of the
// window inside the row (a multiple of 16); rows need KB % 16 == 0 for the alignment.
struct ScaleWindow { uint4 w; float v; };
__device__ __forceinline__ ScaleWindow load_scale_window(const QView& q, uint32_t row_blk0, int base, bool row_ok) {
    ScaleWindow s{make_uint4(0u, 0u, 0u, 0u), 0.0f};
    if (row_ok && base < q.KB) {
        s.w = __ldg(reinterpret_cast<const uint4*>(q.sc + row_blk0 + base));
        s.v = __ldg(q.v + ((row_blk0 + base) >> q.logB1));
    }
    return s;
}
// scale code(s) of block offset b (and b + 1 when two blocks of 16 columns make up the thread's 32 columns)
__device__ __forceinline__ RawScale window_scale(const ScaleWindow& s, int b, bool two) {
    const int i = b & 15;
    const uint32_t word = (i < 8) ? ((i < 4) ? s.w.x : s.w.y) : ((i < 12) ? s.w.z : s.w.w);
    const uint32_t sh = word >> ((i & 3) * 8);
    return RawScale{two ? (sh & 0xFFFFu) : (sh & 0xFFu), s.v};
}

constexpr int kSmemLimit = 232448;   // 227 KB of dynamic shared memory per CTA

// Ring position that advances without divisions: stage index and the parity of the current pass.
template <int S> struct RingPos {
    int s = 0;
    uint32_t ph = 0;
    __device__ __forceinline__ void advance() { if (++s == S) { s = 0; ph ^= 1u; } }
};


// ------------------------------------------------------------------------------------ rank-r pre-product
// T = bf16(A F) with a short output width (r <= 128):  forward  T = X L2^T  (F = L2 [r, K], K-major B operand),
// backward T = dY L1 (F = L1 [N, r], MN-major B operand).  Grid = (row tiles of 128, splits of the
// contraction).  Each CTA accumulates its part in tensor memory; with one split it rounds its tile to bf16 and
// stores it, with several the splits of a tile form a cluster (see CL below).
// Warps: four that issue the copies (warp w those of the steps w, w + 4, ...: one thread sustains a tensor copy per about
// 380 clocks, which made the loop 0.4 us per step with a single one), one that issues the MMAs, four for the epilogue.
constexpr int kLrProducers = 4;
constexpr int kLrThreads = (kLrProducers + 1 + 4) * 32;

struct PreParams {
    __nv_bfloat16* T;      // [M][r]
    int* status;
    int M, r, rp;          // rp = r rounded up to 64 (MMA N)
    int steps;             // contraction steps of 64 in total
    int steps_per_split;
    int stages;
    int clear_status;      // 1: this kernel is the first of a call and clears the status word (no memset in front of it)
};

// Body of the kernel for the CTA (row tile `tile`, split `split` of `nsplit`); the tensor maps are kernel parameters.
// CL: the splits of a tile are the CTAs of a cluster (nsplit = cluster size <= 8, a divisor of 64); their accumulators
// go to the CTA that owns the column through distributed shared memory (own receive buffer behind the ring, rp x 128
// fp32), are added there in rank order and stored as bf16 -- no partial tiles in global memory, no counters.
template <bool BWD, bool CL = false>
__device__ __forceinline__ void lowrank_body(const CUtensorMap& tmA, const CUtensorMap& tmB, const PreParams& p, int tile, int split,
                                             int nsplit) {
    constexpr int A_BYTES = 16384;
    extern __shared__ uint8_t smem_raw[];
    uint8_t* base = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~static_cast<uintptr_t>(1023));
    const int b_bytes = p.rp * 128;
    const int stage_bytes = A_BYTES + b_bytes;
    float* recv = reinterpret_cast<float*>(base + static_cast<size_t>(p.stages) * stage_bytes);
    uint8_t* tail = reinterpret_cast<uint8_t*>(recv) + (CL ? static_cast<size_t>(p.rp) * 512 : 0);
    uint64_t* bars = reinterpret_cast<uint64_t*>(tail);      // full[8], empty[8], acc_full, drain
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(tail + 160);
    volatile int* abort_s = reinterpret_cast<volatile int*>(tmem_slot + 1);
    int* issued = reinterpret_cast<int*>(tmem_slot + 2);      // [kLrProducers] next step of each producer warp

    // The CTAs of a cluster write into each other's shared memory at the end; that is allowed once every CTA of the
    // cluster runs, which the first phase of the cluster barrier establishes: arrive here, wait before the first store.
    if (CL && nsplit > 1) dec::cluster_arrive_relaxed();
    pdl_wait_for_copies();        // started while the previous kernel of the stream ends; everything below comes after it
    // cleared before this CTA lets the dependent kernel start: that kernel is launched once all CTAs have passed here
    if (p.clear_status && tile == 0 && split == 0 && threadIdx.x == 0) *p.status = 0;
    pdl_launch_dependents();      // the linear kernel behind this one needs T only in its last steps
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int m0 = tile * 128;
    const int s_lo = split * p.steps_per_split;
    const int s_hi = min(p.steps, s_lo + p.steps_per_split);
    const int total = s_hi - s_lo;
    const Ctl ctl{abort_s, p.status};
    const uint32_t tmem_cols = (p.rp <= 64) ? 64u : 128u;

    const uint32_t bar0 = smem_u32(bars), ring0 = smem_u32(base);
    auto full = [&](int s) { return bar0 + 8 * s; };
    auto empty = [&](int s) { return bar0 + 64 + 8 * s; };
    const uint32_t acc_full = bar0 + 128, drain = bar0 + 136;

    if (threadIdx.x == 0) {
        for (int s = 0; s < p.stages; ++s) { mbar_init(full(s), 1); mbar_init(empty(s), 1); }
        mbar_init(acc_full, 1);
        mbar_init(drain, 1);
        *abort_s = 0;
        fence_barrier_init();
    }
    if (warp == kLrProducers) { tmem_alloc(smem_u32(tmem_slot), tmem_cols); tmem_relinquish(); }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tmem_slot;
    bool cl_ok = false;          // CL: this thread saw the accumulators complete (epilogue warps)

    if (warp < kLrProducers) {
        int s = warp;                    // stage and pass of step i; advanced without divisions (stages >= kLrProducers)
        uint32_t ph = 0;
        int i = warp;
        for (; i < total; i += kLrProducers) {
            if (!wait(empty(s), ph ^ 1, ctl, 11)) break;
            const uint32_t a_dst = ring0 + s * stage_bytes, b_dst = a_dst + A_BYTES;
            const int c = (s_lo + i) * BK;
            __syncwarp();
            if (elect_one()) {
                mbar_expect_tx(full(s), A_BYTES + b_bytes);
                tma_load_2d(a_dst, &tmA, c, m0, full(s));
                if (!BWD) tma_load_2d(b_dst, &tmB, c, 0, full(s));                       // [rp rows of L2] x 64 columns
                else for (int t = 0; t < p.rp / 64; ++t) tma_load_2d(b_dst + t * 8192, &tmB, t * 64, c, full(s));  // 64 rows of L1
            }
            __syncwarp();
            s += kLrProducers;
            if (s >= p.stages) { s -= p.stages; ph ^= 1u; }
        }
        if (lane == 0) issued[warp] = i;
        __syncwarp();
    } else if (warp == kLrProducers) {
        const uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((BWD ? 1u : 0u) << 16) |
                               (static_cast<uint32_t>(p.rp >> 3) << 17) | (static_cast<uint32_t>(128 >> 4) << 24);
        bool ok = true;
        int s = 0;
        uint32_t ph = 0;
        for (int i = 0; i < total; ++i) {
            ok = wait(full(s), ph, ctl, 12);
            if (!ok) break;
            __syncwarp();
            tc_fence_after();
            const uint32_t a_src = ring0 + s * stage_bytes, b_src = a_src + A_BYTES;
            if (elect_one()) {
#pragma unroll
                for (int k16 = 0; k16 < 4; ++k16) {
                    const uint64_t adesc = make_desc(a_src + k16 * 32, 16, 1024);
                    const uint64_t bdesc = BWD ? make_desc(b_src + k16 * 2048, 8192, 1024) : make_desc(b_src + k16 * 32, 16, 1024);
                    tc_mma(tmem, adesc, bdesc, idesc, (i > 0 || k16 > 0) ? 1u : 0u);
                }
                tc_commit(i + 1 < total ? empty(s) : acc_full);
            }
            __syncwarp();
            if (++s == p.stages) { s = 0; ph ^= 1u; }
        }
        if (!ok) {
            __syncwarp();
            if (elect_one()) tc_commit(drain);
            const long long t0 = clock64();
            while (!mbar_try_wait(drain, 0) && clock64() - t0 < 20000000LL) {}
        }
        __syncwarp();
    } else {
        // epilogue warps, one per TMEM lane quarter (warp % 4)
        const int quarter = warp & 3;
        const int m = m0 + quarter * 32 + lane;
        const bool ok = (total > 0) ? wait(acc_full, 0, ctl, 13) : true;
        cl_ok = ok;
        if (ok && !CL) {
            // one split: the accumulator row of this thread goes straight to T as bf16 (r is a multiple of 16, so a
            // run of eight columns lies inside or outside of it as a whole)
            tc_fence_after();
            for (int col = 0; col < p.rp; col += 32) {
                uint32_t v[32];
                if (total > 0) { tmem_ld32(tmem + (static_cast<uint32_t>(quarter * 32) << 16) + col, v); tmem_ld_wait(); }
                else {
#pragma unroll
                    for (int i = 0; i < 32; ++i) v[i] = 0u;
                }
                if (m < p.M) {
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        if (col + 8 * i < p.r) {
                            uint32_t w[4];
#pragma unroll
                            for (int e = 0; e < 4; ++e) {
                                const __nv_bfloat162 h = __floats2bfloat162_rn(__uint_as_float(v[8 * i + 2 * e]), __uint_as_float(v[8 * i + 2 * e + 1]));
                                w[e] = *reinterpret_cast<const uint32_t*>(&h);
                            }
                            *reinterpret_cast<uint4*>(p.T + static_cast<size_t>(m) * p.r + col + 8 * i) = make_uint4(w[0], w[1], w[2], w[3]);
                        }
                    }
                }
            }
        }
    }
    if constexpr (CL) {
        // all threads of all CTAs of the cluster pass here, whatever happened before
        __syncthreads();
        if (nsplit > 1) dec::cluster_wait();           // every CTA of the cluster has started
        // Four columns at a time: a thread's scalar stores, with a division each to find the column's owner, took longer than the four
        // steps of a short contraction (1024 x 1024 NF3 at 512 rows, whole call: 12.0 us, with this 10.3).  The shares are powers of two from eight columns on.
        const uint32_t recv_addr = smem_u32(recv);         // [split][column / 4 of the share][row] of float4
        const int cols_share = p.rp / nsplit, log_share = 31 - __clz(cols_share);
        if (warp > kLrProducers && cl_ok) {
            tc_fence_after();
            const int quarter = warp & 3;
            const int row = quarter * 32 + lane;
            for (int col = 0; col < p.rp; col += 32) {
                uint32_t v[32];
                if (total > 0) { tmem_ld32(tmem + (static_cast<uint32_t>(quarter * 32) << 16) + col, v); tmem_ld_wait(); }
                else {
#pragma unroll
                    for (int i = 0; i < 32; ++i) v[i] = 0u;
                }
#pragma unroll
                for (int i = 0; i < 32; i += 4) {
                    const int c = col + i, owner = c >> log_share, c4 = (c & (cols_share - 1)) >> 2;
                    dec::st_dsmem_v4(recv_addr + static_cast<uint32_t>((split * (cols_share >> 2) + c4) * 128 + row) * 16u, static_cast<uint32_t>(owner),
                                     v[i], v[i + 1], v[i + 2], v[i + 3]);
                }
            }
        }
        __syncthreads();
        if (nsplit > 1) dec::cluster_sync_all();
        for (int item = threadIdx.x; item < 32 * cols_share; item += kLrThreads) {
            const int row = item & 127, c4 = item >> 7;
            float4 sum = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
            for (int src = 0; src < nsplit; ++src) {
                const float4 x = reinterpret_cast<const float4*>(recv)[(src * (cols_share >> 2) + c4) * 128 + row];
                sum.x += x.x; sum.y += x.y; sum.z += x.z; sum.w += x.w;
            }
            const int m = m0 + row, col = split * cols_share + c4 * 4;
            if (m < p.M && col < p.r) {
                const __nv_bfloat162 lo = __floats2bfloat162_rn(sum.x, sum.y), hi = __floats2bfloat162_rn(sum.z, sum.w);
                *reinterpret_cast<uint2*>(p.T + static_cast<size_t>(m) * p.r + col) =
                    make_uint2(*reinterpret_cast<const uint32_t*>(&lo), *reinterpret_cast<const uint32_t*>(&hi));
            }
        }
    }
    tc_fence_before();
    __syncthreads();
    if (*abort_s && warp == 0) {
        // copies in flight land before the CTA exits: the last step issued into every stage (the producer warps are at most a
        // ring apart, so it is among the last two rings of steps)
        int top = 0;
        for (int w = 0; w < kLrProducers; ++w) top = max(top, min(total, issued[w]));
        for (int i = max(0, top - 2 * p.stages); i < top; ++i)
            if (i < issued[i % kLrProducers] && (i + p.stages >= total || i + p.stages >= issued[(i + p.stages) % kLrProducers]))
                let_land(full(i % p.stages), (i / p.stages) & 1);
    }
    if (warp == kLrProducers) tmem_dealloc(tmem, tmem_cols);
}

template <bool BWD>
__global__ void __launch_bounds__(kLrThreads, 1)
tc_lowrank_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB, const PreParams p) {
    lowrank_body<BWD>(tmA, tmB, p, blockIdx.x, blockIdx.y, gridDim.y);
}

// The same with the splits of a tile as the CTAs of a cluster (grid.y = cluster size, a power of two up to eight).
template <bool BWD>
__global__ void __launch_bounds__(kLrThreads, 1)
tc_lowrank_cl_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB, const PreParams p) {
    lowrank_body<BWD, true>(tmA, tmB, p, blockIdx.x, blockIdx.y, gridDim.y);
}

// Both pre-products of one layer in one launch (the weight-gradient path, which has the GPU to itself): grid.z = 0
// computes T = X L2^T with (tmA0, tmB0, p0), grid.z = 1 computes T' = dY L1 with (tmA1, tmB1, p1); grid.y = splits of
// the contraction = cluster size (the same for both), reduced through distributed shared memory.
__global__ void __launch_bounds__(kLrThreads, 1)
tc_lowrank_both_kernel(const __grid_constant__ CUtensorMap tmA0, const __grid_constant__ CUtensorMap tmB0, const PreParams p0,
                       const __grid_constant__ CUtensorMap tmA1, const __grid_constant__ CUtensorMap tmB1, const PreParams p1) {
    if (blockIdx.z == 0) lowrank_body<false, true>(tmA0, tmB0, p0, blockIdx.x, blockIdx.y, gridDim.y);
    else lowrank_body<true, true>(tmA1, tmB1, p1, blockIdx.x, blockIdx.y, gridDim.y);
}

// ------------------------------------------------------------------------------------ host side
typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*, const cuuint64_t*,
                                  const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle,
                                  CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

inline EncodeTiledFn encode_tiled_fn() {
    static EncodeTiledFn fn = [] {
        void* f = nullptr;
        cudaDriverEntryPointQueryResult qres;
        if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &f, cudaEnableDefault, &qres) != cudaSuccess ||
            qres != cudaDriverEntryPointSuccess) {
            cudaGetLastError();
            f = nullptr;
        }
        return reinterpret_cast<EncodeTiledFn>(f);
    }();
    return fn;
}

// bf16 row-major [rows, cols] matrix, box of 64 columns x box_rows rows, 128-byte swizzle, zero fill.
// A descriptor depends only on (pointer, rows, columns, box rows); a training step issues the same few over and over, so
// the last ones built by this thread are kept (a call needs four to six of them).
inline bool make_map(CUtensorMap* map, const void* ptr, uint64_t rows, uint64_t cols, uint32_t box_rows) {
    struct Entry { const void* ptr; uint64_t rows, cols; uint32_t box_rows; bool valid; CUtensorMap map; };
    constexpr int kEntries = 64;
    thread_local Entry cache[kEntries] = {};
    uint64_t h = reinterpret_cast<uintptr_t>(ptr) >> 4;
    h = (h ^ (h >> 17)) * 0x9E3779B97F4A7C15ull + rows * 31u + cols * 131u + box_rows;
    Entry& e = cache[(h >> 20) % kEntries];
    if (e.valid && e.ptr == ptr && e.rows == rows && e.cols == cols && e.box_rows == box_rows) { *map = e.map; return true; }
    EncodeTiledFn fn = encode_tiled_fn();
    if (!fn) return false;
    const cuuint64_t dims[2] = {cols, rows};
    const cuuint64_t strides[1] = {cols * 2};
    const cuuint32_t box[2] = {64, box_rows};
    const cuuint32_t estr[2] = {1, 1};
    if (fn(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(ptr), dims, strides, box, estr,
           CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
           CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
        return false;
    e.ptr = ptr; e.rows = rows; e.cols = cols; e.box_rows = box_rows; e.map = *map; e.valid = true;
    return true;
}

}  // namespace tc
}  // namespace lq

#include "linear_tc2.cuh"
#include "linear_swap.cuh"

namespace lq {
namespace tc {

struct PrePlan {
    int mtiles, nsplit, steps, steps_per_split, rp;
};

// Number of SMs of the current device (148 on B200; also the answer when no device is present).
inline int sm_count() {
    static const int n = [] {
        int dev = 0, v = 0;
        if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&v, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || v <= 0) {
            cudaGetLastError();
            v = 148;
        }
        return v;
    }();
    return n;
}

// Wave quantisation of the pair kernel: its tiles run in waves of sms / 2 clusters.  When the last wave would hold only a few
// tiles (at most a quarter of a wave), the output columns it would cover are peeled off and computed on
// transposed tiles with the contraction split over clusters, which spreads that small remainder over many SMs (us as a graph,
// all on pairs / peeled: 28672 x 8192 NF3 at 2048 rows, 6 waves + 4 tiles, 674 / 637; 4096 x 4096 NF3 at 2560 rows, 1 wave + 6,
// 95 / 91).  Remainders of three quarters of a wave stay with the pairs (8192 x 8192 at 2048 rows, 1 wave + 54: NF3 186 / 209, 8-bit
// codes 236 / 368; 4096 x 11008 NF4 at 4096 rows, the same: 266 / 297).  In between the line predates the transposed tiles: remainders of
// 22 and 34 of 74 would gain (8192 x 8192 at 1536 rows 176 / 162, 6912 x 8192 at 2048 rows 176 / 167).
// Returns the number of 256-column tiles to peel off.
inline int pair_peel(int64_t M, int64_t out_cols) {
    const int mt = static_cast<int>((M + 511) / 512), pairs = sm_count() / 2, c_tiles = static_cast<int>((out_cols + BN - 1) / BN);
    const long long tiles = static_cast<long long>(mt) * c_tiles;
    const int rem = static_cast<int>(tiles % pairs);
    const int peel = (tiles > pairs && rem > 0 && 4 * rem <= pairs) ? (rem + mt - 1) / mt : 0;
    return peel >= c_tiles ? 0 : peel;
}

// CTA pairs on [512, 256] tiles take over once their tiles fill more than half of the SMs, and below 2048 rows unless the transposed tiles,
// which pad to 16 rows instead of 512 and choose their split, are estimated faster.  The estimate of the pairs is fitted to 448 drawn calls of 257 to 2000 rows
// (spread 6 %): whole waves, whose steps take less time where the last rows or the last wave leave SMs or tensor cores idle.  The side taken is 0.3 % behind the
// faster one on average, more than a tenth in 4 of them (2.1 % and 45 with 6 us per wave and 0.64 per step).  us as a graph, pair / transposed: 8192 x 8192 NF3 at
// 520 rows 87 / 50, 11904 x 8448 NF3 at 546 rows 123 / 80, 4352 x 11008 NF3 at 688 rows 78 / 60, 7160 x 10240 NF2 input gradient at 990 rows 110 / 152;
// 8320 x 4992 NF8 at 825 rows 79 / 100.  Two corrections, both small: long calls run at a lower clock, the transposed tiles more so than the pairs (28672 x 8192 NF3
// measured / estimated at 1024 rows 1.10, at 1500 1.17, at 2047 1.25; pairs 0.97, 1.03, 1.11), 0.4 per 10^12 products; and one wave of pairs
// with at least four fifths of its tiles and nine tenths of its rows stays where they are estimated within a tenth (8192 x 8192 NF3 at 1024 rows 91 / 90, input
// gradient 92.5 / 93.3, 5120 x 5120 NF2 at 1400 rows 60 / 57).
// From 2048 rows on the pairs stay whatever the estimates say.  That line is drawn by hand.  Both sides measured on nine shapes, both passes,
// 3-, 4- and 8-bit codes, 2048 to 4096 rows: where the last wave of pair tiles is well filled the pairs are up to a fifth faster (4096 x 4096 NF3
// at 4096 rows 97 / 120, 28672 x 8192 NF8 at 2048 902 / 1064, 8192 x 8192 NF8 at 2048 273 / 306); where it is between a quarter and a half
// full the transposed tiles would be, by up to a third and on narrow outputs by more (4096 x 11008 NF3 at 2600 rows 240 / 186, NF8 299 / 226; 4392 x
// 26688 NF8 at 2600 726 / 557; 5120 x 5120 NF8 at 2304 148 / 116; 2040 x 27008 NF3 at 2048 274 / 156).
inline double pair_estimate(int b0, int B0, int64_t M, int64_t out_cols, int steps_q, int steps_d) {
    static const double step_us[4] = {0.668, 0.67, 0.693, 0.957};
    const int mt = static_cast<int>((M + 511) / 512), c_tiles = static_cast<int>((out_cols + BN - 1) / BN), peel = pair_peel(M, out_cols);
    const long long pairs = sm_count() / 2, tiles = static_cast<long long>(mt) * (c_tiles - peel), waves = (tiles + pairs - 1) / pairs;
    const double idle = 1.0 - static_cast<double>(tiles) / static_cast<double>(waves * pairs), padding = 1.0 - static_cast<double>(M) / (512.0 * mt);
    const double step = step_us[bits_index(b0)] * (B0 == 16 ? 1.04 : 1.0) * (1.0 - 0.32 * idle) * (1.0 - 0.11 * padding);
    return (steps_d > 0 ? 3.3 : 5.0) + static_cast<double>(waves) * (7.1 + (steps_q + steps_d) * step) + (peel > 0 ? 11.8 + 0.168 * steps_q : 0.0);
}
inline bool tc_use_pair(const QView& q, bool backward, int64_t M, int64_t out_cols, int steps_q, int steps_d) {
    if (M <= 256) return false;
    const long long pair_ctas = 2 * ((M + 511) / 512) * ((out_cols + BN - 1) / BN);
    if (2 * pair_ctas <= sm_count()) return false;
    if (M >= 2048) return true;
    const int64_t rows = (M + 511) / 512 * 512;
    const bool full = pair_ctas <= sm_count() && 5 * pair_ctas >= 4 * sm_count() && 10 * M >= 9 * rows;
    const double products = static_cast<double>(M) * static_cast<double>(out_cols) * BK * steps_q;
    return swap_plan(q.b0, q.B0, backward, M, out_cols, steps_q, steps_d, steps_d > 0).us * (1.0 + 0.4e-12 * products) >=
           (full ? 0.9 : 1.0) * pair_estimate(q.b0, q.B0, M, out_cols, steps_q, steps_d);
}

// The launch on transposed tiles that a call needs: the whole of it, or the output columns from *c_base on that the pair
// kernel leaves (none where *c_base is not below out_cols).
inline SwapPlan call_swap_plan(const QView& q, bool backward, bool pair, int64_t M, int64_t out_cols, int steps_q, int steps_d, int* c_base) {
    *c_base = 0;
    if (!pair) return swap_plan(q.b0, q.B0, backward, M, out_cols, steps_q, steps_d, steps_d > 0);
    const int peel = pair_peel(M, out_cols);
    *c_base = (static_cast<int>((out_cols + BN - 1) / BN) - peel) * BN;
    return peel > 0 ? swap_plan(q.b0, q.B0, backward, M, out_cols - *c_base, steps_q, steps_d, false) : SwapPlan{};
}

// C = contraction length, out_cols = width of the output of the linear kernel that follows.
inline PrePlan pre_plan(const QView& q, bool backward, int64_t C, int r, int64_t M, int64_t out_cols) {
    PrePlan pl;
    pl.mtiles = static_cast<int>((M + 127) / 128);
    pl.steps = static_cast<int>((C + BK - 1) / BK);
    const int steps_d = (r + BK - 1) / BK;
    const long long main_ctas = tc_use_pair(q, backward, M, out_cols, pl.steps, steps_d) ? 2 * ((M + 511) / 512) * ((out_cols + BN - 1) / BN)
                                                                                        : swap_plan(q.b0, q.B0, backward, M, out_cols, pl.steps, steps_d, steps_d > 0).ctas;
    pl.nsplit = pre_splits(pl.mtiles, pl.steps, main_ctas);
    pl.steps_per_split = (pl.steps + pl.nsplit - 1) / pl.nsplit;
    pl.rp = (r <= 64) ? 64 : 128;
    return pl;
}

template <bool BWD>
inline int launch_pre(const CUtensorMap& tA, const CUtensorMap& tB, PreParams p, int mtiles, int nsplit, cudaStream_t st) {
    const int stage = 16384 + p.rp * 128;
    const bool cl = nsplit > 1;            // several splits: reduced inside a cluster
    const int recv_bytes = cl ? p.rp * 512 : 0;
    int stages = (kSmemLimit - 1024 - 256 - recv_bytes) / stage;
    if (stages > 8) stages = 8;
    p.stages = stages;
    const int smem = 1024 + stages * stage + recv_bytes + 256;
    void (*kern)(const CUtensorMap, const CUtensorMap, const PreParams) = cl ? tc_lowrank_cl_kernel<BWD> : tc_lowrank_kernel<BWD>;
    static bool attr_done = false;
    if (!attr_done) {
        if (cudaFuncSetAttribute(tc_lowrank_kernel<BWD>, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemLimit) != cudaSuccess ||
            cudaFuncSetAttribute(tc_lowrank_cl_kernel<BWD>, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemLimit) != cudaSuccess) {
            cudaGetLastError();
            return LQLORA_ERR_CUDA;
        }
        attr_done = true;
    }
    // One split: launched as clusters of two row tiles where possible (the CTAs then fill whole TPCs, and the CTA pairs
    // of the linear kernel that runs beside this one find as many free TPCs as the SM count suggests).
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(mtiles, nsplit);
    cfg.blockDim = dim3(kLrThreads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = (!cl && mtiles % 2 == 0) ? 2 : 1; attr[0].val.clusterDim.y = cl ? nsplit : 1; attr[0].val.clusterDim.z = 1;
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;      // the launch overlaps the end of the kernel in front
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 2;
    const cudaError_t e = cudaLaunchKernelEx(&cfg, kern, tA, tB, p);
    count_launch(1);
    if (e != cudaSuccess) { cudaGetLastError(); return LQLORA_ERR_CUDA; }
    return LQLORA_OK;
}

}  // namespace tc
}  // namespace lq


namespace lq {

constexpr int kTcMinRows = 17;   // up to 16 rows go to the weight-streaming kernels
constexpr int kTcMinRowsBwd = 9;  // input gradient of matrices with at least 2048 rows: up to 8 rows

inline bool tc_supported(const QView& q, int r, int64_t M, bool backward) {
    (void)r;
    // Geometric means of transposed / streaming over some 75 drawn calls for each number of rows (512 .. 28672 rows and columns, 2 to 8 bits): forward 1 row 1.34,
    // 8 rows 1.12, 16 rows 0.98 (8192 x 8192 even, 28672 x 8192 up to a quarter dearer); input gradient 1 to 4 rows 1.05, 8 rows 0.95, 9 rows (a second token
    // group for the streaming kernels) 0.76.  One line for all shapes: around it the faster side depends on the shape, and the streaming kernels keep the even cases.
    const int min_rows = (backward && q.N >= 2048) ? kTcMinRowsBwd : kTcMinRows;
    if (M < min_rows) return false;
    if (q.N % 8 != 0 || q.K % 8 != 0) return false;
    if (static_cast<long long>(q.N) * q.KB >= (1LL << 31)) return false;   // block indices are 32-bit in the kernel
    return true;
}

inline size_t tc_workspace_bytes(int r, int64_t M) {
    return kStatusBytes + round_up(static_cast<size_t>(M) * (r > 0 ? r : 1) * 2, 256);      // [status word][T bf16]
}

inline int tc_launch(const QView& q, const void* L1, const void* L2, int r, const void* A, int M, void* out, char* ws,
                     bool backward, cudaStream_t st) {
    using namespace tc;
    const int C = backward ? q.N : q.K;              // contraction length
    const PrePlan pl = pre_plan(q, backward, C, r, M, backward ? q.K : q.N);
    // workspace: [status word][T bf16]; the status word is cleared by the first kernel of the call (CTA pairs without a rank-r term: by a memset)
    __nv_bfloat16* T = reinterpret_cast<__nv_bfloat16*>(ws + kStatusBytes);
    const bool pair = tc_use_pair(q, backward, M, backward ? q.K : q.N, pl.steps, (r + BK - 1) / BK);      // CTA pairs (cta_group::2) on [512, 256] tiles; boxes of 128 rows
    const int out_cols = backward ? q.K : q.N;
    int c_base = 0;
    const SwapPlan sp = call_swap_plan(q, backward, pair, M, out_cols, pl.steps, (r + BK - 1) / BK, &c_base);
    if (c_base < out_cols && sp.ks < 1) return LQLORA_ERR_INVALID_SHAPE;      // (never: a plan exists for every shape) before any launch
    if (pair && r == 0 && cudaMemsetAsync(ws, 0, kStatusBytes, st) != cudaSuccess) { cudaGetLastError(); return LQLORA_ERR_CUDA; }
    CUtensorMap tA, tA2, tB2;
    if (pair && !make_map(&tA, A, M, C, 128)) return LQLORA_ERR_CUDA;
    if (r > 0) {
        // rank-r pre-product on the tensor cores: T = X L2^T (forward) or dY L1 (backward)
        CUtensorMap tPA, tPB;
        if (!make_map(&tPA, A, M, C, 128)) return LQLORA_ERR_CUDA;
        const bool okp = backward ? make_map(&tPB, L1, q.N, r, 64) : make_map(&tPB, L2, r, q.K, pl.rp);
        if (!okp) return LQLORA_ERR_CUDA;
        PreParams pp;
        pp.T = T; pp.status = reinterpret_cast<int*>(ws);
        pp.M = M; pp.r = r; pp.rp = pl.rp; pp.steps = pl.steps; pp.steps_per_split = pl.steps_per_split; pp.stages = 0;
        pp.clear_status = 1;           // first kernel of the call
        const int rc = backward ? launch_pre<true>(tPA, tPB, pp, pl.mtiles, pl.nsplit, st)
                                : launch_pre<false>(tPA, tPB, pp, pl.mtiles, pl.nsplit, st);
        if (rc != LQLORA_OK) return rc;
    }
    if (!pair) return run_swap(q, L1, L2, r, A, M, out, T, reinterpret_cast<int*>(ws), backward, sp, 0, out_cols, st, true);
    if (r > 0) {
        if (!make_map(&tA2, T, M, r, 128)) return LQLORA_ERR_CUDA;
        const bool okb = backward ? make_map(&tB2, L2, r, q.K, 64) : make_map(&tB2, L1, q.N, r, 128);
        if (!okb) return LQLORA_ERR_CUDA;
    } else {
        tA2 = tA; tB2 = tA;
    }
    Params p;
    p.q = q;
    p.out = static_cast<__nv_bfloat16*>(out);
    p.status = reinterpret_cast<int*>(ws);
    p.M = M;
    p.out_cols = out_cols;
    p.steps_q = (C + BK - 1) / BK;
    p.steps_d = (r + BK - 1) / BK;
    p.c_base = 0;
    p.c_tiles = c_base / BN;
    CUtensorMap tOut;         // output as boxes of 32 rows x 64 columns
    if (!make_map(&tOut, out, M, p.out_cols, 32)) return LQLORA_ERR_CUDA;
    int rc;
    switch (q.b0) {
        case 2: rc = backward ? launch_pair<2, true>(tA, tA2, tB2, tOut, p, st) : launch_pair<2, false>(tA, tA2, tB2, tOut, p, st); break;
        case 3: rc = backward ? launch_pair<3, true>(tA, tA2, tB2, tOut, p, st) : launch_pair<3, false>(tA, tA2, tB2, tOut, p, st); break;
        case 4: rc = backward ? launch_pair<4, true>(tA, tA2, tB2, tOut, p, st) : launch_pair<4, false>(tA, tA2, tB2, tOut, p, st); break;
        default: rc = backward ? launch_pair<8, true>(tA, tA2, tB2, tOut, p, st) : launch_pair<8, false>(tA, tA2, tB2, tOut, p, st); break;
    }
    if (rc != LQLORA_OK || c_base >= out_cols) return rc;
    // the peeled columns run behind the pair kernel (which has waited for the rank-r intermediate), so they need no
    // programmatic dependency of their own
    return run_swap(q, L1, L2, r, A, M, out, T, reinterpret_cast<int*>(ws), backward, sp, c_base, p.out_cols - c_base, st, false);
}

}  // namespace lq
