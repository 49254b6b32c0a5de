// Forward pass for decode-sized inputs (M <= 16 rows): the packed matrix is streamed once, straight from global memory into
// registers.
//
//   - A unit of work is 16 rows x 256 columns of Q (half a slab of four neighbouring 64-column tiles): lane (gid, t) of a warp
//     dequantizes rows 2 gid, 2 gid + 1 of tile t with the byte-table method (bf16 bits identical to the exported dequantized
//     weights; one table per row for blocks of 64 and more) and feeds mma.sync m16n8k16 (weights = the 16-row operand, tokens =
//     the 8-column operand, fp32 accumulators).  The contraction index is permuted so that a lane supplies four consecutive
//     weights of each of its rows per MMA.
//   - Eight warps cover the 128 rows of a tile row; the CTA's run of units (contiguous in memory, across tile rows) is cut into
//     as many phases as there are groups of eight warps.  A warp owns everything that it needs: its packed words are loaded
//     one unit ahead into registers (the word planes of a tile are coalesced as they are), the scales of 16 blocks per row one
//     run ahead, and are laid out in the warp's own corner of shared memory.  There is no ring, no barrier and no wait in the
//     main loop; only the activations are staged once for the CTA.
//   - The runs have the same length for every SM to within one unit.  A tile row that is shared by several runs is added up through
//     global memory: every CTA stores its fp32 sums in its own slot, counts itself on the tile row's arrival counter, and the
//     last one adds the slots in order (the same bits on every run) and writes the bf16 output.
//   - The rank-r intermediate T = X L2^T comes from a small kernel launched in front; the two overlap (programmatic dependent
//     launch), and the warps that work on the last unit of a tile row add T L1^T to their accumulators.  The counters are cleared by
//     that kernel, or by one that does nothing else when there is no rank-r term.
//
// What bounds it: the pipe of byte permutes and logic (64 lanes per clock and SM): about two operations per weight of 3 bits, 2.6 of 4
// bits, 1.2 of 2 bits; busy 53 % of the active cycles of the whole kernel (8192 x 8192 NF3, one row; input gradient 47 %), of which the main
// loop, at 21 weights per clock and SM, is about two thirds.  Around the loop a call takes 6 us: 2.5 from the end of the kernel in front to
// the first unit, 3 for sums, counter and output.  The kernel before this one (tiles and scale tables staged through a ring in shared memory,
// short CTAs in waves) held the pipe at 50 % of its active cycles.
// us per call in a graph, kernels before / these (rank 64): one row of 8192 x 8192 2 bits 19.6 / 16.0, 3 bits 21.2 / 17.7, 4 bits 28.6 / 24.0,
// 8 bits 43.1 / 28.5; 28672 x 8192 3 bits in blocks of 16 68.3 / 57.9; 8192 x 28672 2 bits in blocks of 128 61.5 / 36.0; sixteen rows of 8192 x 8192
// 32.9 / 23.2, 34.1 / 24.6, 41.9 / 30.9, 60.6 / 42.0.  Input gradient, one row: 8192 x 8192 2 bits 26.4 / 24.7, 3 bits 28.6 / 25.4, 4 bits 39.3 / 28.8,
// 8 bits 58.4 / 35.7; 8192 x 28672 2 bits in blocks of 128 80.5 / 57.0.
#pragma once

#include "common.cuh"
#include "device_util.cuh"
#include "linear_decode.cuh"

namespace lq {
namespace stream {
using namespace dev;

constexpr int kUnitTiles = 4;                    // 64-column tiles per unit
constexpr int kXTokenBytes = kUnitTiles * 144;   // one token's 256 activations of a unit: 128 bytes per tile, padded against bank conflicts
constexpr int kStabBytes = 16 * 24 * 4;          // a warp's scales: 16 block columns x 16 rows, padded
constexpr int kMaxSegs = 3;                      // tile rows that a run may touch
constexpr int kSmemLimit = 232448;
// Sixteen warps of at most 104 registers leave room for a CTA of the pre-product in front (256 threads of 48): with 128, the CTAs of the SMs that it
// runs on started 2.5 us late, and the call ended that much later.
constexpr int kMaxRegs = 104;

// Division of numbers below 2^31 by one that the host knows: multiplication by the rounded-up reciprocal (a division takes a
// hundred instructions in front of every run).
struct FastDiv {
    uint32_t d, mul, shr;
    __device__ __forceinline__ int operator()(int x) const { return d == 1u ? x : static_cast<int>(__umulhi(static_cast<uint32_t>(x), mul) >> shr); }
};
inline FastDiv fast_div(int d) {
    FastDiv f{static_cast<uint32_t>(d), 0u, 0u};
    if (d > 1) {
        int l = 0;
        while ((1LL << l) < d) ++l;
        f.mul = static_cast<uint32_t>(((1ULL << (31 + l)) + d - 1) / d);
        f.shr = l - 1;
    }
    return f;
}

// The units of a call in runs: run j has `len` or, for j < rem, len + 1 of them.
struct Runs {
    int pieces, per_cta;       // runs in all, runs per CTA (one after the other)
    int len, rem;
    int L;                     // units per output tile (row of tiles or window)
    int phases;                // warps (or groups of eight) that share a run
    FastDiv by_len, by_len1, by_L, by_phases;
    __device__ __forceinline__ int first(int j) const { return j * len + min(j, rem); }
    __device__ __forceinline__ int of_unit(int s) const {      // run that holds unit s
        const int big = rem * (len + 1);
        return s < big ? by_len1(s) : rem + by_len(s - big);
    }
    // phase ph of a run of n units starts at its unit start(n, ph); the phase that holds its unit u
    __device__ __forceinline__ int start(int n, int ph) const { return by_phases(n * ph); }
    __device__ __forceinline__ int phase_of(int n, int u) const { return n == len ? by_len((u + 1) * phases - 1) : by_len1((u + 1) * phases - 1); }
};
inline Runs make_runs(int total, int pieces, int per_cta, int L, int phases) {
    Runs r;
    r.pieces = pieces; r.per_cta = per_cta; r.len = total / pieces; r.rem = total % pieces; r.L = L; r.phases = phases;
    r.by_len = fast_div(r.len); r.by_len1 = fast_div(r.len + 1); r.by_L = fast_div(L); r.by_phases = fast_div(phases);
    return r;
}
// A run's part in an output tile that it may share: its slot, and how many runs there are (1: it has the tile to itself).
struct Share { int slot, runs; };

// Groups of eight warps of the forward kernel: two.  (Three with 80 registers: 2-bit codes the same, 3-bit codes
// 22.3 instead of 20.7 us on 8192 x 8192, 4-bit codes spill.)
constexpr int kFwdPhases = 2;

struct Params {
    QView q;
    const __nv_bfloat16* X;    // [M][K]
    const __nv_bfloat16* T;    // [M][r], written by the kernel in front of this one (r > 0)
    const __nv_bfloat16* L1;   // [N][r]
    __nv_bfloat16* Y;          // [M][N]
    float* partial;            // [slots][M][ntiles * 128] sums of the runs that share a tile row
    int* counters;             // [ntiles] arrival counters, zero when the kernel starts
    int M, r;
    Runs runs;
    int chunk;                 // units whose activations are staged at a time
    FastDiv by_M;
    int sstr;                  // floats per block column of a warp's scale table
    int vec8;                  // scale codes of eight blocks are one aligned load
    uint32_t zero_off, stab_off, part_off, lut_off;      // shared-memory offsets
};

__device__ __forceinline__ uint2 ldg_codes(const uint32_t* p) {
    uint2 v;
    asm volatile("ld.global.nc.L1::no_allocate.v2.u32 {%0, %1}, [%2];" : "=r"(v.x), "=r"(v.y) : "l"(p));
    return v;
}

// fl(v / levels), levels = 1, 3, 7 or 127: one Newton step on the product with the rounded reciprocal (Markstein 1990; Brisebarre,
// Muller and Raina 2004, division by a constant).  Equal to the IEEE quotient for every mantissa while the residual does not
// underflow; smaller v (and 0) take the division, and so does infinity (an fp16 second-level scale of block maxima above 65504),
// whose residual is not a number.
__device__ __forceinline__ float scale_quotient(float v, float levels) {
    if (v < 1e-27f || v > 3.402823466e38f) return __fdiv_rn(v, levels);
    const float rc = levels == 127.0f ? 1.0f / 127.0f : levels == 7.0f ? 1.0f / 7.0f : levels == 3.0f ? 1.0f / 3.0f : 1.0f;
    const float q0 = __fmul_rn(v, rc);
    return __fmaf_rn(__fmaf_rn(-q0, levels, v), rc, q0);
}

// Chunk c of a row's 32-column group: o[e] holds two weights.  3- and 4-bit codes: columns 8 c + 2 e and the next one.  2-bit codes: the
// four entries of a block are the bytes of two registers, so one permute yields two whole weights; chunk c holds the even (c even) or odd
// (c odd) columns of the 16 columns 8 (c & 2) .. in ascending order (kSplitColumns).
template <int B> constexpr bool kSplitColumns = B == 2;
template <int B>
__device__ __forceinline__ void dequant8(const uint32_t (&w)[B], int c, const BlockTable<B>& tab, uint32_t (&o)[4]) {
    if constexpr (B == 2) {
        // fields of a word: code i of the first eight columns in bits 4 i, 4 i + 1, code 8 + i in the two above; even columns are
        // the even fields.  Byte c of v -> nibbles 2 c, 2 c + 1 of a selector.
        const uint32_t x = w[c >> 1];
        const uint32_t s0 = (((c & 1) ? x >> 4 : x) & 0x03030303u) * 0x22u + 0x10101010u;
        const uint32_t s1 = (((c & 1) ? x >> 6 : x >> 2) & 0x03030303u) * 0x22u + 0x10101010u;
        o[0] = prmt(tab.lo[0], tab.hi[0], s0);
        o[1] = prmt(tab.lo[0], tab.hi[0], s0 >> 16);
        o[2] = prmt(tab.lo[0], tab.hi[0], s1);
        o[3] = prmt(tab.lo[0], tab.hi[0], s1 >> 16);
    } else {
        const uint32_t sel = chunk_selector<B>(w, c);
        uint32_t a = sel, b = 0u;
        if constexpr (B == 4) { a = sel & 0x77777777u; b = ((sel >> 1) & 0x44444444u) | 0x32103210u; }
        tab.lookup4(a, b, o[0], o[1]);
        tab.lookup4(a >> 16, b >> 16, o[2], o[3]);
    }
}
// The table of a block for dequant8.
template <int B>
__device__ __forceinline__ void build_table(BlockTable<B>& tab, float s) {
    if constexpr (B == 2) {
        const float* cb = c_codebook[0];
        const __nv_bfloat162 h0 = __floats2bfloat162_rn(__fmul_rn(cb[0], s), __fmul_rn(cb[1], s)), h1 = __floats2bfloat162_rn(__fmul_rn(cb[2], s), __fmul_rn(cb[3], s));
        tab.lo[0] = *reinterpret_cast<const uint32_t*>(&h0);
        tab.hi[0] = *reinterpret_cast<const uint32_t*>(&h1);
    } else {
        tab.build(s);
    }
}
// Even / odd halves of 16 bf16 numbers in two vectors.
__device__ __forceinline__ void split_columns(uint4& a, uint4& b) {
    const uint4 e = make_uint4(prmt(a.x, a.y, 0x5410u), prmt(a.z, a.w, 0x5410u), prmt(b.x, b.y, 0x5410u), prmt(b.z, b.w, 0x5410u));
    const uint4 o = make_uint4(prmt(a.x, a.y, 0x7632u), prmt(a.z, a.w, 0x7632u), prmt(b.x, b.y, 0x7632u), prmt(b.z, b.w, 0x7632u));
    a = e; b = o;
}
// 8-bit codes: code book in shared memory, one copy per bank; `lut` = address of this lane's copy.
__device__ __forceinline__ float lut8_at(uint32_t lut, uint32_t byte_offset) {
    float v;
    asm volatile("ld.shared.f32 %0, [%1];" : "=f"(v) : "r"(lut + byte_offset));
    return v;
}
// Fills it (256, 384 or 512 threads): a warp reads 32 entries with one load and hands them round.  (Read from constant memory, 16 entries per
// warp one after the other in front of the first codes, 8-bit calls on small matrices were slower than the kernels before; us in a graph, those /
// that / this, rank 64: 1024 x 1024, one row 8.6 / 9.1 / 8.4; 4096 x 1024, one row 8.8 / 9.4 / 8.6, eight rows 11.0 / 13.6 / 11.5.)
__device__ __forceinline__ void fill_lut8(uint8_t* lut) {
    const int lane = threadIdx.x & 31;
    for (int w = threadIdx.x >> 5; w < 16; w += blockDim.x >> 5) {
        const int first = (w & 7) * 32, half = (w >> 3) * 16;
        const float mine = g_codebook8[first + lane];
#pragma unroll
        for (int j = 0; j < 16; ++j)
            reinterpret_cast<float*>(lut)[(first + half + j) * 32 + lane] = __shfl_sync(0xffffffffu, mine, half + j);
    }
}
__device__ __forceinline__ void dequant8_lut(const uint32_t (&w)[8], int c, uint32_t lut, float s, uint32_t (&o)[4]) {
#pragma unroll
    for (int e = 0; e < 4; ++e) {
        const uint32_t x = w[2 * c + (e >> 1)];
        const uint32_t i0 = (e & 1) ? (x >> 9) & 0x7F80u : (x << 7) & 0x7F80u, i1 = (e & 1) ? (x >> 17) & 0x7F80u : (x >> 1) & 0x7F80u;
        const __nv_bfloat162 h = __floats2bfloat162_rn(__fmul_rn(lut8_at(lut, i0), s), __fmul_rn(lut8_at(lut, i1), s));
        o[e] = *reinterpret_cast<const uint32_t*>(&h);
    }
}

__device__ __forceinline__ Share share_of(const Runs& runs, int piece, int tile) {
    const int f = runs.of_unit(tile * runs.L);
    return Share{piece - f, runs.of_unit(tile * runs.L + runs.L - 1) - f + 1};
}

// Four neighbouring sums over the slots, in slot order, eight slots in flight at a time.  The CTA that arrives last at a tile adds them
// alone; one number and four slots at a time, the round trips to L2 took longer than all else in a call on a small matrix.  us per call in a
// graph, the ring kernels before these / that / this (3-bit codes, rank 64): input gradient 4096 x 1024, 8 rows, 20 slots 18.5 / 25.9 / 13.7;
// 768 x 768, 8 rows, 26 slots 16.4 / 20.2 / 10.8; forward 1024 x 4096, 16 rows, 16 slots 15.4 / 21.1 / 10.9; 568 x 11520, 14 rows, no
// rank-r term, 45 slots 22.6 / 32.9 / 16.7.
__device__ __forceinline__ float4 sum_slots(const float* src, size_t stride, int slots) {
    float4 sum = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
    for (int s0 = 0; s0 < slots; s0 += 8) {
        float4 v[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) v[u] = __ldcg(reinterpret_cast<const float4*>(src + min(s0 + u, slots - 1) * stride));
#pragma unroll
        for (int u = 0; u < 8; ++u)
            if (s0 + u < slots) { sum.x += v[u].x; sum.y += v[u].y; sum.z += v[u].z; sum.w += v[u].w; }
    }
    return sum;
}

// The scales of a warp's 16 rows and 16 blocks: lane = (row, half of the blocks), eight codes and the (at most two, since
// B1 >= 16) second-level scales of their groups.
struct ScaleRun {
    uint2 codes;
    float v0, v1;
    int n0;                    // blocks of the first group
};

template <int B, int NT>
__global__ void __maxnreg__(kMaxRegs) stream_fwd_kernel(const Params p) {
    extern __shared__ __align__(16) uint8_t smem[];
    __shared__ Share share_s[kMaxSegs];
    __shared__ int last_s[kMaxSegs];
    const QView& q = p.q;
    const Runs& runs = p.runs;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int hs = warp & 7, phase = warp >> 3;
    const int gid = lane >> 2, t = lane & 3;
    const int M = p.M, L = runs.L, nthr = blockDim.x;
    float* stab = reinterpret_cast<float*>(smem + p.stab_off + warp * kStabBytes);
    float* part = reinterpret_cast<float*>(smem + p.part_off);
    const uint32_t lut8 = smem_u32(smem + p.lut_off) + lane * 4;

    const int row_in_slab = (hs & 1) * 16 + 2 * gid;
    const int off0 = (hs >> 1) * (64 * B) + slab_row_slot(row_in_slab, 0, t);
    const int off1 = (hs >> 1) * (64 * B) + B * 32 + slab_row_slot(row_in_slab, 1, t);
    const int wrap_words = (kUnitTiles * L - q.ktiles) * (256 * B);      // from the end of a ragged tile row to the next one
    const int run_shift = q.logB0 - 4;                                    // units per run of 16 blocks = 1 << run_shift

    auto load_run = [&](int tr, int run) {
        ScaleRun s;
        s.codes = make_uint2(0u, 0u); s.v0 = s.v1 = 0.0f; s.n0 = 8;
        const int grow = tr * 128 + hs * 16 + (lane & 15), kb0 = run * 16 + (lane >> 4) * 8;
        if (grow < q.N && kb0 < q.KB) {
            const uint32_t blk = static_cast<uint32_t>(grow) * q.KB + kb0;
            const int have = min(8, q.KB - kb0);
            if (p.vec8) s.codes = __ldg(reinterpret_cast<const uint2*>(q.sc + blk));
            else {
#pragma unroll
                for (int j = 0; j < 8; ++j) {
                    const uint32_t c = j < have ? static_cast<uint32_t>(__ldg(q.sc + blk + j)) << (8 * (j & 3)) : 0u;
                    if (j < 4) s.codes.x |= c; else s.codes.y |= c;
                }
            }
            const uint32_t g0 = blk >> q.logB1, g1 = (blk + have - 1) >> q.logB1;
            s.v0 = __ldg(q.v + g0);
            if (g1 != g0) { s.v1 = __ldg(q.v + g1); s.n0 = static_cast<int>((g1 << q.logB1) - blk); }
        }
        return s;
    };
    auto build_run = [&](const ScaleRun& s, int run) {
        const float sig0 = scale_quotient(s.v0, q.levels);
        float sig1 = sig0;
        if (s.n0 < 8) sig1 = scale_quotient(s.v1, q.levels);
        float* dst = stab + (lane >> 4) * 8 * p.sstr + (lane & 15);
        const int have = q.KB - run * 16 - (lane >> 4) * 8;    // blocks behind the last column: zero, whatever the group's scale is
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            const uint32_t c = ((j < 4 ? s.codes.x : s.codes.y) >> (8 * (j & 3))) & 255u;
            dst[j * p.sstr] = j < have ? __fmul_rn(static_cast<float>(c), j < s.n0 ? sig0 : sig1) : 0.0f;
        }
    };

    for (int pc = 0; pc < runs.per_cta; ++pc) {
        const int piece = blockIdx.x * runs.per_cta + pc;
        if (piece >= runs.pieces) break;
        const int i0 = runs.first(piece), i1 = runs.first(piece + 1);
        const int tr0 = runs.by_L(i0), nseg = runs.by_L(i1 - 1) - tr0 + 1;
        if (pc > 0) __syncthreads();                          // the sums of the previous run have been read
        for (int e = threadIdx.x; e < nseg * runs.phases * M * 128; e += nthr) part[e] = 0.0f;

        // as many units at a time as there is room for their activations
        for (int r0 = i0; r0 < i1; r0 += p.chunk) {
        const int n = min(p.chunk, i1 - r0);
        const int a = r0 + runs.start(n, phase), b = r0 + runs.start(n, phase + 1);
        const bool whole = n >= L;                           // these units cover every column
        const int s0 = whole ? 0 : r0 - runs.by_L(r0) * L;   // first staged unit column
        const int staged = whole ? L : n;

        // the first unit's codes and scales are requested before the activations are staged
        int tr = 0, ks = 0, run = 0;
        const uint32_t* ptr = q.codes;
        uint2 wb0[B], wb1[B];
        ScaleRun sr;
        if (a < b) {
            tr = runs.by_L(a); ks = a - tr * L;
            ptr += (static_cast<size_t>(tr) * q.ktiles + ks * kUnitTiles + t) * (256 * B);
            // (a tile behind the last column reads the first one instead; its scales and activations are zero)
            const uint32_t* src = ks * kUnitTiles + t < q.ktiles ? ptr : q.codes;
#pragma unroll
            for (int i = 0; i < B; ++i) { wb0[i] = ldg_codes(src + off0 + i * 32); wb1[i] = ldg_codes(src + off1 + i * 32); }
            run = ks >> run_shift;
            sr = load_run(tr, run);
        }
        if (r0 > i0) __syncthreads();                         // everybody has left the staged activations
        if constexpr (B == 8) {
            if (pc == 0 && r0 == i0) fill_lut8(smem + p.lut_off);      // while the first codes are on their way
        }
        for (int e = threadIdx.x; e < staged * M * 16; e += nthr) {
            const int v = e & 15, pm = e >> 4;                 // 16 columns of one token
            const int pos = p.by_M(pm), m = pm - pos * M;
            int u = s0 + pos;
            if (u >= L) u -= L;
            const int col = u * 256 + v * 16;
            uint4 x0 = make_uint4(0u, 0u, 0u, 0u), x1 = x0;
            if (col < q.K) {
                const uint4* src = reinterpret_cast<const uint4*>(p.X + static_cast<size_t>(m) * q.K + col);
                x0 = __ldg(src);
                x1 = __ldg(src + 1);
            }
            if constexpr (kSplitColumns<B>) split_columns(x0, x1);
            uint4* dst = reinterpret_cast<uint4*>(smem + pm * kXTokenBytes + (v >> 2) * 144 + (v & 3) * 32);
            dst[0] = x0;
            dst[1] = x1;
        }
        for (int e = threadIdx.x; e < kXTokenBytes / 16; e += nthr) *reinterpret_cast<uint4*>(smem + p.zero_off + e * 16) = make_uint4(0u, 0u, 0u, 0u);
        __syncthreads();

        // acc[nt][e]: row 2 gid + (e >> 1) of the half slab, token nt * 8 + 2 t + (e & 1)
        float acc[NT][4];
#pragma unroll
        for (int c = 0; c < NT; ++c)
#pragma unroll
            for (int d = 0; d < 4; ++d) acc[c][d] = 0.0f;
        auto flush = [&](int seg) {
#pragma unroll
            for (int nt = 0; nt < NT; ++nt)
#pragma unroll
                for (int e = 0; e < 2; ++e) {
                    const int m = nt * 8 + 2 * t + e;
                    if (m < M) {
                        float2* dst = reinterpret_cast<float2*>(part + (static_cast<size_t>(seg * runs.phases + phase) * M + m) * 128 + hs * 16 + 2 * gid);
                        const float2 old = *dst;
                        *dst = make_float2(old.x + acc[nt][e], old.y + acc[nt][2 + e]);
                    }
                    acc[nt][e] = acc[nt][2 + e] = 0.0f;
                }
        };

        bool fresh = true;                                     // the scale table has to be rebuilt
        for (int i = a; i < b; ++i) {
            if (fresh) {
                __syncwarp();
                build_run(sr, run);
                __syncwarp();
                int ntr = tr, nrun = run + 1;
                if (nrun * 16 >= q.KB) { ntr = tr + 1; nrun = 0; }
                if (ntr * L + (nrun << run_shift) < b) sr = load_run(ntr, nrun);
            }
            // the unit after this one
            const uint32_t* nptr = ptr + 1024 * B;
            int nks = ks + 1, ntr = tr;
            if (nks == L) { nks = 0; ntr = tr + 1; nptr -= wrap_words; }
            const uint32_t* src = i + 1 < b && nks * kUnitTiles + t < q.ktiles ? nptr : q.codes;

            const int pos = whole ? ks : i - r0;
            // activations of the tokens gid and gid + 8 (zeros for tokens past M)
            const bool have0 = gid < M, have1 = NT == 2 && gid + 8 < M;
            const uint8_t* xp = smem + (have0 ? (pos * M + gid) * kXTokenBytes : p.zero_off) + t * 144;
            const uint8_t* xp1 = smem + (have1 ? (pos * M + gid + 8) * kXTokenBytes : p.zero_off) + t * 144;
            const int col = ks * 256 + t * 64;
            BlockTable<B == 8 ? 3 : B> ta, tb;
            float2 s = make_float2(0.0f, 0.0f);
#pragma unroll
            for (int g = 0; g < 2; ++g) {
                uint32_t wa[B], wb[B];
#pragma unroll
                for (int j = 0; j < B; ++j) { const uint2 w = g ? wb1[j] : wb0[j]; wa[j] = w.x; wb[j] = w.y; }
#pragma unroll
                for (int c = 0; c < 4; ++c) {
                    // first columns of a block
                    if ((c == 0 && (g == 0 || q.logB0 < 6)) || (c == 2 && q.logB0 == 4)) {
                        const int kb = ((col + g * 32 + c * 8) >> q.logB0) & 15;
                        s = *reinterpret_cast<const float2*>(stab + kb * p.sstr + 2 * gid);
                        if constexpr (B != 8) { build_table<B>(ta, s.x); build_table<B>(tb, s.y); }
                    }
                    const uint4 x0 = *reinterpret_cast<const uint4*>(xp + (g * 4 + c) * 16);
                    uint32_t oa[4], ob[4];
                    if constexpr (B == 8) { dequant8_lut(wa, c, lut8, s.x, oa); dequant8_lut(wb, c, lut8, s.y, ob); }
                    else { dequant8<B>(wa, c, ta, oa); dequant8<B>(wb, c, tb, ob); }
                    dec::mma16816(acc[0], oa[0], ob[0], oa[1], ob[1], x0.x, x0.y);
                    dec::mma16816(acc[0], oa[2], ob[2], oa[3], ob[3], x0.z, x0.w);
                    if constexpr (NT == 2) {
                        const uint4 x1 = *reinterpret_cast<const uint4*>(xp1 + (g * 4 + c) * 16);
                        dec::mma16816(acc[NT - 1], oa[0], ob[0], oa[1], ob[1], x1.x, x1.y);
                        dec::mma16816(acc[NT - 1], oa[2], ob[2], oa[3], ob[3], x1.z, x1.w);
                    }
                }
#pragma unroll
                for (int j = 0; j < B; ++j) (g ? wb1[j] : wb0[j]) = ldg_codes(src + (g ? off1 : off0) + j * 32);
            }
            if (ntr != tr && p.r > 0) {
                // the last unit of a tile row: T L1^T as more contraction steps, 16 columns of the factors per MMA
                pdl_wait();                                    // T has been written by the kernel in front
                const int na = tr * 128 + hs * 16 + 2 * gid;
#pragma unroll 4
                for (int j = 4 * t; j < p.r; j += 16) {
                    uint2 la = make_uint2(0u, 0u), lb = la, t0 = la;
                    if (na < q.N) la = __ldg(reinterpret_cast<const uint2*>(p.L1 + static_cast<size_t>(na) * p.r + j));
                    if (na + 1 < q.N) lb = __ldg(reinterpret_cast<const uint2*>(p.L1 + static_cast<size_t>(na + 1) * p.r + j));
                    if (have0) t0 = __ldcg(reinterpret_cast<const uint2*>(p.T + static_cast<size_t>(gid) * p.r + j));
                    dec::mma16816(acc[0], la.x, lb.x, la.y, lb.y, t0.x, t0.y);
                    if constexpr (NT == 2) {
                        uint2 t1 = make_uint2(0u, 0u);
                        if (have1) t1 = __ldcg(reinterpret_cast<const uint2*>(p.T + static_cast<size_t>(gid + 8) * p.r + j));
                        dec::mma16816(acc[NT - 1], la.x, lb.x, la.y, lb.y, t1.x, t1.y);
                    }
                }
            }
            if (ntr != tr || i + 1 == b) flush(tr - tr0);
            fresh = ntr != tr || (nks >> run_shift) != run;
            ptr = nptr; ks = nks; tr = ntr; run = nks >> run_shift;
        }

        }

        // ------------------------------------------------------------------ reduction, output
        const int npad = q.ntiles * 128;
        if (threadIdx.x < nseg) share_s[threadIdx.x] = share_of(runs, piece, tr0 + threadIdx.x);
        if (pc + 1 == runs.per_cta || piece + 1 == runs.pieces) pdl_launch_dependents();    // the next call's pre-product may take its place (it waits for this kernel)
        __syncthreads();
        pdl_wait();                                           // the kernel in front has cleared the counters
        auto put_out = [&](int m, int row, float v) {
            if (row < q.N) p.Y[static_cast<size_t>(m) * q.N + row] = __float2bfloat16_rn(v);
        };
        bool shared_any = false;
        for (int seg = 0; seg < nseg; ++seg) {
            const Share sh = share_s[seg];
            const bool alone = sh.runs == 1;
            shared_any |= !alone;
            float* dst = p.partial + static_cast<size_t>(sh.slot) * M * npad;
            for (int e = threadIdx.x; e < 128 * M; e += nthr) {
                const float* src = part + static_cast<size_t>(seg * runs.phases) * M * 128 + e;
                float sum = 0.0f;
                for (int ph = 0; ph < runs.phases; ++ph) sum += src[static_cast<size_t>(ph) * M * 128];
                const int m = e >> 7, row = (tr0 + seg) * 128 + (e & 127);
                if (alone) put_out(m, row, sum);
                else __stcg(dst + static_cast<size_t>(m) * npad + row, sum);
            }
        }
        if (!shared_any) continue;                            // (the same for all threads)
        __threadfence();
        __syncthreads();
        if (threadIdx.x < nseg) {
            const Share sh = share_s[threadIdx.x];
            last_s[threadIdx.x] = sh.runs > 1 && atomicAdd(p.counters + tr0 + threadIdx.x, 1) == sh.runs - 1 ? sh.runs : 0;
        }
        __syncthreads();
        __threadfence();
        for (int seg = 0; seg < nseg; ++seg) {
            const int slots = last_s[seg];
            if (slots == 0) continue;
            for (int e = threadIdx.x; e < 32 * M; e += nthr) {
                const int m = e >> 5, row = (tr0 + seg) * 128 + (e & 31) * 4;
                const float4 sum = sum_slots(p.partial + static_cast<size_t>(m) * npad + row, static_cast<size_t>(M) * npad, slots);
                put_out(m, row, sum.x);
                put_out(m, row + 1, sum.y);
                put_out(m, row + 2, sum.z);
                put_out(m, row + 3, sum.w);
            }
        }
    }
}

// ------------------------------------------------------------------------------------ input gradient for few rows
// dX[m][k] = sum_n dY[m][n] deq16(Q)[n][k] + sum_j T'[m][j] L2[j][k],  M <= 16.
//
// The same structure, transposed: a unit is one slab (32 rows) of a window of 128 columns (two tiles), a run goes down the rows of
// a window and on into the next one.  The contraction runs over rows, so the tensor-core operand needs pairs (W[n][k],
// W[n + 1][k]): lane = row dequantizes the 64 weights of its row of a tile (one table for blocks of 64 and more) into the warp's
// own 4 KB tile in shared memory (16-byte chunks, XOR swizzle), and ldmatrix.trans reads it back as the 16-column operand.
// (Merging the look-ups of two rows with byte permutes instead costs half a permute per weight on the pipe that binds, and 64
// accumulator registers.)  Output gradients and scales are loaded one unit ahead into registers.  The rank-r term T' L2 is r / 32
// more units at the end of a window: rows of L2 in place of dequantized weights, T' in place of dY.
struct BwdParams {
    QView q;
    const __nv_bfloat16* dY;   // [M][N]
    const __nv_bfloat16* T;    // [M][r] = dY L1, written by the kernel in front of this one (r > 0)
    const __nv_bfloat16* L2;   // [r][K]
    __nv_bfloat16* dX;         // [M][K]
    float* partial;            // [slots][M][windows * 128] sums of the runs that share a window
    int* counters;             // [windows] arrival counters, zero when the kernel starts
    int M, r;
    Runs runs;
    int slabs;                 // units of a window that are slabs (the others belong to the rank-r term)
    int windows;
    int nsc;                   // blocks per row of a window (1 for blocks of 128 and more)
    int vec;                   // the scale codes of a row of a window are one aligned load
    uint32_t mid_off, lut_off; // shared-memory offsets
};

// Sixteen warps.  (24 or 20 with 80 or 96 registers: 8192 x 28672 NF2, one row, 81 us instead of 57; 8192 x 8192 NF4 37.4 instead of 31.8, from
// spills.  These spill as well, less: 16 to 60 bytes of stores a thread at up to eight rows with 104 registers, 64 to 232 above with 128.)
constexpr int kBwdWarps = 16;
template <int NT> __host__ __device__ constexpr int bwd_warp_bytes() { return 4096 + 8 * NT * 80; }      // weight tile, 32 output gradients of each token

__device__ __forceinline__ uint32_t ldg_word(const uint32_t* p) {
    uint32_t v;
    asm volatile("ld.global.nc.L1::no_allocate.u32 %0, [%1];" : "=r"(v) : "l"(p));
    return v;
}
__device__ __forceinline__ void ldmatrix_x4_trans(uint32_t addr, uint32_t (&v)[4]) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0, %1, %2, %3}, [%4];"
                 : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]) : "r"(addr) : "memory");
}

template <int B, int NT>
__global__ void __maxnreg__(NT == 1 ? kMaxRegs : 128) stream_bwd_kernel(const BwdParams p) {
    extern __shared__ __align__(16) uint8_t smem[];
    __shared__ Share share_s[kMaxSegs];
    __shared__ int last_s[kMaxSegs];
    const QView& q = p.q;
    const Runs& runs = p.runs;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int gid = lane >> 2, t = lane & 3;
    const int M = p.M, L = runs.L, nthr = blockDim.x;
    const uint32_t wtile = smem_u32(smem) + warp * bwd_warp_bytes<NT>(), ybuf = wtile + 4096;
    float* fin = reinterpret_cast<float*>(smem);                          // [phase][M][128], over the warps' tiles once all are done
    float* mid = reinterpret_cast<float*>(smem + p.mid_off);              // [segment][M][128] of warps whose run goes on in the next window
    const uint32_t lut8 = smem_u32(smem + p.lut_off) + lane * 4;
    // where lane l finds its row of the four 8 x 8 matrices of an ldmatrix: contraction rows (l & 7) + 8 (l / 16), columns 8 (l / 8 % 2)
    const int mrow = (lane & 7) + ((lane >> 4) << 3), mchunk = (lane >> 3) & 1;

    if constexpr (B == 8) {
        fill_lut8(smem + p.lut_off);
        __syncthreads();
    }

    struct RowScale { uint2 codes; float v0, v1; int n0; };
    auto load_scale = [&](int win, int slab) {
        RowScale s;
        s.codes = make_uint2(0u, 0u); s.v0 = s.v1 = 0.0f; s.n0 = 8;
        const int row = slab * 32 + lane, kb0 = (win * 128) >> q.logB0;
        if (row < q.N) {
            const uint32_t blk = static_cast<uint32_t>(row) * q.KB + kb0;
            const int have = min(p.nsc, q.KB - kb0);
            if (p.nsc == 1) s.codes.x = __ldg(q.sc + blk);
            else if (p.vec) {
                if (p.nsc == 2) s.codes.x = __ldg(reinterpret_cast<const uint16_t*>(q.sc + blk));
                else if (p.nsc == 4) s.codes.x = __ldg(reinterpret_cast<const uint32_t*>(q.sc + blk));
                else s.codes = __ldg(reinterpret_cast<const uint2*>(q.sc + blk));
            } else {
#pragma unroll
                for (int j = 0; j < 8; ++j) {
                    const uint32_t c = j < have ? static_cast<uint32_t>(__ldg(q.sc + blk + j)) << (8 * (j & 3)) : 0u;
                    if (j < 4) s.codes.x |= c; else s.codes.y |= c;
                }
            }
            const uint32_t g0 = blk >> q.logB1, g1 = (blk + have - 1) >> q.logB1;
            s.v0 = __ldg(q.v + g0);
            if (g1 != g0) { s.v1 = __ldg(q.v + g1); s.n0 = static_cast<int>((g1 << q.logB1) - blk); }
        }
        return s;
    };
    // eight output gradients per lane: token lane / 4 (+ 8), rows 8 (lane % 4) of the slab
    auto load_y = [&](int slab, uint4 (&y)[NT]) {
#pragma unroll
        for (int nt = 0; nt < NT; ++nt) {
            const int m = nt * 8 + gid, n = slab * 32 + t * 8;
            y[nt] = make_uint4(0u, 0u, 0u, 0u);
            if (m < M && n < q.N) y[nt] = __ldg(reinterpret_cast<const uint4*>(p.dY + static_cast<size_t>(m) * q.N + n));
        }
    };
    auto load_t = [&](int part, uint4 (&y)[NT]) {
#pragma unroll
        for (int nt = 0; nt < NT; ++nt) {
            const int m = nt * 8 + gid, j = part * 32 + t * 8;
            y[nt] = make_uint4(0u, 0u, 0u, 0u);
            if (m < M && j < p.r) y[nt] = __ldcg(reinterpret_cast<const uint4*>(p.T + static_cast<size_t>(m) * p.r + j));
        }
    };
    // 16 bytes of this lane's row of the warp's tile
    auto sts_chunk = [&](int c, uint32_t x, uint32_t y, uint32_t z, uint32_t v) {
        asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(wtile + lane * 128 + ((c * 16) ^ ((lane & 7) << 4))), "r"(x), "r"(y), "r"(z), "r"(v) : "memory");
    };
    // the packed words of this lane's row of tile j of a unit
    auto load_words = [&](int win, int slab, int j, uint32_t (&w)[2][B]) {
        const int kt = 2 * win + j;
        const uint32_t* base = q.codes + (static_cast<size_t>(slab >> 2) * q.ktiles + min(kt, q.ktiles - 1)) * (256 * B) + (slab & 3) * (64 * B);
#pragma unroll
        for (int g = 0; g < 2; ++g)
#pragma unroll
            for (int i = 0; i < B; ++i) w[g][i] = ldg_word(base + (g * B + i) * 32 + ((lane + 8 * g + 16 * j) & 31));
    };

    for (int pc = 0; pc < runs.per_cta; ++pc) {
        const int piece = blockIdx.x * runs.per_cta + pc;
        if (piece >= runs.pieces) break;
        const int i0 = runs.first(piece), i1 = runs.first(piece + 1), n = i1 - i0;
        const int w0 = runs.by_L(i0);
        const int a = warp < runs.phases ? i0 + runs.start(n, warp) : 0, b = warp < runs.phases ? i0 + runs.start(n, warp + 1) : 0;

        float acc[2][4][NT][4];      // [tile][16 columns][8 tokens]: columns gid (+ 8 for e >= 2), tokens 2 t + (e & 1)
        auto clear = [&]() {
#pragma unroll
            for (int j = 0; j < 2; ++j)
#pragma unroll
                for (int c = 0; c < 4; ++c)
#pragma unroll
                    for (int nt = 0; nt < NT; ++nt)
#pragma unroll
                        for (int e = 0; e < 4; ++e) acc[j][c][nt][e] = 0.0f;
        };
        auto flush = [&](float* dst) {
#pragma unroll
            for (int j = 0; j < 2; ++j)
#pragma unroll
                for (int c = 0; c < 4; ++c)
#pragma unroll
                    for (int nt = 0; nt < NT; ++nt)
#pragma unroll
                        for (int e = 0; e < 4; ++e) {
                            const int m = nt * 8 + 2 * t + (e & 1);
                            const int in16 = kSplitColumns<B> ? 2 * gid + (e >> 1) : gid + 8 * (e >> 1);
                            if (m < M) dst[m * 128 + j * 64 + c * 16 + in16] = acc[j][c][nt][e];
                        }
        };
        clear();
        if (pc > 0) __syncthreads();                          // the sums of the previous run have been read
        if (a < b) {
            int win = runs.by_L(a), slab = a - win * L;
            uint32_t words[2][B];
            uint4 yv[NT];
            RowScale sc;
            if (slab < p.slabs) {
                sc = load_scale(win, slab);
                load_words(win, slab, 0, words);
                load_y(slab, yv);
            }
            for (int i = a; i < b; ++i) {
                int nwin = win, nslab = slab + 1;
                if (nslab == L) { nslab = 0; ++nwin; }
                const bool rank = slab >= p.slabs;               // a unit of the rank-r term
                const bool more = i + 1 < b && nslab < p.slabs;   // the next unit's weights are requested now
                if (rank) {
                    pdl_wait();                                   // T' has been written by the kernel in front
                    load_t(slab - p.slabs, yv);
                }
                // output gradients as the 8-column operand
                uint32_t yb[2][NT][2];
                __syncwarp();
#pragma unroll
                for (int nt = 0; nt < NT; ++nt)
                    asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(ybuf + (nt * 8 + gid) * 80 + t * 16), "r"(yv[nt].x), "r"(yv[nt].y), "r"(yv[nt].z), "r"(yv[nt].w) : "memory");
                __syncwarp();
#pragma unroll
                for (int kb = 0; kb < 2; ++kb)
#pragma unroll
                    for (int nt = 0; nt < NT; ++nt)
#pragma unroll
                        for (int h = 0; h < 2; ++h)
                            asm volatile("ld.shared.u32 %0, [%1];" : "=r"(yb[kb][nt][h]) : "r"(ybuf + (nt * 8 + gid) * 80 + (kb * 16 + h * 8 + 2 * t) * 2));
                float sig0 = 0.0f, sig1 = 0.0f;
                if (!rank) {
                    sig0 = scale_quotient(sc.v0, q.levels);
                    sig1 = sc.n0 < 8 ? scale_quotient(sc.v1, q.levels) : sig0;
                }
                const uint2 codes = sc.codes;
                const int n0 = sc.n0;
                if (more) { sc = load_scale(nwin, nslab); load_y(nslab, yv); }
                BlockTable<B == 8 ? 3 : B> tab;
                float s = 0.0f;
#pragma unroll
                for (int j = 0; j < 2; ++j) {
                    uint32_t w[2][B];
#pragma unroll
                    for (int g = 0; g < 2; ++g)
#pragma unroll
                        for (int k = 0; k < B; ++k) w[g][k] = words[g][k];
                    if (j == 0) { if (!rank) load_words(win, slab, 1, words); }
                    else if (more) load_words(nwin, nslab, 0, words);
                    if (2 * win + j >= q.ktiles) continue;      // the last window may have one tile
                    if (rank) {
                        const int row = (slab - p.slabs) * 32 + lane;
                        const uint4* src = reinterpret_cast<const uint4*>(p.L2 + static_cast<size_t>(row) * q.K + (2 * win + j) * 64);
#pragma unroll
                        for (int c = 0; c < 8; c += 2) {
                            uint4 f0 = make_uint4(0u, 0u, 0u, 0u), f1 = f0;
                            if (row < p.r) { f0 = __ldg(src + c); f1 = __ldg(src + c + 1); }
                            if constexpr (kSplitColumns<B>) split_columns(f0, f1);
                            sts_chunk(c, f0.x, f0.y, f0.z, f0.w);
                            sts_chunk(c + 1, f1.x, f1.y, f1.z, f1.w);
                        }
                    } else {
#pragma unroll
                    for (int g = 0; g < 2; ++g)
#pragma unroll
                        for (int c = 0; c < 4; ++c) {
                            // first columns of a block
                            if ((c == 0 && (g == 0 ? (j == 0 || q.logB0 < 7) : q.logB0 < 6)) || (c == 2 && q.logB0 == 4)) {
                                const int idx = p.nsc == 1 ? 0 : (j * 64 + g * 32 + c * 8) >> q.logB0;
                                const uint32_t code = ((idx < 4 ? codes.x : codes.y) >> (8 * (idx & 3))) & 255u;
                                s = __fmul_rn(static_cast<float>(code), idx < n0 ? sig0 : sig1);
                                if constexpr (B != 8) build_table<B>(tab, s);
                            }
                            uint32_t o[4];
                            if constexpr (B == 8) dequant8_lut(w[g], c, lut8, s, o);
                            else dequant8<B>(w[g], c, tab, o);
                            sts_chunk(g * 4 + c, o[0], o[1], o[2], o[3]);
                        }
                    }
                    __syncwarp();
#pragma unroll
                    for (int kb = 0; kb < 2; ++kb)
#pragma unroll
                        for (int c = 0; c < 4; ++c) {
                            uint32_t av[4];
                            ldmatrix_x4_trans(wtile + (kb * 16 + mrow) * 128 + (((2 * c + mchunk) * 16) ^ ((mrow & 7) << 4)), av);
#pragma unroll
                            for (int nt = 0; nt < NT; ++nt) dec::mma16816(acc[j][c][nt], av[0], av[1], av[2], av[3], yb[kb][nt][0], yb[kb][nt][1]);
                        }
                    __syncwarp();
                }
                if (i + 1 < b && nwin != win) { flush(mid + static_cast<size_t>(win - w0) * M * 128); clear(); }
                win = nwin; slab = nslab;
            }
        }

        // ------------------------------------------------------------------ reduction, output
        const int nseg = runs.by_L(i1 - 1) - w0 + 1, kpad = p.windows * 128;
        if (threadIdx.x < nseg) share_s[threadIdx.x] = share_of(runs, piece, w0 + threadIdx.x);
        if (pc + 1 == runs.per_cta || piece + 1 == runs.pieces) pdl_launch_dependents();    // the next call's pre-product may take its place (it waits for this kernel)
        __syncthreads();                                      // the warps' tiles are idle
        if (a < b) flush(fin + static_cast<size_t>(warp) * M * 128);
        pdl_wait();                                           // the kernel in front has cleared the counters
        __syncthreads();
        auto put_out = [&](int m, int col, float v) {
            if (col < q.K) p.dX[static_cast<size_t>(m) * q.K + col] = __float2bfloat16_rn(v);
        };
        bool shared_any = false;
        for (int seg = 0; seg < nseg; ++seg) {
            const Share sh = share_s[seg];
            const bool alone = sh.runs == 1;
            shared_any |= !alone;
            float* dst = p.partial + static_cast<size_t>(sh.slot) * M * kpad;
            // warps that worked on the window: those that hold its first and its last unit, and the ones in between; the last one's
            // sums are in `mid` if it went on to the next window
            const int hi = (w0 + seg + 1) * L;
            const int ph0 = runs.phase_of(n, max(hi - L, i0) - i0), ph1 = runs.phase_of(n, min(hi, i1) - 1 - i0);
            const float* top = i0 + runs.start(n, ph1 + 1) > hi ? mid + static_cast<size_t>(seg) * M * 128 : fin + static_cast<size_t>(ph1) * M * 128;
            for (int e = threadIdx.x; e < 128 * M; e += nthr) {
                float sum = 0.0f;
#pragma unroll 4
                for (int ph = ph0; ph < ph1; ++ph) sum += fin[static_cast<size_t>(ph) * M * 128 + e];
                sum += top[e];
                const int m = e >> 7, col = (w0 + seg) * 128 + (e & 127);
                if (alone) put_out(m, col, sum);
                else __stcg(dst + static_cast<size_t>(m) * kpad + col, sum);
            }
        }
        if (!shared_any) continue;                            // (the same for all threads)
        __threadfence();
        __syncthreads();
        if (threadIdx.x < nseg) {
            const Share sh = share_s[threadIdx.x];
            last_s[threadIdx.x] = sh.runs > 1 && atomicAdd(p.counters + w0 + threadIdx.x, 1) == sh.runs - 1 ? sh.runs : 0;
        }
        __syncthreads();
        __threadfence();
        for (int seg = 0; seg < nseg; ++seg) {
            const int slots = last_s[seg];
            if (slots == 0) continue;
            for (int e = threadIdx.x; e < 32 * M; e += nthr) {
                const int m = e >> 5, col = (w0 + seg) * 128 + (e & 31) * 4;
                const float4 sum = sum_slots(p.partial + static_cast<size_t>(m) * kpad + col, static_cast<size_t>(M) * kpad, slots);
                put_out(m, col, sum.x);
                put_out(m, col + 1, sum.y);
                put_out(m, col + 2, sum.z);
                put_out(m, col + 3, sum.w);
            }
        }
    }
}

// ------------------------------------------------------------------------------------ host side
struct Plan {
    bool ok;
    int NT, L, pieces, per_cta, ctas, phases, slots, chunk;
    uint32_t zero_off, stab_off, part_off, lut_off, smem;
};

// Slots of the runs that share output tiles are kept below this (calls with the library's own scratch have 8 MiB in all).
constexpr size_t kMaxPartialBytes = size_t(6) << 20;

// Runs of equal length, one per SM (several after each other where a run would touch more than three tile rows); whole tile rows
// where the slots of shared ones would take too much room.
inline Plan compute_plan(const QView& q, int M) {
    Plan pl{};
    pl.NT = M <= 8 ? 1 : 2;
    pl.L = (q.ktiles + kUnitTiles - 1) / kUnitTiles;
    const long long total = static_cast<long long>(q.ntiles) * pl.L, sms = dec::sm_count_cached();
    if (total >= (1LL << 31)) return pl;
    const long long need = (total + 2 * pl.L) / (2 * pl.L + 1);             // runs of at most 2 L + 1 units
    pl.per_cta = static_cast<int>((need + sms - 1) / sms);
    pl.pieces = static_cast<int>(total < sms * pl.per_cta ? total : sms * pl.per_cta);
    const int nmin = static_cast<int>(total / pl.pieces);
    pl.slots = (pl.L - 1 + nmin - 1) / nmin + 1;
    const bool whole_rows = static_cast<size_t>(pl.slots) * M * q.ntiles * 512 > kMaxPartialBytes;
    if (whole_rows) {
        pl.pieces = q.ntiles;
        pl.per_cta = static_cast<int>((pl.pieces + sms - 1) / sms);
        pl.slots = 1;
    }
    pl.ctas = (pl.pieces + pl.per_cta - 1) / pl.per_cta;
    const int n = static_cast<int>((total + pl.pieces - 1) / pl.pieces);
    const int segs = whole_rows || n == 1 ? 1 : n <= pl.L + 1 ? 2 : 3;      // tile rows that a run may touch
    pl.phases = n >= kFwdPhases ? kFwdPhases : n;
    const int token = kXTokenBytes * M;
    const int zero = (kXTokenBytes + 127) / 128 * 128, stab = pl.phases * 8 * kStabBytes, part = segs * pl.phases * M * 512, lut = q.b0 == 8 ? 32768 : 0;
    const int room = (kSmemLimit - 1024 - zero - stab - part - lut) / token;
    if (room < 1) return pl;
    pl.chunk = n;
    if (room < (n < pl.L ? n : pl.L)) {
        const int rounds = (n + room - 1) / room;
        pl.chunk = (n + rounds - 1) / rounds;
    }
    const int xs = ((pl.chunk < pl.L ? pl.chunk : pl.L) * token + 127) / 128 * 128;
    pl.zero_off = static_cast<uint32_t>(xs);
    pl.stab_off = pl.zero_off + zero;
    pl.part_off = pl.stab_off + stab;
    pl.lut_off = pl.part_off + part;
    pl.smem = pl.lut_off + lut;
    pl.ok = pl.smem <= static_cast<uint32_t>(kSmemLimit) - 512;
    return pl;
}
inline Plan make_plan(const QView& q, int M) { return dec::cached_plan<Plan>(q, M, 0, [&] { return compute_plan(q, M); }); }

template <int B, int NT>
inline cudaError_t launch_nt(const Params& p, const Plan& pl, cudaStream_t st) {
    auto kern = stream_fwd_kernel<B, NT>;
    static bool attr_done = false;
    if (!attr_done) {
        const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemLimit - 64);
        if (e != cudaSuccess) return e;
        attr_done = true;
    }
    return dec::launch_stream_kernel(kern, p, dim3(pl.ctas), pl.phases * 256, pl.smem, st);
}

// Forward for M <= 16.  The kernel in front (the pre-product, or one that does nothing else) clears the status word and the arrival counters.
template <int B>
inline cudaError_t launch_fwd(const QView& q, const void* L1, const void* L2, int r, const void* X, int M, void* Y, char* ws,
                              cudaStream_t st) {
    const Plan pl = make_plan(q, M);
    const dec::WsLayout w = dec::ws_layout(q.ntiles, M, r, pl.slots, q.ntiles * 128);
    Params p;
    p.q = q;
    p.X = static_cast<const __nv_bfloat16*>(X);
    p.T = reinterpret_cast<const __nv_bfloat16*>(ws + w.t_off);
    p.L1 = static_cast<const __nv_bfloat16*>(L1);
    p.Y = static_cast<__nv_bfloat16*>(Y);
    p.partial = reinterpret_cast<float*>(ws + w.partial_off);
    p.counters = reinterpret_cast<int*>(ws + w.counters_off);
    p.M = M; p.r = r; p.by_M = fast_div(M); p.chunk = pl.chunk;
    p.runs = make_runs(q.ntiles * pl.L, pl.pieces, pl.per_cta, pl.L, pl.phases);
    p.sstr = q.logB0 == 4 ? 18 : q.logB0 == 5 ? 20 : 24;
    p.vec8 = q.KB % 8 == 0 ? 1 : 0;
    p.zero_off = pl.zero_off; p.stab_off = pl.stab_off; p.part_off = pl.part_off; p.lut_off = pl.lut_off;
    if (r > 0) {
        const cudaError_t e = dec::launch_pre<false>(p.X, static_cast<const __nv_bfloat16*>(L2), reinterpret_cast<__nv_bfloat16*>(ws + w.t_off),
                                                     reinterpret_cast<int*>(ws), p.counters, q.ntiles, M, q.K, r, pl.smem, st);
        if (e != cudaSuccess) return e;
    } else {
        const cudaError_t e = dec::launch_clear(reinterpret_cast<int*>(ws), p.counters, q.ntiles, st);
        if (e != cudaSuccess) return e;
    }
    return pl.NT == 1 ? launch_nt<B, 1>(p, pl, st) : launch_nt<B, 2>(p, pl, st);
}


struct BwdPlan {
    bool ok;
    int NT, slabs, L, windows, pieces, per_cta, ctas, phases, nsc, slots;
    uint32_t mid_off, lut_off, smem, threads;
};
inline BwdPlan compute_bwd_plan(const QView& q, int M, int r) {
    BwdPlan pl{};
    pl.NT = M <= 8 ? 1 : 2;
    pl.slabs = (q.N + 31) / 32;
    pl.L = pl.slabs + (r + 31) / 32;
    pl.windows = (q.ktiles + 1) / 2;
    const long long total = static_cast<long long>(pl.windows) * pl.L;
    if (total >= (1LL << 31)) return pl;
    const long long sms = dec::sm_count_cached();
    // a run touches at most three windows (two slots for warps whose run goes on in the next window)
    const long long need = (total + 2 * pl.L - 1) / (2 * pl.L);
    pl.per_cta = static_cast<int>((need + sms - 1) / sms);
    pl.pieces = static_cast<int>(total < sms * pl.per_cta ? total : sms * pl.per_cta);
    pl.slots = static_cast<int>((pl.L - 1 + total / pl.pieces - 1) / (total / pl.pieces) + 1);
    if (static_cast<size_t>(pl.slots) * M * pl.windows * 512 > kMaxPartialBytes) {      // whole windows
        pl.pieces = pl.windows;
        pl.per_cta = static_cast<int>((pl.pieces + sms - 1) / sms);
        pl.slots = 1;
    }
    pl.ctas = (pl.pieces + pl.per_cta - 1) / pl.per_cta;
    const long long n = (total + pl.pieces - 1) / pl.pieces, nmin = total / pl.pieces;
    constexpr int warps = kBwdWarps;
    pl.phases = static_cast<int>(nmin < warps ? nmin : warps);
    pl.threads = 32u * static_cast<uint32_t>(pl.phases <= 8 ? 8 : pl.phases <= 12 ? 12 : pl.phases <= 16 ? 16 : warps);
    pl.nsc = q.B0 >= 128 ? 1 : 128 / q.B0;
    const uint32_t tiles = (pl.threads / 32) * (pl.NT == 1 ? bwd_warp_bytes<1>() : bwd_warp_bytes<2>()), fin = static_cast<uint32_t>(pl.phases * M * 512);
    pl.mid_off = ((tiles > fin ? tiles : fin) + 127) / 128 * 128;
    pl.lut_off = pl.mid_off + static_cast<uint32_t>((n > 1 ? kMaxSegs - 1 : 0) * M * 512);
    pl.smem = pl.lut_off + (q.b0 == 8 ? 32768 : 0);
    pl.ok = n <= 2LL * pl.L && pl.smem + 1024 <= static_cast<uint32_t>(kSmemLimit);
    return pl;
}
inline BwdPlan make_bwd_plan(const QView& q, int M, int r) { return dec::cached_plan<BwdPlan>(q, M, r, [&] { return compute_bwd_plan(q, M, r); }); }

template <int B, int NT>
inline cudaError_t launch_bwd_nt(const BwdParams& p, const BwdPlan& pl, cudaStream_t st) {
    auto kern = stream_bwd_kernel<B, NT>;
    static bool attr_done = false;
    if (!attr_done) {
        const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemLimit - 64);
        if (e != cudaSuccess) return e;
        attr_done = true;
    }
    return dec::launch_stream_kernel(kern, p, dim3(pl.ctas), pl.threads, pl.smem, st);
}

// Input gradient for M <= 16; same conventions as launch_fwd.
template <int B>
inline cudaError_t launch_bwd(const QView& q, const void* L1, const void* L2, int r, const void* dY, int M, void* dX, char* ws,
                              cudaStream_t st) {
    const BwdPlan pl = make_bwd_plan(q, M, r);
    const dec::WsLayout w = dec::ws_layout(pl.windows, M, r, pl.slots, pl.windows * 128);
    BwdParams p;
    p.q = q;
    p.dY = static_cast<const __nv_bfloat16*>(dY);
    p.T = reinterpret_cast<const __nv_bfloat16*>(ws + w.t_off);
    p.L2 = static_cast<const __nv_bfloat16*>(L2);
    p.dX = static_cast<__nv_bfloat16*>(dX);
    p.partial = reinterpret_cast<float*>(ws + w.partial_off);
    p.counters = reinterpret_cast<int*>(ws + w.counters_off);
    p.M = M; p.r = r; p.slabs = pl.slabs; p.windows = pl.windows;
    p.runs = make_runs(pl.windows * pl.L, pl.pieces, pl.per_cta, pl.L, pl.phases);
    p.nsc = pl.nsc; p.vec = q.KB % pl.nsc == 0 ? 1 : 0;
    p.mid_off = pl.mid_off; p.lut_off = pl.lut_off;
    if (r > 0) {
        const cudaError_t e = dec::launch_pre<true>(p.dY, static_cast<const __nv_bfloat16*>(L1), reinterpret_cast<__nv_bfloat16*>(ws + w.t_off),
                                                    reinterpret_cast<int*>(ws), p.counters, pl.windows, M, q.N, r, pl.smem, st);
        if (e != cudaSuccess) return e;
    } else {
        const cudaError_t e = dec::launch_clear(reinterpret_cast<int*>(ws), p.counters, pl.windows, st);
        if (e != cudaSuccess) return e;
    }
    return pl.NT == 1 ? launch_bwd_nt<B, 1>(p, pl, st) : launch_bwd_nt<B, 2>(p, pl, st);
}

inline bool supported(const QView& q, int64_t M) {
    // 40960: as for the kernels before these, which staged a contraction in shared memory.  Nothing here depends on it; longer contractions
    // have been neither timed nor tested on these kernels and take the plain one.
    if (M > 16 || q.K % 8 != 0 || q.K > 40960) return false;
    if (static_cast<long long>(q.N) * q.KB >= (1LL << 31)) return false;
    return make_plan(q, static_cast<int>(M)).ok;
}
inline bool bwd_supported(const QView& q, int r, int64_t M) {
    if (M > 16 || q.N % 8 != 0 || q.K % 8 != 0 || q.N > 40960) return false;      // (see above)
    if (static_cast<long long>(q.N) * q.KB >= (1LL << 31)) return false;
    return make_bwd_plan(q, static_cast<int>(M), r).ok;
}
inline size_t workspace_bytes(const QView& q, int r, int M, bool backward) {
    if (backward) {
        const BwdPlan pl = make_bwd_plan(q, M, r);
        return dec::ws_layout(pl.windows, M, r, pl.slots, pl.windows * 128).total;
    }
    return dec::ws_layout(q.ntiles, M, r, make_plan(q, M).slots, q.ntiles * 128).total;
}
// Bytes at the head of the workspace that must be zero when the linear kernel starts (status word and arrival counters).
inline size_t clear_bytes(const QView& q, bool backward) {
    return kStatusBytes + dec::round_up_ws(static_cast<size_t>(backward ? (q.ktiles + 1) / 2 : q.ntiles) * 4);
}
// Runs that may share an output tile.
inline int slots(const QView& q, int r, int M, bool backward) { return backward ? make_bwd_plan(q, M, r).slots : make_plan(q, M).slots; }

}  // namespace stream

// Decode-sized calls, either direction.
inline bool stream_supported(const QView& q, int r, int64_t M, bool backward) {
    return backward ? stream::bwd_supported(q, r, M) : stream::supported(q, M);
}

}  // namespace lq
