// What the kernels for decode-sized inputs (linear_stream.cuh, M <= 16 rows) and others share: mma.sync and cluster helpers, the
// rank-r pre-product for few rows, workspace layout, plan cache, launch.
#pragma once

#include "common.cuh"
#include "device_util.cuh"

namespace lq {
namespace dec {
using namespace dev;

constexpr int kSmemLimit = 232448;

__device__ __forceinline__ void mma16816(float (&d)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0, uint32_t b1) {
    asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};"
                 : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
                 : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}

__device__ __forceinline__ uint32_t cluster_ctarank() { uint32_t r; asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r)); return r; }
__device__ __forceinline__ void cluster_sync_all() {
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}
// Split cluster barrier: arrive early, wait where the guarantee is needed.
__device__ __forceinline__ void cluster_arrive_relaxed() { asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.aligned;" ::: "memory"); }
__device__ __forceinline__ float ld_dsmem_f32(uint32_t local_addr, uint32_t rank) {
    uint32_t ra;
    float v;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(ra) : "r"(local_addr), "r"(rank));
    asm volatile("ld.shared::cluster.f32 %0, [%1];" : "=f"(v) : "r"(ra) : "memory");
    return v;
}

// Stores v at the shared-memory offset `local_addr` of CTA `rank` of the cluster.
__device__ __forceinline__ void st_dsmem_f32(uint32_t local_addr, uint32_t rank, float v) {
    uint32_t ra;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(ra) : "r"(local_addr), "r"(rank));
    asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(ra), "f"(v) : "memory");
}

__device__ __forceinline__ void st_dsmem_v4(uint32_t local_addr, uint32_t rank, uint32_t a, uint32_t b, uint32_t c, uint32_t d) {
    uint32_t ra;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(ra) : "r"(local_addr), "r"(rank));
    asm volatile("st.shared::cluster.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(ra), "r"(a), "r"(b), "r"(c), "r"(d) : "memory");
}

// ------------------------------------------------------------------------------------ rank-r pre-product for few rows
// T[m][j] = bf16( sum_c A[m][c] * F(j, c) ) for m < M <= 16, j < r <= 128:
//   forward  A = X [M][K],  F(j, c) = L2[j][c]   (T = X L2^T)
//   backward A = dY [M][N], F(j, c) = L1[c][j]   (T = dY L1)
// On the tensor cores (tokens = the 16-row operand, eight columns of T = the 8-column operand): a cluster computes eight columns, each
// of its CTAs a slice of the contraction; its warps take 32 elements at a time, all loads of a warp in flight together.  Sums
// meet in shared memory, those of the CTAs in rank 0 through distributed shared memory, in a fixed order.
struct PreParams {
    const __nv_bfloat16* A;
    const __nv_bfloat16* F;
    __nv_bfloat16* T;
    int* status;       // cleared here: this kernel is the first of a call
    int* counters;     // arrival counters of the linear kernel behind this one, cleared here too
    int ncounters;
    int M, C, r;
    int nranks;
};

constexpr int kPreWarps = 8;
constexpr int kPreThreads = kPreWarps * 32;
constexpr int kPreJ = 8;              // columns of T per cluster

// Grid (ranks, r / 8), cluster (ranks, 1, 1).  NT: groups of eight tokens (1 or 2).
template <bool BWD, int NT>
__global__ void __launch_bounds__(kPreThreads, 5) decode_pre_kernel(const PreParams p) {      // (48 registers, see kMaxRegs of linear_stream.cuh)
    constexpr int kPreAhead = NT == 1 ? 3 : 2;      // steps of 32 elements in flight per warp
    __shared__ __align__(16) uint4 tile[BWD ? kPreWarps : 1][32];     // backward: 32 rows x 8 columns of L1 per warp
    __shared__ float red[kPreWarps][16 * kPreJ];
    __shared__ float part[16 * kPreJ];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int gid = lane >> 2, t = lane & 3;
    const int j0 = blockIdx.y * kPreJ;
    pdl_wait();                   // started while the previous kernel of the stream ends; everything below comes after it
    pdl_launch_dependents();
    if (blockIdx.x == 0 && blockIdx.y == 0) {
        if (threadIdx.x == 0) *p.status = 0;
        for (int i = threadIdx.x; i < p.ncounters; i += kPreThreads) p.counters[i] = 0;
    }
    // lane (gid, t) holds elements 8 t .. 8 t + 7 of a step of 32, of token gid (and gid + 8): the contraction index of the two
    // MMAs of a step is permuted accordingly
    float acc[4] = {0.0f, 0.0f, 0.0f, 0.0f};
    const int stride = p.nranks * kPreWarps * 32;
    for (int c0 = (blockIdx.x * kPreWarps + warp) * 32; c0 < p.C; c0 += kPreAhead * stride) {
        uint4 a[kPreAhead][NT], f[kPreAhead];
#pragma unroll
        for (int u = 0; u < kPreAhead; ++u) {
            const int c = c0 + u * stride;
            f[u] = make_uint4(0u, 0u, 0u, 0u);
            if (!BWD) { if (c + 8 * t < p.C) f[u] = __ldg(reinterpret_cast<const uint4*>(p.F + static_cast<size_t>(j0 + gid) * p.C + c + 8 * t)); }
            else if (c + lane < p.C) f[u] = __ldg(reinterpret_cast<const uint4*>(p.F + static_cast<size_t>(c + lane) * p.r + j0));
#pragma unroll
            for (int nt = 0; nt < NT; ++nt) {
                const int m = nt * 8 + gid;
                a[u][nt] = make_uint4(0u, 0u, 0u, 0u);
                if (m < p.M && c + 8 * t < p.C) a[u][nt] = __ldg(reinterpret_cast<const uint4*>(p.A + static_cast<size_t>(m) * p.C + c + 8 * t));
            }
        }
#pragma unroll
        for (int u = 0; u < kPreAhead; ++u) {
            if (c0 + u * stride >= p.C) break;
            uint32_t b[4] = {f[u].x, f[u].y, f[u].z, f[u].w};
            if constexpr (BWD) {
                // pairs along the rows of L1: through shared memory, row i of matrix m is the element 8 (i / 2) + 2 m + i % 2
                tile[warp][lane] = f[u];
                __syncwarp();
                const int i = lane & 7, n = 8 * (i >> 1) + 2 * (lane >> 3) + (i & 1);
                asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0, %1, %2, %3}, [%4];"
                             : "=r"(b[0]), "=r"(b[1]), "=r"(b[2]), "=r"(b[3]) : "r"(smem_u32(&tile[warp][n])) : "memory");
                __syncwarp();
            }
            const uint4 lo = a[u][0], hi = NT == 2 ? a[u][NT - 1] : make_uint4(0u, 0u, 0u, 0u);
            mma16816(acc, lo.x, hi.x, lo.y, hi.y, b[0], b[1]);
            mma16816(acc, lo.z, hi.z, lo.w, hi.w, b[2], b[3]);
        }
    }
    // token gid (+ 8), columns 2 t, 2 t + 1
    red[warp][gid * kPreJ + 2 * t] = acc[0];
    red[warp][gid * kPreJ + 2 * t + 1] = acc[1];
    red[warp][(gid + 8) * kPreJ + 2 * t] = acc[2];
    red[warp][(gid + 8) * kPreJ + 2 * t + 1] = acc[3];
    __syncthreads();
    if (threadIdx.x < 16 * kPreJ) {
        float sum = 0.0f;
#pragma unroll
        for (int w = 0; w < kPreWarps; ++w) sum += red[w][threadIdx.x];
        part[threadIdx.x] = sum;          // part[m * kPreJ + jl]
    }
    if (p.nranks > 1) cluster_sync_all();
    else __syncthreads();
    if (p.nranks == 1 || cluster_ctarank() == 0) {
        const uint32_t part_addr = smem_u32(part);
        if (threadIdx.x < 16 * kPreJ) {
            const int m = threadIdx.x / kPreJ, jj = j0 + (threadIdx.x & (kPreJ - 1));
            if (m < p.M) {
                float v[8];
#pragma unroll
                for (int rk = 0; rk < 8; ++rk)
                    v[rk] = (rk < p.nranks) ? ld_dsmem_f32(part_addr + static_cast<uint32_t>(threadIdx.x) * 4u, static_cast<uint32_t>(rk)) : 0.0f;
                p.T[static_cast<size_t>(m) * p.r + jj] = __float2bfloat16_rn(((v[0] + v[1]) + (v[2] + v[3])) + ((v[4] + v[5]) + (v[6] + v[7])));
            }
        }
    }
    if (p.nranks > 1) cluster_sync_all();          // the others' sums have been read
}

// ------------------------------------------------------------------------------------ host side
inline size_t round_up_ws(size_t x) { return (x + 255) / 256 * 256; }

inline int sm_count_cached() {
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

// Workspace of a decode-sized call: [status word 256 B][arrival counters][T bf16 [M][r]][slots of the slices, fp32]
struct WsLayout {
    size_t counters_off, counters_bytes, t_off, partial_off, total;
};
inline WsLayout ws_layout(int ncounters, int M, int r, int S, int out_pad) {
    WsLayout w;
    w.counters_off = kStatusBytes;
    w.counters_bytes = round_up_ws(static_cast<size_t>(ncounters) * 4);
    w.t_off = w.counters_off + w.counters_bytes;
    w.partial_off = w.t_off + round_up_ws(static_cast<size_t>(M) * (r > 0 ? r : 1) * 2);
    w.total = w.partial_off + (S > 1 ? round_up_ws(static_cast<size_t>(S) * M * out_pad * 4) : 0);
    return w;
}

// Plans of the last few shapes, kept by the calling thread (pure host arithmetic; a call asks for its plan four times).
template <typename P, typename F>
inline P cached_plan(const QView& q, int M, int r, F&& make) {
    struct Entry { int N = 0, K = 0, b0 = 0, logB0 = 0, M = 0, r = 0; P plan; };
    constexpr int kEntries = 16;
    thread_local Entry cache[kEntries];
    Entry& e = cache[(static_cast<uint32_t>(q.N) * 2654435761u + static_cast<uint32_t>(q.K) * 2246822519u +
                      static_cast<uint32_t>(M * 128 + q.logB0 * 16 + q.b0 + r * 4096) * 3266489917u) >> 28];
    if (e.N != q.N || e.K != q.K || e.b0 != q.b0 || e.logB0 != q.logB0 || e.M != M || e.r != r) {
        e.plan = make();
        e.N = q.N; e.K = q.K; e.b0 = q.b0; e.logB0 = q.logB0; e.M = M; e.r = r;
    }
    return e.plan;
}

// Launches the pre-product kernel for few rows (both directions use it).  It is the first kernel of the call: it clears
// the status word and the arrival counters of the linear kernel behind it.
template <bool BWD>
inline cudaError_t launch_pre(const __nv_bfloat16* A, const __nv_bfloat16* F, __nv_bfloat16* T, int* status, int* counters,
                              int ncounters, int M, int C, int r, size_t beside, cudaStream_t st) {
    PreParams pp;
    pp.A = A; pp.F = F; pp.T = T; pp.status = status; pp.counters = counters; pp.ncounters = ncounters; pp.M = M; pp.C = C; pp.r = r;
    int nranks = 8;
    while (nranks > 1 && C <= (nranks >> 1) * kPreWarps * 32) nranks >>= 1;      // (every warp has a step)
    pp.nranks = nranks;
    void (*kern)(PreParams) = M <= 8 ? decode_pre_kernel<BWD, 1> : decode_pre_kernel<BWD, 2>;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(nranks, r / kPreJ);
    cfg.blockDim = dim3(kPreThreads);
    cfg.stream = st;
    cudaLaunchAttribute attr[3];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = nranks; attr[0].val.clusterDim.y = 1; attr[0].val.clusterDim.z = 1;
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;      // the launch overlaps the end of the kernel in front
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    // Shared memory for the linear CTA that is to join this one on its SM, and no more: a CTA that does not fit waits for this kernel to
    // end, and the rest of the memory is L1 cache (8192 x 8192 NF3 us, default / all of it / this: one row 18.8 / 19.9 / 18.8, eight rows
    // 24.2 / 22.5 / 22.1).
    attr[2].id = cudaLaunchAttributePreferredSharedMemoryCarveout;
    const size_t percent = (beside + 16 * 1024) * 100 / (228 * 1024) + 1;
    attr[2].val.sharedMemCarveout = percent > 100 ? 100 : static_cast<unsigned>(percent);
    cfg.attrs = attr;
    cfg.numAttrs = 3;
    count_launch(1);
    return cudaLaunchKernelEx(&cfg, kern, pp);
}

// Without a rank-r term: clears the status word and the arrival counters for the linear kernel behind it, which is launched while this one runs.  (With a
// memset in front the linear kernel starts when the memset has ended, and the memset when the kernel before it has.  us per call in a graph, that / this,
// 3-bit codes: one row of 4096 x 4096 12.3 / 8.8, input gradient 14.3 / 10.9, 8192 x 8192 20.4 / 17.2; four rows of 1024 x 1024 9.1 / 6.7.)
__global__ void __launch_bounds__(128) decode_clear_kernel(int* status, int* counters, int ncounters) {
    pdl_wait();                   // started while the previous kernel of the stream ends
    pdl_launch_dependents();
    if (threadIdx.x == 0) *status = 0;
    for (int i = threadIdx.x; i < ncounters; i += 128) counters[i] = 0;
}
inline cudaError_t launch_clear(int* status, int* counters, int ncounters, cudaStream_t st) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(1);
    cfg.blockDim = dim3(128);
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    count_launch(1);
    return cudaLaunchKernelEx(&cfg, decode_clear_kernel, status, counters, ncounters);
}

// Launch of a linear kernel behind the kernel that clears: programmatic dependent launch lets the two overlap.
template <typename Kern, typename P>
inline cudaError_t launch_stream_kernel(Kern kern, const P& p, dim3 grid, int threads, size_t smem, cudaStream_t st) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    count_launch(1);
    return cudaLaunchKernelEx(&cfg, kern, p);
}

}  // namespace dec
}  // namespace lq
