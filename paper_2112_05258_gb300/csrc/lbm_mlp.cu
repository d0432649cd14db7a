// Warm-start network on the GPU: BF16 tensor-core matrix products (tcgen05
// MMA with the accumulator in tensor memory, FP32 accumulation) with fused
// epilogues, SiLU hidden layers, mean-squared-error loss, backpropagation
// and Adam, all in the kernels below.  Contract in include/lbm_mlp.h.
//
// Every product is C[M][N] = A[M][K] * Bt[N][K]^T with both operands stored
// K-contiguous ("NT"):
//   forward     act_out[B][N]  = act_in[B][K]  * Wt[N][K]^T   (+ bias, SiLU)
//   input grad  g_in[B][K]     = g_out[B][N]   * W[K][N]^T    (x SiLU'(pre))
//   weight grad dWt[N][K]      = g_out^T[N][B] * act_in^T[K][B]^T
// so each layer keeps its weights in both layouts (Wt and W), and activations
// and output gradients are written in both by the kernel that makes them.
// One Adam step of the 8-256-256-256-64 network on 512 rows is 11 launches and
// 57 us (35 launches and 291 us before; 64-wide, one hidden layer, 64 rows: 96
// -> 18 us), with the same bits: every sum keeps its order.
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <cmath>
#include <cstdio>
#include <string>
#include <vector>

#include "../../include/lbm_mlp.h"

namespace {

using bf16 = __nv_bfloat16;
constexpr int K0 = 16;       // padded input width

enum { EPI_HIDDEN = 0, EPI_OUT = 1, EPI_DX = 2, EPI_DW = 3 };

struct Epi {
    const float *bias;   // EPI_HIDDEN, EPI_OUT
    float *pre;          // EPI_HIDDEN: pre-activation out
    bf16 *out_bf;        // EPI_HIDDEN: SiLU(pre); EPI_DX: gradient (bf16)
    float *out_f;        // EPI_OUT: y; EPI_DX: gradient (fp32); EPI_DW: dWt
    const float *pre_in; // EPI_DX: pre-activation of the layer below
    bf16 *out_t;         // EPI_HIDDEN, EPI_DX: out_bf transposed (N x M) for the weight gradients, or null
    int n_keep;          // EPI_DW: columns kept (the layer's inputs without padding; the row stride of out_f)
};

__device__ __forceinline__ float silu_f(float z) { return z / (1.f + __expf(-z)); }
__device__ __forceinline__ float silu_grad_f(float z) {
    const float s = 1.f / (1.f + __expf(-z));
    return s * (1.f + z * (1.f - s));
}

// ---------------------------------------------------------------------------
// tcgen05 product C[M][N] = A[M][K] * Bt[N][K]^T (BF16 operands, FP32
// accumulator in tensor memory).  One CTA of 256 threads per 128 x NT tile of
// C (NT = 32 or 16 columns).  The K range is walked in chunks of 64 through
// a ring of TC_STAGES shared-memory stages: the warps start the
// asynchronous copies (cp.async, 16 bytes each) of the first stages' chunks of
// the A tile (128 rows) and B tile (NT rows) at once and refill a stage once
// its MMAs are done.  The products are small (256 x 256 weights, 512 rows) and
// bound by latency, not by the tensor cores: clocks of a CTA of the 512 x 256 x
// 256 layer before were 8,500 copies (4-way conflicts of 8-row core matrices
// and a round trip per chunk) and 5,600 epilogue (32 SiLU values a thread); with
// swizzled rows, four stages, twice the threads and tiles of 16 columns 3,500
// and 1,500.
// The tiles are laid out K-major with the 128-byte swizzle: row r of a chunk is
// 128 bytes (64 columns) at r * 128, its 16-byte piece p at p ^ (r % 8), so that
// a warp's copy writes whole rows without bank conflicts; 16 columns of K are
// 32 bytes on in the descriptor's start address.  One
// thread issues one MMA (M = 128, N = NT, K = 16) per 16 columns of the chunk
// and commits them to the stage's mbarrier, which the copy that reuses the
// stage waits for.  After the last chunk each warp reads its 32 rows of the
// accumulator (tensor-memory lanes 32 w .. 32 w + 31) with tcgen05.ld and
// applies the epilogue, 16 consecutive columns of a row per thread with
// 16-byte loads and stores.  Rows >= M and columns >= N are computed from zeros
// and not stored.  Every wait is bounded: on a time-out the kernel sets
// *err, waits (bounded) for its own MMAs, frees its tensor memory and leaves.
constexpr int TC_M = 128, TC_K = 64;
constexpr int TC_STAGES = 4;
constexpr int TC_SMEM = TC_STAGES * (TC_M + 32) * TC_K * 2 + 1024;  // and the 1024-byte alignment of the tiles
constexpr int TC_THREADS = 256;
constexpr long long TC_SPIN = 1ll << 22;  // mbarrier polls before a time-out

// The kernels of a pass follow one another at once (programmatic dependent
// launch): a kernel lets its successor start its set-up early and itself waits,
// before it touches memory, until its predecessor has finished.  Every thread
// waits, so that a finished kernel means that all before it have finished too.
__device__ __forceinline__ void let_next_start() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void wait_for_previous() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

__device__ __forceinline__ uint32_t smem_u32(const void *p) {
    return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

// shared-memory matrix descriptor of a K-major tile with 128-byte swizzle: start
// address, leading offset (unused with this swizzle), stride offset 1024 bytes
// (8 rows), the fixed 0b001 at bits 46-48, swizzle mode 2 at bits 61-63
__device__ __forceinline__ uint64_t tc_desc(uint32_t addr) {
    return (uint64_t)((addr & 0x3FFFFu) >> 4) | (1ull << 16) | ((uint64_t)(1024u >> 4) << 32) | (1ull << 46) | (2ull << 61);
}

// instruction descriptor of kind::f16: FP32 accumulator (bits 4-5 = 1), BF16 A
// and B (bits 7-9, 10-12 = 1), both K-major, N >> 3 at bits 17-22, M >> 4 at
// bits 24-28
template <int NT> __device__ __forceinline__ uint32_t tc_idesc() {
    return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(NT >> 3) << 17) | ((uint32_t)(TC_M >> 4) << 24);
}

__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t phase) {
    for (long long it = 0; it < TC_SPIN; it++) {
        uint32_t done;
        asm volatile(
            "{\n.reg .pred p;\n"
            "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n"
            "selp.u32 %0, 1, 0, p;\n}\n"
            : "=r"(done)
            : "r"(bar), "r"(phase)
            : "memory");
        if (done) return true;
    }
    return false;
}

// Epilogue of W (8 or 16) consecutive columns col .. col + W - 1 of one row (col
// a multiple of W, N of 16): 16-byte vector loads and stores; x holds the
// columns' biases or pre-activations, read before the product was ready.
template <int EPI, int W> __device__ __forceinline__ void epi_load(const Epi &e, int row, int col, int N, float (&x)[W]) {
    if (EPI == EPI_DW) return;
    const float4 *p = reinterpret_cast<const float4 *>(EPI == EPI_DX ? e.pre_in + (size_t)row * N + col : e.bias + col);
#pragma unroll
    for (int q = 0; q < W / 4; q++) {
        const float4 v = p[q];
        x[4 * q] = v.x;
        x[4 * q + 1] = v.y;
        x[4 * q + 2] = v.z;
        x[4 * q + 3] = v.w;
    }
}
template <int EPI, int W>
__device__ __forceinline__ void epi_store(const Epi &e, int row, int col, int M, int N, const uint32_t (&r)[W],
                                          const float (&x)[W]) {
    const size_t idx = (size_t)row * N + col;
    float v[W];
#pragma unroll
    for (int j = 0; j < W; j++) {
        v[j] = __uint_as_float(r[j]);
        if (EPI == EPI_HIDDEN || EPI == EPI_OUT) v[j] += x[j];
        if (EPI == EPI_DX) v[j] *= silu_grad_f(x[j]);
    }
    if (EPI == EPI_DW && e.n_keep != N) {  // an input layer narrower than its padding
#pragma unroll
        for (int j = 0; j < W; j++)
            if (col + j < e.n_keep) e.out_f[(size_t)row * e.n_keep + col + j] = v[j];
        return;
    }
    float *of = EPI == EPI_HIDDEN ? e.pre : e.out_f;
    float4 *o4 = reinterpret_cast<float4 *>(of + idx);
#pragma unroll
    for (int q = 0; q < W / 4; q++) o4[q] = make_float4(v[4 * q], v[4 * q + 1], v[4 * q + 2], v[4 * q + 3]);
    if (EPI == EPI_HIDDEN || EPI == EPI_DX) {
        uint32_t w[W / 2];
#pragma unroll
        for (int q = 0; q < W / 2; q++) {
            const float a = EPI == EPI_HIDDEN ? silu_f(v[2 * q]) : v[2 * q];
            const float b = EPI == EPI_HIDDEN ? silu_f(v[2 * q + 1]) : v[2 * q + 1];
            const __nv_bfloat162 h = __floats2bfloat162_rn(a, b);
            w[q] = *reinterpret_cast<const uint32_t *>(&h);
        }
        uint4 *b4 = reinterpret_cast<uint4 *>(e.out_bf + idx);
#pragma unroll
        for (int q = 0; q < W / 8; q++) b4[q] = make_uint4(w[4 * q], w[4 * q + 1], w[4 * q + 2], w[4 * q + 3]);
        if (e.out_t) {  // the warp's rows are consecutive: 64 bytes per column
            uint16_t *t = reinterpret_cast<uint16_t *>(e.out_t) + (size_t)col * M + row;
#pragma unroll
            for (int q = 0; q < W / 2; q++) {
                t[(size_t)(2 * q) * M] = (uint16_t)w[q];
                t[(size_t)(2 * q + 1) * M] = (uint16_t)(w[q] >> 16);
            }
        }
    }
}

// tcgen05.ld of W consecutive accumulator columns, lane l of the warp row l of its quadrant
template <int W> __device__ __forceinline__ void tmem_ld(uint32_t addr, uint32_t (&r)[W]);
template <> __device__ __forceinline__ void tmem_ld<8>(uint32_t ta, uint32_t (&r)[8]) {
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];\n"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
                 : "r"(ta));
}
template <> __device__ __forceinline__ void tmem_ld<16>(uint32_t ta, uint32_t (&r)[16]) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, "
        "[%16];\n"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(ta));
}

__device__ __forceinline__ void cp_async16(uint32_t dst, const void *src, bool valid) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(valid ? 16 : 0)
                 : "memory");
}

template <int EPI, int NT>
__device__ __forceinline__ void gemm_tile(const bf16 *__restrict__ A, const bf16 *__restrict__ Bt, int M, int N, int K,
                                          const Epi &e, int *err, int mt, int nt) {
    constexpr int TMEM_COLS = 32;  // NT <= 32 accumulator columns (the minimum allocation)
    constexpr int A_BYTES = TC_M * TC_K * 2, B_BYTES = NT * TC_K * 2;
    static_assert(NT == 16 || NT == 32, "tile width");
    extern __shared__ uint8_t tiles[];
    __shared__ __align__(8) uint64_t bar[TC_STAGES];
    __shared__ uint32_t tmem_base;
    __shared__ int failed;
    const uint32_t sA = (smem_u32(tiles) + 1023u) & ~1023u, sB = sA + TC_STAGES * A_BYTES;
    static_assert(TC_THREADS / 32 >= 32 / 4, "one piece of the B tile per warp");
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int m0 = mt * TC_M, n0 = nt * NT;
    const uint32_t bar0 = smem_u32(&bar[0]);
    if (tid == 0) {
        failed = 0;
#pragma unroll
        for (int k = 0; k < TC_STAGES; k++) asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(bar0 + 8 * k));
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_base)),
                     "r"(TMEM_COLS));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem = tmem_base;
    wait_for_previous();
    const uint32_t idesc = tc_idesc<NT>();
    const int nchunk = (K + TC_K - 1) / TC_K;
    // asynchronous copy of chunk j into its stage (rows or columns past the
    // matrix are zero-filled): A tile 128 rows x 8 pieces of 16 bytes, B tile NT rows
    auto copy_chunk = [&](int j) {
        const int st = j % TC_STAGES, k0 = j * TC_K;
        const uint32_t a_s = sA + st * A_BYTES, b_s = sB + st * B_BYTES;
        // a warp copies 4 rows of 128 bytes at a time (whole lines of both memories)
        auto piece = [&](uint32_t tile, const bf16 *X, int row0, int rows, int idx) {
            const int r = 4 * idx + (lane >> 3), kc = lane & 7;
            const int grow = row0 + r, gk = k0 + kc * 8;
            const bool valid = grow < rows && gk < K;
            cp_async16(tile + (uint32_t)(r * 128 + ((kc ^ (r & 7)) << 4)), valid ? X + (size_t)grow * K + gk : X, valid);
        };
#pragma unroll
        for (int u = 0; u < TC_M / 4; u += TC_THREADS / 32) piece(a_s, A, m0, M, warp + u);
        if (warp < NT / 4) piece(b_s, Bt, n0, N, warp);
    };
    // this thread's part of the epilogue
    constexpr int W = NT / 2;
    const int row = m0 + (warp & 3) * 32 + lane, col = n0 + (warp >> 2) * W;
    const bool mine = row < M && col < N;  // N is a multiple of 16
    float x[W];
    bool ok = true;
    int last = -1;  // the last chunk whose MMAs were committed
#pragma unroll
    for (int j = 0; j < TC_STAGES - 1; j++) {  // one group per chunk, empty past the last
        if (j < nchunk) copy_chunk(j);
        asm volatile("cp.async.commit_group;" ::: "memory");
    }
    if (mine) epi_load<EPI, W>(e, row, col, N, x);
    for (int j = 0; j < nchunk && ok; j++) {
        const int st = j % TC_STAGES, k0 = j * TC_K;
        const int jn = j + TC_STAGES - 1;  // the chunk to start now
        if (jn < nchunk) {
            // its stage was last read by the MMAs of chunk j - 1
            if (j >= 1 && !mbar_wait(bar0 + 8 * ((j - 1) % TC_STAGES), ((j - 1) / TC_STAGES) & 1)) atomicExch(&failed, 1);
            if (!failed) copy_chunk(jn);
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
        asm volatile("cp.async.wait_group %0;" ::"n"(TC_STAGES - 1) : "memory");  // chunk j has landed
        // make the copies visible to the tensor core
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        __syncthreads();
        if (failed) {
            ok = false;
            break;
        }
        if (tid == 0) {
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            const uint32_t a_base = sA + st * A_BYTES, b_base = sB + st * B_BYTES;
            const int nk = min(TC_K / 16, (K - k0 + 15) / 16);
            for (int kk = 0; kk < nk; kk++) {
                const uint64_t ad = tc_desc(a_base + kk * 32);
                const uint64_t bd = tc_desc(b_base + kk * 32);
                const uint32_t acc = (k0 > 0 || kk > 0) ? 1u : 0u;
                asm volatile(
                    "{\n.reg .pred p;\n"
                    "setp.ne.b32 p, %4, 0;\n"
                    "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(tmem),
                    "l"(ad), "l"(bd), "r"(idesc), "r"(acc));
            }
            asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
                             bar0 + 8 * st)
                         : "memory");
        }
        last = j;
    }
    asm volatile("cp.async.wait_group 0;" ::: "memory");  // no copy outlives the kernel
    // the last commit completes when all MMAs issued before it have completed
    if (last >= 0 && !mbar_wait(bar0 + 8 * (last % TC_STAGES), (last / TC_STAGES) & 1)) atomicExch(&failed, 1);
    __syncthreads();
    if (failed) ok = false;
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    if (ok) {
        // warps w and w + 4 hold the rows 32 (w % 4) .. + 31 (their quadrant of the
        // tensor memory) and one half of the tile's columns each
        uint32_t r[W];
        tmem_ld<W>(tmem + ((uint32_t)((warp & 3) * 32) << 16) + (uint32_t)((warp >> 2) * W), r);
        asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
        if (mine) epi_store<EPI, W>(e, row, col, M, N, r, x);
    } else {
        if (tid == 0) atomicExch(err, 1);
        // the MMAs still in flight (bounded; their commit was the last one)
        if (last >= 0) mbar_wait(bar0 + 8 * (last % TC_STAGES), (last / TC_STAGES) & 1);
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (warp == 0) {
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(TMEM_COLS));
    }
}

// one forward layer
template <int EPI, int NT>
__global__ void __launch_bounds__(TC_THREADS) k_gemm_tc(const bf16 *__restrict__ A, const bf16 *__restrict__ Bt, int M,
                                                        int N, int K, Epi e, int *err) {
    let_next_start();
    gemm_tile<EPI, NT>(A, Bt, M, N, K, e, err, blockIdx.y, blockIdx.x);
}

// db[n] = sum over the batch of g[b][n] for 32 columns, in the order of the
// rows: the block stages 128 rows at a time in shared memory (the next rows in
// flight in registers meanwhile), one warp adds them column by column.  Bound
// by the chain of FP32 additions, 4 cycles each; one thread per column reading
// global memory row by row took 31 us for 512 rows.
__device__ __forceinline__ void bias_columns(const float *__restrict__ g, int batch, int n, float *db, int c0, float *tile) {
    constexpr int ROWS = 128;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, c = c0 + lane;
    constexpr int WARPS = TC_THREADS / 32;
    float v[ROWS / WARPS], s = 0.f;
    auto load = [&](int r0) {
#pragma unroll
        for (int k = 0; k < ROWS / WARPS; k++) {
            const int r = r0 + w + WARPS * k;
            v[k] = r < batch && c < n ? g[(size_t)r * n + c] : 0.f;
        }
    };
    load(0);
    for (int r0 = 0; r0 < batch; r0 += ROWS) {
#pragma unroll
        for (int k = 0; k < ROWS / WARPS; k++) tile[(w + WARPS * k) * 32 + lane] = v[k];
        __syncthreads();
        if (r0 + ROWS < batch) load(r0 + ROWS);
        if (w == 0) {
            const int m = min(ROWS, batch - r0);
            if (m == ROWS) {
#pragma unroll 32
                for (int r = 0; r < ROWS; r++) s += tile[r * 32 + lane];
            } else {
                for (int r = 0; r < m; r++) s += tile[r * 32 + lane];
            }
        }
        __syncthreads();
    }
    if (w == 0 && c < n) db[c] = s;
}

// The loss: the rows' sums added in a fixed tree of 256 threads.
__device__ __forceinline__ void sum_loss(const float *row_loss, int batch, int n_out, float *loss, float *red) {
    static_assert(TC_THREADS == 256, "the tree's threads");
    float s = 0.f;
    for (int b = threadIdx.x; b < batch; b += 256) s += row_loss[b];
    red[threadIdx.x] = s;
    __syncthreads();
    for (int o = 128; o > 0; o >>= 1) {
        if ((int)threadIdx.x < o) red[threadIdx.x] += red[threadIdx.x + o];
        __syncthreads();
    }
    if (threadIdx.x == 0) *loss = red[0] / (float)(batch * n_out);
}

// One layer of the backward pass in one launch (five and a product before: two
// transposes, now written by the epilogues, bias sums, weight product, copy
// without padding); the blocks take, in this order,
// the tiles of the input gradient (the longest chain: the next layer waits for
// it), the tiles of the weight gradient, 32 columns each of the bias gradient,
// and, with loss, the loss.  All of them only need the layer's output gradient.
struct Backward {
    int B, N, K;                      // rows, outputs, padded inputs
    const bf16 *g, *g_t, *W, *in_t;   // output gradient (B x N), transposed; weights (K x N); inputs transposed (K x B)
    const float *g_f;
    float *db;
    Epi dx, dw;
    int n_dx, dx_cols, n_dw, dw_cols; // tiles, and tiles per row of tiles
    int n_bias;
    const float *row_loss;
    float *loss;
    int n_out;
};
template <int NT>
__global__ void __launch_bounds__(TC_THREADS) k_backward(Backward q, int *err) {
    extern __shared__ uint8_t tiles[];
    let_next_start();
    int k = blockIdx.x;
    if (k < q.n_dx) {
        gemm_tile<EPI_DX, NT>(q.g, q.W, q.B, q.K, q.N, q.dx, err, k / q.dx_cols, k % q.dx_cols);
        return;
    }
    k -= q.n_dx;
    if (k < q.n_dw) {
        gemm_tile<EPI_DW, NT>(q.g_t, q.in_t, q.N, q.K, q.B, q.dw, err, k / q.dw_cols, k % q.dw_cols);
        return;
    }
    k -= q.n_dw;
    wait_for_previous();
    if (k < q.n_bias) bias_columns(q.g_f, q.B, q.N, q.db, 32 * k, reinterpret_cast<float *>(tiles));
    else sum_loss(q.row_loss, q.B, q.n_out, q.loss, reinterpret_cast<float *>(tiles));
}

__global__ void k_transpose_bf16(const bf16 *__restrict__ in, bf16 *__restrict__ out, int R, int C) {
    __shared__ bf16 tile[32][33];
    const int c = blockIdx.x * 32 + threadIdx.x, r0 = blockIdx.y * 32;
    for (int k = threadIdx.y; k < 32; k += 8)
        if (r0 + k < R && c < C) tile[k][threadIdx.x] = in[(size_t)(r0 + k) * C + c];
    __syncthreads();
    const int r = r0 + threadIdx.x, c0 = blockIdx.x * 32;
    for (int k = threadIdx.y; k < 32; k += 8)
        if (c0 + k < C && r < R) out[(size_t)(c0 + k) * R + r] = tile[threadIdx.x][k];
}

// Gathers minibatch rows into the padded BF16 input (both layouts) and the FP32 target.
__global__ void k_gather_batch(const float *__restrict__ xd, const float *__restrict__ td,
                               const int32_t *__restrict__ idx, int batch, int n_in, int n_out, bf16 *x_bf,
                               bf16 *x_t, float *t) {
    let_next_start();
    wait_for_previous();
    const int b = blockIdx.x, j = threadIdx.x;
    const int r = idx[b];
    if (j < K0) {
        const bf16 v = __float2bfloat16_rn(j < n_in ? xd[(size_t)r * n_in + j] : 0.f);
        x_bf[(size_t)b * K0 + j] = v;
        x_t[(size_t)j * batch + b] = v;
    }
    for (int k = j; k < n_out; k += blockDim.x) t[(size_t)b * n_out + k] = td[(size_t)r * n_out + k];
}

// d loss / d y for the mean squared error, and per-row partial sums of the loss.
__global__ void k_mse_grad(const float *__restrict__ y, const float *__restrict__ t, int batch, int n_out,
                           float *g_f, bf16 *g_bf, bf16 *g_t, float *row_loss) {
    let_next_start();
    wait_for_previous();
    const int b = blockIdx.x;
    float s = 0.f;
    const float scale = 2.f / (float)(batch * n_out);
    for (int k = threadIdx.x; k < n_out; k += blockDim.x) {
        const size_t i = (size_t)b * n_out + k;
        const float d = y[i] - t[i];
        s += d * d;
        g_f[i] = scale * d;
        const bf16 v = __float2bfloat16_rn(scale * d);
        g_bf[i] = v;
        g_t[(size_t)k * batch + b] = v;
    }
    __shared__ float red[64];
    red[threadIdx.x] = s;
    __syncthreads();
    for (int o = blockDim.x / 2; o > 0; o >>= 1) {
        if (threadIdx.x < o) red[threadIdx.x] += red[threadIdx.x + o];
        __syncthreads();
    }
    if (threadIdx.x == 0) row_loss[b] = red[0];
}

// Master FP32 layer weights (flat, n_out x n_in) -> BF16 Wt (n_out x K pad) and W (K pad x n_out).
__global__ void k_refresh_bf16(const float *__restrict__ wt, int n_out, int n_in, int kpad, bf16 *Wt_bf,
                               bf16 *W_bf) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n_out * kpad) return;
    const int r = i / kpad, c = i % kpad;
    const bf16 v = __float2bfloat16_rn(c < n_in ? wt[(size_t)r * n_in + c] : 0.f);
    Wt_bf[i] = v;
    W_bf[(size_t)c * n_out + r] = v;
}

// Adam on the flat parameters, and the BF16 copies of the new weights in both
// layouts (their padding stays zero).
struct LayerTab {
    int64_t woff, boff;  // weights, biases in the flat vector
    int n_in, n_out, kpad;
    bf16 *Wt, *W;
};
__global__ void k_adam(float *theta, const float *g, float *m, float *v, int64_t n, float lr, float b1, float b2,
                       float c1, float c2, float eps, const LayerTab *tab) {
    let_next_start();
    wait_for_previous();
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const float gi = g[i];
    const float mi = b1 * m[i] + (1.f - b1) * gi;
    const float vi = b2 * v[i] + (1.f - b2) * gi * gi;
    m[i] = mi;
    v[i] = vi;
    const float t = theta[i] - lr * (mi / c1) / (sqrtf(vi / c2) + eps);
    theta[i] = t;
    int l = 0;
    while (i >= tab[l].boff + tab[l].n_out) l++;
    const LayerTab &q = tab[l];
    if (i >= q.boff) return;
    const int k = (int)(i - q.woff), r = k / q.n_in, c = k - r * q.n_in;
    const bf16 h = __float2bfloat16_rn(t);
    q.Wt[(size_t)r * q.kpad + c] = h;
    q.W[(size_t)c * q.n_out + r] = h;
}

}  // namespace

struct lbm_mlp {
    int device = 0;
    cudaStream_t stream = nullptr;
    bool own_stream = false;
    int n_in = 0, n_out = 0, hidden = 0, n_layers = 0, max_batch = 0;
    std::vector<int> nin, nout, kpad;     // per layer
    std::vector<int64_t> woff, boff;      // offsets into the flat parameter vector
    int64_t np = 0;
    float *theta = nullptr, *grad = nullptr, *m = nullptr, *v = nullptr;
    std::vector<bf16 *> Wt, W;            // per layer
    std::vector<bf16 *> act;              // act[l]: input of layer l (B x kpad[l]) ; act[L] unused
    std::vector<float *> pre;             // pre-activation of hidden layer l (B x nout[l])
    std::vector<bf16 *> actT;             // transposed inputs (kpad[l] x B)
    float *y = nullptr, *t = nullptr, *row_loss = nullptr, *losses = nullptr;
    std::vector<float *> gf;              // gradient w.r.t. layer l output (B x nout[l]), fp32
    std::vector<bf16 *> gbf, gT;          // bf16 copy and transpose
    LayerTab *tab = nullptr;
    int32_t *ord = nullptr;               // training: order of the rows and losses of a call (grown as needed)
    float *dl = nullptr;
    size_t ord_cap = 0, dl_cap = 0;
    float *xd = nullptr, *td = nullptr;   // training set
    int n_data = 0;
    int32_t *idx = nullptr;
    int64_t adam_steps = 0;
    int *err = nullptr;                   // device: set by a tensor-core product that timed out
    std::vector<void *> allocs;
};

namespace {

template <class T> cudaError_t dal(lbm_mlp *h, T **p, size_t n) {
    void *q = nullptr;
    cudaError_t e = cudaMalloc(&q, (n ? n : 1) * sizeof(T));
    if (e == cudaSuccess) {
        h->allocs.push_back(q);
        cudaMemset(q, 0, (n ? n : 1) * sizeof(T));
    }
    *p = static_cast<T *>(q);
    return e;
}

// a workspace of at least n entries (the stream must not be using the old one)
template <class T> cudaError_t grow(T **p, size_t *cap, size_t n) {
    if (n <= *cap) return cudaSuccess;
    if (*p) cudaFree(*p);
    *p = nullptr;
    *cap = 0;
    void *q = nullptr;
    const cudaError_t e = cudaMalloc(&q, n * sizeof(T));
    if (e != cudaSuccess) return e;
    *p = static_cast<T *>(q);
    *cap = n;
    return cudaSuccess;
}

#define MCK(call)                                                                   \
    do {                                                                            \
        cudaError_t e_ = (call);                                                    \
        if (e_ != cudaSuccess) {                                                    \
            fprintf(stderr, "lbm_mlp: %s: %s\n", #call, cudaGetErrorString(e_));  \
            return e_ == cudaErrorMemoryAllocation ? LBM_ERR_OOM : LBM_ERR_CUDA;    \
        }                                                                           \
    } while (0)

// a launch that may start while its predecessor on the stream finishes
template <class... P, class... A>
cudaError_t follow(lbm_mlp *h, void (*k)(P...), dim3 grid, int threads, size_t smem, A... args) {
    cudaLaunchConfig_t cfg{};
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    cfg.gridDim = grid;
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = h->stream;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, k, static_cast<P>(args)...);
}

// Tile width of a product of mt tiles of rows and N columns: 16 while tiles of
// 32 would leave SMs idle (the epilogue, whose SiLU divisions take longer than
// the product, then spreads over twice as many CTAs), else 32.
int tile_cols(int mt, int N) { return N % 32 == 0 && mt * (N / 32) >= 148 ? 32 : 16; }

template <int EPI> cudaError_t gemm(lbm_mlp *h, const bf16 *A, const bf16 *Bt, int M, int N, int K, const Epi &e) {
    const int mt = (M + TC_M - 1) / TC_M;
    if (tile_cols(mt, N) == 32)
        return follow(h, k_gemm_tc<EPI, 32>, dim3(N / 32, mt), TC_THREADS, TC_SMEM, A, Bt, M, N, K, e, h->err);
    return follow(h, k_gemm_tc<EPI, 16>, dim3(N / 16, mt), TC_THREADS, TC_SMEM, A, Bt, M, N, K, e, h->err);
}

// the products' shared memory exceeds the 48 KB that need no request
cudaError_t prepare_products() {
    const void *k[] = {(const void *)k_gemm_tc<EPI_HIDDEN, 32>, (const void *)k_gemm_tc<EPI_HIDDEN, 16>,
                       (const void *)k_gemm_tc<EPI_OUT, 32>,    (const void *)k_gemm_tc<EPI_OUT, 16>,
                       (const void *)k_backward<32>,            (const void *)k_backward<16>};
    cudaError_t e = cudaSuccess;
    for (const void *f : k)
        if (e == cudaSuccess) e = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, TC_SMEM);
    return e;
}

cudaError_t transpose(lbm_mlp *h, const bf16 *in, bf16 *out, int R, int C) {
    dim3 grid((C + 31) / 32, (R + 31) / 32), block(32, 8);
    k_transpose_bf16<<<grid, block, 0, h->stream>>>(in, out, R, C);
    return cudaGetLastError();
}

cudaError_t refresh(lbm_mlp *h) {
    for (int l = 0; l < h->n_layers; l++) {
        const int n = h->nout[l] * h->kpad[l];
        k_refresh_bf16<<<(n + 255) / 256, 256, 0, h->stream>>>(h->theta + h->woff[l], h->nout[l], h->nin[l],
                                                               h->kpad[l], h->Wt[l], h->W[l]);
    }
    return cudaGetLastError();
}

// forward pass from act[0] (already filled, B x 16); output in h->y; with
// train, the activations' transposes for the backward pass too
cudaError_t forward(lbm_mlp *h, int B, bool train) {
    for (int l = 0; l < h->n_layers; l++) {
        Epi e{};
        e.bias = h->theta + h->boff[l];
        if (l < h->n_layers - 1) {
            e.pre = h->pre[l];
            e.out_bf = h->act[l + 1];
            e.out_t = train ? h->actT[l + 1] : nullptr;
            cudaError_t r = gemm<EPI_HIDDEN>(h, h->act[l], h->Wt[l], B, h->nout[l], h->kpad[l], e);
            if (r != cudaSuccess) return r;
        } else {
            e.out_f = h->y;
            cudaError_t r = gemm<EPI_OUT>(h, h->act[l], h->Wt[l], B, h->nout[l], h->kpad[l], e);
            if (r != cudaSuccess) return r;
        }
    }
    return cudaSuccess;
}

// backward pass from gf, gbf and gT of the output layer; fills h->grad and,
// where loss is given, *loss from h->row_loss
cudaError_t backward(lbm_mlp *h, int B, float *loss) {
    for (int l = h->n_layers - 1; l >= 0; l--) {
        Backward q{};
        q.B = B;
        q.N = h->nout[l];
        q.K = h->kpad[l];
        q.g = h->gbf[l];
        q.g_t = h->gT[l];
        q.W = h->W[l];
        q.in_t = h->actT[l];
        q.g_f = h->gf[l];
        q.db = h->grad + h->boff[l];
        q.dw.out_f = h->grad + h->woff[l];
        q.dw.n_keep = h->nin[l];
        const int nt = tile_cols((B + TC_M - 1) / TC_M + (q.N + TC_M - 1) / TC_M, q.K);
        q.dw_cols = q.K / nt;
        q.n_dw = q.dw_cols * ((q.N + TC_M - 1) / TC_M);
        q.n_bias = (q.N + 31) / 32;
        if (l > 0) {
            q.dx.out_f = h->gf[l - 1];
            q.dx.out_bf = h->gbf[l - 1];
            q.dx.out_t = h->gT[l - 1];
            q.dx.pre_in = h->pre[l - 1];
            q.dx_cols = q.dw_cols;
            q.n_dx = q.dx_cols * ((B + TC_M - 1) / TC_M);
        }
        const bool with_loss = loss && l == h->n_layers - 1;
        if (with_loss) {
            q.row_loss = h->row_loss;
            q.loss = loss;
            q.n_out = h->n_out;
        }
        const int grid = q.n_dx + q.n_dw + q.n_bias + (with_loss ? 1 : 0);
        const cudaError_t e = follow(h, nt == 32 ? k_backward<32> : k_backward<16>, dim3(grid), TC_THREADS, TC_SMEM, q, h->err);
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

lbm_status load_input(lbm_mlp *h, const float *x, int B) {
    std::vector<bf16> xb((size_t)B * K0);
    for (int b = 0; b < B; b++)
        for (int j = 0; j < K0; j++) xb[(size_t)b * K0 + j] = __float2bfloat16_rn(j < h->n_in ? x[(size_t)b * h->n_in + j] : 0.f);
    MCK(cudaMemcpyAsync(h->act[0], xb.data(), xb.size() * sizeof(bf16), cudaMemcpyHostToDevice, h->stream));
    MCK(cudaStreamSynchronize(h->stream));
    return LBM_OK;
}

bool bad_batch(const lbm_mlp *h, int B) { return !h || B < 16 || B % 16 || B > h->max_batch; }

// after a synchronisation: a tensor-core product that gave up waiting
lbm_status check_err(lbm_mlp *h) {
    int e = 0;
    MCK(cudaMemcpy(&e, h->err, sizeof e, cudaMemcpyDeviceToHost));
    if (e) {
        fprintf(stderr, "lbm_mlp: a tensor-core product timed out waiting for its MMAs\n");
        return LBM_ERR_CUDA;
    }
    return LBM_OK;
}

}  // namespace

extern "C" {

lbm_status lbm_mlp_create(int n_in, int hidden, int n_hidden, int n_out, int max_batch, int device, void *stream,
                          lbm_mlp **out) {
    if (!out) return LBM_ERR_ARG;
    *out = nullptr;
    if (n_in < 1 || n_in > K0 || hidden < 64 || hidden % 64 || n_hidden < 1 || n_out < 16 || n_out % 16 ||
        max_batch < 64 || max_batch % 64) {
        fprintf(stderr, "lbm_mlp_create: invalid shape\n");
        return LBM_ERR_ARG;
    }
    if (cudaSetDevice(device) != cudaSuccess) return LBM_ERR_CUDA;
    lbm_mlp *h = new lbm_mlp();
    h->device = device;
    h->n_in = n_in;
    h->n_out = n_out;
    h->hidden = hidden;
    h->n_layers = n_hidden + 1;
    h->max_batch = max_batch;
    if (stream) {
        h->stream = static_cast<cudaStream_t>(stream);
    } else {
        cudaStreamCreateWithFlags(&h->stream, cudaStreamNonBlocking);
        h->own_stream = true;
    }
    int64_t off = 0;
    for (int l = 0; l < h->n_layers; l++) {
        const int ni = l == 0 ? n_in : hidden, no = l == h->n_layers - 1 ? n_out : hidden;
        h->nin.push_back(ni);
        h->nout.push_back(no);
        h->kpad.push_back(l == 0 ? K0 : hidden);
        h->woff.push_back(off);
        off += (int64_t)ni * no;
        h->boff.push_back(off);
        off += no;
    }
    h->np = off;
    bool ok = dal(h, &h->theta, off) == cudaSuccess && dal(h, &h->grad, off) == cudaSuccess &&
              dal(h, &h->m, off) == cudaSuccess && dal(h, &h->v, off) == cudaSuccess &&
              dal(h, &h->tab, h->n_layers) == cudaSuccess && dal(h, &h->y, (size_t)max_batch * n_out) == cudaSuccess &&
              dal(h, &h->t, (size_t)max_batch * n_out) == cudaSuccess &&
              dal(h, &h->row_loss, max_batch) == cudaSuccess && dal(h, &h->idx, max_batch) == cudaSuccess &&
              dal(h, &h->err, 1) == cudaSuccess;
    h->Wt.resize(h->n_layers);
    h->W.resize(h->n_layers);
    h->act.resize(h->n_layers + 1);
    h->actT.resize(h->n_layers);
    h->pre.resize(h->n_layers);
    h->gf.resize(h->n_layers);
    h->gbf.resize(h->n_layers);
    h->gT.resize(h->n_layers);
    for (int l = 0; l < h->n_layers && ok; l++) {
        const size_t B = max_batch;
        ok = dal(h, &h->Wt[l], (size_t)h->nout[l] * h->kpad[l]) == cudaSuccess &&
             dal(h, &h->W[l], (size_t)h->nout[l] * h->kpad[l]) == cudaSuccess &&
             dal(h, &h->act[l], B * h->kpad[l]) == cudaSuccess &&
             dal(h, &h->actT[l], B * h->kpad[l]) == cudaSuccess &&
             dal(h, &h->pre[l], B * h->nout[l]) == cudaSuccess &&
             dal(h, &h->gf[l], B * h->nout[l]) == cudaSuccess &&
             dal(h, &h->gbf[l], B * h->nout[l]) == cudaSuccess &&
             dal(h, &h->gT[l], B * h->nout[l]) == cudaSuccess;
    }
    if (!ok) {
        lbm_mlp_destroy(h);
        return LBM_ERR_OOM;
    }
    std::vector<LayerTab> tab;
    for (int l = 0; l < h->n_layers; l++)
        tab.push_back({h->woff[l], h->boff[l], h->nin[l], h->nout[l], h->kpad[l], h->Wt[l], h->W[l]});
    if (cudaMemcpy(h->tab, tab.data(), tab.size() * sizeof(LayerTab), cudaMemcpyHostToDevice) != cudaSuccess ||
        prepare_products() != cudaSuccess) {
        lbm_mlp_destroy(h);
        return LBM_ERR_CUDA;
    }
    *out = h;
    return LBM_OK;
}

int64_t lbm_mlp_num_params(const lbm_mlp *m) { return m ? m->np : 0; }

lbm_status lbm_mlp_set_params(lbm_mlp *h, const float *theta, int64_t n) {
    if (!h || !theta || n != h->np) return LBM_ERR_ARG;
    for (int64_t i = 0; i < n; i++)
        if (!std::isfinite(theta[i])) return LBM_ERR_ARG;
    MCK(cudaSetDevice(h->device));
    MCK(cudaMemcpyAsync(h->theta, theta, n * sizeof(float), cudaMemcpyHostToDevice, h->stream));
    MCK(cudaMemsetAsync(h->m, 0, n * sizeof(float), h->stream));
    MCK(cudaMemsetAsync(h->v, 0, n * sizeof(float), h->stream));
    h->adam_steps = 0;
    MCK(refresh(h));
    MCK(cudaStreamSynchronize(h->stream));
    return LBM_OK;
}

lbm_status lbm_mlp_get_params(lbm_mlp *h, float *theta, int64_t n) {
    if (!h || !theta || n != h->np) return LBM_ERR_ARG;
    MCK(cudaSetDevice(h->device));
    MCK(cudaMemcpyAsync(theta, h->theta, n * sizeof(float), cudaMemcpyDeviceToHost, h->stream));
    MCK(cudaStreamSynchronize(h->stream));
    return LBM_OK;
}

lbm_status lbm_mlp_forward(lbm_mlp *h, const float *x, int B, float *y) {
    if (bad_batch(h, B) || !x || !y) return LBM_ERR_ARG;
    MCK(cudaSetDevice(h->device));
    lbm_status s = load_input(h, x, B);
    if (s != LBM_OK) return s;
    MCK(forward(h, B, false));
    MCK(cudaMemcpyAsync(y, h->y, (size_t)B * h->n_out * sizeof(float), cudaMemcpyDeviceToHost, h->stream));
    MCK(cudaStreamSynchronize(h->stream));
    return check_err(h);
}

lbm_status lbm_mlp_grad(lbm_mlp *h, const float *x, const float *dy, int B, float *g) {
    if (bad_batch(h, B) || !x || !dy || !g) return LBM_ERR_ARG;
    MCK(cudaSetDevice(h->device));
    lbm_status s = load_input(h, x, B);
    if (s != LBM_OK) return s;
    MCK(forward(h, B, true));
    const int L = h->n_layers - 1;
    const size_t n = (size_t)B * h->n_out;
    std::vector<bf16> db(n);
    for (size_t i = 0; i < n; i++) db[i] = __float2bfloat16_rn(dy[i]);
    MCK(cudaMemcpyAsync(h->gf[L], dy, n * sizeof(float), cudaMemcpyHostToDevice, h->stream));
    MCK(cudaMemcpyAsync(h->gbf[L], db.data(), n * sizeof(bf16), cudaMemcpyHostToDevice, h->stream));
    MCK(transpose(h, h->gbf[L], h->gT[L], B, h->n_out));
    MCK(transpose(h, h->act[0], h->actT[0], B, K0));
    MCK(backward(h, B, nullptr));
    MCK(cudaMemcpyAsync(g, h->grad, h->np * sizeof(float), cudaMemcpyDeviceToHost, h->stream));
    MCK(cudaStreamSynchronize(h->stream));
    return check_err(h);
}

lbm_status lbm_mlp_set_data(lbm_mlp *h, const float *x, const float *t, int n) {
    if (!h || !x || !t || n < 1) return LBM_ERR_ARG;
    MCK(cudaSetDevice(h->device));
    MCK(cudaStreamSynchronize(h->stream));
    if (h->xd) cudaFree(h->xd);
    if (h->td) cudaFree(h->td);
    h->xd = h->td = nullptr;
    MCK(cudaMalloc(&h->xd, (size_t)n * h->n_in * sizeof(float)));
    MCK(cudaMalloc(&h->td, (size_t)n * h->n_out * sizeof(float)));
    MCK(cudaMemcpy(h->xd, x, (size_t)n * h->n_in * sizeof(float), cudaMemcpyHostToDevice));
    MCK(cudaMemcpy(h->td, t, (size_t)n * h->n_out * sizeof(float), cudaMemcpyHostToDevice));
    h->n_data = n;
    return LBM_OK;
}

lbm_status lbm_mlp_train(lbm_mlp *h, const int32_t *order, int n_steps, int B, float lr, float *losses) {
    if (bad_batch(h, B) || !order || n_steps < 1 || !h->xd) return LBM_ERR_ARG;
    for (int64_t i = 0; i < (int64_t)n_steps * B; i++)
        if (order[i] < 0 || order[i] >= h->n_data) return LBM_ERR_ARG;
    MCK(cudaSetDevice(h->device));
    MCK(grow(&h->ord, &h->ord_cap, (size_t)n_steps * B));
    MCK(grow(&h->dl, &h->dl_cap, (size_t)n_steps));
    int32_t *ord = h->ord;
    float *dl = h->dl;
    MCK(cudaMemcpyAsync(ord, order, (size_t)n_steps * B * sizeof(int32_t), cudaMemcpyHostToDevice, h->stream));
    const int L = h->n_layers - 1;
    const float b1 = 0.9f, b2 = 0.999f;
    cudaError_t e = cudaSuccess;
    for (int s = 0; s < n_steps && e == cudaSuccess; s++) {
        e = follow(h, k_gather_batch, dim3(B), 64, 0, h->xd, h->td, ord + (size_t)s * B, B, h->n_in, h->n_out, h->act[0],
                   h->actT[0], h->t);
        if (e == cudaSuccess) e = forward(h, B, true);
        if (e == cudaSuccess)
            e = follow(h, k_mse_grad, dim3(B), 64, 0, h->y, h->t, B, h->n_out, h->gf[L], h->gbf[L], h->gT[L], h->row_loss);
        if (e == cudaSuccess) e = backward(h, B, dl + s);
        if (e != cudaSuccess) break;
        h->adam_steps++;
        const float c1 = 1.f - powf(b1, (float)h->adam_steps), c2 = 1.f - powf(b2, (float)h->adam_steps);
        e = follow(h, k_adam, dim3((unsigned)((h->np + 255) / 256)), 256, 0, h->theta, h->grad, h->m, h->v, h->np, lr, b1,
                   b2, c1, c2, 1e-8f, h->tab);
    }
    if (e == cudaSuccess) e = cudaGetLastError();
    if (e == cudaSuccess && losses)
        e = cudaMemcpyAsync(losses, dl, (size_t)n_steps * sizeof(float), cudaMemcpyDeviceToHost, h->stream);
    const cudaError_t es = cudaStreamSynchronize(h->stream);  // also before the host's arrays may go
    MCK(e);
    MCK(es);
    return check_err(h);
}

void lbm_mlp_destroy(lbm_mlp *h) {
    if (!h) return;
    cudaSetDevice(h->device);
    if (h->stream) cudaStreamSynchronize(h->stream);
    for (void *p : h->allocs) cudaFree(p);
    if (h->ord) cudaFree(h->ord);
    if (h->dl) cudaFree(h->dl);
    if (h->xd) cudaFree(h->xd);
    if (h->td) cudaFree(h->td);
    if (h->own_stream) cudaStreamDestroy(h->stream);
    delete h;
}

}  // extern "C"
