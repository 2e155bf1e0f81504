// Learned warm start for the mass solve (no counterpart in the paper).
//
// A small fully convolutional network on the periodic mesh predicts the mass
// assignment (Sec. 2.4, Eqs. proj and phi_def) from the delta assignment
// (Sec. 2.2, Eq. delta) and the lumped-mass solution b / h^2 (b the exact
// right-hand side of Eq. proj);
// its prediction starts the conjugate-gradient solve, which still finishes to
// the requested residual. Layers: 3x3 periodic convolutions 2 -> 32 -> 32 ->
// 32 -> 1 with bias, ReLU after the first three. Activations are stored in
// BF16 (NHWC, 32 channels = 64 bytes per pixel), products accumulate in FP32.
//
// The two 32 -> 32 layers run on the 5th-generation tensor cores: an implicit
// GEMM per tile of 128 output pixels of one mesh row, M = 128 pixels, N = 32
// output channels, K = 9 taps x 32 input channels = 288 (18 MMAs of K = 16),
// FP32 accumulators in tensor memory. The input rows y-1, y, y+1 of the tile
// (130 pixels each, periodic) are staged in shared memory as planes of 8
// channels x 130 pixels, so that the A operand of tap (dy, dx) is the plane
// of row y+dy shifted by dx pixels: a 16-byte offset of the descriptor start.
// The same kernel computes the data gradient of these layers (weights
// transposed in channels and flipped in taps), with the ReLU mask of the
// layer below fused into its epilogue. The thin first and last layers and the
// weight gradients run on the CUDA cores (deterministic two-stage sums).
#include <cuda_bf16.h>

#include <cstring>
#include <vector>

#include "internal.cuh"
#include "tc.cuh"

#define NCH 32
#define NPARAM 19393
// parameter offsets (layer l: W [Co][Ci][3][3], b [Co])
#define P_W0 0
#define P_B0 576
#define P_W1 608
#define P_B1 9824
#define P_W2 9856
#define P_B2 19072
#define P_W3 19104
#define P_B3 19392

typedef __nv_bfloat16 bf16;

namespace {

__device__ __forceinline__ int wrapn(int i, int n) { return i < 0 ? i + n : (i >= n ? i - n : i); }

// ---------------------------------------------------------------------------
// weight packing
// ---------------------------------------------------------------------------
struct Packed {
    float *w0, *b0;        // [32][2][9] (bf16-rounded), [32]
    bf16 *f1, *d1, *f2, *d2;  // [32][288]: forward (k = tap*32 + ci) and data-gradient (k = tap*32 + co)
    float *b1, *b2;        // [32]
    float *w3, *b3;        // [32][9] (bf16-rounded), [1]
};

__global__ void k_pack(const float *__restrict__ th, Packed P) {
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < 576) P.w0[i] = __bfloat162float(__float2bfloat16(th[P_W0 + i]));
    if (i < 32) {
        P.b0[i] = th[P_B0 + i];
        P.b1[i] = th[P_B1 + i];
        P.b2[i] = th[P_B2 + i];
    }
    if (i < 288) P.w3[i] = __bfloat162float(__float2bfloat16(th[P_W3 + i]));
    if (i == 0) P.b3[0] = th[P_B3];
    if (i < 9216) {
        // i = co*288 + tap*32 + ci  (forward B matrix row co, column k)
        int co = i / 288, k = i % 288, tap = k / 32, ci = k % 32;
        P.f1[i] = __float2bfloat16(th[P_W1 + (co * 32 + ci) * 9 + tap]);
        P.f2[i] = __float2bfloat16(th[P_W2 + (co * 32 + ci) * 9 + tap]);
        // data gradient: row ci' = co (of this matrix), column k = tap'*32 + c, weight W[c][co][8 - tap']
        int r = co, tp = tap, c = ci;
        P.d1[i] = __float2bfloat16(th[P_W1 + (c * 32 + r) * 9 + (8 - tp)]);
        P.d2[i] = __float2bfloat16(th[P_W2 + (c * 32 + r) * 9 + (8 - tp)]);
    }
}

// ---------------------------------------------------------------------------
// first layer (2 -> 32) and last layer (32 -> 1) on CUDA cores
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(256) k_first(const float *__restrict__ x, int B, int n, const float *__restrict__ w0,
                                               const float *__restrict__ b0, bf16 *__restrict__ out) {
    // weights transposed to [c][tap][co] so that 4 output channels' weights
    // are one 16-byte shared-memory read
    __shared__ __align__(16) float sw[18 * 32];
    __shared__ float sb[32];
    for (int i = threadIdx.x; i < 576; i += blockDim.x) {
        const int co = i % 32, ct = i / 32;  // ct = c * 9 + tap
        sw[i] = w0[co * 18 + ct];
    }
    if (threadIdx.x < 32) sb[threadIdx.x] = b0[threadIdx.x];
    __syncthreads();
    ll p = (ll)blockIdx.x * blockDim.x + threadIdx.x;
    const ll npx = (ll)n * n;
    if (p >= npx * B) return;
    const int img = (int)(p / npx), yx = (int)(p % npx), y = yx / n, xx = yx % n;
    float s[32];
#pragma unroll
    for (int co = 0; co < 32; ++co) s[co] = sb[co];
#pragma unroll
    for (int c = 0; c < 2; ++c)
#pragma unroll
        for (int t = 0; t < 9; ++t) {
            const int yy = wrapn(y + t / 3 - 1, n), xs = wrapn(xx + t % 3 - 1, n);
            const float in = __bfloat162float(__float2bfloat16(x[((ll)img * 2 + c) * npx + (ll)yy * n + xs]));
            const float4 *w4 = (const float4 *)(sw + (c * 9 + t) * 32);
#pragma unroll
            for (int q = 0; q < 8; ++q) {
                const float4 w = w4[q];
                s[4 * q] = fmaf(w.x, in, s[4 * q]);
                s[4 * q + 1] = fmaf(w.y, in, s[4 * q + 1]);
                s[4 * q + 2] = fmaf(w.z, in, s[4 * q + 2]);
                s[4 * q + 3] = fmaf(w.w, in, s[4 * q + 3]);
            }
        }
    alignas(16) bf16 o[32];
#pragma unroll
    for (int co = 0; co < 32; ++co) o[co] = __float2bfloat16(fmaxf(s[co], 0.0f));
    uint4 *dst = (uint4 *)(out + p * 32);
    const uint4 *src = (const uint4 *)o;
#pragma unroll
    for (int q = 0; q < 4; ++q) dst[q] = src[q];
}

// 32 -> 1: one block per tile of LTX x LTY output pixels; the tile's input
// with its one-pixel periodic halo is staged in shared memory (80-byte pixel
// stride against bank conflicts), then every thread sums its 9 x 32 products
// in the same order as before (tap, then channel).
#define LTX 32
#define LTY 8
__global__ void __launch_bounds__(256) k_last(const bf16 *__restrict__ a, int B, int n, const float *__restrict__ w3,
                                              const float *__restrict__ b3, float *__restrict__ out) {
    __shared__ float sw[9 * 32 + 1];
    __shared__ uint4 tile[(LTX + 2) * (LTY + 2)][5];
    for (int i = threadIdx.x; i < 289; i += blockDim.x) sw[i] = i < 288 ? w3[(i % 32) * 9 + i / 32] : b3[0];
    const int tiles_x = n / LTX, tiles_y = n / LTY;
    const int img = blockIdx.x / (tiles_x * tiles_y), rem = blockIdx.x % (tiles_x * tiles_y);
    const int x0 = (rem % tiles_x) * LTX, y0 = (rem / tiles_x) * LTY;
    const ll npx = (ll)n * n;
    for (int i = threadIdx.x; i < (LTX + 2) * (LTY + 2) * 4; i += blockDim.x) {
        const int px = i >> 2, q = i & 3;
        const int ty = px / (LTX + 2), tx = px % (LTX + 2);
        const int gy = wrapn(y0 + ty - 1, n), gx = wrapn(x0 + tx - 1, n);
        tile[px][q] = __ldg((const uint4 *)(a + ((ll)img * npx + (ll)gy * n + gx) * 32) + q);
    }
    __syncthreads();
    const int tx = threadIdx.x % LTX, ty = threadIdx.x / LTX;
    float s = sw[288];
#pragma unroll 1
    for (int t = 0; t < 9; ++t) {
        const int px = (ty + t / 3) * (LTX + 2) + tx + t % 3;
        const float *wt = sw + t * 32;
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const uint4 u = tile[px][q];
            const uint32_t w4[4] = {u.x, u.y, u.z, u.w};
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const float lo = __uint_as_float(w4[j] << 16), hi = __uint_as_float(w4[j] & 0xffff0000u);
                s = fmaf(wt[q * 8 + 2 * j], lo, s);
                s = fmaf(wt[q * 8 + 2 * j + 1], hi, s);
            }
        }
    }
    out[(ll)img * npx + (ll)(y0 + ty) * n + x0 + tx] = s;
}

// ---------------------------------------------------------------------------
// 32 -> 32 layer on the tensor cores
// ---------------------------------------------------------------------------
#define CT 128           // output pixels per tile
#define CPW 130          // staged pixels per row (1 halo each side)
#define PLANE (CPW * 16) // bytes of one 8-channel plane

struct ConvArgs {
    const bf16 *in;    // [B][n][n][32]
    bf16 *out;         // [B][n][n][32]
    const bf16 *w;     // [32][288]
    const float *bias; // [32] or null
    const bf16 *mask;  // [B][n][n][32] or null: out = acc if mask > 0 else 0
    int relu;
    int B, n;
    int rows;  // output rows per work item (conv_rows)
    int *status;
};

// One work item is a strip of `rows` output rows of CT pixels. Input rows live in
// a ring of 4 slots in shared memory, each slot 4 planes of 8 channels x CPW
// pixels (16 bytes per pixel); a row is staged once and serves the three
// output rows that need it. Two accumulators of 32 TMEM columns alternate
// between rows: while the tensor cores run the 18 MMAs of row y (issued by
// one thread), the block stores row y-1 from the other accumulator and stages
// row y+2 into the slot that row y-2 used (free once the MMAs of row y-1, the
// last to read it, have signalled their mbarrier).
#define RING (4 * 4 * PLANE)       // 4 row slots of 4 planes (33,280 B)
#define RING_PAD 33792             // ring rounded up to 1 KB
// Dynamic shared memory: ring, B (18,432 B), and 4 KB of slack so that every
// address an operand descriptor can reach stays inside this CTA's allocation.
#define CONV_SMEM (RING_PAD + 18432 + 4096)

// Stage one input row into a ring slot with 16-byte asynchronous copies
// (cp.async): the copies proceed while the block stores the previous output
// row; cp.async.wait_all before the next barrier makes them complete.
__device__ __forceinline__ void stage_row(uint8_t *sA, const bf16 *in, ll img_off, int n, int gy, int x0, int slot,
                                          int tid) {
    for (int i = tid; i < CPW * 4; i += 128) {
        const int px = i >> 2, c = i & 3;
        const int gx = wrapn(x0 + px - 1, n);
        const bf16 *src = in + (img_off + (ll)gy * n + gx) * 32 + c * 8;
        const uint32_t dst = tc::smem_u32(sA + (slot * 4 + c) * PLANE + px * 16);
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
}

__device__ __forceinline__ void stage_wait() { asm volatile("cp.async.wait_all;" ::: "memory"); }

__global__ void __launch_bounds__(128) k_conv_mma(ConvArgs a) {
    extern __shared__ __align__(1024) uint8_t conv_smem[];
    uint8_t *sA = conv_smem;
    uint8_t *sB = conv_smem + RING_PAD;
    __shared__ __align__(8) uint64_t mbar[2];
    __shared__ uint32_t tmem_base;
    __shared__ int abort_flag;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    if (warp == 0) tc::alloc(&tmem_base, 64);
    if (tid == 0) {
        tc::mbar_init(&mbar[0], 1);
        tc::mbar_init(&mbar[1], 1);
        abort_flag = 0;
    }
    // weights: B operand, 36 chunks of [32 rows][8 k] (16 bytes per row)
    for (int i = tid; i < 32 * 36; i += blockDim.x) {
        int row = i / 36, ch = i % 36;
        *(uint4 *)(sB + ch * 512 + row * 16) = *(const uint4 *)(a.w + row * 288 + ch * 8);
    }
    tc::fence_proxy_async();
    tc::fence_before();
    __syncthreads();
    tc::fence_after();
    const uint32_t tmem = tmem_base;
    const int n = a.n, R = a.rows, strips = n / CT, groups = n / R;
    const ll nitems = (ll)a.B * strips * groups;
    const uint32_t idesc = tc::idesc_bf16(128, 32);
    const uint32_t sa = tc::smem_u32(sA), sb = tc::smem_u32(sB);
    uint32_t phase[2] = {0u, 0u};
    bool pend[2] = {false, false};  // a commit on this mbarrier not yet waited for
    float bias[32];
    for (int c = 0; c < 32; ++c) bias[c] = a.bias ? a.bias[c] : 0.0f;

    // epilogue of output row yo from accumulator buf: warp w owns TMEM lanes
    // (pixels) 32w .. 32w+31
    // completion of the MMAs of accumulator buf (bounded wait)
    auto mma_wait = [&](int buf) {
        if (!tc::mbar_wait(&mbar[buf], phase[buf], 1LL << 24)) {
            atomicOr(a.status, ST_TIMEOUT);
            abort_flag = 1;
        }
        phase[buf] ^= 1u;
        pend[buf] = false;
        tc::fence_after();
    };
    // epilogue of output row yo from accumulator buf: warp w owns TMEM lanes
    // (pixels) 32w .. 32w+31
    auto epilogue = [&](int buf, ll img_off, int yo, int x0) {
        float acc[32];
        tc::ld32(tmem + ((uint32_t)(warp * 32) << 16) + (uint32_t)(buf * 32), acc);
        const ll p = img_off + (ll)yo * n + x0 + warp * 32 + lane;
        alignas(16) bf16 o[32];
        if (a.mask) {
            alignas(16) bf16 mk[32];
            const uint4 *ms = (const uint4 *)(a.mask + p * 32);
            for (int q = 0; q < 4; ++q) ((uint4 *)mk)[q] = ms[q];
            for (int c = 0; c < 32; ++c) o[c] = __float2bfloat16(__bfloat162float(mk[c]) > 0.0f ? acc[c] : 0.0f);
        } else {
            for (int c = 0; c < 32; ++c) {
                const float v = acc[c] + bias[c];
                o[c] = __float2bfloat16(a.relu ? fmaxf(v, 0.0f) : v);
            }
        }
        uint4 *dst = (uint4 *)(a.out + p * 32);
        for (int q = 0; q < 4; ++q) dst[q] = ((const uint4 *)o)[q];
    };

    for (ll item = blockIdx.x; item < nitems && !abort_flag; item += gridDim.x) {
        const int img = (int)(item / ((ll)strips * groups));
        const int rem = (int)(item % ((ll)strips * groups));
        const int y0 = (rem / strips) * R, x0 = (rem % strips) * CT;
        const ll img_off = (ll)img * n * n;
        // prologue: rows y0-1, y0, y0+1
        for (int r = -1; r <= 1; ++r) stage_row(sA, a.in, img_off, n, wrapn(y0 + r, n), x0, (y0 + r) & 3, tid);
        stage_wait();
        tc::fence_proxy_async();
        tc::fence_before();
        __syncthreads();
        for (int i = 0; i < R; ++i) {
            const int y = y0 + i, buf = i & 1;
            if (tid == 0) {
                tc::fence_after();
                for (int kb = 0; kb < 18; ++kb) {
                    const int t = kb >> 1, h = kb & 1, dy = t / 3, dx = t % 3;  // dy, dx in 0..2
                    const int slot = (y + dy - 1) & 3;
                    const uint64_t ad = tc::desc(sa + (slot * 4 + 2 * h) * PLANE + dx * 16, PLANE, 128);
                    const uint64_t bd = tc::desc(sb + (2 * kb) * 512, 512, 128);
                    tc::mma_bf16(tmem + (uint32_t)(buf * 32), ad, bd, idesc, kb > 0 ? 1u : 0u);
                }
                tc::commit(&mbar[buf]);
            }
            pend[buf] = true;
            __syncwarp();
            // once the MMAs of row y-1 are done, the ring slot of row y-2 is
            // free: start staging row y+2 there, then store row y-1 out of
            // the other accumulator while the copies are in flight
            if (i > 0) mma_wait(buf ^ 1);
            if (i + 1 < R) stage_row(sA, a.in, img_off, n, wrapn(y + 2, n), x0, (y + 2) & 3, tid);
            if (i > 0) epilogue(buf ^ 1, img_off, y - 1, x0);
            stage_wait();
            tc::fence_proxy_async();
            tc::fence_before();
            __syncthreads();
            if (abort_flag) break;
        }
        if (abort_flag) break;
        mma_wait((R - 1) & 1);
        epilogue((R - 1) & 1, img_off, y0 + R - 1, x0);
        tc::fence_before();
        __syncthreads();
    }
    // after an abort, give MMAs still in flight a bounded time to finish
    // before the accumulators are freed
    for (int b = 0; b < 2; ++b)
        if (pend[b]) tc::mbar_wait(&mbar[b], phase[b], 1LL << 20);
    tc::fence_after();
    __syncthreads();
    if (warp == 0) tc::dealloc(tmem, 64);
}

// ---------------------------------------------------------------------------
// training: loss, backward of the thin layers, weight gradients, Adam
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(256) k_loss(const float *__restrict__ out, const float *__restrict__ tgt, ll m,
                                              float *__restrict__ g, double *__restrict__ part) {
    __shared__ double sh[8];
    double s = 0.0;
    const float inv = 1.0f / (float)m;
    for (ll i = (ll)blockIdx.x * blockDim.x + threadIdx.x; i < m; i += (ll)gridDim.x * blockDim.x) {
        float r = out[i] - tgt[i];
        g[i] = r * inv;
        s += (double)(r * r);
    }
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = s;
    __syncthreads();
    if (threadIdx.x == 0) {
        double t = 0;
        for (int w = 0; w < 8; ++w) t += sh[w];
        part[blockIdx.x] = t;
    }
}

// g_a3[p][c] = sum_tap w3[c][tap] g_out[p - tap], masked by a3 > 0.
__global__ void __launch_bounds__(256) k_last_back(const float *__restrict__ gout, const bf16 *__restrict__ a3, int B,
                                                   int n, const float *__restrict__ w3, bf16 *__restrict__ gz) {
    __shared__ float sw[288];
    for (int i = threadIdx.x; i < 288; i += blockDim.x) sw[i] = w3[i];
    __syncthreads();
    ll p = (ll)blockIdx.x * blockDim.x + threadIdx.x;
    const ll npx = (ll)n * n;
    if (p >= npx * B) return;
    const int img = (int)(p / npx), yx = (int)(p % npx), y = yx / n, xx = yx % n;
    float gt[9];
    for (int t = 0; t < 9; ++t) {
        int yy = wrapn(y - (t / 3 - 1), n), xs = wrapn(xx - (t % 3 - 1), n);
        gt[t] = gout[(ll)img * npx + (ll)yy * n + xs];
    }
    alignas(16) bf16 mk[32];
    for (int q = 0; q < 4; ++q) ((uint4 *)mk)[q] = ((const uint4 *)(a3 + p * 32))[q];
    alignas(16) bf16 o[32];
    for (int c = 0; c < 32; ++c) {
        float s = 0.0f;
        for (int t = 0; t < 9; ++t) s = fmaf(sw[c * 9 + t], gt[t], s);
        o[c] = __float2bfloat16(__bfloat162float(mk[c]) > 0.0f ? s : 0.0f);
    }
    for (int q = 0; q < 4; ++q) ((uint4 *)(gz + p * 32))[q] = ((const uint4 *)o)[q];
}

// Weight gradient of a 32 -> 32 layer:
// dW[co][ci][tap] = sum_p g[p][co] a[p + tap][ci], db[co] = sum_p g[p][co],
// a contraction over all pixels (M = 32 co, N = 9 taps x 32 ci, K = pixels)
// of 9 GFLOP on 67 MB of activations (8 images of 256^2), so the floor is
// reading them. Both operands are stored pixel-major (K-major rows of 64
// bytes), the layout ldmatrix.trans turns into fragments of the warp-level
// m16n8k16 MMA; the accumulators (72 registers per lane) stay in registers
// over all of a block's rows, so nothing but the staging touches shared memory.
// A unit is one row of 128 pixels. A block takes a contiguous range of units,
// (image, column strip, row), keeps the input rows y-1, y, y+1 in a ring of 4
// and prefetches the next row and gradient row with cp.async while it
// multiplies. Warp w takes input channels 8 (w & 3) .. + 7, all taps and all 32
// outputs, over pixels 64 (w >> 2) .. + 63 of the row. A pixel takes 80 bytes of
// shared memory: the 8 rows of an ldmatrix then fall in distinct banks.
// The bias gradient is one more column of ones (warps w & 3 = 0).
// 8 images of 256^2: 48 us, where FP32 sums on the CUDA cores took 615 us (one
// pixel at a time, every operand from shared memory). What bounds it now is the
// latency of the MMAs at 13 warps per SM. Error of W and b against 64-bit sums of
// the same operands, 1 to 8 images of 128^2 to 1024^2, rms: 6.1e-8 and 2.7e-8
// (FP32 sums on the CUDA cores: 1.0e-7 and 2.9e-8); first layer 7.2e-8 (1.8e-7), last
// 1.0e-7 (3.4e-7).
#define WG_PX 80                     // bytes of a staged pixel
#define WG_ROW (CPW * WG_PX)         // an input row with its halo
#define WG_GROW (CT * WG_PX)         // a gradient row
#define WG_SMEM (4 * WG_ROW + 2 * WG_GROW)

__device__ __forceinline__ void cp16(void *dst, const void *src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(tc::smem_u32(dst)), "l"(src) : "memory");
}
__device__ __forceinline__ void ldmat4t(uint32_t (&r)[4], uint32_t addr) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                 : "r"(addr)
                 : "memory");
}
__device__ __forceinline__ void ldmat2t(uint32_t (&r)[2], uint32_t addr) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x2.trans.shared.b16 {%0,%1}, [%2];"
                 : "=r"(r[0]), "=r"(r[1])
                 : "r"(addr)
                 : "memory");
}
__device__ __forceinline__ void mma16816(float (&d)[4], const uint32_t (&a)[4], const uint32_t (&b)[2]) {
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
        : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b[0]), "r"(b[1]));
}

__global__ void __launch_bounds__(256, 2) k_wgrad_mid(const bf16 *__restrict__ g, const bf16 *__restrict__ a, int B,
                                                      int n, int per_block, float *__restrict__ part) {
    extern __shared__ __align__(128) uint8_t wg_smem[];
    uint8_t *sa = wg_smem, *sg = wg_smem + 4 * WG_ROW;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, cit = warp & 3, half = warp >> 2;
    const int strips = n / CT, units = B * strips * n;
    const int u0 = blockIdx.x * per_block, u1 = min(u0 + per_block, units);
    float acc[2][10][4];  // [output half][tap, or 9: ones][fragment]
#pragma unroll
    for (int i = 0; i < 2; ++i)
#pragma unroll
        for (int t = 0; t < 10; ++t)
#pragma unroll
            for (int q = 0; q < 4; ++q) acc[i][t][q] = 0.0f;
    // input row y of a strip (unwrapped, -1 .. n) into ring slot y & 3
    auto stage_in = [&](int img, int x0, int y) {
        const bf16 *row = a + ((ll)img * n + wrapn(y, n)) * n * 32;
        uint8_t *dst = sa + (y & 3) * WG_ROW;
        for (int i = tid; i < CPW * 4; i += 256)
            cp16(dst + (i >> 2) * WG_PX + (i & 3) * 16, row + wrapn(x0 + (i >> 2) - 1, n) * 32 + (i & 3) * 8);
    };
    auto stage_g = [&](int img, int x0, int y) {
        const bf16 *row = g + (((ll)img * n + y) * n + x0) * 32;
        uint8_t *dst = sg + (y & 1) * WG_GROW;
        for (int i = tid; i < CT * 4; i += 256) cp16(dst + (i >> 2) * WG_PX + (i & 3) * 16, row + i * 8);
    };
    const uint32_t sau = tc::smem_u32(sa), sgu = tc::smem_u32(sg);
    // ldmatrix row addresses: A blocks (co 0-7, px 0-7), (co 8-15, px 0-7),
    // (co 0-7, px 8-15), (co 8-15, px 8-15); B blocks px 0-7, px 8-15
    const uint32_t aoff = ((lane & 7) + ((lane >> 4) & 1) * 8) * WG_PX + ((lane >> 3) & 1) * 16;
    const uint32_t boff = (lane & 15) * WG_PX + cit * 16;
    for (int u = u0; u < u1; ++u) {
        const int y = u % n, run = u / n, img = run / strips, x0 = (run % strips) * CT;
        if (u == u0 || y == 0) {  // a new strip: nothing staged yet
            for (int r = -1; r <= 1; ++r) stage_in(img, x0, y + r);
            stage_g(img, x0, y);
        }
        asm volatile("cp.async.wait_all;" ::: "memory");
        __syncthreads();
        if (u + 1 < u1 && y + 1 < n) {
            stage_in(img, x0, y + 2);
            stage_g(img, x0, y + 1);
        }
#pragma unroll 1
        for (int k = 0; k < 4; k += 2) {
            const int px = half * 64 + k * 16;
            uint32_t A[2][2][4];  // [pixel step][output half]
            const uint32_t ga = sgu + (y & 1) * WG_GROW + px * WG_PX + aoff;
#pragma unroll
            for (int q = 0; q < 2; ++q) {
                ldmat4t(A[q][0], ga + q * 16 * WG_PX);
                ldmat4t(A[q][1], ga + q * 16 * WG_PX + 32);
            }
            // 32 pixels in the tensor cores, whose sums truncate, then one
            // rounded addition: the error stays that of FP32 sums
#pragma unroll
            for (int t = 0; t < 10; ++t) {
                if (t == 9 && cit != 0) break;
                float d[2][4];
#pragma unroll
                for (int q = 0; q < 4; ++q) d[0][q] = d[1][q] = 0.0f;
#pragma unroll
                for (int q = 0; q < 2; ++q) {
                    uint32_t Bf[2] = {0x3f803f80u, 0x3f803f80u};  // ones: the bias gradient
                    if (t < 9)
                        ldmat2t(Bf, sau + ((y + t / 3 - 1) & 3) * WG_ROW + (px + q * 16 + t % 3) * WG_PX + boff);
                    mma16816(d[0], A[q][0], Bf);
                    mma16816(d[1], A[q][1], Bf);
                }
#pragma unroll
                for (int i = 0; i < 2; ++i)
#pragma unroll
                    for (int q = 0; q < 4; ++q) acc[i][t][q] += d[i][q];
            }
        }
        __syncthreads();
    }
    // the two pixel halves, then this block's partial in parameter order
    float *sx = (float *)wg_smem;
    asm volatile("cp.async.wait_all;" ::: "memory");
    __syncthreads();
    if (half == 1) {
#pragma unroll
        for (int i = 0; i < 2; ++i)
#pragma unroll
            for (int t = 0; t < 10; ++t)
#pragma unroll
                for (int q = 0; q < 4; ++q) sx[((i * 10 + t) * 4 + q) * 128 + cit * 32 + lane] = acc[i][t][q];
    }
    __syncthreads();
    if (half == 0) {
        float *dst = part + (ll)blockIdx.x * 9248;
#pragma unroll
        for (int i = 0; i < 2; ++i)
#pragma unroll
            for (int t = 0; t < 10; ++t)
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    const float v = acc[i][t][q] + sx[((i * 10 + t) * 4 + q) * 128 + cit * 32 + lane];
                    const int co = i * 16 + (lane >> 2) + (q >> 1) * 8, c = (lane & 3) * 2 + (q & 1);
                    if (t < 9) dst[(co * 32 + cit * 8 + c) * 9 + t] = v;
                    else if (cit == 0 && c == 0) dst[9216 + co] = v;
                }
    }
}

// Weight gradients of the first (2 -> 32) and last (32 -> 1) layers in FP32:
//   dW0[co][c][tap] = sum_p gz1[p][co] bf16(x[c][p + tap]), db0[co] = sum_p gz1[p][co]
//   dW3[ci][tap] = sum_q a3[q][ci] gout[q - tap],           db3 = sum_p gout[p].
// A lane holds two channels (one 4-byte load per pixel and array) and packed
// FP32 accumulators for all taps; a half-warp walks along a row of 32 pixels
// with the taps' values sliding through registers, so a pixel costs it two
// loads, 9 shared-memory reads and 28 packed FMAs. The x and gout rows of a
// 64 x 4 pixel tile are staged in shared memory, duplicated into pairs for the
// packed FMA. 8 images of 256^2: 36 us, against 2.49 ms with one thread per
// weight walking over all pixels. Per-block partials [608 + 289].
#define WTX 64
#define WTY 4
__device__ __forceinline__ f32x2 bf2(uint32_t v) {  // two BF16 -> two FP32
    f32x2 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "r"(v << 16), "r"(v & 0xffff0000u));
    return r;
}
__global__ void __launch_bounds__(256, 2) k_wgrad_thin(const bf16 *__restrict__ gz1, const float *__restrict__ x,
                                                    const float *__restrict__ gout, const bf16 *__restrict__ a3, int B,
                                                    int n, float *__restrict__ part) {
    __shared__ f32x2 sx[2][WTY + 2][WTX + 2], so[WTY + 2][WTX + 2];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, hw = lane >> 4, cp = lane & 15;
    const int tiles_x = n / WTX, tiles_y = n / WTY, ntiles = B * tiles_x * tiles_y;
    const ll npx = (ll)n * n;
    auto twice = [](float v) { return pk2(v, v); };
    f32x2 w0[2][9], b0 = 0, w3[9];
    KSum b3;
#pragma unroll
    for (int t = 0; t < 9; ++t) w0[0][t] = w0[1][t] = w3[t] = 0;
    const int ty = warp >> 1, tx0 = (warp & 1) * 32 + hw * 16;  // this half-warp's 16 pixels
    for (int tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
        const int img = tile / (tiles_x * tiles_y), rem = tile % (tiles_x * tiles_y);
        const int y0 = (rem / tiles_x) * WTY, x0 = (rem % tiles_x) * WTX;
        __syncthreads();
        for (int i = tid; i < (WTY + 2) * (WTX + 2); i += 256) {
            const int ly = i / (WTX + 2), lx = i % (WTX + 2);
            const ll o = (ll)wrapn(y0 + ly - 1, n) * n + wrapn(x0 + lx - 1, n);
            sx[0][ly][lx] = twice(__bfloat162float(__float2bfloat16(x[((ll)img * 2) * npx + o])));
            sx[1][ly][lx] = twice(__bfloat162float(__float2bfloat16(x[((ll)img * 2 + 1) * npx + o])));
            so[ly][lx] = twice(gout[(ll)img * npx + o]);
        }
        __syncthreads();
        const ll p0 = (ll)img * npx + (ll)(y0 + ty) * n + x0 + tx0;
        const uint32_t *gp = (const uint32_t *)(gz1 + p0 * 32) + cp, *ap = (const uint32_t *)(a3 + p0 * 32) + cp;
        float bt = 0.0f;
        // columns lx - 1, lx, lx + 1 of the three rows around the pixel
        f32x2 v0[3][3], v1[3][3], vo[3][3];
#pragma unroll
        for (int r = 0; r < 3; ++r)
#pragma unroll
            for (int c = 0; c < 2; ++c) {
                v0[r][c] = sx[0][ty + r][tx0 + c];
                v1[r][c] = sx[1][ty + r][tx0 + c];
                vo[r][c] = so[ty + r][tx0 + c];
            }
#pragma unroll
        for (int k = 0; k < 16; ++k) {
            const f32x2 gv = bf2(__ldg(gp + k * 16)), av = bf2(__ldg(ap + k * 16));
#pragma unroll
            for (int r = 0; r < 3; ++r) {
                v0[r][(k + 2) % 3] = sx[0][ty + r][tx0 + k + 2];
                v1[r][(k + 2) % 3] = sx[1][ty + r][tx0 + k + 2];
                vo[r][(k + 2) % 3] = so[ty + r][tx0 + k + 2];
            }
#pragma unroll
            for (int t = 0; t < 9; ++t) {
                w0[0][t] = fma2(gv, v0[t / 3][(k + t % 3) % 3], w0[0][t]);
                w0[1][t] = fma2(gv, v1[t / 3][(k + t % 3) % 3], w0[1][t]);
                w3[t] = fma2(av, vo[2 - t / 3][(k + 2 - t % 3) % 3], w3[t]);
            }
            b0 = add2(b0, gv);
            bt += __uint_as_float((unsigned)vo[1][(k + 1) % 3]);
        }
        b3.add(bt);
    }
    // half-warps, then warps in order, through shared memory
    __syncthreads();
    float *sr = (float *)sx;  // [8 warps][58][16]: 3 rounds of what fits
    auto lo = [](f32x2 v) { return __uint_as_float((unsigned)v); };
    auto hi = [](f32x2 v) { return __uint_as_float((unsigned)(v >> 32)); };
    float *dst = part + (ll)blockIdx.x * 897;
    // one packed accumulator at a time: slot q of the list w0[0], w0[1], b0, w3
#pragma unroll
    for (int q = 0; q < 28; ++q) {
        f32x2 v = q < 9 ? w0[0][q] : (q < 18 ? w0[1][q - 9] : (q == 18 ? b0 : w3[q - 19]));
        v = add2(v, __shfl_xor_sync(0xffffffffu, v, 16));
        if (hw == 0) {
            sr[(q & 3) * 256 + warp * 32 + cp * 2] = lo(v);
            sr[(q & 3) * 256 + warp * 32 + cp * 2 + 1] = hi(v);
        }
        if ((q & 3) == 3) {
            __syncthreads();
            if (tid < 128) {
                const int qq = q - 3 + (tid >> 5), ch = tid & 31;
                float s = 0.0f;
                for (int w = 0; w < 8; ++w) s += sr[(tid >> 5) * 256 + w * 32 + ch];
                const int o = qq < 18 ? ch * 18 + qq : (qq == 18 ? 576 + ch : 608 + ch * 9 + (qq - 19));
                dst[o] = s;
            }
            __syncthreads();
        }
    }
    // every lane of a half-warp holds the same sum of gout
    if (cp == 0) sr[warp * 2 + hw] = b3.get();
    __syncthreads();
    if (tid == 0) {
        KSum s;
        for (int w = 0; w < 16; ++w) s.add(sr[w]);
        dst[896] = s.get();
    }
}

// grad[map(i)] = sum over the blocks of part[b][i] in a fixed order, in Sum3 (no
// fewer bits than FP64, which would bound the kernel): 32 threads per parameter
// take every 32nd block, then FP64 over the 32 sums (up to 256 dependent
// additions by one thread had taken 44 us, this 8).
#define RED_T 32
template <class Map>
__device__ __forceinline__ void reduce_parts(const float *__restrict__ part, int nblk, int len, float *__restrict__ grad,
                                             Map map) {
    __shared__ double sh[RED_T][33];
    const int i = blockIdx.x * 32 + threadIdx.x;
    Sum3 s{0.0f, 0.0f, 0.0f, 0};
    if (i < len) {
#pragma unroll 5
        for (int b = threadIdx.y; b < nblk; b += RED_T) add_parts(s, part[(ll)b * len + i], 0.0f, 0.0f);
    }
    sh[threadIdx.y][threadIdx.x] = ((double)s.a + (double)s.b) + (double)s.c;
    __syncthreads();
    if (threadIdx.y == 0 && i < len) {
        double t = 0.0;
        for (int k = 0; k < RED_T; ++k) t += sh[k][threadIdx.x];
        grad[map(i)] = (float)t;
    }
}
__global__ void __launch_bounds__(32 * RED_T) k_reduce_thin(const float *__restrict__ part, int nblk,
                                                            float *__restrict__ grad) {
    reduce_parts(part, nblk, 897, grad, [](int i) { return i < 608 ? P_W0 + i : P_W3 + (i - 608); });
}
// middle layers: partial layout [9216 W then 32 b]
__global__ void __launch_bounds__(32 * RED_T) k_reduce_mid(const float *__restrict__ part, int nblk,
                                                           float *__restrict__ grad, int offW, int offB) {
    reduce_parts(part, nblk, 9248, grad, [=](int i) { return i < 9216 ? offW + i : offB + (i - 9216); });
}

__global__ void k_adam(float *__restrict__ th, const float *__restrict__ g, float *__restrict__ m, float *__restrict__ v,
                       int np, float lr, float b1, float b2, float c1, float c2, float eps) {
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= np) return;
    float gi = g[i];
    float mi = b1 * m[i] + (1.0f - b1) * gi, vi = b2 * v[i] + (1.0f - b2) * gi * gi;
    m[i] = mi;
    v[i] = vi;
    th[i] -= lr * (mi / c1) / (sqrtf(vi / c2) + eps);
}

}  // namespace

// ---------------------------------------------------------------------------
// host side
// ---------------------------------------------------------------------------
struct pm_net {
    int max_n, max_b;
    cudaStream_t st;
    float *theta, *grad, *m, *v;
    Packed P;
    bf16 *a1, *a2, *a3, *g1, *g2;  // activations and gradients [B][n][n][32]
    float *out, *gout;             // [B][n][n]
    float *part_mid, *part_thin;
    double *loss_part;
    double *h_loss;
    int *status;
    long long step;
    int nsm;
    std::vector<void *> allocs;
};

namespace {

template <class T>
bool nalloc(pm_net *t, T **p, size_t count) {
    if (cudaMalloc((void **)p, sizeof(T) * (count ? count : 1)) != cudaSuccess) return false;
    t->allocs.push_back((void *)*p);
    return true;
}

const int WG_BLOCKS = 304;   // weight-gradient partial blocks (two per SM)
const int LOSS_BLOCKS = 256;

void net_pack(pm_net *t) {
    k_pack<<<div_up(9216, 256), 256, 0, t->st>>>(t->theta, t->P);
    count_launches(1);
}

// Output rows per work item: a taller strip reads fewer halo rows and fills its
// pipeline once, but leaves SMs idle when there are few strips. An item costs
// about rows + 2 row times (the first rows have nothing to overlap with), so
// the number of waves over the resident CTAs decides. 8 images of 256^2 take 8
// rows (512 items): 37 us a layer, 41 us with 16 (256 items).
int conv_rows(const pm_net *t, int B, int n) {
    int best = 16;
    ll cost = -1;
    for (int r : {16, 8, 4}) {
        const ll items = (ll)B * (n / CT) * (n / r), waves = (items + 4LL * t->nsm - 1) / (4LL * t->nsm);
        if (cost < 0 || waves * (r + 2) < cost) {
            cost = waves * (r + 2);
            best = r;
        }
    }
    return best;
}

// One 32 -> 32 layer. At most 4 CTAs per SM (shared memory bound), so at most
// 128 of the 512 tensor-memory columns of an SM are ever requested.
void conv_layer(pm_net *t, const bf16 *in, bf16 *out, const bf16 *w, const float *bias, const bf16 *mask, int relu,
                int B, int n) {
    const int rows = conv_rows(t, B, n);
    const ll items = (ll)B * (n / CT) * (n / rows), cap = (ll)t->nsm * 4;
    const ConvArgs a{in, out, w, bias, mask, relu, B, n, rows, t->status};
    k_conv_mma<<<(int)(items < cap ? items : cap), 128, CONV_SMEM, t->st>>>(a);
}

void net_forward(pm_net *t, const float *x, int B, int n, float *out) {
    const ll m = (ll)B * n * n;
    net_pack(t);
    k_first<<<div_up(m, 256), 256, 0, t->st>>>(x, B, n, t->P.w0, t->P.b0, t->a1);
    conv_layer(t, t->a1, t->a2, t->P.f1, t->P.b1, nullptr, 1, B, n);
    conv_layer(t, t->a2, t->a3, t->P.f2, t->P.b2, nullptr, 1, B, n);
    k_last<<<B * (n / LTX) * (n / LTY), LTX * LTY, 0, t->st>>>(t->a3, B, n, t->P.w3, t->P.b3, out);
    count_launches(4);
}

}  // namespace

extern "C" {

int pm_net_num_params(void) { return NPARAM; }

pm_status pm_net_create(pm_net **out, int max_n, int max_batch, void *stream) {
    if (!out || max_n < CT || max_n % CT || max_batch < 1) return PM_EINVAL;
    *out = nullptr;
    pm_net *t = new pm_net();
    t->max_n = max_n;
    t->max_b = max_batch;
    t->st = (cudaStream_t)stream;
    t->step = 0;
    int dev = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&t->nsm, cudaDevAttrMultiProcessorCount, dev);
    const size_t m = (size_t)max_n * max_n * max_batch;
    bool ok = nalloc(t, &t->theta, NPARAM) && nalloc(t, &t->grad, NPARAM) && nalloc(t, &t->m, NPARAM) &&
              nalloc(t, &t->v, NPARAM) && nalloc(t, &t->P.w0, 576) && nalloc(t, &t->P.b0, 32) &&
              nalloc(t, &t->P.f1, 9216) && nalloc(t, &t->P.d1, 9216) && nalloc(t, &t->P.f2, 9216) &&
              nalloc(t, &t->P.d2, 9216) && nalloc(t, &t->P.b1, 32) && nalloc(t, &t->P.b2, 32) &&
              nalloc(t, &t->P.w3, 288) && nalloc(t, &t->P.b3, 1) && nalloc(t, &t->a1, m * 32) &&
              nalloc(t, &t->a2, m * 32) && nalloc(t, &t->a3, m * 32) && nalloc(t, &t->g1, m * 32) &&
              nalloc(t, &t->g2, m * 32) && nalloc(t, &t->out, m) && nalloc(t, &t->gout, m) &&
              nalloc(t, &t->part_mid, (size_t)WG_BLOCKS * 9248) && nalloc(t, &t->part_thin, (size_t)WG_BLOCKS * 897) && nalloc(t, &t->loss_part, LOSS_BLOCKS) &&
              nalloc(t, &t->status, 1);
    if (ok && cudaMallocHost((void **)&t->h_loss, sizeof(double) * (LOSS_BLOCKS + 1)) != cudaSuccess) ok = false;
    if (!ok) {
        pm_net_destroy(t);
        cudaGetLastError();
        return PM_ENOMEM;
    }
    cudaMemset(t->theta, 0, sizeof(float) * NPARAM);
    cudaMemset(t->m, 0, sizeof(float) * NPARAM);
    cudaMemset(t->v, 0, sizeof(float) * NPARAM);
    cudaMemset(t->status, 0, sizeof(int));
    cudaFuncSetAttribute(k_wgrad_mid, cudaFuncAttributeMaxDynamicSharedMemorySize, WG_SMEM);
    cudaFuncSetAttribute(k_conv_mma, cudaFuncAttributeMaxDynamicSharedMemorySize, CONV_SMEM);
    if (cudaDeviceSynchronize() != cudaSuccess) {
        pm_net_destroy(t);
        return PM_ECUDA;
    }
    *out = t;
    return PM_OK;
}

void pm_net_destroy(pm_net *t) {
    if (!t) return;
    for (void *p : t->allocs) cudaFree(p);
    if (t->h_loss) cudaFreeHost(t->h_loss);
    delete t;
}

pm_status pm_net_set_stream(pm_net *t, void *stream) {
    if (!t) return PM_EINVAL;
    t->st = (cudaStream_t)stream;
    return PM_OK;
}

pm_status pm_net_state(pm_net *t, float *host_out, long long *step_out) {
    if (!t || !host_out) return PM_EINVAL;
    cudaStreamSynchronize(t->st);
    if (cudaMemcpy(host_out, t->theta, sizeof(float) * NPARAM, cudaMemcpyDeviceToHost) != cudaSuccess ||
        cudaMemcpy(host_out + NPARAM, t->m, sizeof(float) * NPARAM, cudaMemcpyDeviceToHost) != cudaSuccess ||
        cudaMemcpy(host_out + 2 * NPARAM, t->v, sizeof(float) * NPARAM, cudaMemcpyDeviceToHost) != cudaSuccess)
        return PM_ECUDA;
    if (step_out) *step_out = t->step;
    return PM_OK;
}

pm_status pm_net_load(pm_net *t, const float *host_in, int with_moments, long long step) {
    if (!t || !host_in) return PM_EINVAL;
    cudaStreamSynchronize(t->st);
    if (cudaMemcpy(t->theta, host_in, sizeof(float) * NPARAM, cudaMemcpyHostToDevice) != cudaSuccess) return PM_ECUDA;
    if (with_moments) {
        if (cudaMemcpy(t->m, host_in + NPARAM, sizeof(float) * NPARAM, cudaMemcpyHostToDevice) != cudaSuccess ||
            cudaMemcpy(t->v, host_in + 2 * NPARAM, sizeof(float) * NPARAM, cudaMemcpyHostToDevice) != cudaSuccess)
            return PM_ECUDA;
    } else {
        cudaMemset(t->m, 0, sizeof(float) * NPARAM);
        cudaMemset(t->v, 0, sizeof(float) * NPARAM);
    }
    t->step = step;
    return PM_OK;
}

pm_status pm_net_forward(pm_net *t, const float *x, int B, int n, float *out) {
    if (!t || !x || !out || B < 1 || B > t->max_b || n < CT || n % CT || n > t->max_n) return PM_EINVAL;
    net_forward(t, x, B, n, out);
    return cudaGetLastError() == cudaSuccess ? PM_OK : PM_ECUDA;
}

pm_status pm_net_train_step(pm_net *t, const float *x, const float *target, int B, int n, float lr, double *loss) {
    if (!t || !x || !target || B < 1 || B > t->max_b || n < CT || n % CT || n > t->max_n) return PM_EINVAL;
    const ll m = (ll)B * n * n;
    net_forward(t, x, B, n, t->out);
    k_loss<<<LOSS_BLOCKS, 256, 0, t->st>>>(t->out, target, m, t->gout, t->loss_part);
    k_last_back<<<div_up(m, 256), 256, 0, t->st>>>(t->gout, t->a3, B, n, t->P.w3, t->g2);  // g2 = dL/dz3 (pre-ReLU)
    // rows of 128 pixels per weight-gradient block, and the blocks that have any
    const int units = B * (n / CT) * n, per = (units + WG_BLOCKS - 1) / WG_BLOCKS, wblk = (units + per - 1) / per;
    const dim3 rblk(32, RED_T);
    // layer 2 (input a2, output gradient g2)
    k_wgrad_mid<<<wblk, 256, WG_SMEM, t->st>>>(t->g2, t->a2, B, n, per, t->part_mid);
    k_reduce_mid<<<div_up(9248, 32), rblk, 0, t->st>>>(t->part_mid, wblk, t->grad, P_W2, P_B2);
    conv_layer(t, t->g2, t->g1, t->P.d2, nullptr, t->a2, 0, B, n);  // g1 = dL/dz2
    // layer 1 (input a1, output gradient g1)
    k_wgrad_mid<<<wblk, 256, WG_SMEM, t->st>>>(t->g1, t->a1, B, n, per, t->part_mid);
    k_reduce_mid<<<div_up(9248, 32), rblk, 0, t->st>>>(t->part_mid, wblk, t->grad, P_W1, P_B1);
    conv_layer(t, t->g1, t->g2, t->P.d1, nullptr, t->a1, 0, B, n);  // g2 = dL/dz1
    // first and last layers
    const int tblk = min(WG_BLOCKS, B * (n / WTX) * (n / WTY));
    k_wgrad_thin<<<tblk, 256, 0, t->st>>>(t->g2, x, t->gout, t->a3, B, n, t->part_thin);
    k_reduce_thin<<<div_up(897, 32), rblk, 0, t->st>>>(t->part_thin, tblk, t->grad);
    t->step += 1;
    const float b1 = 0.9f, b2 = 0.999f;
    const float c1 = 1.0f - powf(b1, (float)t->step), c2 = 1.0f - powf(b2, (float)t->step);
    k_adam<<<div_up(NPARAM, 256), 256, 0, t->st>>>(t->theta, t->grad, t->m, t->v, NPARAM, lr, b1, b2, c1, c2, 1e-8f);
    count_launches(11);
    if (cudaGetLastError() != cudaSuccess) return PM_ECUDA;
    if (loss) {
        if (cudaMemcpyAsync(t->h_loss, t->loss_part, sizeof(double) * LOSS_BLOCKS, cudaMemcpyDeviceToHost, t->st) !=
                cudaSuccess ||
            cudaStreamSynchronize(t->st) != cudaSuccess)
            return PM_ECUDA;
        double s = 0.0;
        for (int b = 0; b < LOSS_BLOCKS; ++b) s += t->h_loss[b];
        *loss = 0.5 * s / (double)m;
        int st = 0;
        cudaMemcpy(&st, t->status, sizeof(int), cudaMemcpyDeviceToHost);
        if (st & ST_TIMEOUT) return PM_ETIMEOUT;
    }
    return PM_OK;
}

// Gradient of the last train step (host, NPARAM floats), for tests.
pm_status pm_net_grad(pm_net *t, float *host_out) {
    if (!t || !host_out) return PM_EINVAL;
    cudaStreamSynchronize(t->st);
    return cudaMemcpy(host_out, t->grad, sizeof(float) * NPARAM, cudaMemcpyDeviceToHost) == cudaSuccess ? PM_OK
                                                                                                           : PM_ECUDA;
}

}  // extern "C"
