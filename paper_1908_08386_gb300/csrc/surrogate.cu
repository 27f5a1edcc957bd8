// Kernels of the learned warm start (include/surrogate.h).
//
// The forward and adjoint 3x3 convolutions run on the fifth-generation tensor
// cores (conv_tc.cu: tcgen05.mma with tensor-memory accumulators, TMA-staged
// operands).  This file holds the rest:
// weight and bias gradient (wgrad_kernel): one block owns 32 output x 16 input
//   channels and a strided share of the pixels (split K); products on the
//   tensor cores by warp-level mma (m16n8k16, BF16, FP32 accumulation) from
//   operands staged by cp.async and read transposed with ldmatrix (rows of
//   16 bytes XOR-swizzled so that the eight rows one ldmatrix phase reads fall
//   in distinct bank groups); partial sums end in FP32 atomics.
// Everything else is small and elementwise.

#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <cstdarg>
#include <cstdio>

#include "conv_tc.h"
#include "surrogate.h"

namespace {

thread_local char g_sg_err[256] = "";

int sg_fail(int code, const char *fmt, ...) {
    va_list ap;
    va_start(ap, fmt);
    vsnprintf(g_sg_err, sizeof(g_sg_err), fmt, ap);
    va_end(ap);
    return code;
}

constexpr int kOk = 0, kErrArg = -1, kErrCuda = -3;

int launched(const char *what) {
    const cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return sg_fail(kErrCuda, "%s: %s", what, cudaGetErrorString(e));
    return kOk;
}

using bf16 = __nv_bfloat16;
constexpr float kLeak = 1.0f / 16.0f;

__device__ __forceinline__ float dleaky(float y) { return y > 0.0f ? 1.0f : kLeak; }

__device__ __forceinline__ uint32_t smem_addr(const void *p) {
    return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

// 16-byte asynchronous copy global -> shared; src_bytes = 0 fills zeros.
__device__ __forceinline__ void cp_async16(void *dst, const void *src, int src_bytes) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(smem_addr(dst)), "l"(src), "r"(src_bytes)
                 : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() {
    asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

__device__ __forceinline__ void ldsm_x4_t(uint32_t &r0, uint32_t &r1, uint32_t &r2, uint32_t &r3, const void *p) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0, %1, %2, %3}, [%4];"
                 : "=r"(r0), "=r"(r1), "=r"(r2), "=r"(r3)
                 : "r"(smem_addr(p)));
}

// d += a (16x16, row) * b (16x8, col), BF16 inputs, FP32 accumulators.
__device__ __forceinline__ void mma16816(float d[4], const uint32_t a[4], const uint32_t b[2]) {
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, "
        "{%0, %1, %2, %3};"
        : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b[0]), "r"(b[1]));
}

// Element offset of 16-byte chunk `c` of a 32-byte row `r` (two chunks per
// row): chunks swap on every other group of four rows.
__device__ __forceinline__ int sw32(int r, int c) { return r * 16 + ((c ^ ((r >> 2) & 1)) << 3); }
// The same for 64-byte rows (four chunks).
__device__ __forceinline__ int sw64(int r, int c) { return r * 32 + ((c ^ ((r >> 1) & 3)) << 3); }

// ---------------------------------------------------------------------------
// weight gradient of the 3x3 convolution
// ---------------------------------------------------------------------------
// A block owns 32 output x 16 input channels of all nine taps and a share of
// the pieces (8 rows x 16 pixels of one image); each of its eight warps takes
// pieces of its own and keeps the whole 9 x 32 x 16 accumulator in registers.
// A row of a piece is one K step of 16 pixels: the output-gradient fragments
// (two ldmatrix) stay in registers for the three input rows that meet them and
// the three shifted input fragments of a row serve the three output rows around
// it, so 36 MMAs follow five ldmatrix (a warp per tap needed three for four).
// Rows arrive through a five-slot ring per warp filled by cp.async four rows
// ahead; the warps never wait for one another until the sums are folded.
// Bound by the warp-level MMA rate and the L2 traffic of re-reading dy for
// every block of 16 input channels.
// The bias gradient adds up the same fragments (in FP32): the Cin / 16 blocks
// that read a piece's dy take turns, one per piece (a kernel of its own walked
// 1024 pixels per thread).
// Measured (ncu, 32 maps of 128^2, the network's 14 layers summed): weight and
// bias gradients 761 + 2450 -> 447 us.
constexpr int kTH = 8, kTW = 16;       // piece: 8 rows x 16 pixels
constexpr int kWCo = 32, kWCi = 16;    // channels per block
constexpr int kWarps = 8;
constexpr int kItems = kTH + 2;        // input rows of a piece
constexpr int kSlots = 5;              // kItems % kSlots == 0: slots are compile-time constants
constexpr int kDRow = kTW * kWCo * 2;  // bytes of a staged dy row: [16 pixels][32 co]
constexpr int kXRow = 640;             // of an input row: [18 pixels][16 ci], rounded up to 128 bytes
constexpr int kAcc = 9 * 2 * 2 * 4;    // accumulators per lane
constexpr int kWgradSmem = kWarps * kSlots * (kDRow + kXRow) > 4 * kAcc * 32 * 4 + kWarps * 32 * 4
                               ? kWarps * kSlots * (kDRow + kXRow)
                               : 4 * kAcc * 32 * 4 + kWarps * 32 * 4;

struct WgradArgs {
    const bf16 *x;
    const bf16 *dy;
    float *dw, *db;
    int ldx, lddy, B, H, W, Cin, pieces;
};

__global__ void __launch_bounds__(32 * kWarps, 1) wgrad_kernel(const WgradArgs a) {
    static_assert(kItems % kSlots == 0, "static slots");
    extern __shared__ __align__(128) unsigned char wsm[];
    const int co0 = blockIdx.x * kWCo, ci0 = blockIdx.y * kWCi;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    unsigned char *ring = wsm + warp * kSlots * (kDRow + kXRow);
    auto dslot = [&](int s) { return reinterpret_cast<bf16 *>(ring + s * (kDRow + kXRow)); };
    auto xslot = [&](int s) { return reinterpret_cast<bf16 *>(ring + s * (kDRow + kXRow) + kDRow); };

    // Piece -> image, first row, first column; pieces of one column follow one another.
    const int rows8 = a.H / kTH, strips = a.W / kTW, stride = gridDim.z * kWarps;
    struct Piece {
        const bf16 *x, *dy;  // pixel (y0, x0), this block's first channel
        int y0, x0;
    };
    auto piece_at = [&](int p) {
        Piece r;
        const int col = p / rows8;
        r.y0 = (p - col * rows8) * kTH;
        const int b = col / strips;
        r.x0 = (col - b * strips) * kTW;
        const long long pix = ((long long)b * a.H + r.y0) * a.W + r.x0;
        r.x = a.x + pix * a.ldx + ci0;
        r.dy = a.dy + pix * a.lddy + co0;
        return r;
    };
    // Item i of a piece: input row y0 + i - 1 (18 pixels from x0 - 1, zeros
    // outside the image) and, up to i = 7, output-gradient row y0 + i.
    auto issue = [&](const Piece &r, int i) {
        const int y = r.y0 + i - 1;
        const bool row = y >= 0 && y < a.H;
        bf16 *xs = xslot(i % kSlots);
#pragma unroll
        for (int h = 0; h < 2; h++) {
            const int c = lane + 32 * h;
            if (c < 2 * (kTW + 2)) {
                const int px = c >> 1, half = c & 1, gx = r.x0 + px - 1;
                const bool in = row && gx >= 0 && gx < a.W;
                const bf16 *src = in ? r.x + ((long long)(i - 1) * a.W + px - 1) * a.ldx + half * 8 : a.x;
                cp_async16(xs + sw32(px, half), src, in ? 16 : 0);
            }
        }
        if (i < kTH) {
            bf16 *ds = dslot(i % kSlots);
#pragma unroll
            for (int h = 0; h < 2; h++) {
                const int c = lane + 32 * h, px = c >> 2, ch = c & 3;
                cp_async16(ds + sw64(px, ch), r.dy + ((long long)i * a.W + px) * a.lddy + ch * 8, 16);
            }
        }
    };

    float acc[9][2][2][4];
    float bsum[4] = {0.0f, 0.0f, 0.0f, 0.0f};
#pragma unroll
    for (int t = 0; t < 9; t++)
#pragma unroll
        for (int i = 0; i < 2; i++)
#pragma unroll
            for (int j = 0; j < 2; j++)
#pragma unroll
                for (int k = 0; k < 4; k++) acc[t][i][j][k] = 0.0f;

    const int mi = lane >> 3, lr = lane & 7;
    int p = blockIdx.z * kWarps + warp;
    Piece cur = piece_at(p < a.pieces ? p : 0), nxt = cur;
#pragma unroll
    for (int i = 0; i < kSlots - 1; i++) {
        if (p < a.pieces) issue(cur, i);
        cp_async_commit();
    }
    uint32_t afr[3][2][4];  // output-gradient fragments of the last three rows
    for (; p < a.pieces; p += stride) {
        const bool more = p + stride < a.pieces;
        if (more) nxt = piece_at(p + stride);
        const bool bias = a.db && p % (int)gridDim.y == (int)blockIdx.y;
#pragma unroll
        for (int i = 0; i < kItems; i++) {
            cp_async_wait<kSlots - 2>();  // item i has landed
            __syncwarp();
            if (i < kTH) {
                // A (co x pixel), transposed on load: (px 0..7, co +0..7),
                // (px 0..7, co +8..15), (px 8..15, co +0..7), (px 8..15, co +8..15)
                const bf16 *D = dslot(i % kSlots);
#pragma unroll
                for (int mt = 0; mt < 2; mt++) {
                    uint32_t *f = afr[i % 3][mt];
                    ldsm_x4_t(f[0], f[1], f[2], f[3], D + sw64((mi >> 1) * 8 + lr, mt * 2 + (mi & 1)));
                }
            }
            // B (pixel x ci) at the three horizontal shifts, transposed on load:
            // (px 0..7, ci 0..7), (px 8..15, ci 0..7), (px 0..7, ci 8..15), (px 8..15, ci 8..15)
            const bf16 *X = xslot(i % kSlots);
            uint32_t bfr[3][4];
#pragma unroll
            for (int kx = 0; kx < 3; kx++)
                ldsm_x4_t(bfr[kx][0], bfr[kx][1], bfr[kx][2], bfr[kx][3], X + sw32((mi & 1) * 8 + lr + kx, mi >> 1));
            // the slot read one item ago takes the item four ahead
            const int ahead = i + kSlots - 1;
            if (ahead < kItems) issue(cur, ahead);
            else if (more) issue(nxt, ahead - kItems);
            cp_async_commit();
            if (i < kTH && bias) {
#pragma unroll
                for (int mt = 0; mt < 2; mt++)
#pragma unroll
                    for (int h = 0; h < 2; h++) {
                        const uint32_t q = afr[i % 3][mt][h], r = afr[i % 3][mt][h + 2];
                        bsum[2 * mt + h] += (__uint_as_float(q << 16) + __uint_as_float(q & 0xffff0000u)) +
                                            (__uint_as_float(r << 16) + __uint_as_float(r & 0xffff0000u));
                    }
            }
            // input row y0 + i - 1 meets output rows y0 + i - ky at tap row ky
#pragma unroll
            for (int ky = 0; ky < 3; ky++)
                if (i - ky >= 0 && i - ky < kTH) {
#pragma unroll
                    for (int kx = 0; kx < 3; kx++)
#pragma unroll
                        for (int mt = 0; mt < 2; mt++)
#pragma unroll
                            for (int nt = 0; nt < 2; nt++)
                                mma16816(acc[3 * ky + kx][mt][nt], afr[(i - ky + 3) % 3][mt], bfr[kx] + 2 * nt);
                }
        }
        cur = nxt;
    }
    // Fold the eight warps' sums: the upper four into the lower four, then four
    // areas element by element; one atomic per weight and block.
    cp_async_wait<0>();
    __syncthreads();
    float *red = reinterpret_cast<float *>(wsm);
    float *bred = red + 4 * kAcc * 32;
    auto each = [&](auto f) {
#pragma unroll
        for (int t = 0; t < 9; t++)
#pragma unroll
            for (int i = 0; i < 2; i++)
#pragma unroll
                for (int j = 0; j < 2; j++)
#pragma unroll
                    for (int k = 0; k < 4; k++) f(((t * 2 + i) * 2 + j) * 4 + k, acc[t][i][j][k]);
    };
    float *mine = red + (warp & 3) * kAcc * 32 + lane;
    if (warp >= 4) each([&](int e, float &v) { mine[e * 32] = v; });
    // co = 16 mt + 8 h + lane / 4; the four lanes of a co hold different pixels
#pragma unroll
    for (int k = 0; k < 4; k++) {
        bsum[k] += __shfl_xor_sync(0xffffffffu, bsum[k], 1);
        bsum[k] += __shfl_xor_sync(0xffffffffu, bsum[k], 2);
        if ((lane & 3) == 0) bred[warp * 32 + (k >> 1) * 16 + (k & 1) * 8 + (lane >> 2)] = bsum[k];
    }
    __syncthreads();
    if (warp < 4) each([&](int e, float &v) { mine[e * 32] += v; });
    __syncthreads();
    for (int e = tid; e < kAcc * 32; e += 32 * kWarps) {
        const float v = (red[e] + red[e + kAcc * 32]) + (red[e + 2 * kAcc * 32] + red[e + 3 * kAcc * 32]);
        const int l = e & 31, q = e >> 5, k = q & 3, j = (q >> 2) & 1, i = (q >> 3) & 1, t = q >> 4;
        const int co = co0 + i * 16 + (l >> 2) + (k >> 1) * 8, ci = ci0 + j * 8 + 2 * (l & 3) + (k & 1);
        atomicAdd(a.dw + ((long long)co * 9 + t) * a.Cin + ci, v);
    }
    if (a.db && tid < kWCo) {
        float v = 0.0f;
#pragma unroll
        for (int w = 0; w < kWarps; w++) v += bred[w * 32 + tid];
        atomicAdd(a.db + co0 + tid, v);
    }
}

__global__ void flip_kernel(const bf16 *w, bf16 *wt, int Cin, int Cout) {
    const long long n = (long long)Cout * 9 * Cin;
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
        const int ci = (int)(i % Cin);
        const int tap = (int)((i / Cin) % 9);
        const int co = (int)(i / (9LL * Cin));
        wt[((long long)ci * 9 + (8 - tap)) * Cout + co] = w[i];
    }
}

// ---------------------------------------------------------------------------
// pooling, up-sampling
// ---------------------------------------------------------------------------
__global__ void pool2_kernel(const bf16 *x, int ldx, bf16 *y, int ldy, int B, int H, int W, int C) {
    const int Ho = H / 2, Wo = W / 2;
    const long long n = (long long)B * Ho * Wo * C;
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
        const int c = (int)(i % C);
        const long long p = i / C;
        const int xo = (int)(p % Wo), yo = (int)((p / Wo) % Ho), b = (int)(p / ((long long)Wo * Ho));
        const long long q = ((long long)(b * H + 2 * yo) * W + 2 * xo) * ldx + c;
        const float s = __bfloat162float(x[q]) + __bfloat162float(x[q + ldx]) + __bfloat162float(x[q + (long long)W * ldx]) +
                        __bfloat162float(x[q + (long long)W * ldx + ldx]);
        y[p * ldy + c] = __float2bfloat16_rn(0.25f * s);
    }
}

__global__ void pool2_backward_kernel(const bf16 *dy, int lddy, const bf16 *add, int ldadd, const bf16 *m, int ldm,
                                      bf16 *dx, int lddx, int B, int H, int W, int C) {
    const long long n = (long long)B * H * W * C;
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
        const int c = (int)(i % C);
        const long long p = i / C;
        const int xx = (int)(p % W), yy = (int)((p / W) % H), b = (int)(p / ((long long)W * H));
        float v = 0.25f * __bfloat162float(dy[((long long)(b * (H / 2) + yy / 2) * (W / 2) + xx / 2) * lddy + c]);
        if (add) v += __bfloat162float(add[p * ldadd + c]);
        if (m) v *= dleaky(__bfloat162float(m[p * ldm + c]));
        dx[p * lddx + c] = __float2bfloat16_rn(v);
    }
}

__global__ void upsample2_kernel(const bf16 *x, int ldx, bf16 *y, int ldy, int B, int H, int W, int C) {
    const int Ho = 2 * H, Wo = 2 * W;
    const long long n = (long long)B * Ho * Wo * C;
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
        const int c = (int)(i % C);
        const long long p = i / C;
        const int xo = (int)(p % Wo), yo = (int)((p / Wo) % Ho), b = (int)(p / ((long long)Wo * Ho));
        y[p * ldy + c] = x[((long long)(b * H + yo / 2) * W + xo / 2) * ldx + c];
    }
}

__global__ void upsample2_backward_kernel(const bf16 *dy, int lddy, const bf16 *m, int ldm, bf16 *dx, int lddx, int B,
                                          int H, int W, int C) {
    const long long n = (long long)B * H * W * C;
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
        const int c = (int)(i % C);
        const long long p = i / C;
        const int xx = (int)(p % W), yy = (int)((p / W) % H), b = (int)(p / ((long long)W * H));
        const long long q = ((long long)(b * 2 * H + 2 * yy) * (2 * W) + 2 * xx) * lddy + c;
        const long long row = 2LL * W * lddy;
        float s = __bfloat162float(dy[q]) + __bfloat162float(dy[q + lddy]) + __bfloat162float(dy[q + row]) +
                  __bfloat162float(dy[q + row + lddy]);
        if (m) s *= dleaky(__bfloat162float(m[p * ldm + c]));
        dx[p * lddx + c] = __float2bfloat16_rn(s);
    }
}

// Eight BF16 channels as one 16-byte word.  The kernels above move two bytes
// per thread and spend a 64-bit division per channel; on the network's maps
// (C a multiple of 32, strides and slices 16-byte aligned) a thread takes
// eight channels of a pixel instead: the same arithmetic per element in the
// same order, an eighth of the index arithmetic, 16-byte accesses.  They are
// bound by L2 / DRAM bytes.  Every other form takes the kernels above.
// Measured (ncu, 32 maps of 128^2, the network's three levels summed): pooling
// 53 -> 23 us, its adjoint 167 -> 46, up-sampling 242 -> 24, its adjoint
// 88 -> 35; the input encoding below 48 -> 7.
struct Vec8 {
    uint4 v;
    __device__ __forceinline__ float get(int k) const {
        const uint32_t w = k < 2 ? v.x : (k < 4 ? v.y : (k < 6 ? v.z : v.w));
        return __uint_as_float((k & 1) ? (w & 0xffff0000u) : (w << 16));
    }
    __device__ __forceinline__ void set(const float (&f)[8]) {
        __nv_bfloat162 *o = reinterpret_cast<__nv_bfloat162 *>(&v);
#pragma unroll
        for (int k = 0; k < 4; k++) o[k] = __floats2bfloat162_rn(f[2 * k], f[2 * k + 1]);
    }
};
__device__ __forceinline__ Vec8 ld8(const bf16 *p) { return Vec8{*reinterpret_cast<const uint4 *>(p)}; }
__device__ __forceinline__ void st8(bf16 *p, const Vec8 &v) { *reinterpret_cast<uint4 *>(p) = v.v; }

// Output pixel and first channel of thread i of n = (pixels) * (C / 8).
struct PixelChunk {
    uint32_t x, y, b, p;
    int c;
    __device__ __forceinline__ PixelChunk(uint32_t i, uint32_t C8, uint32_t W, uint32_t H) {
        p = i / C8;
        c = (int)(i - p * C8) * 8;
        const uint32_t r = p / W;
        x = p - r * W;
        b = r / H;
        y = r - b * H;
    }
};

__global__ void __launch_bounds__(256) pool2_vec_kernel(const bf16 *x, int ldx, bf16 *y, int ldy, int H, int W, int C8,
                                                        uint32_t n) {
    const uint32_t i = blockIdx.x * 256u + threadIdx.x;
    if (i >= n) return;
    const PixelChunk o(i, C8, W / 2, H / 2);
    const bf16 *q = x + ((long long)(o.b * H + 2 * o.y) * W + 2 * o.x) * ldx + o.c;
    const Vec8 a = ld8(q), b = ld8(q + ldx), c = ld8(q + (long long)W * ldx), d = ld8(q + (long long)W * ldx + ldx);
    float f[8];
#pragma unroll
    for (int k = 0; k < 8; k++) f[k] = 0.25f * (a.get(k) + b.get(k) + c.get(k) + d.get(k));
    Vec8 r;
    r.set(f);
    st8(y + (long long)o.p * ldy + o.c, r);
}

__global__ void __launch_bounds__(256) pool2_backward_vec_kernel(const bf16 *dy, int lddy, const bf16 *add, int ldadd,
                                                                 const bf16 *m, int ldm, bf16 *dx, int lddx, int H,
                                                                 int W, int C8, uint32_t n) {
    const uint32_t i = blockIdx.x * 256u + threadIdx.x;
    if (i >= n) return;
    const PixelChunk o(i, C8, W, H);
    const Vec8 d = ld8(dy + ((long long)(o.b * (H / 2) + o.y / 2) * (W / 2) + o.x / 2) * lddy + o.c);
    float f[8];
#pragma unroll
    for (int k = 0; k < 8; k++) f[k] = 0.25f * d.get(k);
    if (add) {
        const Vec8 a = ld8(add + (long long)o.p * ldadd + o.c);
#pragma unroll
        for (int k = 0; k < 8; k++) f[k] += a.get(k);
    }
    if (m) {
        const Vec8 a = ld8(m + (long long)o.p * ldm + o.c);
#pragma unroll
        for (int k = 0; k < 8; k++) f[k] *= dleaky(a.get(k));
    }
    Vec8 r;
    r.set(f);
    st8(dx + (long long)o.p * lddx + o.c, r);
}

// One thread per input pixel and chunk: read once, written to its four children.
__global__ void __launch_bounds__(256) upsample2_vec_kernel(const bf16 *x, int ldx, bf16 *y, int ldy, int H, int W,
                                                            int C8, uint32_t n) {
    const uint32_t i = blockIdx.x * 256u + threadIdx.x;
    if (i >= n) return;
    const PixelChunk o(i, C8, W, H);
    const Vec8 v = ld8(x + (long long)o.p * ldx + o.c);
    bf16 *q = y + ((long long)(o.b * 2 * H + 2 * o.y) * (2 * W) + 2 * o.x) * ldy + o.c;
    const long long row = 2LL * W * ldy;
    st8(q, v);
    st8(q + ldy, v);
    st8(q + row, v);
    st8(q + row + ldy, v);
}

__global__ void __launch_bounds__(256) upsample2_backward_vec_kernel(const bf16 *dy, int lddy, const bf16 *m, int ldm,
                                                                     bf16 *dx, int lddx, int H, int W, int C8,
                                                                     uint32_t n) {
    const uint32_t i = blockIdx.x * 256u + threadIdx.x;
    if (i >= n) return;
    const PixelChunk o(i, C8, W, H);
    const bf16 *q = dy + ((long long)(o.b * 2 * H + 2 * o.y) * (2 * W) + 2 * o.x) * lddy + o.c;
    const long long row = 2LL * W * lddy;
    const Vec8 a = ld8(q), b = ld8(q + lddy), c = ld8(q + row), d = ld8(q + row + lddy);
    float f[8];
#pragma unroll
    for (int k = 0; k < 8; k++) f[k] = a.get(k) + b.get(k) + c.get(k) + d.get(k);
    if (m) {
        const Vec8 g = ld8(m + (long long)o.p * ldm + o.c);
#pragma unroll
        for (int k = 0; k < 8; k++) f[k] *= dleaky(g.get(k));
    }
    Vec8 r;
    r.set(f);
    st8(dx + (long long)o.p * lddx + o.c, r);
}

// ---------------------------------------------------------------------------
// output layer (1x1 convolution), loss, optimiser
// ---------------------------------------------------------------------------
constexpr int kMaxCin1 = 64, kMaxCout1 = 8;

__global__ void conv1x1_kernel(const bf16 *x, int ldx, const float *w, const float *bias, float *y, long long P,
                               int Cin, int Cout) {
    __shared__ float ws[kMaxCout1 * kMaxCin1];
    for (int i = threadIdx.x; i < Cin * Cout; i += blockDim.x) ws[i] = w[i];
    __syncthreads();
    for (long long p = blockIdx.x * (long long)blockDim.x + threadIdx.x; p < P; p += (long long)gridDim.x * blockDim.x) {
        float acc[kMaxCout1];
        for (int o = 0; o < Cout; o++) acc[o] = bias[o];
        for (int c = 0; c < Cin; c++) {
            const float xv = __bfloat162float(x[p * ldx + c]);
            for (int o = 0; o < Cout; o++) acc[o] += ws[o * Cin + c] * xv;
        }
        for (int o = 0; o < Cout; o++) y[p * Cout + o] = acc[o];
    }
}

__global__ void conv1x1_dx_kernel(const bf16 *x, int ldx, const float *w, const float *dy, bf16 *dx, int lddx,
                                  long long P, int Cin, int Cout) {
    __shared__ float ws[kMaxCout1 * kMaxCin1];
    for (int i = threadIdx.x; i < Cin * Cout; i += blockDim.x) ws[i] = w[i];
    __syncthreads();
    for (long long p = blockIdx.x * (long long)blockDim.x + threadIdx.x; p < P; p += (long long)gridDim.x * blockDim.x) {
        for (int c = 0; c < Cin; c++) {
            float s = 0.0f;
            for (int o = 0; o < Cout; o++) s += dy[p * Cout + o] * ws[o * Cin + c];
            dx[p * lddx + c] = __float2bfloat16_rn(s * dleaky(__bfloat162float(x[p * ldx + c])));
        }
    }
}

// dw[o][c] += sum_p dy[p][o] x[p][c]; db[o] += sum_p dy[p][o]: thread j owns
// (o, c) = (j / Cin, j % Cin) over the block's share of the pixels.
__global__ void conv1x1_dw_kernel(const bf16 *x, int ldx, const float *dy, float *dw, float *db, long long P, int Cin,
                                  int Cout) {
    const long long per = (P + gridDim.x - 1) / gridDim.x;
    const long long p0 = blockIdx.x * per, p1 = p0 + per < P ? p0 + per : P;
    const int j = threadIdx.x;
    if (j >= Cin * Cout) return;
    const int o = j / Cin, c = j % Cin;
    float s = 0.0f, sb = 0.0f;
    for (long long p = p0; p < p1; p++) {
        const float d = dy[p * Cout + o];
        s += d * __bfloat162float(x[p * ldx + c]);
        sb += d;
    }
    atomicAdd(dw + j, s);
    if (c == 0 && db) atomicAdd(db + o, sb);
}

// The output layer with 16-byte accesses (Cin a multiple of 8, stride and
// pointers 16-byte aligned; every other form takes the kernels above).
// Forward: a thread per pixel, the products summed in channel order as above.
// Backward: dx, dw and db from one pass over x and dy (the split kernels read
// both twice, and a thread of the dw kernel walked 1024 pixels one after the
// other).  Cin / 8 lanes share a pixel, one 8-channel chunk each, so that a
// warp reads whole rows of consecutive pixels; each thread keeps its chunk's
// Cout x 8 sums, a warp folds the lanes of equal chunk by shuffles, a block
// its warps in shared memory, and one thread per weight adds to the gradient.
// Measured (ncu, 524288 pixels, 32 channels, 3 outputs): forward 57 -> 12 us,
// backward 382 (dx 121, dw and db 261) -> 23; the bytes alone take 11.
template <int CO>
__global__ void __launch_bounds__(256) conv1x1_vec_kernel(const bf16 *x, int ldx, const float *w, const float *bias,
                                                          float *y, long long P, int Cin) {
    __shared__ float ws[CO * kMaxCin1];
    for (int i = threadIdx.x; i < Cin * CO; i += 256) ws[i] = w[i];
    __syncthreads();
    for (long long p = blockIdx.x * 256LL + threadIdx.x; p < P; p += gridDim.x * 256LL) {
        float acc[CO];
#pragma unroll
        for (int o = 0; o < CO; o++) acc[o] = bias[o];
        for (int c = 0; c < Cin; c += 8) {
            const Vec8 v = ld8(x + p * ldx + c);
#pragma unroll
            for (int k = 0; k < 8; k++)
#pragma unroll
                for (int o = 0; o < CO; o++) acc[o] += ws[o * Cin + c + k] * v.get(k);
        }
#pragma unroll
        for (int o = 0; o < CO; o++) y[p * CO + o] = acc[o];
    }
}

// DX: dx is wanted.  C8 = Cin / 8 chunks (1, 2, 4 or 8: a divisor of a warp).
template <int CO, int C8, bool DX>
__global__ void __launch_bounds__(256) conv1x1_backward_vec_kernel(const bf16 *x, int ldx, const float *w,
                                                                   const float *dy, bf16 *dx, int lddx, float *dw,
                                                                   float *db, long long P) {
    constexpr int Cin = 8 * C8, PW = 256 / C8;  // pixels per block and pass
    __shared__ float red[8][C8 * CO * 8 + CO];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int ch = tid % C8;
    float wr[CO][8], acc[CO][8], sb[CO];
#pragma unroll
    for (int o = 0; o < CO; o++) {
        sb[o] = 0.0f;
#pragma unroll
        for (int k = 0; k < 8; k++) {
            wr[o][k] = w[o * Cin + ch * 8 + k];
            acc[o][k] = 0.0f;
        }
    }
    for (long long p = blockIdx.x * (long long)PW + tid / C8; p < P; p += gridDim.x * (long long)PW) {
        const Vec8 v = ld8(x + p * ldx + ch * 8);
        float d[CO], f[8];
#pragma unroll
        for (int o = 0; o < CO; o++) {
            d[o] = dy[p * CO + o];
            sb[o] += d[o];
        }
#pragma unroll
        for (int k = 0; k < 8; k++) {
            const float xv = v.get(k);
            float s = 0.0f;
#pragma unroll
            for (int o = 0; o < CO; o++) {
                s += d[o] * wr[o][k];
                acc[o][k] += d[o] * xv;
            }
            f[k] = s * dleaky(xv);
        }
        if (DX) {
            Vec8 r;
            r.set(f);
            st8(dx + p * lddx + ch * 8, r);
        }
    }
    // lanes of equal chunk sit C8 apart
#pragma unroll
    for (int o = 0; o < CO; o++) {
#pragma unroll
        for (int sh = C8; sh < 32; sh <<= 1) {
#pragma unroll
            for (int k = 0; k < 8; k++) acc[o][k] += __shfl_xor_sync(0xffffffffu, acc[o][k], sh);
            sb[o] += __shfl_xor_sync(0xffffffffu, sb[o], sh);
        }
        if (lane < C8)
#pragma unroll
            for (int k = 0; k < 8; k++) red[warp][o * Cin + lane * 8 + k] = acc[o][k];
        if (lane == 0) red[warp][CO * Cin + o] = sb[o];
    }
    __syncthreads();
    for (int j = tid; j < CO * Cin + CO; j += 256) {
        float s = 0.0f;
#pragma unroll
        for (int q = 0; q < 8; q++) s += red[q][j];
        if (j < CO * Cin) atomicAdd(dw + j, s);
        else if (db) atomicAdd(db + j - CO * Cin, s);
    }
}

__global__ void mse_kernel(const float *pred, const float *target, const uint8_t *fluid, long long P, int C,
                           double n_inv, float *dpred, double *loss) {
    __shared__ double red[32];
    double s = 0.0;
    for (long long p = blockIdx.x * (long long)blockDim.x + threadIdx.x; p < P; p += (long long)gridDim.x * blockDim.x) {
        const bool f = fluid[p] != 0;
        for (int c = 0; c < C; c++) {
            const long long i = p * C + c;
            const double d = f ? (double)pred[i] - (double)target[i] : 0.0;
            s += d * d;
            dpred[i] = (float)(2.0 * d * n_inv);
        }
    }
    for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = s;
    __syncthreads();
    if (threadIdx.x == 0) {
        double t = 0.0;
        for (int w = 0; w < (int)(blockDim.x >> 5); w++) t += red[w];
        atomicAdd(loss, t * n_inv);
    }
}

__global__ void adam_kernel(float *p, const float *g, float *m, float *v, bf16 *pb, long long n, float lr, float b1,
                            float b2, float eps, float c1, float c2) {
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
        const float gi = g[i];
        const float mi = b1 * m[i] + (1.0f - b1) * gi;
        const float vi = b2 * v[i] + (1.0f - b2) * gi * gi;
        m[i] = mi;
        v[i] = vi;
        const float pi = p[i] - lr * (mi * c1) / (sqrtf(vi * c2) + eps);
        p[i] = pi;
        if (pb) pb[i] = __float2bfloat16_rn(pi);
    }
}

__global__ void encode_kernel(const uint8_t *mask, const float *scalars, bf16 *x, int B, int H, int W, bool vec) {
    const long long n = (long long)B * H * W;
    for (long long p = blockIdx.x * (long long)blockDim.x + threadIdx.x; p < n; p += (long long)gridDim.x * blockDim.x) {
        const int b = (int)(p / ((long long)H * W));
        const float f[8] = {mask[p] ? 1.0f : 0.0f, scalars[2 * b], scalars[2 * b + 1], 0.0f, 0.0f, 0.0f, 0.0f, 0.0f};
        if (vec) {  // the pixel's 32 bytes as two 16-byte words
            Vec8 v;
            v.set(f);
            st8(x + p * 16, v);
            st8(x + p * 16 + 8, Vec8{make_uint4(0, 0, 0, 0)});
        } else {
            bf16 *o = x + p * 16;
            for (int c = 0; c < 16; c++) o[c] = __float2bfloat16_rn(c < 3 ? f[c] : 0.0f);
        }
    }
}

__global__ void resample_mask_kernel(const uint8_t *mask, int nx, int ny, uint8_t *out, int H, int W) {
    const int n = H * W;
    for (int p = blockIdx.x * blockDim.x + threadIdx.x; p < n; p += gridDim.x * blockDim.x) {
        const int y = p / W, x = p % W;
        int sy = (int)(((double)y + 0.5) * ny / H), sx = (int)(((double)x + 0.5) * nx / W);
        sy = sy < ny ? sy : ny - 1;
        sx = sx < nx ? sx : nx - 1;
        out[p] = mask[(long long)sy * nx + sx];
    }
}

__global__ void resample_fields_kernel(const float *pred, int H, int W, const uint8_t *mask, int nx, int ny, float U0,
                                       float *u, float *v, float *T) {
    const long long n = (long long)nx * ny;
    for (long long k = blockIdx.x * (long long)blockDim.x + threadIdx.x; k < n; k += (long long)gridDim.x * blockDim.x) {
        const int i = (int)(k % nx), j = (int)(k / nx);
        float fx = ((float)i + 0.5f) * W / nx - 0.5f, fy = ((float)j + 0.5f) * H / ny - 0.5f;
        fx = fminf(fmaxf(fx, 0.0f), (float)(W - 1));
        fy = fminf(fmaxf(fy, 0.0f), (float)(H - 1));
        const int x0 = (int)fx, y0 = (int)fy;
        const int x1 = x0 + 1 < W ? x0 + 1 : W - 1, y1 = y0 + 1 < H ? y0 + 1 : H - 1;
        const float ax = fx - x0, ay = fy - y0;
        float out[3];
        for (int c = 0; c < 3; c++) {
            const float a00 = pred[((long long)y0 * W + x0) * 3 + c], a01 = pred[((long long)y0 * W + x1) * 3 + c];
            const float a10 = pred[((long long)y1 * W + x0) * 3 + c], a11 = pred[((long long)y1 * W + x1) * 3 + c];
            out[c] = (1 - ay) * ((1 - ax) * a00 + ax * a01) + ay * ((1 - ax) * a10 + ax * a11);
        }
        const bool still = (mask && mask[k]) || i == 0 || j == 0 || i == nx - 1 || j == ny - 1;
        u[k] = still ? 0.0f : out[0] * U0;
        v[k] = still ? 0.0f : out[1] * U0;
        T[k] = fminf(fmaxf(out[2], 0.0f), 1.0f);
    }
}

int grid_for(long long n, int block = 256) {
    long long g = (n + block - 1) / block;
    return (int)(g < 4096 ? (g > 0 ? g : 1) : 4096);
}

bool aligned16(const void *p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }

// Whether a channel slice can be read and written in 16-byte words (a NULL
// one is not touched).
bool words16(const void *p, int ld) { return !p || (aligned16(p) && ld % 8 == 0); }
// Threads of a vector launch over `pixels` pixels of C channels, one per eight
// channels; 0 where the counts do not fit the kernels' 32-bit indices or the
// channels do not come in eights.
uint32_t vec_threads(long long pixels, int C) {
    if (C % 8 || pixels * (C / 8) > (1LL << 31)) return 0;
    return (uint32_t)(pixels * (C / 8));
}
unsigned vec_blocks(uint32_t n) { return (n + 255u) / 256u; }

}  // namespace

extern "C" {

const char *lbmfvm_sg_last_error(void) { return g_sg_err; }

int lbmfvm_sg_conv3x3(const uint16_t *x, int32_t ldx, const uint16_t *w, const float *bias, uint16_t *y, int32_t ldy,
                      const uint16_t *m, int32_t ldm, int32_t B, int32_t H, int32_t W, int32_t Cin, int32_t Cout,
                      int32_t mode, void *stream) {
    if (!x || !w || !y || (mode == LBMFVM_SG_DLEAKY && !m)) return sg_fail(kErrArg, "conv3x3: NULL tensor");
    if (mode < LBMFVM_SG_LINEAR || mode > LBMFVM_SG_DLEAKY) return sg_fail(kErrArg, "conv3x3: mode %d", mode);
    if (B < 1 || H < 8 || W < 16 || H % 8 || W % 16 || Cin < 16 || Cin % 16 || Cout < 32 || Cout % 32)
        return sg_fail(kErrArg, "conv3x3: shape B=%d H=%d W=%d Cin=%d Cout=%d breaks the tile rules", B, H, W, Cin,
                       Cout);
    if (ldx < Cin || ldy < Cout || ldx % 8 || ldy % 8 || (m && (ldm < Cout || ldm % 8)) || !aligned16(x) ||
        !aligned16(w) || !aligned16(y) || (m && !aligned16(m)))
        return sg_fail(kErrArg, "conv3x3: strides or alignment");
    return lbmfvm_sg_tc::conv3x3(x, ldx, w, bias, y, ldy, m, ldm, B, H, W, Cin, Cout, mode, (cudaStream_t)stream,
                                 g_sg_err, sizeof(g_sg_err));
}

int lbmfvm_sg_inject_stall(void) {
    lbmfvm_sg_tc::inject_stall();
    return kOk;
}

int lbmfvm_sg_check(void *stream) {
    const int r = lbmfvm_sg_tc::check((cudaStream_t)stream);
    if (r == -4) return sg_fail(-4, "a bounded wait of the tensor-core convolution ran out");
    if (r) return sg_fail(kErrCuda, "status check failed");
    return kOk;
}

int lbmfvm_sg_flip(const uint16_t *w, uint16_t *wt, int32_t Cin, int32_t Cout, void *stream) {
    if (!w || !wt || Cin < 1 || Cout < 1) return sg_fail(kErrArg, "flip: arguments");
    flip_kernel<<<grid_for(9LL * Cin * Cout), 256, 0, (cudaStream_t)stream>>>(
        reinterpret_cast<const bf16 *>(w), reinterpret_cast<bf16 *>(wt), Cin, Cout);
    return launched("flip");
}

int lbmfvm_sg_conv3x3_wgrad(const uint16_t *x, int32_t ldx, const uint16_t *dy, int32_t lddy, float *dw, float *db,
                            int32_t B, int32_t H, int32_t W, int32_t Cin, int32_t Cout, void *stream) {
    if (!x || !dy || !dw) return sg_fail(kErrArg, "wgrad: NULL tensor");
    if (B < 1 || H < 8 || W < 16 || H % 8 || W % 16 || Cin < 16 || Cin % 16 || Cout < 32 || Cout % 32)
        return sg_fail(kErrArg, "wgrad: shape B=%d H=%d W=%d Cin=%d Cout=%d breaks the tile rules", B, H, W, Cin, Cout);
    if (ldx < Cin || lddy < Cout || ldx % 8 || lddy % 8 || !aligned16(x) || !aligned16(dy))
        return sg_fail(kErrArg, "wgrad: strides or alignment");
    const int pieces = B * (H / kTH) * (W / kTW);
    const int gx = Cout / kWCo, gy = Cin / kWCi;
    // one block per SM (the accumulators fill its registers), fewer where the
    // pieces would not give every warp one
    int split = 152 / (gx * gy);
    if (split < 1) split = 1;
    if (split > (pieces + kWarps - 1) / kWarps) split = (pieces + kWarps - 1) / kWarps;
    WgradArgs a{reinterpret_cast<const bf16 *>(x), reinterpret_cast<const bf16 *>(dy), dw, db, ldx, lddy, B, H, W, Cin,
                pieces};
    const cudaError_t e = cudaFuncSetAttribute(wgrad_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kWgradSmem);
    if (e != cudaSuccess) return sg_fail(kErrCuda, "wgrad: %s", cudaGetErrorString(e));
    wgrad_kernel<<<dim3(gx, gy, split), 32 * kWarps, kWgradSmem, (cudaStream_t)stream>>>(a);
    return launched("wgrad");
}

int lbmfvm_sg_pool2(const uint16_t *x, int32_t ldx, uint16_t *y, int32_t ldy, int32_t B, int32_t H, int32_t W,
                    int32_t C, void *stream) {
    if (!x || !y || B < 1 || H < 2 || W < 2 || H % 2 || W % 2 || C < 1 || ldx < C || ldy < C)
        return sg_fail(kErrArg, "pool2: arguments");
    const uint32_t n8 = vec_threads((long long)B * (H / 2) * (W / 2), C);
    if (n8 && words16(x, ldx) && words16(y, ldy)) {
        pool2_vec_kernel<<<vec_blocks(n8), 256, 0, (cudaStream_t)stream>>>(
            reinterpret_cast<const bf16 *>(x), ldx, reinterpret_cast<bf16 *>(y), ldy, H, W, C / 8, n8);
        return launched("pool2");
    }
    pool2_kernel<<<grid_for((long long)B * H * W * C / 4), 256, 0, (cudaStream_t)stream>>>(
        reinterpret_cast<const bf16 *>(x), ldx, reinterpret_cast<bf16 *>(y), ldy, B, H, W, C);
    return launched("pool2");
}

int lbmfvm_sg_pool2_backward(const uint16_t *dy, int32_t lddy, const uint16_t *add, int32_t ldadd, const uint16_t *m,
                             int32_t ldm, uint16_t *dx, int32_t lddx, int32_t B, int32_t H, int32_t W, int32_t C,
                             void *stream) {
    if (!dy || !dx || B < 1 || H < 2 || W < 2 || H % 2 || W % 2 || C < 1 || lddy < C || lddx < C ||
        (add && ldadd < C) || (m && ldm < C))
        return sg_fail(kErrArg, "pool2_backward: arguments");
    const uint32_t n8 = vec_threads((long long)B * H * W, C);
    if (n8 && words16(dy, lddy) && words16(add, ldadd) && words16(m, ldm) && words16(dx, lddx)) {
        pool2_backward_vec_kernel<<<vec_blocks(n8), 256, 0, (cudaStream_t)stream>>>(
            reinterpret_cast<const bf16 *>(dy), lddy, reinterpret_cast<const bf16 *>(add), ldadd,
            reinterpret_cast<const bf16 *>(m), ldm, reinterpret_cast<bf16 *>(dx), lddx, H, W, C / 8, n8);
        return launched("pool2_backward");
    }
    pool2_backward_kernel<<<grid_for((long long)B * H * W * C), 256, 0, (cudaStream_t)stream>>>(
        reinterpret_cast<const bf16 *>(dy), lddy, reinterpret_cast<const bf16 *>(add), ldadd,
        reinterpret_cast<const bf16 *>(m), ldm, reinterpret_cast<bf16 *>(dx), lddx, B, H, W, C);
    return launched("pool2_backward");
}

int lbmfvm_sg_upsample2(const uint16_t *x, int32_t ldx, uint16_t *y, int32_t ldy, int32_t B, int32_t H, int32_t W,
                        int32_t C, void *stream) {
    if (!x || !y || B < 1 || H < 1 || W < 1 || C < 1 || ldx < C || ldy < C) return sg_fail(kErrArg, "upsample2: arguments");
    const uint32_t n8 = vec_threads((long long)B * H * W, C);
    if (n8 && words16(x, ldx) && words16(y, ldy)) {
        upsample2_vec_kernel<<<vec_blocks(n8), 256, 0, (cudaStream_t)stream>>>(
            reinterpret_cast<const bf16 *>(x), ldx, reinterpret_cast<bf16 *>(y), ldy, H, W, C / 8, n8);
        return launched("upsample2");
    }
    upsample2_kernel<<<grid_for(4LL * B * H * W * C), 256, 0, (cudaStream_t)stream>>>(
        reinterpret_cast<const bf16 *>(x), ldx, reinterpret_cast<bf16 *>(y), ldy, B, H, W, C);
    return launched("upsample2");
}

int lbmfvm_sg_upsample2_backward(const uint16_t *dy, int32_t lddy, const uint16_t *m, int32_t ldm, uint16_t *dx,
                                 int32_t lddx, int32_t B, int32_t H, int32_t W, int32_t C, void *stream) {
    if (!dy || !dx || B < 1 || H < 1 || W < 1 || C < 1 || lddy < C || lddx < C || (m && ldm < C))
        return sg_fail(kErrArg, "upsample2_backward: arguments");
    const uint32_t n8 = vec_threads((long long)B * H * W, C);
    if (n8 && words16(dy, lddy) && words16(m, ldm) && words16(dx, lddx)) {
        upsample2_backward_vec_kernel<<<vec_blocks(n8), 256, 0, (cudaStream_t)stream>>>(
            reinterpret_cast<const bf16 *>(dy), lddy, reinterpret_cast<const bf16 *>(m), ldm,
            reinterpret_cast<bf16 *>(dx), lddx, H, W, C / 8, n8);
        return launched("upsample2_backward");
    }
    upsample2_backward_kernel<<<grid_for((long long)B * H * W * C), 256, 0, (cudaStream_t)stream>>>(
        reinterpret_cast<const bf16 *>(dy), lddy, reinterpret_cast<const bf16 *>(m), ldm, reinterpret_cast<bf16 *>(dx),
        lddx, B, H, W, C);
    return launched("upsample2_backward");
}

int lbmfvm_sg_conv1x1(const uint16_t *x, int32_t ldx, const float *w, const float *b, float *y, int64_t P,
                      int32_t Cin, int32_t Cout, void *stream) {
    if (!x || !w || !b || !y || P < 1 || Cin < 1 || Cin > kMaxCin1 || Cout < 1 || Cout > kMaxCout1 || ldx < Cin)
        return sg_fail(kErrArg, "conv1x1: arguments");
    // three outputs (the network's u, v, T) from a 16-byte aligned slice
    if (Cout == 3 && Cin % 8 == 0 && words16(x, ldx)) {
        conv1x1_vec_kernel<3><<<grid_for(P), 256, 0, (cudaStream_t)stream>>>(reinterpret_cast<const bf16 *>(x), ldx, w,
                                                                             b, y, P, Cin);
        return launched("conv1x1");
    }
    conv1x1_kernel<<<grid_for(P), 256, 0, (cudaStream_t)stream>>>(reinterpret_cast<const bf16 *>(x), ldx, w, b, y, P,
                                                                   Cin, Cout);
    return launched("conv1x1");
}

int lbmfvm_sg_conv1x1_backward(const uint16_t *x, int32_t ldx, const float *w, const float *dy, uint16_t *dx,
                               int32_t lddx, float *dw, float *db, int64_t P, int32_t Cin, int32_t Cout,
                               void *stream) {
    if (!x || !w || !dy || !dw || P < 1 || Cin < 1 || Cin > kMaxCin1 || Cout < 1 || Cout > kMaxCout1 || ldx < Cin ||
        (dx && lddx < Cin) || Cin * Cout > 1024)
        return sg_fail(kErrArg, "conv1x1_backward: arguments");
    cudaStream_t s = (cudaStream_t)stream;
    // three outputs and 32 or 64 channels in 16-byte aligned slices: one pass
    if (Cout == 3 && (Cin == 32 || Cin == 64) && words16(x, ldx) && words16(dx, lddx)) {
        const bf16 *xb = reinterpret_cast<const bf16 *>(x);
        bf16 *dxb = reinterpret_cast<bf16 *>(dx);
        const long long passes = (P + 256 / (Cin / 8) - 1) / (256 / (Cin / 8));
        const int blocks = (int)(passes < 4 * 152 ? passes : 4 * 152);
        if (Cin == 32 && dx) conv1x1_backward_vec_kernel<3, 4, true><<<blocks, 256, 0, s>>>(xb, ldx, w, dy, dxb, lddx, dw, db, P);
        else if (Cin == 32) conv1x1_backward_vec_kernel<3, 4, false><<<blocks, 256, 0, s>>>(xb, ldx, w, dy, dxb, lddx, dw, db, P);
        else if (dx) conv1x1_backward_vec_kernel<3, 8, true><<<blocks, 256, 0, s>>>(xb, ldx, w, dy, dxb, lddx, dw, db, P);
        else conv1x1_backward_vec_kernel<3, 8, false><<<blocks, 256, 0, s>>>(xb, ldx, w, dy, dxb, lddx, dw, db, P);
        return launched("conv1x1 backward");
    }
    if (dx) {
        conv1x1_dx_kernel<<<grid_for(P), 256, 0, s>>>(reinterpret_cast<const bf16 *>(x), ldx, w, dy,
                                                      reinterpret_cast<bf16 *>(dx), lddx, P, Cin, Cout);
        if (int r = launched("conv1x1 dx")) return r;
    }
    const int threads = (Cin * Cout + 31) / 32 * 32;
    const int blocks = (int)((P + 1023) / 1024 < 1024 ? (P + 1023) / 1024 : 1024);
    conv1x1_dw_kernel<<<blocks, threads, 0, s>>>(reinterpret_cast<const bf16 *>(x), ldx, dy, dw, db, P, Cin, Cout);
    return launched("conv1x1 dw");
}

int lbmfvm_sg_mse(const float *pred, const float *target, const uint8_t *fluid, int64_t P, int32_t C, double n_inv,
                  float *dpred, double *loss, void *stream) {
    if (!pred || !target || !fluid || !dpred || !loss || P < 1 || C < 1) return sg_fail(kErrArg, "mse: arguments");
    mse_kernel<<<grid_for(P) < 1024 ? grid_for(P) : 1024, 256, 0, (cudaStream_t)stream>>>(pred, target, fluid, P, C,
                                                                                         n_inv, dpred, loss);
    return launched("mse");
}

int lbmfvm_sg_adam(float *p, const float *g, float *m, float *v, uint16_t *p_bf16, int64_t n, float lr, float beta1,
                   float beta2, float eps, int32_t t, void *stream) {
    if (!p || !g || !m || !v || n < 1 || t < 1) return sg_fail(kErrArg, "adam: arguments");
    const float c1 = 1.0f / (1.0f - powf(beta1, (float)t)), c2 = 1.0f / (1.0f - powf(beta2, (float)t));
    adam_kernel<<<grid_for(n), 256, 0, (cudaStream_t)stream>>>(p, g, m, v, reinterpret_cast<bf16 *>(p_bf16), n, lr,
                                                                beta1, beta2, eps, c1, c2);
    return launched("adam");
}

int lbmfvm_sg_encode(const uint8_t *mask, const float *scalars, uint16_t *x, int32_t B, int32_t H, int32_t W,
                     void *stream) {
    if (!mask || !scalars || !x || B < 1 || H < 1 || W < 1) return sg_fail(kErrArg, "encode: arguments");
    encode_kernel<<<grid_for((long long)B * H * W), 256, 0, (cudaStream_t)stream>>>(
        mask, scalars, reinterpret_cast<bf16 *>(x), B, H, W, aligned16(x));
    return launched("encode");
}

int lbmfvm_sg_resample_mask(const uint8_t *mask, int32_t nx, int32_t ny, uint8_t *out, int32_t H, int32_t W,
                            void *stream) {
    if (!mask || !out || nx < 1 || ny < 1 || H < 1 || W < 1) return sg_fail(kErrArg, "resample_mask: arguments");
    resample_mask_kernel<<<grid_for((long long)H * W), 256, 0, (cudaStream_t)stream>>>(mask, nx, ny, out, H, W);
    return launched("resample_mask");
}

int lbmfvm_sg_resample_fields(const float *pred, int32_t H, int32_t W, const uint8_t *mask, int32_t nx, int32_t ny,
                              float U0, float *u, float *v, float *T, void *stream) {
    if (!pred || !u || !v || !T || H < 1 || W < 1 || nx < 1 || ny < 1) return sg_fail(kErrArg, "resample_fields: arguments");
    resample_fields_kernel<<<grid_for((long long)nx * ny), 256, 0, (cudaStream_t)stream>>>(pred, H, W, mask, nx, ny,
                                                                                            U0, u, v, T);
    return launched("resample_fields");
}

}  // extern "C"
