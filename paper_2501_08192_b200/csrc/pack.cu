// Weight packing, run once at layer creation.  Sources are the caller's
// [in, out] row-major matrices; destinations are laid out so that the GEMM
// kernels stream them in address order with perfectly coalesced loads.
//
// GEMV path ("fragment-major"): the matrix is cut into tiles of 16 output rows
// x 32 k; tile (rb, kc) occupies 1 KiB at ((rb * K/32) + kc) * 1024.  Inside a
// tile lane L = 4g + t owns 32 contiguous bytes: 16 B of row g (k = 8t..8t+7)
// then 16 B of row g + 8 (same k), which is exactly the A-operand fragment of two
// m16n8k16 MMAs (up to a permutation of k shared with the activations).
//
// Tensor path: the tcgen05 A operand's 128-row x 64-k tiles, each 16 KiB in one piece and already in the 128-byte
// swizzle of shared memory: tile (row tile, k block) at ((row tile) * K/64 + k block) * 16384, row r at r * 128,
// its eight 16-byte groups in the order q ^ (r % 8).  A CTA's stream of k blocks is one contiguous run,
// fetched by plain bulk copies.
#include <cuda_fp16.h>

#include "epilogue.cuh"

namespace prsv {

struct PackParams {
    const bf16 *src[3];
    int cols[3];
    int n_srcs;
    int N, K, kind;
    bf16 *dst;
};

__global__ void k_pack_gemv(const __grid_constant__ PackParams p)
{
    // one thread per (k, packed row); packed rows fastest so source reads coalesce
    const size_t idx = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    const size_t total = (size_t)p.N * p.K;
    if (idx >= total)
        return;
    const int row = (int)(idx % p.N);
    const int k = (int)(idx / p.N);
    int src, col;
    packed_row_source(p.kind, false, row, p.cols, src, col);
    const bf16 v = p.src[src][(size_t)k * p.cols[src] + col];
    const int rb = row >> 4, r = row & 15, g = r & 7, hi = r >> 3;
    const int kc = k >> 5, t = (k & 31) >> 3, e = k & 7;
    p.dst[((size_t)rb * (p.K >> 5) + kc) * 512 + (size_t)(g * 4 + t) * 16 + hi * 8 + e] = v;
}

// One CTA per tile of 128 packed rows x 64 k: read along the source rows, turned in shared memory, written in one piece.
// (Written element by element the tiles of four 70B-shaped TP=8 layers took 115 ms to prepare, as rows 70 ms.)
constexpr int kPackPitch = 129;      // elements per k row in shared memory: odd, so that neither side has bank conflicts
__global__ void __launch_bounds__(256) k_pack_tiles(const __grid_constant__ PackParams p)
{
    __shared__ uint16_t tile[64 * kPackPitch];
    const int row0 = blockIdx.y * 128, k0 = blockIdx.x * 64;
    const int row = threadIdx.x & 127;
    int src, col;
    packed_row_source(p.kind, true, row0 + row, p.cols, src, col);
    const bf16 *from = p.src[src] + (size_t)k0 * p.cols[src] + col;
#pragma unroll 8
    for (int k = threadIdx.x >> 7; k < 64; k += 2) {
        // Both operands of a tcgen05 kind::f16 MMA must have the same 16-bit format, and the activations are fp16
        // planes, so the weights are stored as fp16: exact for every bf16 weight of magnitude
        // 2^-17 .. 65504 (fp16 has the longer mantissa); smaller ones round to a multiple of 2^-24 (error
        // <= 2^-25, far below one bf16 ulp of any output), larger ones saturate
        const bf16 v = from[(size_t)k * p.cols[src]];
        tile[k * kPackPitch + row] = __half_as_ushort(__float2half_rn(fminf(fmaxf(__bfloat162float(v), -65504.f), 65504.f)));
    }
    __syncthreads();
    uint4 *dst = reinterpret_cast<uint4 *>(p.dst) + ((size_t)blockIdx.y * (p.K >> 6) + blockIdx.x) * 1024;
    for (int i = threadIdx.x; i < 1024; i += 256) {
        const int r = i >> 3, q = (i & 7) ^ (r & 7);      // the row's group q lies at q ^ (r % 8)
        uint16_t e[8];
#pragma unroll
        for (int j = 0; j < 8; ++j)
            e[j] = tile[(q * 8 + j) * kPackPitch + r];
        dst[i] = make_uint4(e[0] | (uint32_t)e[1] << 16, e[2] | (uint32_t)e[3] << 16, e[4] | (uint32_t)e[5] << 16, e[6] | (uint32_t)e[7] << 16);
    }
}

static cudaError_t launch_pack(bool tensor, const void *const *srcs, const int *src_cols, int n_srcs, int K,
                               int kind, void *dst, cudaStream_t s)
{
    PackParams p = {};
    int N = 0;
    for (int i = 0; i < n_srcs; ++i) {
        p.src[i] = reinterpret_cast<const bf16 *>(srcs[i]);
        p.cols[i] = src_cols[i];
        N += src_cols[i];
    }
    p.n_srcs = n_srcs;
    p.N = N;
    p.K = K;
    p.kind = kind;
    p.dst = reinterpret_cast<bf16 *>(dst);
    if (tensor) {
        if (N % 128 || K % 64)
            return cudaErrorInvalidValue;
        k_pack_tiles<<<dim3(K / 64, N / 128), 256, 0, s>>>(p);
    } else {
        const size_t total = (size_t)N * K;
        k_pack_gemv<<<(unsigned)((total + 255) / 256), 256, 0, s>>>(p);
    }
    return cudaGetLastError();
}

// ---- int8 weights (GEMV path: fragment-major tiles; tensor path: contiguous blocks of codes, see launch_pack_tiles_w8)
struct PackW8Params {
    const bf16 *src[3];
    int cols[3];
    int N, K, kind;
    int tensor;       // tensor-path row order and layout: 128-row tiles per block (1 or 2), 0 = GEMV path
    int8_t *codes;
    float *scales;
};

// scale of every packed row: max |w| over the row's source column, divided by 127 (fp32)
__global__ void k_w8_scales(const __grid_constant__ PackW8Params p)
{
    const int row = blockIdx.x * blockDim.x + threadIdx.x;
    if (row >= p.N)
        return;
    int src, col;
    packed_row_source(p.kind, p.tensor != 0, row, p.cols, src, col);
    float mx = 0.f;
    for (int k = 0; k < p.K; ++k)
        mx = fmaxf(mx, fabsf(__bfloat162float(p.src[src][(size_t)k * p.cols[src] + col])));
    p.scales[row] = __fdiv_rn(mx, 127.0f);
}

__global__ void k_pack_w8(const __grid_constant__ PackW8Params p)
{
    const size_t idx = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    const size_t total = (size_t)p.N * p.K;
    if (idx >= total)
        return;
    const int row = (int)(idx % p.N);
    const int k = (int)(idx / p.N);
    int src, col;
    packed_row_source(p.kind, p.tensor != 0, row, p.cols, src, col);
    const float v = __bfloat162float(p.src[src][(size_t)k * p.cols[src] + col]);
    const float sc = p.scales[row];
    // the code is decided in fp32: one correctly rounded division, round to nearest even, clamp
    float r = sc > 0.f ? rintf(__fdiv_rn(v, sc)) : 0.f;
    r = fminf(fmaxf(r, -127.f), 127.f);
    size_t o;
    if (p.tensor) {
        // the tensor path keeps the codes biased by 128 (unsigned bytes): its widening stage then needs
        // no sign handling
        const int block_rows = p.tensor * 128;
        const size_t block = (size_t)(row / block_rows) * (p.K >> 7) + (k >> 7);
        // (the eight 16-byte groups of a row's 128 k are stored in the order q ^ (row % 8): the widening
        // warps read one group per lane, 32 consecutive rows at a time, without bank conflicts)
        const int rr = row % block_rows, kk = k & 127;
        const int grp = (kk >> 4) ^ (rr & 7);
        p.codes[(block * block_rows + rr) * 128 + grp * 16 + (kk & 15)] = (int8_t)(uint8_t)((int)r + 128);
        return;
    } else {
        const int rb = row >> 4, rr = row & 15, g = rr & 7, hi = rr >> 3;
        const int kc = k >> 6, t = (k & 63) >> 4, e = k & 15;
        o = ((size_t)rb * (p.K >> 6) + kc) * 1024 + (size_t)(g * 4 + t) * 32 + hi * 16 + e;
    }
    p.codes[o] = (int8_t)(int)r;
}

static cudaError_t launch_pack_w8(int tensor, const void *const *srcs, const int *src_cols, int n_srcs, int K, int kind,
                                  void *dst_codes, float *dst_scales, cudaStream_t s)
{
    if (K % 64)
        return cudaErrorInvalidValue;
    PackW8Params p = {};
    int N = 0;
    for (int i = 0; i < n_srcs; ++i) {
        p.src[i] = reinterpret_cast<const bf16 *>(srcs[i]);
        p.cols[i] = src_cols[i];
        N += src_cols[i];
    }
    p.N = N; p.K = K; p.kind = kind;
    p.tensor = tensor;
    p.codes = reinterpret_cast<int8_t *>(dst_codes);
    p.scales = dst_scales;
    k_w8_scales<<<(N + 127) / 128, 128, 0, s>>>(p);
    const size_t total = (size_t)N * K;
    k_pack_w8<<<(unsigned)((total + 255) / 256), 256, 0, s>>>(p);
    return cudaGetLastError();
}

cudaError_t launch_pack_gemv_w8(const void *const *srcs, const int *src_cols, int n_srcs, int K, int kind,
                                void *dst_codes, float *dst_scales, cudaStream_t s)
{
    return launch_pack_w8(0, srcs, src_cols, n_srcs, K, kind, dst_codes, dst_scales, s);
}
cudaError_t launch_pack_tiles_w8(const void *const *srcs, const int *src_cols, int n_srcs, int K, int kind,
                                 void *dst_codes, float *dst_scales, int tiles, cudaStream_t s)
{
    if ((tiles != 1 && tiles != 2) || K % 128)
        return cudaErrorInvalidValue;
    return launch_pack_w8(tiles, srcs, src_cols, n_srcs, K, kind, dst_codes, dst_scales, s);
}

cudaError_t launch_pack_gemv(const void *const *srcs, const int *src_cols, int n_srcs, int K, int kind, void *dst,
                             cudaStream_t s)
{
    return launch_pack(false, srcs, src_cols, n_srcs, K, kind, dst, s);
}
cudaError_t launch_pack_tiles(const void *const *srcs, const int *src_cols, int n_srcs, int K, int kind, void *dst,
                              cudaStream_t s)
{
    return launch_pack(true, srcs, src_cols, n_srcs, K, kind, dst, s);
}

}  // namespace prsv
