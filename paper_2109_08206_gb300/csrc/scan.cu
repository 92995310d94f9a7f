// Exclusive prefix sums of int32 counts (CSR row pointers, cell starts), one
// array or two of the same length at once (grid.y), and the zeroing of count
// arrays.  Small steps are bound by their launches (about 3 us each, most of
// it the launch), so each of these is one where it can be.
// Up to kScanSmall entries one block scans an array tile after tile (1.6e4
// entries: 4 us; two launches 6 to 9).  More: per-tile totals, then per-tile
// scans, each block adding the totals of the tiles before it (a few thousand at
// most) for its offset.  Integer sums: exact and deterministic.
#include "internal.cuh"

namespace alens {

constexpr int kScanThreads = 512;
constexpr int kScanItems = 8;                       // per thread
constexpr int kScanTile = kScanThreads * kScanItems;

__device__ __forceinline__ int block_exclusive_scan(int v, int* smem, int& total)
{
    // warp inclusive scan
    int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int x = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        int y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) smem[warp] = x;
    __syncthreads();
    if (warp == 0) {
        int nw = blockDim.x >> 5;
        int w = lane < nw ? smem[lane] : 0;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            int y = __shfl_up_sync(0xffffffffu, w, o);
            if (lane >= o) w += y;
        }
        smem[32 + lane] = w;   // inclusive warp totals
    }
    __syncthreads();
    total = smem[32 + ((blockDim.x >> 5) - 1)];
    int before = warp > 0 ? smem[32 + warp - 1] : 0;
    int r = before + x - v;
    __syncthreads();
    return r;
}

constexpr int kScanSmall = 4 * kScanTile;

struct ScanArrays {
    const int* in[2];
    int* out[2];
};

__global__ void __launch_bounds__(kScanThreads) k_scan_small(ScanArrays s, int n)
{
    __shared__ int smem[64];
    const int* __restrict__ in = s.in[blockIdx.x];
    int* __restrict__ out = s.out[blockIdx.x];
    int before = 0;
    for (int t = 0; t < n; t += kScanTile) {
        const int base = t + (int)threadIdx.x * kScanItems;
        int v[kScanItems], acc = 0;
#pragma unroll
        for (int k = 0; k < kScanItems; ++k) {
            v[k] = base + k < n ? in[base + k] : 0;
            acc += v[k];
        }
        int total;
        int ex = block_exclusive_scan(acc, smem, total) + before;
#pragma unroll
        for (int k = 0; k < kScanItems; ++k) {
            if (base + k < n) out[base + k] = ex;
            ex += v[k];
        }
        before += total;
    }
    if (threadIdx.x == 0) out[n] = before;
}

// sums: [arrays][gridDim.x] tile totals
__global__ void k_tile_sums(ScanArrays s, int n, int* __restrict__ sums)
{
    __shared__ int smem[64];
    const int* __restrict__ in = s.in[blockIdx.y];
    long long base = (long long)blockIdx.x * kScanTile;
    int acc = 0;
    for (int k = 0; k < kScanItems; ++k) {
        long long idx = base + (long long)k * kScanThreads + threadIdx.x;
        if (idx < n) acc += in[idx];
    }
    int total;
    block_exclusive_scan(acc, smem, total);
    if (threadIdx.x == 0) sums[blockIdx.y * gridDim.x + blockIdx.x] = total;
}

__global__ void k_tile_scan(ScanArrays s, int n, const int* __restrict__ sums)
{
    __shared__ int smem[64];
    __shared__ int pre;
    const int* __restrict__ in = s.in[blockIdx.y];
    int* __restrict__ out = s.out[blockIdx.y];
    if (threadIdx.x < 32) {   // this tile's offset: the totals of the tiles before it
        int a = 0;
        for (int t = threadIdx.x; t < (int)blockIdx.x; t += 32) a += sums[blockIdx.y * gridDim.x + t];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) a += __shfl_xor_sync(0xffffffffu, a, o);
        if (threadIdx.x == 0) pre = a;
    }
    __syncthreads();
    long long base = (long long)blockIdx.x * kScanTile + (long long)threadIdx.x * kScanItems;
    int v[kScanItems];
    int acc = 0;
    for (int k = 0; k < kScanItems; ++k) {
        long long idx = base + k;
        v[k] = idx < n ? in[idx] : 0;
        acc += v[k];
    }
    int total;
    int ex = block_exclusive_scan(acc, smem, total) + pre;
    for (int k = 0; k < kScanItems; ++k) {
        long long idx = base + k;
        if (idx < n) out[idx] = ex;
        ex += v[k];
    }
    if (blockIdx.x == gridDim.x - 1 && threadIdx.x == 0) out[n] = pre + total;
}

// k_tile_sums sums a tile in strided order and k_tile_scan scans it in
// blocked order; both cover the same kScanTile elements, so the tile totals agree.
static cudaError_t scan_arrays(aLENS_ctx* ctx, const ScanArrays& s, int arrays, int n)
{
    if (n <= kScanSmall) {
        k_scan_small<<<arrays, kScanThreads, 0, ctx->stream>>>(s, n);
        ++ctx->launches;
        return cudaGetLastError();
    }
    const int ntiles = (n + kScanTile - 1) / kScanTile;
    if (arrays * ntiles > ctx->scan_tmp_len) return cudaErrorInvalidValue;
    k_tile_sums<<<dim3(ntiles, arrays), kScanThreads, 0, ctx->stream>>>(s, n, ctx->scan_tmp);
    ++ctx->launches;
    k_tile_scan<<<dim3(ntiles, arrays), kScanThreads, 0, ctx->stream>>>(s, n, ctx->scan_tmp);
    ++ctx->launches;
    return cudaGetLastError();
}

cudaError_t exclusive_scan(aLENS_ctx* ctx, const int* counts, int* out, int n)
{
    return scan_arrays(ctx, ScanArrays{{counts, nullptr}, {out, nullptr}}, 1, n);
}

cudaError_t exclusive_scan2(aLENS_ctx* ctx, const int* counts0, int* out0, const int* counts1, int* out1, int n)
{
    return scan_arrays(ctx, ScanArrays{{counts0, counts1}, {out0, out1}}, 2, n);
}

struct ZeroArrays {
    int* p[4];
    int n[4];
};

__global__ void k_zero_ints(ZeroArrays z)
{
    int* const p = z.p[blockIdx.y];
    for (int k = blockIdx.x * blockDim.x + threadIdx.x; k < z.n[blockIdx.y]; k += gridDim.x * blockDim.x) p[k] = 0;
}

cudaError_t zero_ints(aLENS_ctx* ctx, int arrays, int* const* p, const int* n)
{
    ZeroArrays z = {};
    int most = 1;
    for (int k = 0; k < arrays; ++k) {
        z.p[k] = p[k];
        z.n[k] = n[k];
        if (n[k] > most) most = n[k];
    }
    const int blocks = (most + 1023) / 1024;
    k_zero_ints<<<dim3(blocks < 1024 ? blocks : 1024, arrays), 256, 0, ctx->stream>>>(z);
    ++ctx->launches;
    return cudaGetLastError();
}

}  // namespace alens
