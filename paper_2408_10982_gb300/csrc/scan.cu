// scan.cu -- device-wide exclusive scan of int32 counts into int64 offsets.
//
// out[0] = base, out[i+1] = base + in[0] + ... + in[i]  (count+1 outputs).
// Per-tile sums, then a rescan of every tile that adds the tile's prefix, which
// each block sums up itself: from the tile sums, or, in a scan of a few tiles,
// from the counts in front of it without a first pass.  Beyond kScanSumTiles
// tiles a single-block scan of the tile sums runs in between.
// The scans of a small call are launches and gaps, not bytes: with three launches
// each, a call on 16,384 sets at scale 10 spent .062 ms on three scans, now .031;
// a pool of 4.2 M sets .129 and .100 ms.
#include "internal.cuh"

namespace im {

namespace {

constexpr int kScanThreads = 512;
constexpr int kScanItems = 8;                      // per thread
constexpr int kScanTile = kScanThreads * kScanItems;
constexpr int64_t kScanDirectTiles = 8;            // prefixes straight from the counts
constexpr int64_t kScanSumTiles = 8192;            // ... from the tile sums, 16 per thread

__device__ __forceinline__ int64_t block_excl_scan(int64_t v, int64_t *total, int64_t *sh) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int64_t incl = warp_incl_scan<int64_t>(v, lane);
    if (lane == 31) sh[warp] = incl;
    __syncthreads();
    if (warp == 0) {
        int64_t s = lane < (kScanThreads / 32) ? sh[lane] : 0;
        int64_t si = warp_incl_scan<int64_t>(s, lane);
        if (lane < kScanThreads / 32) sh[lane] = si - s;
        if (lane == 31) sh[32] = si;
    }
    __syncthreads();
    int64_t r = sh[warp] + incl - v;
    *total = sh[32];
    __syncthreads();
    return r;
}

__global__ void __launch_bounds__(kScanThreads) k_tile_sums(const int32_t *in, int64_t count,
                                                            int64_t *sums) {
    __shared__ int64_t sh[33];
    const int64_t base = (int64_t)blockIdx.x * kScanTile;
    int64_t s = 0;
    if (base + kScanTile <= count && ((uintptr_t)in & 15) == 0) {
        const int4 *in4 = reinterpret_cast<const int4 *>(in + base);
#pragma unroll
        for (int i = 0; i < kScanItems / 4; ++i) {
            const int4 x = in4[i * kScanThreads + threadIdx.x];
            s += (int64_t)x.x + x.y + ((int64_t)x.z + x.w);
        }
    } else {
#pragma unroll
        for (int i = 0; i < kScanItems; ++i) {
            int64_t idx = base + (int64_t)i * kScanThreads + threadIdx.x;
            if (idx < count) s += in[idx];
        }
    }
    int64_t total;
    block_excl_scan(s, &total, sh);
    if (threadIdx.x == 0) sums[blockIdx.x] = total;
}

__global__ void __launch_bounds__(kScanThreads) k_scan_sums(int64_t *sums, int64_t ntiles,
                                                            const int64_t *base, int64_t *grand) {
    __shared__ int64_t sh[33];
    int64_t carry = base ? *base : 0;
    for (int64_t b0 = 0; b0 < ntiles; b0 += kScanThreads) {
        int64_t idx = b0 + threadIdx.x;
        int64_t v = idx < ntiles ? sums[idx] : 0;
        int64_t total;
        int64_t ex = block_excl_scan(v, &total, sh);
        if (idx < ntiles) sums[idx] = carry + ex;
        carry += total;
    }
    if (threadIdx.x == 0) *grand = carry;
}

// FROM: what a tile's prefix comes from: 0 the counts, 1 the tile sums, 2 the
// scanned tile sums (which hold *base already).
template <int FROM>
__global__ void __launch_bounds__(kScanThreads) k_tile_scan(const int32_t *in, int64_t count,
                                                            const int64_t *sums,
                                                            const int64_t *base, int64_t *out) {
    __shared__ int64_t sh[33];
    const int64_t first = (int64_t)blockIdx.x * kScanTile;
    int64_t total;
    int64_t prefix;
    if (FROM == 2) {
        prefix = sums[blockIdx.x];
    } else {
        int64_t s = threadIdx.x == 0 && base ? *base : 0;
        if (FROM == 0) {
#pragma unroll 8
            for (int64_t i = threadIdx.x; i < first; i += kScanThreads) s += in[i];
        } else {
#pragma unroll 8
            for (int64_t i = threadIdx.x; i < (int64_t)blockIdx.x; i += kScanThreads) s += sums[i];
        }
        block_excl_scan(s, &prefix, sh);
    }
    // each thread owns kScanItems consecutive items, read and written 16 bytes at
    // a time where the arrays' alignment allows
    const int64_t at = first + (int64_t)threadIdx.x * kScanItems;
    const bool whole = at + kScanItems <= count;
    int32_t v[kScanItems];
    int64_t s = 0;
    if (whole && ((uintptr_t)in & 15) == 0) {
#pragma unroll
        for (int i = 0; i < kScanItems; i += 4) {
            const int4 x = *reinterpret_cast<const int4 *>(in + at + i);
            v[i] = x.x;
            v[i + 1] = x.y;
            v[i + 2] = x.z;
            v[i + 3] = x.w;
        }
    } else {
#pragma unroll
        for (int i = 0; i < kScanItems; ++i) v[i] = at + i < count ? in[at + i] : 0;
    }
#pragma unroll
    for (int i = 0; i < kScanItems; ++i) s += v[i];
    int64_t run = prefix + block_excl_scan(s, &total, sh);
    if (whole && ((uintptr_t)out & 15) == 0) {
#pragma unroll
        for (int i = 0; i < kScanItems; i += 2) {
            const int64_t next = run + v[i];
            *reinterpret_cast<longlong2 *>(out + at + i) = make_longlong2(run, next);
            run = next + v[i + 1];
        }
    } else {
#pragma unroll
        for (int i = 0; i < kScanItems; ++i) {
            if (at + i < count) out[at + i] = run;
            run += v[i];
        }
    }
    // (*base may be out[0]: it is read before, or stays what it is)
    if (blockIdx.x == gridDim.x - 1 && threadIdx.x == 0) out[count] = prefix + total;
}

}  // namespace

size_t scan_tmp_bytes(int64_t count) {
    int64_t ntiles = (count + kScanTile - 1) / kScanTile;
    return (size_t)(ntiles + 2) * sizeof(int64_t);
}

im_status exclusive_scan_i32_to_i64(const int32_t *in, int64_t *out, int64_t count,
                                    const int64_t *base, void *tmp, size_t tmp_bytes,
                                    cudaStream_t st) {
    int64_t ntiles = (count + kScanTile - 1) / kScanTile;
    if (tmp_bytes < scan_tmp_bytes(count)) return IM_ERR_INVALID_ARG;
    int64_t *sums = (int64_t *)tmp;
    int64_t *grand = sums + ntiles + 1;
    if (count == 0) {
        // out[0] = base
        {
            KernelTimer kt(st, "scan");
            k_scan_sums<<<1, kScanThreads, 0, st>>>(sums, 0, base, grand);
        }
        IM_CUDA(cudaMemcpyAsync(out, grand, sizeof(int64_t), cudaMemcpyDeviceToDevice, st));
        return IM_OK;
    }
    KernelTimer kt(st, "scan");
    if (ntiles <= kScanDirectTiles) {
        k_tile_scan<0><<<(unsigned)ntiles, kScanThreads, 0, st>>>(in, count, nullptr, base, out);
    } else {
        k_tile_sums<<<(unsigned)ntiles, kScanThreads, 0, st>>>(in, count, sums);
        if (ntiles <= kScanSumTiles) {
            k_tile_scan<1><<<(unsigned)ntiles, kScanThreads, 0, st>>>(in, count, sums, base, out);
        } else {
            k_scan_sums<<<1, kScanThreads, 0, st>>>(sums, ntiles, base, grand);
            k_tile_scan<2><<<(unsigned)ntiles, kScanThreads, 0, st>>>(in, count, sums, nullptr, out);
        }
    }
    IM_CUDA(cudaGetLastError());
    return IM_OK;
}

}  // namespace im
