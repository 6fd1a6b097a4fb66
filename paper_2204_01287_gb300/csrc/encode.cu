// encode.cu — the encoder of pc_upload_cloud on the device (Sec. 3.1, Eq. 1,
// Listing 2): raw points in device memory to the batches, words and colours of a
// resident cloud, bit for bit what encode_host makes of them.
//
//   k_bounds     binary32 box of the cloud; notes coordinates that are not finite
//   k_codes      63-bit Morton code per point, the host encoder's binary64 formula
//   k_digits, k_chunk_sums, k_scan_chunks, k_scan, k_scatter
//                one pass of a stable radix sort on 8 bits of the codes: counts per
//                tile, exclusive scan over (digit, tile), scatter by rank
//   k_quantize   per batch of consecutive sorted points: box, Eq. 1 in binary64,
//                word split, colours
//
// Every binary64 operation is an explicit round-to-nearest intrinsic in the
// host encoder's order, or certified to give its result (quantize). For 4M points
// the kernels take 0.8 ms: the sort 0.5 (63 us a pass, 41 of them k_scatter, whose integer
// pipe is 52 % busy), k_quantize 0.17 and k_codes 0.11, both at the binary64 rate (that
// pipe 69 and 84 % busy; GB300 has 2 binary64 FMAs per clock and SM). From some ten million
// points on k_quantize waits for its gathers of 12 bytes by index instead (50M points:
// 3.2 ms, 363 bytes a point read from memory, the binary64 pipe 42 %).
#include <algorithm>
#include <cstdint>

#include "pc_internal.h"

namespace pcr {

namespace {

constexpr unsigned FULL = 0xFFFFFFFFu;
constexpr uint32_t kThreads = 256, kWarps = kThreads / 32;
constexpr uint32_t kItems = 16;                       // points per thread of a sort tile
constexpr uint32_t kTilePoints = kThreads * kItems;   // a warp owns 512 consecutive ones
constexpr uint32_t kDigits = 256, kPasses = 8;
constexpr uint32_t kChunk = 2048;                     // counts per block of the scan
constexpr uint32_t kBlocksPerSm = 8;                  // of the kernels that stride over the points

// What k_bounds leaves: the box's minima and maxima as ordered integers, and
// whether some coordinate is NaN or infinite.
struct Bounds {
    uint32_t lo[3], hi[3], not_finite;
};

// Unsigned integers in the order of the binary32 numbers.
__device__ __forceinline__ uint32_t ordered(float f) {
    const uint32_t u = __float_as_uint(f);
    return u ^ ((u >> 31) ? 0xFFFFFFFFu : 0x80000000u);
}
__device__ __forceinline__ float unordered(uint32_t u) {
    return __uint_as_float(u ^ ((u >> 31) ? 0x80000000u : 0xFFFFFFFFu));
}

__global__ void __launch_bounds__(kThreads) k_bounds(const float* xyz, uint32_t n, Bounds* out) {
    uint32_t lo[3] = {~0u, ~0u, ~0u}, hi[3] = {0u, 0u, 0u};
    bool bad = false;
    for (uint64_t i = (uint64_t)blockIdx.x * kThreads + threadIdx.x; i < n; i += (uint64_t)gridDim.x * kThreads) {
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            const float f = xyz[3 * i + a];
            bad |= !isfinite(f);
            const uint32_t u = ordered(f);
            lo[a] = min(lo[a], u);
            hi[a] = max(hi[a], u);
        }
    }
    // one atomic per block and value: thousands on one address cost more than the reads
    __shared__ uint32_t s_lo[3], s_hi[3];
    if (threadIdx.x < 3) {
        s_lo[threadIdx.x] = ~0u;
        s_hi[threadIdx.x] = 0u;
    }
    __syncthreads();
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        lo[a] = __reduce_min_sync(FULL, lo[a]);
        hi[a] = __reduce_max_sync(FULL, hi[a]);
        if ((threadIdx.x & 31) == 0) {
            atomicMin(&s_lo[a], lo[a]);
            atomicMax(&s_hi[a], hi[a]);
        }
    }
    if (__any_sync(FULL, bad) && (threadIdx.x & 31) == 0) out->not_finite = 1u;
    __syncthreads();
    if (threadIdx.x < 3) {
        atomicMin(&out->lo[threadIdx.x], s_lo[threadIdx.x]);
        atomicMax(&out->hi[threadIdx.x], s_hi[threadIdx.x]);
    }
}

// floor(scale * (p - lo) / size) in the host encoder's binary64 operations, clamped
// to [0, scale - 1]; scale is 2^21 or 2^30 and inv is scale / size, rounded. With
// d = p - lo, rounded, as both take it, and t = scale d / size exact: the definition's
// quotient is t within 2^-53 t (scale d is exact, one rounding), t' = d inv is t within
// 2 * 2^-53 t, so for t up to 2^30 the two are within 3 * 2^-23 = 0.375 * 2^-20 of each
// other. (d is at most hi - lo, so t passes 2^30 only by the rounding of a binary32 size;
// both results are then scale - 1.) Added to 2^32, t' is rounded to a multiple of 2^-20,
// off by at most 0.5 of them: 0.875 in all. So when the sum's fraction is none of 0 and
// 2^20 - 1 of these steps, the whole part is the definition's. Otherwise, and for every t'
// that is not in [0, 2^32), the definition decides. Three binary64 operations in place of a
// division: k_codes 370 -> 114 us and k_quantize 422 -> 174 us for 4M points.
__device__ __noinline__ uint32_t quantize_exact(double d, double size, double scale) {
    double t = 0.0;
    if (size > 0.0) t = floor(__ddiv_rn(__dmul_rn(scale, d), size));
    t = t < 0.0 ? 0.0 : (t > scale - 1.0 ? scale - 1.0 : t);
    return (uint32_t)t;
}
__device__ __forceinline__ uint32_t quantize(float p, double lo, double size, double inv, double scale) {
    const double d = __dsub_rn((double)p, lo);
    const uint64_t bits = (uint64_t)__double_as_longlong(__dadd_rn(__dmul_rn(d, inv), 4294967296.0));
    const uint32_t fraction = (uint32_t)bits & 0xFFFFFu;
    const bool sure = (uint32_t)(bits >> 52) == 1023u + 32u && fraction - 1u < 0xFFFFEu;
    return sure ? min((uint32_t)(bits >> 20), (uint32_t)scale - 1u) : quantize_exact(d, size, scale);
}

// Spread the low 21 bits of v so that bit i lands on bit 3i.
__device__ __forceinline__ uint64_t spread3(uint64_t v) {
    v &= 0x1FFFFFull;
    v = (v | (v << 32)) & 0x001F00000000FFFFull;
    v = (v | (v << 16)) & 0x001F0000FF0000FFull;
    v = (v | (v << 8)) & 0x100F00F00F00F00Full;
    v = (v | (v << 4)) & 0x10C30C30C30C30C3ull;
    v = (v | (v << 2)) & 0x1249249249249249ull;
    return v;
}

__global__ void __launch_bounds__(kThreads) k_codes(const float* xyz, uint32_t n, const Bounds* bounds,
                                                  uint64_t* key, uint32_t* idx) {
    constexpr double scale = 2097152.0;   // 2^21
    double lo[3], size[3], inv[3];
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        lo[a] = (double)unordered(bounds->lo[a]);
        size[a] = __dsub_rn((double)unordered(bounds->hi[a]), lo[a]);
        inv[a] = __ddiv_rn(scale, size[a]);
    }
    for (uint64_t i = (uint64_t)blockIdx.x * kThreads + threadIdx.x; i < n; i += (uint64_t)gridDim.x * kThreads) {
        uint64_t code = 0;
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            code |= spread3(quantize(xyz[3 * i + a], lo[a], size[a], inv[a], scale)) << a;
        }
        key[i] = code;
        idx[i] = (uint32_t)i;
    }
}

__global__ void __launch_bounds__(kThreads) k_identity(uint32_t n, uint32_t* idx) {
    for (uint64_t i = (uint64_t)blockIdx.x * kThreads + threadIdx.x; i < n; i += (uint64_t)gridDim.x * kThreads)
        idx[i] = (uint32_t)i;
}

// Ranks of a warp's 32 digits of one round among the digits the warp has seen:
// counter[d] counts them. Lanes past the end (in false) take no part.
__device__ __forceinline__ uint32_t rank_digit(uint32_t* counter, uint32_t d, bool in) {
    const uint32_t lane = threadIdx.x & 31;
    // lanes of the same digit, bit by bit (a match over 32 values takes longer)
    uint32_t same = __ballot_sync(FULL, in);
#pragma unroll
    for (int b = 0; b < 8; ++b) {
        const uint32_t set = __ballot_sync(FULL, (d >> b) & 1u);
        same &= ((d >> b) & 1u) ? set : ~set;
    }
    uint32_t before = 0;
    const uint32_t leader = in ? __ffs(same) - 1 : lane;
    if (in && lane == leader) {
        before = counter[d];
        counter[d] = before + __popc(same);
    }
    before = __shfl_sync(FULL, before, leader);
    __syncwarp();
    return before + __popc(same & ((1u << lane) - 1u));
}

__global__ void __launch_bounds__(kThreads) k_digits(const uint64_t* key, uint32_t n, uint32_t shift,
                                                   uint32_t tiles, uint32_t* counts) {
    __shared__ uint32_t h[kDigits];
    h[threadIdx.x] = 0;
    __syncthreads();
    const uint64_t first = (uint64_t)blockIdx.x * kTilePoints;
#pragma unroll
    for (uint32_t j = 0; j < kItems; ++j) {
        const uint64_t i = first + j * kThreads + threadIdx.x;
        if (i < n) atomicAdd(&h[(uint32_t)(key[i] >> shift) & (kDigits - 1u)], 1u);
    }
    __syncthreads();
    counts[(uint64_t)threadIdx.x * tiles + blockIdx.x] = h[threadIdx.x];
}

// Exclusive sum over the block's threads of v; total: the block's sum.
__device__ __forceinline__ uint32_t block_exclusive(uint32_t v, uint32_t& total) {
    __shared__ uint32_t warp[kWarps];
    const uint32_t lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    uint32_t incl = v;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        const uint32_t t = __shfl_up_sync(FULL, incl, d);
        if (lane >= (uint32_t)d) incl += t;
    }
    __syncthreads();   // the previous call's readers are done
    if (lane == 31) warp[w] = incl;
    __syncthreads();
    uint32_t base = 0;
    total = 0;
#pragma unroll
    for (uint32_t j = 0; j < kWarps; ++j) {
        if (j < w) base += warp[j];
        total += warp[j];
    }
    return base + incl - v;
}

__global__ void __launch_bounds__(kThreads) k_chunk_sums(const uint32_t* counts, uint64_t m, uint32_t* sums) {
    uint32_t v = 0;
    const uint64_t first = (uint64_t)blockIdx.x * kChunk;
#pragma unroll
    for (uint32_t j = 0; j < kChunk / kThreads; ++j) {
        const uint64_t i = first + j * kThreads + threadIdx.x;
        if (i < m) v += counts[i];
    }
    uint32_t total;
    block_exclusive(v, total);
    if (threadIdx.x == 0) sums[blockIdx.x] = total;
}

// One block: exclusive scan of the chunks' sums in place (their total is below 2^32).
__global__ void __launch_bounds__(kThreads) k_scan_chunks(uint32_t* sums, uint32_t chunks) {
    uint32_t base = 0;
    for (uint32_t c0 = 0; c0 < chunks; c0 += kThreads) {
        const uint32_t i = c0 + threadIdx.x;
        const uint32_t v = i < chunks ? sums[i] : 0u;
        uint32_t total;
        const uint32_t e = block_exclusive(v, total);
        if (i < chunks) sums[i] = base + e;
        base += total;
    }
}

__global__ void __launch_bounds__(kThreads) k_scan(uint32_t* counts, uint64_t m, const uint32_t* sums) {
    constexpr uint32_t per = kChunk / kThreads;
    const uint64_t first = (uint64_t)blockIdx.x * kChunk + threadIdx.x * per;
    uint32_t v[per], sum = 0;
#pragma unroll
    for (uint32_t j = 0; j < per; ++j) {
        v[j] = first + j < m ? counts[first + j] : 0u;
        sum += v[j];
    }
    uint32_t total;
    uint32_t at = sums[blockIdx.x] + block_exclusive(sum, total);
#pragma unroll
    for (uint32_t j = 0; j < per; ++j) {
        if (first + j < m) counts[first + j] = at;
        at += v[j];
    }
}

// A warp takes 512 consecutive points of the tile in rounds of 32, so equal digits
// keep their order: rounds within a warp, warps within the tile, tiles by the
// scan. The tile is put in order in shared memory first, so that a digit's points
// leave as one run: stored from where they are ranked, every 8-byte store was
// a transaction of its own (82 us a pass for 4M points, 41 us this way).
struct ScatterShared {
    uint64_t key[kTilePoints];
    uint32_t idx[kTilePoints];
    uint32_t count[kWarps][kDigits];
    uint32_t out[kDigits];   // place of the digit's first point, less its place in the tile
};

__global__ void __launch_bounds__(kThreads, 3) k_scatter(const uint64_t* key, const uint32_t* idx, uint32_t n,
                                                    uint32_t shift, uint32_t tiles,
                                                    const uint32_t* offsets, uint64_t* key_out,
                                                    uint32_t* idx_out) {
    extern __shared__ __align__(16) unsigned char shared_bytes[];
    ScatterShared& sh = *reinterpret_cast<ScatterShared*>(shared_bytes);
    const uint32_t lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    for (uint32_t j = threadIdx.x; j < kWarps * kDigits; j += kThreads) (&sh.count[0][0])[j] = 0;
    __syncthreads();
    const uint64_t tile = (uint64_t)blockIdx.x * kTilePoints;
    const uint64_t first = tile + w * (kTilePoints / kWarps) + lane;
    uint64_t k[kItems];
    uint32_t rank[kItems];
#pragma unroll
    for (uint32_t j = 0; j < kItems; ++j) {
        const uint64_t i = first + 32u * j;
        k[j] = i < n ? key[i] : 0ull;
    }
#pragma unroll
    for (uint32_t j = 0; j < kItems; ++j)
        rank[j] = rank_digit(sh.count[w], (uint32_t)(k[j] >> shift) & (kDigits - 1u), first + 32u * j < n);
    __syncthreads();
    // count[w][d] becomes the place in the tile of warp w's first point with digit d
    uint32_t total = 0, all;
#pragma unroll
    for (uint32_t j = 0; j < kWarps; ++j) total += sh.count[j][threadIdx.x];
    uint32_t at = block_exclusive(total, all);
    sh.out[threadIdx.x] = offsets[(uint64_t)threadIdx.x * tiles + blockIdx.x] - at;
#pragma unroll
    for (uint32_t j = 0; j < kWarps; ++j) {
        const uint32_t c = sh.count[j][threadIdx.x];
        sh.count[j][threadIdx.x] = at;
        at += c;
    }
    __syncthreads();
#pragma unroll
    for (uint32_t j = 0; j < kItems; ++j) {
        if (first + 32u * j >= n) continue;
        const uint32_t p = sh.count[w][(uint32_t)(k[j] >> shift) & (kDigits - 1u)] + rank[j];
        sh.key[p] = k[j];
        sh.idx[p] = idx[first + 32u * j];
    }
    __syncthreads();
    const uint32_t points = (uint32_t)min((uint64_t)kTilePoints, n - tile);
#pragma unroll
    for (uint32_t j = 0; j < kItems; ++j) {
        const uint32_t p = j * kThreads + threadIdx.x;
        if (p >= points) continue;
        const uint64_t v = sh.key[p];
        const uint32_t to = sh.out[(uint32_t)(v >> shift) & (kDigits - 1u)] + p;
        key_out[to] = v;
        idx_out[to] = sh.idx[p];
    }
}

// One block per batch. The host's running minimum keeps the first of equal
// values, which shows in the sign of a zero: `zero` finds the first zero.
__global__ void __launch_bounds__(kThreads) k_quantize(const float* xyz, const uint32_t* rgba,
                                                     const uint32_t* idx, uint32_t n,
                                                     uint32_t batch_size, pc_batch* batches,
                                                     uint32_t* w1, uint32_t* w2, uint32_t* w3,
                                                     uint32_t* color) {
    __shared__ uint32_t lo[3], hi[3], zero[3];
    if (threadIdx.x < 3) {
        lo[threadIdx.x] = zero[threadIdx.x] = ~0u;
        hi[threadIdx.x] = 0u;
    }
    __syncthreads();
    const uint64_t f = (uint64_t)blockIdx.x * batch_size;
    const uint32_t count = (uint32_t)min((uint64_t)batch_size, n - f);
    uint32_t l[3] = {~0u, ~0u, ~0u}, h[3] = {0u, 0u, 0u}, z[3] = {~0u, ~0u, ~0u};
    for (uint32_t j = threadIdx.x; j < count; j += kThreads) {
        const float* p = xyz + 3ull * idx[f + j];
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            const uint32_t u = ordered(p[a]);
            l[a] = min(l[a], u);
            h[a] = max(h[a], u);
            if (p[a] == 0.0f) z[a] = min(z[a], j);
        }
    }
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        l[a] = __reduce_min_sync(FULL, l[a]);
        h[a] = __reduce_max_sync(FULL, h[a]);
        z[a] = __reduce_min_sync(FULL, z[a]);
        if ((threadIdx.x & 31) == 0) {
            atomicMin(&lo[a], l[a]);
            atomicMax(&hi[a], h[a]);
            atomicMin(&zero[a], z[a]);
        }
    }
    __syncthreads();
    constexpr double scale = 1073741824.0;   // 2^30, Eq. 1
    float mn[3], size[3];
    double inv[3];
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        mn[a] = unordered(lo[a]);
        const float mx = unordered(hi[a]);
        if (mn[a] == 0.0f) mn[a] = xyz[3ull * idx[f + zero[a]] + a];
        size[a] = mx == mn[a] ? 0.0f : __fsub_rn(mx, mn[a]);
        inv[a] = __ddiv_rn(scale, (double)size[a]);
    }
    if (threadIdx.x == 0) {
        pc_batch b;
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            b.min[a] = mn[a];
            b.size[a] = size[a];
        }
        b.first = (uint32_t)f;
        b.count = count;
        batches[blockIdx.x] = b;
    }
    for (uint32_t j = threadIdx.x; j < count; j += kThreads) {
        const uint32_t i = idx[f + j];
        const float* p = xyz + 3ull * i;
        const uint32_t q0 = quantize(p[0], (double)mn[0], (double)size[0], inv[0], scale);
        const uint32_t q1 = quantize(p[1], (double)mn[1], (double)size[1], inv[1], scale);
        const uint32_t q2 = quantize(p[2], (double)mn[2], (double)size[2], inv[2], scale);
        w1[f + j] = (q0 >> 20) | ((q1 >> 20) << 10) | ((q2 >> 20) << 20);
        w2[f + j] = ((q0 >> 10) & 1023u) | (((q1 >> 10) & 1023u) << 10) | (((q2 >> 10) & 1023u) << 20);
        w3[f + j] = (q0 & 1023u) | ((q1 & 1023u) << 10) | ((q2 & 1023u) << 20);
        color[f + j] = rgba ? rgba[i] : 0u;
    }
}

uint64_t up256(uint64_t x) { return (x + 255) & ~255ull; }

// Parts of the scratch memory.
struct Layout {
    uint64_t xyz, rgba, key[2], idx[2], counts, sums, bounds, bytes;
    uint32_t tiles, chunks;
    Layout(uint64_t n, bool colours, bool sort) {
        tiles = (uint32_t)((n + kTilePoints - 1) / kTilePoints);
        chunks = (uint32_t)(((uint64_t)kDigits * tiles + kChunk - 1) / kChunk);
        uint64_t at = 0;
        auto part = [&](uint64_t size) {
            const uint64_t p = at;
            at += up256(size);
            return p;
        };
        bounds = part(sizeof(Bounds));
        xyz = part(12 * n);
        rgba = part(colours ? 4 * n : 0);
        idx[0] = part(4 * n);
        idx[1] = part(sort ? 4 * n : 0);
        key[0] = part(sort ? 8 * n : 0);
        key[1] = part(sort ? 8 * n : 0);
        counts = part(sort ? 4ull * kDigits * tiles : 0);
        sums = part(sort ? 4ull * chunks : 0);
        bytes = at;
    }
};

}  // namespace

uint64_t encode_device_scratch(uint64_t n, bool colours, bool keep_order) {
    return Layout(n, colours, !keep_order).bytes;
}

cudaError_t encode_device(const float* xyz, const uint32_t* rgba, uint64_t n64, uint32_t batch_size,
                          bool keep_order, void* scratch, pc_batch* batches, uint32_t* w1,
                          uint32_t* w2, uint32_t* w3, uint32_t* color, cudaStream_t st,
                          bool* finite) {
    const uint32_t n = (uint32_t)n64;
    const Layout L(n, rgba != nullptr, !keep_order);
    uint8_t* base = static_cast<uint8_t*>(scratch);
    float* d_xyz = reinterpret_cast<float*>(base + L.xyz);
    uint32_t* d_rgba = rgba ? reinterpret_cast<uint32_t*>(base + L.rgba) : nullptr;
    Bounds* bounds = reinterpret_cast<Bounds*>(base + L.bounds);
    uint64_t* key[2] = {reinterpret_cast<uint64_t*>(base + L.key[0]), reinterpret_cast<uint64_t*>(base + L.key[1])};
    uint32_t* idx[2] = {reinterpret_cast<uint32_t*>(base + L.idx[0]), reinterpret_cast<uint32_t*>(base + L.idx[1])};
    uint32_t* counts = reinterpret_cast<uint32_t*>(base + L.counts);
    uint32_t* sums = reinterpret_cast<uint32_t*>(base + L.sums);
    cudaError_t e = cudaMemcpyAsync(d_xyz, xyz, 12ull * n, cudaMemcpyHostToDevice, st);
    if (e == cudaSuccess && rgba) e = cudaMemcpyAsync(d_rgba, rgba, 4ull * n, cudaMemcpyHostToDevice, st);
    if (e == cudaSuccess) e = cudaMemsetAsync(bounds, 0, sizeof(Bounds), st);
    if (e == cudaSuccess) e = cudaMemsetAsync(bounds->lo, 0xFF, sizeof bounds->lo, st);
    if (e != cudaSuccess) return e;
    int dev = 0, sms = 0;
    e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return e;
    const uint32_t grid = (uint32_t)std::min<uint64_t>((n64 + kThreads - 1) / kThreads, (uint64_t)sms * kBlocksPerSm);
    k_bounds<<<grid, kThreads, 0, st>>>(d_xyz, n, bounds);
    if (keep_order) {
        k_identity<<<grid, kThreads, 0, st>>>(n, idx[0]);
    } else {
        k_codes<<<grid, kThreads, 0, st>>>(d_xyz, n, bounds, key[0], idx[0]);
        const uint64_t m = (uint64_t)kDigits * L.tiles;
        e = cudaFuncSetAttribute(k_scatter, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)sizeof(ScatterShared));
        if (e != cudaSuccess) return e;
        for (uint32_t pass = 0; pass < kPasses; ++pass) {
            const uint32_t s = pass & 1u, shift = 8u * pass;
            k_digits<<<L.tiles, kThreads, 0, st>>>(key[s], n, shift, L.tiles, counts);
            k_chunk_sums<<<L.chunks, kThreads, 0, st>>>(counts, m, sums);
            k_scan_chunks<<<1, kThreads, 0, st>>>(sums, L.chunks);
            k_scan<<<L.chunks, kThreads, 0, st>>>(counts, m, sums);
            k_scatter<<<L.tiles, kThreads, sizeof(ScatterShared), st>>>(key[s], idx[s], n, shift, L.tiles, counts,
                                                    key[s ^ 1u], idx[s ^ 1u]);
        }
        static_assert(kPasses % 2 == 0, "the sorted order ends in idx[0]");
    }
    const uint32_t nb = (uint32_t)((n64 + batch_size - 1) / batch_size);
    k_quantize<<<nb, kThreads, 0, st>>>(d_xyz, d_rgba, idx[0], n, batch_size, batches, w1, w2, w3, color);
    e = cudaGetLastError();
    uint32_t bad = 0;
    if (e == cudaSuccess)
        e = cudaMemcpyAsync(&bad, &bounds->not_finite, sizeof bad, cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    *finite = bad == 0;
    return e;
}

}  // namespace pcr
