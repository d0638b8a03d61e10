// Device-wide exclusive scan and stable LSD radix sort (reduce-then-scan).
//
// The radix sort orders (key, value) pairs by 8-bit digits, least significant
// first.  Each pass: (1) every block histograms the digits of its 4096-key
// tile, (2) one exclusive scan over the histograms laid out
// [segment][digit][block] gives every (block, digit) its output base, (3)
// every block re-reads its tile, ranks each key among the equal digits before
// it in the tile (warp match/popc, then a prefix over the warps), sorts the
// tile by digit in shared memory and writes each digit's run to its base.
// Segment-major histogram order keeps equal-length segments apart, so one
// launch sorts many views.
#include "common.cuh"

namespace ludvig {

namespace {

constexpr int kScanThreads = 1024;
constexpr int kScanItems = 4;
constexpr int kScanTile = kScanThreads * kScanItems;

__device__ __forceinline__ uint32_t warp_incl_scan(uint32_t v) {
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        uint32_t t = __shfl_up_sync(0xffffffffu, v, o);
        if (lane >= o) v += t;
    }
    return v;
}

// Block-wide exclusive scan of one value per thread; returns the block total.
__device__ __forceinline__ uint32_t block_excl_scan(uint32_t v, uint32_t* out_excl) {
    __shared__ uint32_t warp_tot[32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int nwarps = (blockDim.x + 31) >> 5;
    uint32_t incl = warp_incl_scan(v);
    if (lane == 31) warp_tot[warp] = incl;
    __syncthreads();
    if (warp == 0) {
        uint32_t t = lane < nwarps ? warp_tot[lane] : 0u;
        t = warp_incl_scan(t);
        warp_tot[lane] = t;   // inclusive over warps
    }
    __syncthreads();
    const uint32_t before = warp > 0 ? warp_tot[warp - 1] : 0u;
    *out_excl = before + incl - v;
    const uint32_t total = warp_tot[nwarps - 1];
    __syncthreads();
    return total;
}

__device__ __forceinline__ unsigned long long warp_incl_scan64(unsigned long long v) {
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        unsigned long long t = __shfl_up_sync(0xffffffffu, v, o);
        if (lane >= o) v += t;
    }
    return v;
}

// 64-bit block sum (a tile of 4096 counts may exceed 32 bits).
__device__ __forceinline__ unsigned long long block_sum64(unsigned long long v) {
    __shared__ unsigned long long part[32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    if (lane == 0) part[warp] = v;
    __syncthreads();
    unsigned long long t = 0;
    if (warp == 0) {
        t = lane < (int)((blockDim.x + 31) >> 5) ? part[lane] : 0ull;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
    }
    __syncthreads();
    return t;   // valid in warp 0
}

__global__ void k_scan_reduce(const uint32_t* __restrict__ in, int64_t n,
                              unsigned long long* __restrict__ sums) {
    const int64_t base = (int64_t)blockIdx.x * kScanTile + (int64_t)threadIdx.x * kScanItems;
    unsigned long long s = 0;
#pragma unroll
    for (int i = 0; i < kScanItems; ++i)
        if (base + i < n) s += in[base + i];
    const unsigned long long tot = block_sum64(s);
    if (threadIdx.x == 0) sums[blockIdx.x] = tot;
}

// Single block: exclusive scan of the block sums in place, carrying across chunks.
__global__ void k_scan_sums(unsigned long long* __restrict__ sums, int64_t nb,
                            unsigned long long* __restrict__ total) {
    __shared__ unsigned long long wt[32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int nwarps = (blockDim.x + 31) >> 5;
    unsigned long long carry = 0;
    for (int64_t c0 = 0; c0 < nb; c0 += blockDim.x) {
        const int64_t i = c0 + threadIdx.x;
        const unsigned long long v = i < nb ? sums[i] : 0ull;
        const unsigned long long incl = warp_incl_scan64(v);
        if (lane == 31) wt[warp] = incl;
        __syncthreads();
        if (warp == 0) {
            unsigned long long t = lane < nwarps ? wt[lane] : 0ull;
            wt[lane] = warp_incl_scan64(t);
        }
        __syncthreads();
        const unsigned long long before = warp > 0 ? wt[warp - 1] : 0ull;
        if (i < nb) sums[i] = carry + before + incl - v;
        carry += wt[nwarps - 1];
        __syncthreads();
    }
    if (threadIdx.x == 0 && total) *total = carry;
}

__global__ void k_scan_apply(const uint32_t* __restrict__ in, uint32_t* __restrict__ out, int64_t n,
                             const unsigned long long* __restrict__ sums) {
    const int64_t base = (int64_t)blockIdx.x * kScanTile + (int64_t)threadIdx.x * kScanItems;
    uint32_t v[kScanItems];
    uint32_t s = 0;
#pragma unroll
    for (int i = 0; i < kScanItems; ++i) {
        v[i] = base + i < n ? in[base + i] : 0u;
        s += v[i];
    }
    uint32_t excl;
    block_excl_scan(s, &excl);
    uint32_t run = (uint32_t)sums[blockIdx.x] + excl;
#pragma unroll
    for (int i = 0; i < kScanItems; ++i) {
        if (base + i < n) out[base + i] = run;
        run += v[i];
    }
}

// The whole scan in one block, for inputs so short that the launches are the
// cost: a call on 8 views of 20k Gaussians runs six of them, 10k to 20k counts
// each, and took 12 launches more.  All of a thread's counts are loaded before
// anything is added (four from each part of 4096), so the block waits for memory
// once (4.4 us; 8.7 when it took the parts one after the other).
constexpr int kSmallParts = 8;
constexpr int64_t kScanSmall = (int64_t)kSmallParts * kScanTile;

__global__ void __launch_bounds__(kScanThreads) k_scan_small(const uint32_t* in, uint32_t* out, int64_t n,
                                                             unsigned long long* __restrict__ total) {
    constexpr int kWarps = kScanThreads / 32;
    __shared__ unsigned long long wt[kSmallParts * kWarps];   // each part's warp sums, then their prefix
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    uint32_t v[kSmallParts][kScanItems];
    // (16-byte accesses where the arrays are aligned; the last counts one by one)
    const bool vec = ((reinterpret_cast<uintptr_t>(in) | reinterpret_cast<uintptr_t>(out)) & 15) == 0;
    const int parts = (int)((n + kScanTile - 1) / kScanTile);
#pragma unroll
    for (int p = 0; p < kSmallParts; ++p) {
        const int64_t k = (int64_t)p * kScanTile + (int64_t)threadIdx.x * kScanItems;
        if (vec && k + kScanItems <= n) {
            const uint4 q = *reinterpret_cast<const uint4*>(in + k);
            v[p][0] = q.x;
            v[p][1] = q.y;
            v[p][2] = q.z;
            v[p][3] = q.w;
        } else {
#pragma unroll
            for (int i = 0; i < kScanItems; ++i) v[p][i] = k + i < n ? in[k + i] : 0u;
        }
    }
    uint32_t excl[kSmallParts];   // (a prefix is meaningful below 2^32, as the scan's contract has it)
#pragma unroll
    for (int p = 0; p < kSmallParts; ++p) {
        if (p >= parts) {   // (whole block)
            if (lane == 31) wt[p * kWarps + warp] = 0;
            continue;
        }
        unsigned long long s = 0;
#pragma unroll
        for (int i = 0; i < kScanItems; ++i) s += v[p][i];
        const unsigned long long incl = warp_incl_scan64(s);
        excl[p] = (uint32_t)(incl - s);
        if (lane == 31) wt[p * kWarps + warp] = incl;
    }
    __syncthreads();
    if (warp == 0) {   // the sums' exclusive prefix, eight consecutive ones per lane
        constexpr int kPer = kSmallParts * kWarps / 32;
        unsigned long long s = 0, part[kPer];
#pragma unroll
        for (int i = 0; i < kPer; ++i) {
            part[i] = s;
            s += wt[lane * kPer + i];
        }
        const unsigned long long incl = warp_incl_scan64(s);
#pragma unroll
        for (int i = 0; i < kPer; ++i) wt[lane * kPer + i] = incl - s + part[i];
        if (lane == 31 && total) *total = incl;
    }
    __syncthreads();
#pragma unroll
    for (int p = 0; p < kSmallParts; ++p) {
        if (p >= parts) continue;
        const int64_t k = (int64_t)p * kScanTile + (int64_t)threadIdx.x * kScanItems;
        uint32_t run[kScanItems];
        run[0] = (uint32_t)wt[p * kWarps + warp] + excl[p];
#pragma unroll
        for (int i = 1; i < kScanItems; ++i) run[i] = run[i - 1] + v[p][i - 1];
        if (vec && k + kScanItems <= n) {
            *reinterpret_cast<uint4*>(out + k) = make_uint4(run[0], run[1], run[2], run[3]);
        } else {
#pragma unroll
            for (int i = 0; i < kScanItems; ++i)
                if (k + i < n) out[k + i] = run[i];
        }
    }
}

// ------------------------------------------------------------------ radix

// Keys of a sort whose length lives in device memory (`len`, one segment):
// entries at or past the length read as the largest key (they sort last), and
// blocks that start past it take no part (zero histogram, no output).
__device__ __forceinline__ int64_t radix_valid(const uint64_t* len, int64_t seg_len) {
    return len ? (int64_t)min((uint64_t)seg_len, *len) : seg_len;
}

// Keys are 32-bit or 16-bit (KeyT); entries past the valid length read as the
// type's largest key.
template <class KeyT>
__global__ void __launch_bounds__(kRadixThreads)
k_radix_upsweep(const KeyT* __restrict__ keys, int shift, uint32_t* __restrict__ hist, int64_t bps,
                const uint64_t* __restrict__ len) {
    constexpr uint32_t kFill = (uint32_t)(KeyT)~(KeyT)0;
    __shared__ uint32_t h[256];
    h[threadIdx.x] = 0;
    __syncthreads();
    const int64_t base = (int64_t)blockIdx.x * kRadixTile;
    // positions within the block's segment are compared with the valid length
    const int64_t seg_base = (int64_t)(blockIdx.x % bps) * kRadixTile;
    const int64_t valid = radix_valid(len, bps * kRadixTile);
    if (seg_base < valid) {
#pragma unroll 4
        for (int i = 0; i < kRadixItems; ++i) {
            const int64_t off = i * kRadixThreads + threadIdx.x;
            const uint32_t k = seg_base + off < valid ? (uint32_t)keys[base + off] : kFill;
            atomicAdd(&h[(k >> shift) & 0xffu], 1u);
        }
    }
    __syncthreads();
    const int64_t seg = blockIdx.x / bps, b = blockIdx.x % bps;
    hist[(seg * 256 + threadIdx.x) * bps + b] = h[threadIdx.x];
}

// Warp w owns keys [512 w, 512 w + 512) of the block's tile (16 rounds of 32
// consecutive keys), so per-digit counts accumulate warp-locally in tile order;
// one block prefix over the warps then gives every key its place in the tile
// sorted by digit (stable).  The tile is sorted in shared memory and written
// out in digit runs, so the stores coalesce.
template <class KeyT>
__global__ void __launch_bounds__(kRadixThreads)
k_radix_downsweep(const KeyT* __restrict__ kin, const uint32_t* __restrict__ vin,
                  KeyT* __restrict__ kout, uint32_t* __restrict__ vout, int shift,
                  const uint32_t* __restrict__ hist, int64_t bps, const uint64_t* __restrict__ len) {
    constexpr int kWarps = kRadixThreads / 32;
    constexpr uint32_t kFill = (uint32_t)(KeyT)~(KeyT)0;
    __shared__ uint32_t s_key[kRadixTile];
    __shared__ uint32_t s_val[kRadixTile];
    __shared__ uint32_t wcnt[kWarps][256];   // per-warp digit counts, then their prefix
    __shared__ uint32_t dstart[256];          // first tile position of each digit
    __shared__ uint32_t obase[256];           // output position of each digit's first key
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int64_t seg = blockIdx.x / bps, b = blockIdx.x % bps;
    const int64_t base = (int64_t)blockIdx.x * kRadixTile;
    const int64_t seg_base = b * kRadixTile;   // the block's position within its segment
    const int64_t valid = radix_valid(len, bps * kRadixTile);
    if (seg_base >= valid) return;   // (whole block uniform)
    const uint32_t lt_mask = (1u << lane) - 1u;
#pragma unroll
    for (int w = 0; w < kWarps; ++w) wcnt[w][tid] = 0;
    __syncthreads();
    uint32_t k[kRadixItems], v[kRadixItems], rk[kRadixItems];
#pragma unroll
    for (int i = 0; i < kRadixItems; ++i) {
        const int64_t off = warp * (32 * kRadixItems) + i * 32 + lane;
        k[i] = seg_base + off < valid ? (uint32_t)kin[base + off] : kFill;
        v[i] = seg_base + off < valid ? vin[base + off] : 0u;
    }
#pragma unroll
    for (int i = 0; i < kRadixItems; ++i) {
        const uint32_t d = (k[i] >> shift) & 0xffu;
        const uint32_t peers = __match_any_sync(0xffffffffu, d);
        const uint32_t before = wcnt[warp][d];   // equal digits in this warp's earlier rounds
        rk[i] = before + __popc(peers & lt_mask);
        __syncwarp();
        if ((peers & lt_mask) == 0) wcnt[warp][d] = before + __popc(peers);
        __syncwarp();
    }
    __syncthreads();
    // digit tid: exclusive prefix over the warps, tile total
    uint32_t tot = 0;
#pragma unroll
    for (int w = 0; w < kWarps; ++w) {
        const uint32_t c = wcnt[w][tid];
        wcnt[w][tid] = tot;
        tot += c;
    }
    obase[tid] = hist[(seg * 256 + tid) * bps + b];
    uint32_t ex;
    {
        // exclusive scan of tot over the 256 digits
        __shared__ uint32_t wsum[kWarps];
        uint32_t incl = tot;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t t = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += t;
        }
        if (lane == 31) wsum[warp] = incl;
        __syncthreads();
        uint32_t before = 0;
#pragma unroll
        for (int w = 0; w < kWarps; ++w)
            if (w < warp) before += wsum[w];
        ex = before + incl - tot;
    }
    dstart[tid] = ex;
    __syncthreads();
#pragma unroll
    for (int i = 0; i < kRadixItems; ++i) {
        const uint32_t d = (k[i] >> shift) & 0xffu;
        const uint32_t pos = dstart[d] + wcnt[warp][d] + rk[i];
        s_key[pos] = k[i];
        s_val[pos] = v[i];
    }
    __syncthreads();
#pragma unroll 4
    for (int i = 0; i < kRadixItems; ++i) {
        const int p = i * kRadixThreads + tid;
        const uint32_t kk = s_key[p];
        const uint32_t d = (kk >> shift) & 0xffu;
        const uint32_t o = obase[d] + (uint32_t)p - dstart[d];
        kout[o] = (KeyT)kk;
        vout[o] = s_val[p];
    }
}

}  // namespace

ludvig_status scan_exclusive_u32(const uint32_t* in, uint32_t* out, int64_t n, uint64_t* total_dev,
                                 Arena& ws, cudaStream_t st, bool side) {
    if (n <= 0) {
        if (total_dev) LV_CUDA(cudaMemsetAsync(total_dev, 0, sizeof(uint64_t), st));
        return LUDVIG_OK;
    }
    if (n <= kScanSmall) {
        k_scan_small<<<1, kScanThreads, 0, st>>>(in, out, n, reinterpret_cast<unsigned long long*>(total_dev));
        LV_LAUNCH();
        return LUDVIG_OK;
    }
    const int64_t nb = ceil_div(n, kScanTile);
    unsigned long long* sums = nullptr;
    LV_TRY(ws.get(side ? "scan.sums.side" : "scan.sums", (size_t)nb, &sums));
    k_scan_reduce<<<(unsigned)nb, kScanThreads, 0, st>>>(in, n, sums);
    LV_LAUNCH();
    k_scan_sums<<<1, kScanThreads, 0, st>>>(sums, nb, reinterpret_cast<unsigned long long*>(total_dev));
    LV_LAUNCH();
    k_scan_apply<<<(unsigned)nb, kScanThreads, 0, st>>>(in, out, n, sums);
    LV_LAUNCH();
    return LUDVIG_OK;
}

namespace {
template <class KeyT>
ludvig_status radix_sort_impl(KeyT** keys, uint32_t** vals, KeyT* keys_alt, uint32_t* vals_alt, int64_t nseg,
                              int64_t seg_len, const uint64_t* len, int nbits, Arena& ws, cudaStream_t st,
                              bool side = false) {
    if (len && nseg != 1) {
        set_error("radix_sort_pairs_len: a device length needs one segment");
        return LUDVIG_ERR_INTERNAL;
    }
    if (nseg <= 0 || seg_len <= 0 || nbits <= 0) return LUDVIG_OK;
    if (seg_len % kRadixTile != 0) {
        set_error("radix_sort_pairs: segment length %lld not a multiple of %d", (long long)seg_len,
                  kRadixTile);
        return LUDVIG_ERR_INTERNAL;
    }
    const int64_t bps = seg_len / kRadixTile;
    const int64_t nblocks = bps * nseg;
    if (nblocks > 0x7fffffff) {
        set_error("radix_sort_pairs: too many blocks");
        return LUDVIG_ERR_ARG;
    }
    const int64_t nh = nseg * 256 * bps;
    uint32_t* hist = nullptr;
    LV_TRY(ws.get(side ? "radix.hist.side" : "radix.hist", (size_t)nh, &hist));
    KeyT *kin = *keys, *kout = keys_alt;
    uint32_t *vin = *vals, *vout = vals_alt;
    for (int shift = 0; shift < nbits; shift += 8) {
        k_radix_upsweep<KeyT><<<(unsigned)nblocks, kRadixThreads, 0, st>>>(kin, shift, hist, bps, len);
        LV_LAUNCH();
        LV_TRY(scan_exclusive_u32(hist, hist, nh, nullptr, ws, st, side));
        k_radix_downsweep<KeyT><<<(unsigned)nblocks, kRadixThreads, 0, st>>>(kin, vin, kout, vout, shift,
                                                                             hist, bps, len);
        LV_LAUNCH();
        KeyT* tk = kin;
        kin = kout;
        kout = tk;
        uint32_t* tv = vin;
        vin = vout;
        vout = tv;
    }
    *keys = kin;
    *vals = vin;
    return LUDVIG_OK;
}
}  // namespace

ludvig_status radix_sort_pairs(uint32_t** keys, uint32_t** vals, uint32_t* keys_alt,
                               uint32_t* vals_alt, int64_t nseg, int64_t seg_len, int nbits,
                               Arena& ws, cudaStream_t st, bool side) {
    return radix_sort_impl<uint32_t>(keys, vals, keys_alt, vals_alt, nseg, seg_len, nullptr, nbits, ws, st, side);
}

ludvig_status radix_sort_pairs_len(uint32_t** keys, uint32_t** vals, uint32_t* keys_alt,
                                   uint32_t* vals_alt, int64_t nseg, int64_t seg_len, const uint64_t* len,
                                   int nbits, Arena& ws, cudaStream_t st) {
    return radix_sort_impl<uint32_t>(keys, vals, keys_alt, vals_alt, nseg, seg_len, len, nbits, ws, st);
}

ludvig_status radix_sort_pairs_len16(uint16_t** keys, uint32_t** vals, uint16_t* keys_alt, uint32_t* vals_alt,
                                     int64_t nseg, int64_t seg_len, const uint64_t* len, int nbits, Arena& ws,
                                     cudaStream_t st) {
    if (nbits > 16) {
        set_error("radix_sort_pairs_len16: %d key bits", nbits);
        return LUDVIG_ERR_INTERNAL;
    }
    return radix_sort_impl<uint16_t>(keys, vals, keys_alt, vals_alt, nseg, seg_len, len, nbits, ws, st);
}

}  // namespace ludvig
