// Stable LSD radix sort of (key, value) pairs, hand-written.
//
// Each pass sorts by one 8-bit digit with three kernels ("reduce, then scan,
// then scatter"):
//   upsweep   : per tile digit histogram, written digit-major [256][n_tiles]
//   scan      : one block per digit turns its row into exclusive offsets and
//               leaves the digit's total
//   downsweep : per tile stable ranking and scatter to the digit's base + the
//               tile's offset + rank
// A warp takes kSortItems x 32 consecutive keys of the tile, 32 at a time, so
// ordering by (warp, step, lane) is the input order and the pass is stable.
// Up to kSmallSort pairs one block sorts in shared memory, in one launch.
//
// What bounds it: launches and latency (1M pairs are 12 MB, in L2 all along).
// 4-bit digits took 16 passes, with a block-wide barrier per 256 keys and all
// counts scanned by one block: 0.51 ms for 1M 63-bit keys; 8-bit digits, eight
// passes ranked warp by warp and a scan block per digit: 0.17 ms.
#include "common.cuh"

namespace lidar {
namespace {

constexpr int kSortThreads = 256;
constexpr int kSortItems = 8;
constexpr int kSortTile = kSortThreads * kSortItems;
constexpr int kRadixBits = 8;
constexpr int kRadix = 1 << kRadixBits;
constexpr int kSortWarps = kSortThreads / 32;

template <typename K>
__device__ __forceinline__ uint32_t digit_of(K key, int shift)
{
    return (uint32_t)(key >> shift) & (uint32_t)(kRadix - 1);
}

// lanes of the warp with the same digit (the ones past the end, kRadix, form a
// group of their own).  Out of ballots of the digit's bits: __match_any_sync
// takes longer (a downsweep of 1M pairs 14.9 us with it, 12.6 us so).
__device__ __forceinline__ uint32_t peers_of(uint32_t dg)
{
    uint32_t peers = 0xffffffffu;
#pragma unroll
    for (int b = 0; b <= kRadixBits; ++b) {
        const bool bit = (dg >> b) & 1u;
        const uint32_t m = __ballot_sync(0xffffffffu, bit);
        peers &= bit ? m : ~m;
    }
    return peers;
}

// Start of a pass's kernel: it may be resident before the kernel ahead of it
// has ended (launch_pass), so the next is let in and it waits for that one's
// results before it touches memory.  No pointer below is __restrict__: a load
// taken for read-only could be moved above the wait.
__device__ __forceinline__ void pass_begin()
{
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    asm volatile("griddepcontrol.wait;" ::: "memory");
}

template <typename K>
__global__ void __launch_bounds__(kSortThreads) k_upsweep(const K* keys, int64_t n, int shift, int n_tiles,
                                                          uint32_t* counts)
{
    pass_begin();
    __shared__ uint32_t s_cnt[kRadix];
    s_cnt[threadIdx.x] = 0;
    const int64_t base = (int64_t)blockIdx.x * kSortTile;
    uint32_t dg[kSortItems];
#pragma unroll
    for (int i = 0; i < kSortItems; ++i) {
        const int64_t idx = base + (int64_t)i * kSortThreads + threadIdx.x;
        dg[i] = idx < n ? digit_of(keys[idx], shift) : (uint32_t)kRadix;
    }
    __syncthreads();
    // (one addition per group of equal digits, found by __match_any_sync, took
    // 10.0 us a pass for 1M keys; an addition per key 4.7 us)
#pragma unroll
    for (int i = 0; i < kSortItems; ++i)
        if (dg[i] < (uint32_t)kRadix) atomicAdd(&s_cnt[dg[i]], 1u);
    __syncthreads();
    counts[(int64_t)threadIdx.x * n_tiles + blockIdx.x] = s_cnt[threadIdx.x];
}

// Exclusive scan of one digit's counts in place; its total to totals[digit].
__global__ void __launch_bounds__(kSortThreads) k_scan_digit(uint32_t* counts, int n_tiles, uint32_t* totals)
{
    pass_begin();
    __shared__ uint32_t s_sum[kSortWarps];
    uint32_t* row = counts + (int64_t)blockIdx.x * n_tiles;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    uint32_t carry = 0;
    for (int base = 0; base < n_tiles; base += kSortThreads) {
        const int i = base + threadIdx.x;
        const uint32_t v = i < n_tiles ? row[i] : 0u;
        uint32_t x = v;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
            if (lane >= o) x += y;
        }
        __syncthreads();
        if (lane == 31) s_sum[warp] = x;
        __syncthreads();
        uint32_t before = 0, sum = 0;
#pragma unroll
        for (int w = 0; w < kSortWarps; ++w) {
            const uint32_t y = s_sum[w];
            if (w < warp) before += y;
            sum += y;
        }
        if (i < n_tiles) row[i] = carry + before + x - v;
        carry += sum;
    }
    if (threadIdx.x == 0) totals[blockIdx.x] = carry;
}

// exclusive prefix over the 256 threads of a block
__device__ __forceinline__ uint32_t digit_prefix(uint32_t v, uint32_t* s_sum)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    uint32_t x = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) s_sum[warp] = x;
    __syncthreads();
    uint32_t before = 0;
    for (int w = 0; w < warp; ++w) before += s_sum[w];
    return before + x - v;
}

template <typename K>
__global__ void __launch_bounds__(kSortThreads) k_downsweep(const K* keys_in, const uint32_t* vals_in, K* keys_out,
                                                            uint32_t* vals_out, int64_t n, int shift, int n_tiles,
                                                            const uint32_t* offsets, const uint32_t* totals)
{
    pass_begin();
    __shared__ uint32_t s_at[kSortWarps][kRadix];  // per warp: keys of a digit so far, then where its next ones go
    __shared__ uint32_t s_out[kRadix];
    __shared__ K s_key[kSortTile];
    __shared__ uint32_t s_val[kSortTile];
    __shared__ uint32_t s_sum[kSortWarps];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t total = totals[threadIdx.x];
    const uint32_t tile_off = offsets[(int64_t)threadIdx.x * n_tiles + blockIdx.x];
    const int64_t base = (int64_t)blockIdx.x * kSortTile + warp * (32 * kSortItems) + lane;
    K key[kSortItems];
    uint32_t val[kSortItems], rank[kSortItems];
#pragma unroll
    for (int i = 0; i < kSortItems; ++i) {
        const int64_t idx = base + i * 32;
        key[i] = idx < n ? keys_in[idx] : (K)0;
        val[i] = idx < n ? vals_in[idx] : 0u;
    }
#pragma unroll
    for (int w = 0; w < kSortWarps; ++w) s_at[w][threadIdx.x] = 0;
    __syncthreads();
    const uint32_t lt_mask = (1u << lane) - 1u;
#pragma unroll
    for (int i = 0; i < kSortItems; ++i) {
        const bool ok = base + i * 32 < n;
        const uint32_t dg = ok ? digit_of(key[i], shift) : (uint32_t)kRadix;
        const uint32_t peers = peers_of(dg);
        rank[i] = 0;
        if (ok) rank[i] = s_at[warp][dg] + __popc(peers & lt_mask);
        __syncwarp();
        if (ok && lane == __ffs(peers) - 1) s_at[warp][dg] += __popc(peers);
        __syncwarp();
    }
    // thread d: digit d's first place in the sorted tile and of each warp's
    // share, and how far from there the output is
    const uint32_t first = digit_prefix(total, s_sum) + tile_off;  // (its barrier ends the counting)
    uint32_t mine = 0;
#pragma unroll
    for (int w = 0; w < kSortWarps; ++w) {
        const uint32_t c = s_at[w][threadIdx.x];
        s_at[w][threadIdx.x] = mine;
        mine += c;
    }
    __syncthreads();
    const uint32_t local = digit_prefix(mine, s_sum);
#pragma unroll
    for (int w = 0; w < kSortWarps; ++w) s_at[w][threadIdx.x] += local;
    s_out[threadIdx.x] = first - local;
    __syncthreads();
    // sorted in shared memory first, so that a digit's keys leave side by side
    // (scattered from registers: 19 us a pass for 1M pairs, against 15)
#pragma unroll
    for (int i = 0; i < kSortItems; ++i) {
        if (base + i * 32 >= n) continue;
        const uint32_t pos = s_at[warp][digit_of(key[i], shift)] + rank[i];
        s_key[pos] = key[i];
        s_val[pos] = val[i];
    }
    __syncthreads();
    const int count = (int)min((int64_t)kSortTile, n - (int64_t)blockIdx.x * kSortTile);
#pragma unroll
    for (int i = 0; i < kSortItems; ++i) {
        const int k = i * kSortThreads + threadIdx.x;
        if (k >= count) break;
        const K x = s_key[k];
        const uint32_t pos = s_out[digit_of(x, shift)] + k;
        keys_out[pos] = x;
        vals_out[pos] = s_val[k];
    }
}

// Up to kSmallSort pairs in one block: every pass ranks out of registers and
// scatters through shared memory.  (770 pairs of 63-bit keys: 24 launches
// would take 55 us; 48 launches of 4-bit passes took 270 us, this one 16.)
constexpr int kSmallSort = 4096;
constexpr int kSmallThreads = 512;
constexpr int kSmallWarps = kSmallThreads / 32;
constexpr int kSmallItems = kSmallSort / kSmallThreads;

template <typename K>
constexpr size_t small_sort_smem()
{
    return kSmallSort * (sizeof(K) + sizeof(uint32_t)) + kSmallWarps * kRadix * sizeof(uint32_t);
}

template <typename K>
__global__ void __launch_bounds__(kSmallThreads) k_sort_small(K* __restrict__ keys, uint32_t* __restrict__ vals, int n,
                                                              int key_bits)
{
    extern __shared__ __align__(16) unsigned char smem[];
    K* s_key = (K*)smem;
    uint32_t* s_val = (uint32_t*)(s_key + kSmallSort);
    uint32_t(*s_at)[kRadix] = (uint32_t(*)[kRadix])(s_val + kSmallSort);
    __shared__ uint32_t s_sum[kRadix / 32];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    // the fewest whole steps of 32 per warp that hold n
    const int items = (n + kSmallThreads - 1) / kSmallThreads;
    const int base = warp * (32 * items) + lane;
    const uint32_t lt_mask = (1u << lane) - 1u;
    K key[kSmallItems];
    uint32_t val[kSmallItems], rank[kSmallItems];
#pragma unroll
    for (int i = 0; i < kSmallItems; ++i) {
        const int idx = base + i * 32;
        const bool ok = i < items && idx < n;
        key[i] = ok ? keys[idx] : (K)0;
        val[i] = ok ? vals[idx] : 0u;
    }
    for (int shift = 0; shift < key_bits; shift += kRadixBits) {
        for (int k = threadIdx.x; k < kSmallWarps * kRadix; k += kSmallThreads) (&s_at[0][0])[k] = 0;
        __syncthreads();
#pragma unroll
        for (int i = 0; i < kSmallItems; ++i) {
            if (i >= items) break;
            const bool ok = base + i * 32 < n;
            const uint32_t dg = ok ? digit_of(key[i], shift) : (uint32_t)kRadix;
            const uint32_t peers = peers_of(dg);
            rank[i] = 0;
            if (ok) rank[i] = s_at[warp][dg] + __popc(peers & lt_mask);
            __syncwarp();
            if (ok && lane == __ffs(peers) - 1) s_at[warp][dg] += __popc(peers);
            __syncwarp();
        }
        __syncthreads();
        // thread d < 256: counts before each warp, then the digit's base added
        uint32_t total = 0, x = 0;
        if (threadIdx.x < kRadix) {
#pragma unroll
            for (int w = 0; w < kSmallWarps; ++w) {
                const uint32_t c = s_at[w][threadIdx.x];
                s_at[w][threadIdx.x] = total;
                total += c;
            }
            x = total;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
                if (lane >= o) x += y;
            }
            if (lane == 31) s_sum[warp] = x;
        }
        __syncthreads();
        if (threadIdx.x < kRadix) {
            uint32_t first = x - total;
            for (int w = 0; w < warp; ++w) first += s_sum[w];
#pragma unroll
            for (int w = 0; w < kSmallWarps; ++w) s_at[w][threadIdx.x] += first;
        }
        __syncthreads();
#pragma unroll
        for (int i = 0; i < kSmallItems; ++i) {
            if (i >= items) break;
            if (base + i * 32 < n) {
                const uint32_t pos = s_at[warp][digit_of(key[i], shift)] + rank[i];
                s_key[pos] = key[i];
                s_val[pos] = val[i];
            }
        }
        __syncthreads();
#pragma unroll
        for (int i = 0; i < kSmallItems; ++i) {
            const int idx = base + i * 32;
            if (i < items && idx < n) {
                key[i] = s_key[idx];
                val[i] = s_val[idx];
            }
        }
    }
#pragma unroll
    for (int i = 0; i < kSmallItems; ++i) {
        const int idx = base + i * 32;
        if (i < items && idx < n) {
            keys[idx] = key[i];
            vals[idx] = val[i];
        }
    }
}

// Launches a pass's kernel so that its blocks may become resident while the
// kernel ahead of it in the stream drains; `first` waits for that one's end.
// (24 kernels of 4 to 13 us: 1M pairs' rebuild and cast 1,402 us with plain
// launches, 1,358 us so.)  A kernel is let in once all blocks of the one ahead
// have started, so none that waits keeps an earlier one's from running.
template <typename... P, typename... A>
cudaError_t launch_pass(cudaStream_t s, bool first, void (*fn)(P...), int blocks, A... args)
{
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((unsigned)blocks);
    cfg.blockDim = dim3(kSortThreads);
    cfg.stream = s;
    cfg.attrs = attr;
    cfg.numAttrs = first ? 0 : 1;
    return cudaLaunchKernelEx(&cfg, fn, P(args)...);
}

template <typename K>
cudaError_t radix_sort_pairs(cudaStream_t s, K* keys, uint32_t* vals, int64_t n, int key_bits, void* scratch,
                             size_t scratch_bytes)
{
    if (n <= 1) return cudaSuccess;
    if (scratch_bytes < radix_sort_scratch_bytes(n)) return cudaErrorInvalidValue;
    if (n <= kSmallSort) {
        constexpr size_t smem = small_sort_smem<K>();
        cudaError_t e = cudaFuncSetAttribute(k_sort_small<K>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
        k_sort_small<K><<<1, kSmallThreads, smem, s>>>(keys, vals, (int)n, key_bits);
        return cudaGetLastError();
    }
    const int n_tiles = (int)((n + kSortTile - 1) / kSortTile);
    char* p = (char*)scratch;
    K* alt_keys = (K*)p;
    p += ((n * sizeof(uint64_t) + 255) / 256) * 256;
    uint32_t* alt_vals = (uint32_t*)p;
    p += ((n * sizeof(uint32_t) + 255) / 256) * 256;
    uint32_t* totals = (uint32_t*)p;
    p += kRadix * sizeof(uint32_t);
    uint32_t* counts = (uint32_t*)p;
    const int passes = (key_bits + kRadixBits - 1) / kRadixBits;
    K* kin = keys;
    K* kout = alt_keys;
    uint32_t* vin = vals;
    uint32_t* vout = alt_vals;
    for (int pass = 0; pass < passes; ++pass) {
        const int shift = pass * kRadixBits;
        cudaError_t e = launch_pass(s, pass == 0, k_upsweep<K>, n_tiles, kin, n, shift, n_tiles, counts);
        if (e == cudaSuccess) e = launch_pass(s, false, k_scan_digit, kRadix, counts, n_tiles, totals);
        if (e == cudaSuccess)
            e = launch_pass(s, false, k_downsweep<K>, n_tiles, kin, vin, kout, vout, n, shift, n_tiles, counts, totals);
        if (e != cudaSuccess) return e;
        K* tk = kin; kin = kout; kout = tk;
        uint32_t* tv = vin; vin = vout; vout = tv;
    }
    if (kin != keys) {
        cudaMemcpyAsync(keys, kin, n * sizeof(K), cudaMemcpyDeviceToDevice, s);
        cudaMemcpyAsync(vals, vin, n * sizeof(uint32_t), cudaMemcpyDeviceToDevice, s);
    }
    return cudaGetLastError();
}

}  // namespace

size_t radix_sort_scratch_bytes(int64_t n)
{
    const int64_t n_tiles = (n + kSortTile - 1) / kSortTile;
    return ((n * sizeof(uint64_t) + 255) / 256) * 256 + ((n * sizeof(uint32_t) + 255) / 256) * 256 +
           (size_t)kRadix * (n_tiles + 1) * sizeof(uint32_t) + 256;
}

cudaError_t radix_sort_pairs_u64(cudaStream_t s, uint64_t* keys, uint32_t* vals, int64_t n, int key_bits,
                                 void* scratch, size_t scratch_bytes)
{
    return radix_sort_pairs<uint64_t>(s, keys, vals, n, key_bits, scratch, scratch_bytes);
}

cudaError_t radix_sort_pairs_u32(cudaStream_t s, uint32_t* keys, uint32_t* vals, int64_t n, int key_bits,
                                 void* scratch, size_t scratch_bytes)
{
    return radix_sort_pairs<uint32_t>(s, keys, vals, n, key_bits, scratch, scratch_bytes);
}

}  // namespace lidar
