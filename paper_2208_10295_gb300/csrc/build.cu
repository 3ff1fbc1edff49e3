// Linear BVH build (Karras, "Maximizing Parallelism in the Construction of
// BVHs, Octrees, and k-d Trees", HPG 2012), hand-written:
//   1. centroid bounds (block reduction + ordered-int atomics), index check
//   2. 63-bit Morton keys of the triangle centroids (21 bits per axis)
//   3. stable radix sort of (key, triangle index)
//   4. leaf-ordered triangle gather (vertices + original index, material, instance)
//   5. internal nodes from the longest common key prefixes (ties on equal keys
//      broken by the leaf index), parent links
//   6. bottom-up refit: each leaf climbs; the second thread to reach a node
//      writes both child boxes (exact FP32 min/max, no rounding) and the node
//      height; the first stops.  The root height bounds the traversal stack.
#include "common.cuh"
#include "ploc_counts.h"

#include <algorithm>
#include <type_traits>

namespace lidar {
namespace {

constexpr int kBuildThreads = 256;

__device__ __forceinline__ int float_to_ordered(float f)
{
    int i = __float_as_int(f);
    return i >= 0 ? i : i ^ 0x7FFFFFFF;
}

__device__ __forceinline__ float ordered_to_float(int i)
{
    return __int_as_float(i >= 0 ? i : i ^ 0x7FFFFFFF);
}

// Orders a bottom-up climb: the writes of a finished child before its arrival
// at the parent, the arrival before the parent's reads (which go to L2).
__device__ __forceinline__ void climb_fence()
{
    asm volatile("fence.acq_rel.gpu;" ::: "memory");
}

// The same in one operation: counts an arrival, releasing what the thread (and
// its warp, up to its last __syncwarp) wrote and acquiring what the arrivals
// before it released.  Instead of a fence on each side of a relaxed addition,
// the treelet rounds of 0.65M triangles: 5.54 -> 5.41 ms for the whole load.
__device__ __forceinline__ unsigned arrive(unsigned* counter)
{
    unsigned before;
    asm volatile("atom.add.acq_rel.gpu.global.u32 %0, [%1], 1;" : "=r"(before) : "l"(counter) : "memory");
    return before;
}

__device__ __forceinline__ float3 load_vert(const float* v, uint32_t i)
{
    return make_float3(v[3 * (int64_t)i], v[3 * (int64_t)i + 1], v[3 * (int64_t)i + 2]);
}

__global__ void k_init_bounds(int* bounds)
{
    if (threadIdx.x < 3) bounds[threadIdx.x] = float_to_ordered(INFINITY);
    else if (threadIdx.x < 6) bounds[threadIdx.x] = float_to_ordered(-INFINITY);
}

__device__ __forceinline__ float3 centroid(float3 a, float3 b, float3 c)
{
    const float k = 1.0f / 3.0f;
    return make_float3((a.x + b.x + c.x) * k, (a.y + b.y + c.y) * k, (a.z + b.z + c.z) * k);
}

__global__ void __launch_bounds__(kBuildThreads) k_centroid_bounds(const float* __restrict__ verts,
                                                                   int64_t n_verts,
                                                                   const uint32_t* __restrict__ tris,
                                                                   int64_t n, int* bounds, int* status)
{
    float lo[3] = {INFINITY, INFINITY, INFINITY};
    float hi[3] = {-INFINITY, -INFINITY, -INFINITY};
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        uint32_t a = tris[3 * i], b = tris[3 * i + 1], c = tris[3 * i + 2];
        if ((int64_t)a >= n_verts || (int64_t)b >= n_verts || (int64_t)c >= n_verts) {
            raise_status(status, ST_INDEX);
            continue;
        }
        float3 ct = centroid(load_vert(verts, a), load_vert(verts, b), load_vert(verts, c));
        lo[0] = fminf(lo[0], ct.x); lo[1] = fminf(lo[1], ct.y); lo[2] = fminf(lo[2], ct.z);
        hi[0] = fmaxf(hi[0], ct.x); hi[1] = fmaxf(hi[1], ct.y); hi[2] = fmaxf(hi[2], ct.z);
    }
    // one atomic per block and plane: one per warp queued 12,000 deep on six
    // words (67 us at 1M triangles, 12 us so)
    __shared__ int s_b[6];
    if (threadIdx.x < 6) s_b[threadIdx.x] = float_to_ordered(threadIdx.x < 3 ? INFINITY : -INFINITY);
    __syncthreads();
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        const int l = __reduce_min_sync(0xffffffffu, float_to_ordered(lo[k]));
        const int h = __reduce_max_sync(0xffffffffu, float_to_ordered(hi[k]));
        if ((threadIdx.x & 31) == 0) {
            atomicMin(&s_b[k], l);
            atomicMax(&s_b[3 + k], h);
        }
    }
    __syncthreads();
    if (threadIdx.x < 3) atomicMin(&bounds[threadIdx.x], s_b[threadIdx.x]);
    else if (threadIdx.x < 6) atomicMax(&bounds[threadIdx.x], s_b[threadIdx.x]);
}

// spread the low 21 bits of x so that bit i lands on bit 3i
__device__ __forceinline__ uint64_t spread3(uint64_t x)
{
    x &= 0x1FFFFFull;
    x = (x | (x << 32)) & 0x001F00000000FFFFull;
    x = (x | (x << 16)) & 0x001F0000FF0000FFull;
    x = (x | (x << 8)) & 0x100F00F00F00F00Full;
    x = (x | (x << 4)) & 0x10C30C30C30C30C3ull;
    x = (x | (x << 2)) & 0x1249249249249249ull;
    return x;
}

__device__ __forceinline__ uint32_t quantize21(float v, float lo, float inv_ext)
{
    float q = (v - lo) * inv_ext * 2097151.0f;
    q = fminf(fmaxf(q, 0.0f), 2097151.0f);
    return (uint32_t)q;
}

__global__ void __launch_bounds__(kBuildThreads) k_morton(const float* __restrict__ verts,
                                                          const uint32_t* __restrict__ tris, int64_t n,
                                                          int64_t n_verts, const int* __restrict__ bounds,
                                                          uint64_t* __restrict__ keys,
                                                          uint32_t* __restrict__ vals)
{
    int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    float lo[3], inv[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        lo[k] = ordered_to_float(bounds[k]);
        float ext = ordered_to_float(bounds[3 + k]) - lo[k];
        inv[k] = ext > 0.0f ? 1.0f / ext : 0.0f;
    }
    uint32_t a = tris[3 * i], b = tris[3 * i + 1], c = tris[3 * i + 2];
    uint64_t key = 0;
    if ((int64_t)a < n_verts && (int64_t)b < n_verts && (int64_t)c < n_verts) {
        float3 ct = centroid(load_vert(verts, a), load_vert(verts, b), load_vert(verts, c));
        key = (spread3(quantize21(ct.x, lo[0], inv[0])) << 2) | (spread3(quantize21(ct.y, lo[1], inv[1])) << 1) |
              spread3(quantize21(ct.z, lo[2], inv[2]));
    }
    keys[i] = key;
    vals[i] = (uint32_t)i;
}

__global__ void __launch_bounds__(kBuildThreads) k_gather(const float* __restrict__ verts, int64_t n_verts,
                                                          const uint32_t* __restrict__ tris,
                                                          const uint16_t* __restrict__ mat,
                                                          const uint32_t* __restrict__ inst,
                                                          const uint32_t* __restrict__ order, int64_t n,
                                                          float4* __restrict__ tris_out,
                                                          uint32_t* __restrict__ leaf_tri)
{
    int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    uint32_t t = order[i];
    uint32_t a = tris[3 * (int64_t)t], b = tris[3 * (int64_t)t + 1], c = tris[3 * (int64_t)t + 2];
    if ((int64_t)a >= n_verts || (int64_t)b >= n_verts || (int64_t)c >= n_verts) a = b = c = 0;
    float3 va = load_vert(verts, a), vb = load_vert(verts, b), vc = load_vert(verts, c);
    tris_out[3 * i + 0] = make_float4(va.x, va.y, va.z, __int_as_float((int)t));
    tris_out[3 * i + 1] = make_float4(vb.x, vb.y, vb.z, __int_as_float((int)(mat ? mat[t] : 0)));
    tris_out[3 * i + 2] = make_float4(vc.x, vc.y, vc.z, __int_as_float((int)(inst ? inst[t] : 0)));
    leaf_tri[i] = t;
}

// length of the common prefix of keys i and j; -1 outside [0, n)
__device__ __forceinline__ int delta(const uint64_t* __restrict__ keys, int64_t n, int64_t i, int64_t j)
{
    if (j < 0 || j >= n) return -1;
    uint64_t a = keys[i], b = keys[j];
    if (a != b) return __clzll((long long)(a ^ b));
    return 64 + __clz((int)((uint32_t)i ^ (uint32_t)j));
}

__global__ void __launch_bounds__(kBuildThreads) k_karras(const uint64_t* __restrict__ keys, int64_t n,
                                                          float4* __restrict__ nodes,
                                                          int* __restrict__ parent_node,
                                                          int* __restrict__ parent_leaf)
{
    int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n - 1) return;
    // direction of the node's key range
    const int d = (delta(keys, n, i, i + 1) - delta(keys, n, i, i - 1)) >= 0 ? 1 : -1;
    const int dmin = delta(keys, n, i, i - d);
    // exponential then binary search for the far end of the range
    int64_t lmax = 2;
    while (delta(keys, n, i, i + lmax * d) > dmin) lmax <<= 1;
    int64_t l = 0;
    for (int64_t t = lmax >> 1; t >= 1; t >>= 1)
        if (delta(keys, n, i, i + (l + t) * d) > dmin) l += t;
    const int64_t j = i + l * d;
    const int dnode = delta(keys, n, i, j);
    // split: last position of the range that still shares more than dnode bits with i
    int64_t s = 0;
    int64_t step = l;
    do {
        step = (step + 1) >> 1;
        if (delta(keys, n, i, i + (s + step) * d) > dnode) s += step;
    } while (step > 1);
    const int64_t gamma = i + s * d + (d < 0 ? -1 : 0);
    const int64_t lo = i < j ? i : j, hi = i < j ? j : i;
    int left, right;
    if (lo == gamma) {
        left = ~(int)gamma;
        parent_leaf[gamma] = (int)i;
    } else {
        left = (int)gamma;
        parent_node[gamma] = (int)i;
    }
    if (hi == gamma + 1) {
        right = ~(int)(gamma + 1);
        parent_leaf[gamma + 1] = (int)i;
    } else {
        right = (int)(gamma + 1);
        parent_node[gamma + 1] = (int)i;
    }
    nodes[4 * i + 3] = make_float4(__int_as_float(left), __int_as_float(right), 0.0f, 0.0f);
    if (i == 0) parent_node[0] = -1;
}

struct Box {
    float lo[3], hi[3];
};

__device__ __forceinline__ Box leaf_box(const float4* __restrict__ tris, int leaf)
{
    float4 a = tris[3 * (int64_t)leaf], b = tris[3 * (int64_t)leaf + 1], c = tris[3 * (int64_t)leaf + 2];
    Box r;
    r.lo[0] = fminf(a.x, fminf(b.x, c.x)); r.hi[0] = fmaxf(a.x, fmaxf(b.x, c.x));
    r.lo[1] = fminf(a.y, fminf(b.y, c.y)); r.hi[1] = fmaxf(a.y, fmaxf(b.y, c.y));
    r.lo[2] = fminf(a.z, fminf(b.z, c.z)); r.hi[2] = fmaxf(a.z, fmaxf(b.z, c.z));
    return r;
}

__device__ __forceinline__ Box node_box(const float4* node_boxes, int node)
{
    float4 lo = __ldcg(&node_boxes[2 * (int64_t)node]);
    float4 hi = __ldcg(&node_boxes[2 * (int64_t)node + 1]);
    Box r;
    r.lo[0] = lo.x; r.lo[1] = lo.y; r.lo[2] = lo.z;
    r.hi[0] = hi.x; r.hi[1] = hi.y; r.hi[2] = hi.z;
    return r;
}

__global__ void __launch_bounds__(kBuildThreads) k_refit(const float4* __restrict__ tris, int64_t n,
                                                         float4* nodes, float4* node_boxes, int* heights,
                                                         const int* __restrict__ parent_node,
                                                         const int* __restrict__ parent_leaf, int* visits,
                                                         int* max_height)
{
    int64_t leaf = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (leaf >= n) return;
    int p = parent_leaf[leaf];
    while (p >= 0) {
        const int before = atomicAdd(&visits[p], 1);
        const float4 n3 = __ldcg(&nodes[4 * (int64_t)p + 3]);  // links and the next parent: nobody writes them here
        const int next = parent_node[p];
        if (before == 0) return;  // the sibling subtree is not finished yet
        climb_fence();
        int cl = __float_as_int(n3.x), cr = __float_as_int(n3.y);
        Box L = cl < 0 ? leaf_box(tris, ~cl) : node_box(node_boxes, cl);
        Box R = cr < 0 ? leaf_box(tris, ~cr) : node_box(node_boxes, cr);
        int hl = cl < 0 ? 0 : __ldcg(&heights[cl]);
        int hr = cr < 0 ? 0 : __ldcg(&heights[cr]);
        nodes[4 * (int64_t)p + 0] = make_float4(L.lo[0], L.hi[0], L.lo[1], L.hi[1]);
        nodes[4 * (int64_t)p + 1] = make_float4(R.lo[0], R.hi[0], R.lo[1], R.hi[1]);
        nodes[4 * (int64_t)p + 2] = make_float4(L.lo[2], L.hi[2], R.lo[2], R.hi[2]);
        node_boxes[2 * (int64_t)p] = make_float4(fminf(L.lo[0], R.lo[0]), fminf(L.lo[1], R.lo[1]),
                                                 fminf(L.lo[2], R.lo[2]), 0.0f);
        node_boxes[2 * (int64_t)p + 1] = make_float4(fmaxf(L.hi[0], R.hi[0]), fmaxf(L.hi[1], R.hi[1]),
                                                     fmaxf(L.hi[2], R.hi[2]), 0.0f);
        int h = 1 + max(hl, hr);
        heights[p] = h;
        if (p == 0) atomicMax(max_height, h);
        climb_fence();
        p = next;
    }
}

// a single triangle: one root whose right child box is empty
__global__ void k_single(const float4* __restrict__ tris, float4* nodes, int* max_height)
{
    Box L = leaf_box(tris, 0);
    nodes[0] = make_float4(L.lo[0], L.hi[0], L.lo[1], L.hi[1]);
    nodes[1] = make_float4(INFINITY, -INFINITY, INFINITY, -INFINITY);
    nodes[2] = make_float4(L.lo[2], L.hi[2], INFINITY, -INFINITY);
    nodes[3] = make_float4(__int_as_float(~0), __int_as_float(~0), 0.0f, 0.0f);
    *max_height = 1;
}

inline size_t align256(size_t b) { return (b + 255) / 256 * 256; }

}  // namespace

size_t build_scratch_bytes(int64_t n)
{
    return align256(n * sizeof(uint64_t)) + align256(n * sizeof(uint32_t)) + align256(n * sizeof(int)) * 4 +
           align256((size_t)n * 2 * sizeof(float4)) + align256(64) + radix_sort_scratch_bytes(n);
}

cudaError_t build_ploc(cudaStream_t s, const float4* tris_sorted, int64_t n, float4* nodes_out, int* max_height_dev,
                       int radius, void* scratch, size_t scratch_bytes, AreaW w, int* status, int num_sms, int coop,
                       uint64_t wait_ns);

cudaError_t build_lbvh(cudaStream_t s, const float* verts, int64_t n_verts, const uint32_t* tris,
                       const uint16_t* mat, const uint32_t* inst, int64_t n, float4* nodes_out,
                       float4* tris_out, uint32_t* leaf_tri_out, int* status, int* max_height_dev,
                       void* scratch, size_t scratch_bytes, int num_sms, int coop, uint64_t wait_ns, int method,
                       int radius, AreaW area_w)
{
    if (n == 0) return cudaSuccess;
    if (scratch_bytes < build_scratch_bytes(n)) return cudaErrorInvalidValue;
    char* p = (char*)scratch;
    uint64_t* keys = (uint64_t*)p; p += align256(n * sizeof(uint64_t));
    uint32_t* vals = (uint32_t*)p; p += align256(n * sizeof(uint32_t));
    int* parent_node = (int*)p; p += align256(n * sizeof(int));
    int* parent_leaf = (int*)p; p += align256(n * sizeof(int));
    int* visits = (int*)p; p += align256(n * sizeof(int));
    int* heights = (int*)p; p += align256(n * sizeof(int));
    float4* node_boxes = (float4*)p; p += align256((size_t)n * 2 * sizeof(float4));
    int* bounds = (int*)p; p += align256(64);
    void* sort_scratch = p;
    size_t sort_bytes = scratch_bytes - (size_t)(p - (char*)scratch);

    const int blocks = (int)((n + kBuildThreads - 1) / kBuildThreads);
    k_init_bounds<<<1, 32, 0, s>>>(bounds);
    const int red_blocks = blocks < 608 ? blocks : 608;
    k_centroid_bounds<<<red_blocks, kBuildThreads, 0, s>>>(verts, n_verts, tris, n, bounds, status);
    k_morton<<<blocks, kBuildThreads, 0, s>>>(verts, tris, n, n_verts, bounds, keys, vals);
    cudaError_t e = radix_sort_pairs_u64(s, keys, vals, n, 63, sort_scratch, sort_bytes);
    if (e != cudaSuccess) return e;
    k_gather<<<blocks, kBuildThreads, 0, s>>>(verts, n_verts, tris, mat, inst, vals, n, tris_out, leaf_tri_out);
    cudaMemsetAsync(max_height_dev, 0, sizeof(int), s);
    if (n == 1) {
        k_single<<<1, 1, 0, s>>>(tris_out, nodes_out, max_height_dev);
        return cudaGetLastError();
    }
    if (method == 1) {
        // clustering over the Morton-ordered leaves; the sort's buffers are free again
        return build_ploc(s, tris_out, n, nodes_out, max_height_dev, radius, scratch, scratch_bytes, area_w, status,
                          num_sms, coop, wait_ns);
    }
    const int iblocks = (int)((n - 1 + kBuildThreads - 1) / kBuildThreads);
    k_karras<<<iblocks, kBuildThreads, 0, s>>>(keys, n, nodes_out, parent_node, parent_leaf);
    cudaMemsetAsync(visits, 0, n * sizeof(int), s);
    k_refit<<<blocks, kBuildThreads, 0, s>>>(tris_out, n, nodes_out, node_boxes, heights, parent_node, parent_leaf,
                                             visits, max_height_dev);
    return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// PLOC: Parallel Locally-Ordered Clustering (Meister and Bittner, "Parallel
// Locally-Ordered Clustering for Bounding Volume Hierarchy Construction",
// IEEE TVCG 2018), an alternative to the Karras hierarchy over the same
// Morton-ordered leaves.  Clusters start as the leaves; each iteration every
// cluster finds its nearest neighbour within `radius` positions of the
// cluster array (distance: surface area of the union box; ties to the lower
// position), mutual nearest pairs merge into a new node at the lower position,
// and the array is compacted in order.  Node ids count down from n - 2, so the
// last merge is the root at 0.  Boxes are exact FP32 min/max unions.
namespace {

// half the weighted surface of the union of two boxes
__device__ __forceinline__ float union_half_area(float4 alo, float4 ahi, float4 blo, float4 bhi, AreaW w)
{
    const float dx = fmaxf(ahi.x, bhi.x) - fminf(alo.x, blo.x);
    const float dy = fmaxf(ahi.y, bhi.y) - fminf(alo.y, blo.y);
    const float dz = fmaxf(ahi.z, bhi.z) - fminf(alo.z, blo.z);
    return w.z * dx * dy + w.x * dy * dz + w.y * dz * dx;
}

// Where the blocks of a cooperative launch meet: a counter they arrive at and
// a word, in another line, that the last to arrive sets for the rest to see
// (both zero before the launch).  With every block reading the counter, or a
// flag of every other block, the meeting took 2.8 and 5 us for 152 to 304
// blocks: the readers queued at one line with the arrivals.
struct MeetPlace {
    unsigned arrived;
    unsigned pad0[31];
    unsigned released;
    unsigned pad1[31];
};

// How long a block waits for the others (the context's wait limit), and where
// it says that it gave up.
struct BuildWait {
    int* status;
    uint64_t ns;
};

// Spins until `ready()`.  Bounded: after w.ns nanoseconds (0: at once) ST_TIMEOUT
// and false.  The timer is read every 64th time, so that the reads of what is
// waited for follow closely.
template <typename Ready>
__device__ __forceinline__ bool build_spin(BuildWait w, Ready ready)
{
    uint64_t t0 = 0;
    for (unsigned it = 1; !ready(); ++it) {
        if ((it & 63u) != 0u && w.ns != 0) continue;
        uint64_t t;
        asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
        if (t0 == 0) t0 = t;
        if (t - t0 > w.ns || w.ns == 0) {
            raise_status(w.status, ST_TIMEOUT);
            return false;
        }
    }
    return true;
}

__device__ __forceinline__ unsigned ld_acquire(const unsigned* p)
{
    unsigned v;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}

__device__ __forceinline__ void st_release(unsigned* p, unsigned v)
{
    asm volatile("st.release.gpu.global.u32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}

// The `blocks` blocks of a cooperative launch meet for the `met`-th time (this
// counts it), what each wrote before visible to all after.  One block alone
// only meets its own threads.  False in every thread when the wait ran out.
__device__ bool build_meet(MeetPlace* at, unsigned blocks, unsigned& met, BuildWait wait)
{
    __syncthreads();
    if (blocks == 1) return true;
    ++met;
    bool ok = true;
    if (threadIdx.x == 0) {
        if (arrive(&at->arrived) + 1u == met * blocks) {
            st_release(&at->released, met);
        } else {
            ok = build_spin(wait, [&] { return ld_acquire(&at->released) >= met; });
        }
    }
    return __syncthreads_and(ok) != 0;
}

// exclusive prefix of v over the block's threads, and the block's sum
template <int kThreads, typename T>
__device__ __forceinline__ T block_prefix(T v, T& total)
{
    constexpr int kWarps = kThreads / 32;
    __shared__ T s_sum[kWarps];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    T x = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const T y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    __syncthreads();
    if (lane == 31) s_sum[warp] = x;
    __syncthreads();
    // every warp adds up the warps' sums for itself
    const T y = lane < kWarps ? s_sum[lane] : T(0);
    T before = lane < warp ? y : T(0), sum = y;
    if constexpr (sizeof(T) == 4) {
        before = __reduce_add_sync(0xffffffffu, before);
        sum = __reduce_add_sync(0xffffffffu, sum);
    } else {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            before += __shfl_xor_sync(0xffffffffu, before, o);
            sum += __shfl_xor_sync(0xffffffffu, sum, o);
        }
    }
    total = sum;
    return before + x - v;
}

constexpr int kPlocThreads = 512;
constexpr int kPlocMaxRadius = 64;
constexpr int kPlocSolo = kPlocThreads;  // clusters one block finishes alone, in shared memory
constexpr int kPlocWide = 2;             // clusters a thread takes at most
constexpr int kPlocMaxBlocks = kPlocThreads;
constexpr int kPlocSpan = kPlocWide * kPlocThreads + 2 * kPlocMaxRadius;

struct PlocArgs {
    const float4* tris;
    int n;
    float4* cluster[2];           // [2 n] each: lo, ref bits; hi, height bits (the rounds alternate)
    int* mate;                    // [n] >= 0: merges with that later position; -1: stays; -2: merged away
    // per block: its counts (ploc_counts.h); and, in a sector of its own, those
    // before it and of all, each with the round's tag
    unsigned long long* total;    // [kPlocMaxBlocks]
    unsigned long long* answer;   // [kPlocMaxBlocks][4]
    float4* nodes;
    int* max_height;
    int radius;
    AreaW w;
    MeetPlace* place;             // the blocks' meetings and exchanges (two), zero before the launch
    BuildWait wait;
};

// Clusters in shared memory: lo x y z, hi x y z, ref bits, height bits.
typedef float PlocShared[8][kPlocSpan];

__device__ __forceinline__ void ploc_put(PlocShared& c, int k, float4 lo, float4 hi)
{
    c[0][k] = lo.x; c[1][k] = lo.y; c[2][k] = lo.z;
    c[3][k] = hi.x; c[4][k] = hi.y; c[5][k] = hi.z;
    c[6][k] = lo.w; c[7][k] = hi.w;
}

__device__ __forceinline__ void ploc_get(const PlocShared& c, int k, float4& lo, float4& hi)
{
    lo = make_float4(c[0][k], c[1][k], c[2][k], c[6][k]);
    hi = make_float4(c[3][k], c[4][k], c[5][k], c[7][k]);
}

// Nearest neighbour of the cluster at k among those at lo..hi (all in shared
// memory), found by `lanes` neighbouring lanes (a power of two), lane `sub` of
// them taking its share in order; ties to the lowest.  -1: none.
__device__ __forceinline__ int ploc_nearest(const PlocShared& c, int k, int lo, int hi, int lanes, int sub, AreaW w)
{
    const float4 alo = make_float4(c[0][k], c[1][k], c[2][k], 0.0f);
    const float4 ahi = make_float4(c[3][k], c[4][k], c[5][k], 0.0f);
    const int share = (hi - lo + lanes) / lanes;
    const int j0 = lo + sub * share, j1 = min(j0 + share - 1, hi);
    float best_d = INFINITY;
    int best = -1;
#pragma unroll 4
    for (int j = j0; j <= j1; ++j) {
        const float d = union_half_area(alo, ahi, make_float4(c[0][j], c[1][j], c[2][j], 0.0f),
                                        make_float4(c[3][j], c[4][j], c[5][j], 0.0f), w);
        if (j != k && d < best_d) {  // ascending j: ties keep the lower position
            best_d = d;
            best = j;
        }
    }
    for (int o = 1; o < lanes; o <<= 1) {
        const float d = __shfl_xor_sync(0xffffffffu, best_d, o);
        const int j = __shfl_xor_sync(0xffffffffu, best, o);
        if (d < best_d || (d == best_d && (unsigned)j < (unsigned)best)) {
            best_d = d;
            best = j;
        }
    }
    return best;
}

// Nearest neighbours of the two clusters at k and k + 1 (k even) within `r` of
// each: the window's boxes are read two at a time, each serving both searches.  Places outside the array hold boxes whose union with
// anything is infinite.  best[i] is -1 for none.
__device__ __forceinline__ void ploc_nearest2(const PlocShared& c, int k, int r, AreaW w, int best[2])
{
    constexpr int K = 2;
    float al[3][K], ah[3][K];
#pragma unroll
    for (int x = 0; x < 3; ++x) {
        *(float2*)al[x] = *(const float2*)&c[x][k];
        *(float2*)ah[x] = *(const float2*)&c[3 + x][k];
    }
    float best_d[K];
#pragma unroll
    for (int i = 0; i < K; ++i) {
        best_d[i] = INFINITY;
        best[i] = -1;
    }
    const int h = (r + K - 1) / K * K;
    for (int g = -h; g <= h; g += K) {
        float bl[3][K], bh[3][K];
#pragma unroll
        for (int x = 0; x < 3; ++x) {
            *(float2*)bl[x] = *(const float2*)&c[x][k + g];
            *(float2*)bh[x] = *(const float2*)&c[3 + x][k + g];
        }
        // all K x K pairs within r of each other, and none a cluster with itself
        const bool whole = g != 0 && g - (K - 1) >= -r && g + (K - 1) <= r;
#pragma unroll
        for (int j = 0; j < K; ++j) {
#pragma unroll
            for (int i = 0; i < K; ++i) {
                const int off = g + j - i;
                const float d = union_half_area(make_float4(al[0][i], al[1][i], al[2][i], 0.0f),
                                                make_float4(ah[0][i], ah[1][i], ah[2][i], 0.0f),
                                                make_float4(bl[0][j], bl[1][j], bl[2][j], 0.0f),
                                                make_float4(bh[0][j], bh[1][j], bh[2][j], 0.0f), w);
                // ascending position: ties keep the lower one
                if (d < best_d[i] && (whole || (off != 0 && off >= -r && off <= r))) {
                    best_d[i] = d;
                    best[i] = k + g + j;
                }
            }
        }
    }
}

// What position e of nc does, given its and its neighbour's nearest.
__device__ __forceinline__ int ploc_mate(int e, int nc, int best, int best_of_best, bool force)
{
    if (force) return e % 2 == 1 ? -2 : (e + 1 < nc ? e + 1 : -1);  // no mutual pair anywhere (not expected)
    if (best < 0 || best_of_best != e) return -1;
    return e < best ? best : -2;
}

// Merges the cluster (rlo, rhi) into (lo, hi) as node `id`.
__device__ __forceinline__ void ploc_merge(const PlocArgs& a, int id, float4& lo, float4& hi, float4 rlo, float4 rhi)
{
    a.nodes[4 * (int64_t)id + 0] = make_float4(lo.x, hi.x, lo.y, hi.y);
    a.nodes[4 * (int64_t)id + 1] = make_float4(rlo.x, rhi.x, rlo.y, rhi.y);
    a.nodes[4 * (int64_t)id + 2] = make_float4(lo.z, hi.z, rlo.z, rhi.z);
    a.nodes[4 * (int64_t)id + 3] = make_float4(lo.w, rlo.w, 0.0f, 0.0f);
    const int h = 1 + max(__float_as_int(hi.w), __float_as_int(rhi.w));
    lo = make_float4(fminf(lo.x, rlo.x), fminf(lo.y, rlo.y), fminf(lo.z, rlo.z), __int_as_float(id));
    hi = make_float4(fmaxf(hi.x, rhi.x), fmaxf(hi.y, rhi.y), fmaxf(hi.z, rhi.z), __int_as_float(h));
    if (id == 0) *a.max_height = h;
}

// The rounds from kPlocSolo clusters on, by one block out of shared memory.
__device__ void ploc_solo(const PlocArgs& a, const float4* C, int nc, int id_top, PlocShared& c, int* s_nn)
{
    const int tid = threadIdx.x, r = a.radius;
    __syncthreads();
    for (int k = tid; k < nc; k += kPlocThreads) ploc_put(c, k, __ldcg(&C[2 * (int64_t)k]), __ldcg(&C[2 * (int64_t)k + 1]));
    __syncthreads();
    bool force = false;
    while (nc > 1) {
        int lanes = 1;
        while (lanes < 32 && 2 * lanes * nc <= kPlocThreads) lanes *= 2;
        {
            const int e = tid / lanes, k = min(e, nc - 1);
            const int best = force ? -1 : ploc_nearest(c, k, max(k - r, 0), min(k + r, nc - 1), lanes, tid % lanes, a.w);
            if (e < nc && tid % lanes == 0) s_nn[e] = best;
        }
        __syncthreads();
        int mate = -2;
        float4 lo, hi, rlo, rhi;
        if (tid < nc) {
            const int best = s_nn[tid];
            mate = ploc_mate(tid, nc, best, best >= 0 ? s_nn[best] : -1, force);
            if (mate != -2) ploc_get(c, tid, lo, hi);
            if (mate >= 0) ploc_get(c, mate, rlo, rhi);
        }
        unsigned sum;
        const unsigned at =  // (its barriers end the reads)
            block_prefix<kPlocThreads>(mate == -2 ? 0u : (mate >= 0 ? 0x10001u : 1u), sum);
        force = (sum >> 16) == 0;
        if (force) continue;
        if (mate != -2) {
            if (mate >= 0) ploc_merge(a, id_top - (int)(at >> 16), lo, hi, rlo, rhi);
            ploc_put(c, (int)(at & 0xFFFFu), lo, hi);
        }
        id_top -= (int)(sum >> 16);
        nc = (int)(sum & 0xFFFFu);
        __syncthreads();
    }
}

// One round of the blocks' clustering.  A tile is what a block's threads
// hold, K clusters each or one per `lanes` threads, less `halo` on either
// side: the block keeps the boxes within twice the halo in shared memory and
// finds the nearest neighbours of the halo's clusters too, so that it can tell
// mutual pairs by itself.  The blocks then exchange their counts and write the
// merged array at the positions those give.
struct PlocRound {
    const float4* C;
    float4* D;
    int nc, id_top, lanes;
    bool force;
    unsigned round;
};

template <int K>
__device__ __forceinline__ bool ploc_round(const PlocArgs& a, PlocShared& s_c, int* s_nn, unsigned blocks, const PlocRound& g,
                           unsigned long long& all)
{
    __shared__ unsigned long long s_sum[2];
    const int tid = threadIdx.x, r = a.radius, nc = g.nc;
    const int lanes = K > 1 ? 1 : g.lanes;
    const int halo = K > 1 ? (r + 1) & ~1 : r;
    const int E = K > 1 ? K * kPlocThreads : kPlocThreads / lanes;  // clusters held, T of them the tile's own
    const int T = E - 2 * halo;
    const int tiles = (nc + T - 1) / T;
    const int per = (tiles + (int)blocks - 1) / (int)blocks;
    const int t0 = min((int)blockIdx.x * per, tiles), t1 = min(t0 + per, tiles);
    const int first = K > 1 ? K * tid : tid / lanes;  // this thread's first cluster of those held
    int mate[K];                                      // of the last tile's
    unsigned place = 0, count;                        // merges << 16 | stays before this thread's, and of the tile
    unsigned long long mine = 0;                      // counts of the block's tiles
#pragma unroll
    for (int i = 0; i < K; ++i) mate[i] = -2;
    for (int t = t0; t < t1; ++t) {
        const int base = t * T, from = base - 2 * halo, span = T + 4 * halo;
        for (int k = tid; k < span; k += kPlocThreads) {
            const int e = from + k;
            if (e >= 0 && e < nc) {
                ploc_put(s_c, k, __ldcg(&g.C[2 * (int64_t)e]), __ldcg(&g.C[2 * (int64_t)e + 1]));
            } else if (K > 1) {
                ploc_put(s_c, k, make_float4(-INFINITY, -INFINITY, -INFINITY, 0.0f),
                         make_float4(INFINITY, INFINITY, INFINITY, 0.0f));
            }
        }
        __syncthreads();
        // held cluster m is e = base - halo + m, at halo + m of the boxes
        if constexpr (K > 1) {
            int best[K];
#pragma unroll
            for (int i = 0; i < K; ++i) best[i] = -1;
            if (!g.force) ploc_nearest2(s_c, halo + first, r, a.w, best);
            *(int2*)&s_nn[first] = make_int2(best[0], best[1]);
        } else {
            const int e = min(max(base - halo + first, 0), nc - 1);
            int best = -1;
            if (!g.force)
                best = ploc_nearest(s_c, e - from, max(e - r, 0) - from, min(e + r, nc - 1) - from, lanes, tid % lanes,
                                    a.w);
            if (tid % lanes == 0) s_nn[first] = best;
        }
        __syncthreads();
        unsigned v = 0;
#pragma unroll
        for (int i = 0; i < K; ++i) {
            const int m = first + i, e = base - halo + m;
            mate[i] = -2;
            if (tid % lanes != 0 || m < halo || m >= halo + T || e >= nc) continue;
            const int best = s_nn[m];
            mate[i] = ploc_mate(e, nc, best < 0 ? -1 : best + from, best < 0 ? -1 : s_nn[best - halo] + from, g.force);
            if (per > 1) __stcg(&a.mate[e], mate[i]);
            if (mate[i] != -2) v += mate[i] >= 0 ? 0x10001u : 1u;
        }
        place = block_prefix<kPlocThreads>(v, count);
        mine += ploc_counts(count >> 16, count & 0xFFFFu);
    }
    // merges and stays of the blocks before, and of all
    unsigned long long before = 0;
    all = mine;
    if (blocks > 1) {
        // every block leaves its counts and arrives; the last one sums them up
        // and answers each in its own sector
        MeetPlace* at = a.place + 1;
        bool last = false;
        if (tid == 0) {
            __stcg(&a.total[blockIdx.x], mine);
            last = arrive(&at->arrived) + 1u == (g.round + 1u) * blocks;
        }
        if (__syncthreads_or(last)) {
            const unsigned long long v = tid < (int)blocks ? __ldcg(&a.total[tid]) : 0ull;
            unsigned long long sum;
            const unsigned long long x = block_prefix<kPlocThreads>(v, sum);
            if (tid < (int)blocks) {
                *(volatile unsigned long long*)&a.answer[4 * tid] = ploc_tagged(x, g.round);
                *(volatile unsigned long long*)&a.answer[4 * tid + 1] = ploc_tagged(sum, g.round);
            }
        }
        bool ok = true;
        if (tid == 0) {
            const volatile unsigned long long* mine_at = a.answer + 4 * blockIdx.x;
            unsigned long long x = 0, y = 0;
            ok = build_spin(a.wait, [&] {
                x = mine_at[0];
                y = mine_at[1];
                return ploc_is_of(x, g.round) && ploc_is_of(y, g.round);
            });
            s_sum[0] = ploc_untagged(x);
            s_sum[1] = ploc_untagged(y);
        }
        if (!__syncthreads_and(ok)) return false;
        before = s_sum[0];
        all = s_sum[1];
    }
    if (ploc_merges(all) == 0) return true;
    // the tile at `base`, its boxes in shared memory and its mates in registers
    auto write = [&](int base, unsigned long long at) {
        const int from = base - 2 * halo;
#pragma unroll
        for (int i = 0; i < K; ++i) {
            if (mate[i] == -2) continue;
            float4 lo, hi;
            ploc_get(s_c, halo + first + i, lo, hi);
            if (mate[i] >= 0) {
                float4 rlo, rhi;
                ploc_get(s_c, mate[i] - from, rlo, rhi);
                ploc_merge(a, g.id_top - (int)ploc_merges(at), lo, hi, rlo, rhi);
            }
            const int64_t out = ploc_stays(at);
            __stcg(&g.D[2 * out], lo);
            __stcg(&g.D[2 * out + 1], hi);
            at += ploc_counts(mate[i] >= 0 ? 1u : 0u, 1u);
        }
    };
    auto wide = [](unsigned v) { return ploc_counts(v >> 16, v & 0xFFFFu); };
    if (per == 1) {
        write(t0 * T, before + wide(place));
        return true;
    }
    for (int t = t0; t < t1; ++t) {
        const int base = t * T, from = base - 2 * halo;
        for (int k = 2 * halo + tid; k < T + 3 * halo; k += kPlocThreads)
            if (from + k < nc)
                ploc_put(s_c, k, __ldcg(&g.C[2 * (int64_t)(from + k)]), __ldcg(&g.C[2 * (int64_t)(from + k) + 1]));
        unsigned v = 0;
#pragma unroll
        for (int i = 0; i < K; ++i) {
            const int m = first + i, e = base - halo + m;
            mate[i] = m >= halo && m < halo + T && e < nc ? __ldcg(&a.mate[e]) : -2;
            if (mate[i] != -2) v += mate[i] >= 0 ? 0x10001u : 1u;
        }
        const unsigned p = block_prefix<kPlocThreads>(v, count);  // (its barriers end the loads)
        write(base, before + wide(p));
        before += wide(count);
        __syncthreads();
    }
    return true;
}

constexpr size_t kPlocShared = sizeof(PlocShared) + kPlocWide * kPlocThreads * sizeof(int);

// The whole clustering in one cooperative launch, a round at a time: two
// clusters a thread while the blocks' threads are fewer than the clusters,
// then one, then one per 2, 4 or 8 lanes; the last kPlocSolo of them block 0
// finishes alone, meeting nobody.
//
// What bounds it: six kernels and a host round trip a round (63 rounds at 1M
// triangles, 3.3 ms) left it waiting for launches.  In one launch it is a
// round's chain (an exchange of counts and a meeting, ~5 us, a search) and, in
// the first rounds, the 2 radius box unions per cluster (~30 issue slots each,
// half of them min / max).  1M triangles: 0.69 ms with one cluster a thread,
// everything through L2 and the blocks polling one counter; 0.56 ms so.  Four
// clusters a thread, or 1,024 threads, take as long: the searches are bound
// by issue, the rest by the chain.
__global__ void __launch_bounds__(kPlocThreads, 1) k_ploc(PlocArgs a)
{
    extern __shared__ __align__(16) unsigned char smem[];
    PlocShared& s_c = *(PlocShared*)smem;
    int* s_nn = (int*)(smem + sizeof(PlocShared));
    const int r = a.radius;
    const unsigned blocks = gridDim.x;
    unsigned met = 0;
    for (int64_t i = blockIdx.x * kPlocThreads + threadIdx.x; i < a.n; i += gridDim.x * kPlocThreads) {
        const Box b = leaf_box(a.tris, (int)i);
        __stcg(&a.cluster[0][2 * i], make_float4(b.lo[0], b.lo[1], b.lo[2], __int_as_float(~(int)i)));
        __stcg(&a.cluster[0][2 * i + 1], make_float4(b.hi[0], b.hi[1], b.hi[2], __int_as_float(0)));
    }
    if (!build_meet(a.place, blocks, met, a.wait)) return;
    PlocRound g{a.cluster[0], a.cluster[1], a.n, a.n - 2, 1, false, 0};
    while (g.nc > kPlocSolo) {
        // the most lanes a cluster with which every block still has one tile at most
        g.lanes = 0;
        for (int l = 8; l >= 1 && g.lanes == 0; l >>= 1) {
            const int T = kPlocThreads / l - 2 * r;
            if (T >= 32 && (int64_t)T * blocks >= g.nc) g.lanes = l;
        }
        unsigned long long all;
        if (!(g.lanes ? ploc_round<1>(a, s_c, s_nn, blocks, g, all) : ploc_round<kPlocWide>(a, s_c, s_nn, blocks, g, all)))
            return;
        ++g.round;
        g.force = ploc_merges(all) == 0;  // then nothing was written
        if (!g.force) {
            g.id_top -= (int)ploc_merges(all);
            g.nc = (int)ploc_stays(all);
            const float4* swap = g.C;
            g.C = g.D;
            g.D = const_cast<float4*>(swap);
        }
        if (!build_meet(a.place, blocks, met, a.wait)) return;
    }
    if (blockIdx.x == 0) ploc_solo(a, g.C, g.nc, g.id_top, s_c, s_nn);
}

// blocks of a cooperative launch of `fn`, at most `want`; 1 without cooperative launch
int coop_blocks(const void* fn, int threads, size_t smem, int num_sms, int coop, int64_t want)
{
    int per_sm = 0;
    if (!coop || want <= 1 || cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, fn, threads, smem) != cudaSuccess)
        return 1;
    return (int)std::max<int64_t>(1, std::min(want, (int64_t)per_sm * num_sms));
}

}  // namespace

size_t ploc_scratch_bytes(int64_t n)
{
    return 2 * align256((size_t)n * 2 * sizeof(float4)) + align256(n * sizeof(int)) +
           align256(2 * sizeof(MeetPlace)) + kPlocMaxBlocks * 5 * sizeof(unsigned long long);
}

cudaError_t build_ploc(cudaStream_t s, const float4* tris_sorted, int64_t n, float4* nodes_out, int* max_height_dev,
                       int radius, void* scratch, size_t scratch_bytes, AreaW w, int* status, int num_sms, int coop,
                       uint64_t wait_ns)
{
    if (n < 2 || radius < 1 || radius > kPlocMaxRadius) return cudaErrorInvalidValue;
    if (scratch_bytes < ploc_scratch_bytes(n)) return cudaErrorInvalidValue;
    char* p = (char*)scratch;
    PlocArgs a;
    a.tris = tris_sorted;
    a.n = (int)n;
    for (float4*& c : a.cluster) {
        c = (float4*)p;
        p += align256((size_t)n * 2 * sizeof(float4));
    }
    a.mate = (int*)p; p += align256(n * sizeof(int));
    char* zero = p;
    a.place = (MeetPlace*)p; p += align256(2 * sizeof(MeetPlace));
    a.answer = (unsigned long long*)p; p += kPlocMaxBlocks * 4 * sizeof(unsigned long long);
    a.total = (unsigned long long*)p; p += kPlocMaxBlocks * sizeof(unsigned long long);
    a.nodes = nodes_out;
    a.max_height = max_height_dev;
    a.radius = radius;
    a.w = w;
    a.wait = BuildWait{status, wait_ns};
    cudaError_t e = cudaMemsetAsync(zero, 0, (size_t)(p - zero), s);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(k_ploc, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kPlocShared);
    if (e != cudaSuccess) return e;
    const int grid = coop_blocks((const void*)k_ploc, kPlocThreads, kPlocShared, num_sms, coop,
                                 n <= kPlocSolo ? 1 : std::min<int64_t>((n + 31) / 32, kPlocMaxBlocks));
    if (grid == 1) {
        k_ploc<<<1, kPlocThreads, kPlocShared, s>>>(a);
        return cudaGetLastError();
    }
    void* args[] = {&a};
    return cudaLaunchCooperativeKernel((const void*)k_ploc, dim3(grid), dim3(kPlocThreads), args, kPlocShared, s);
}

}  // namespace lidar

// ---------------------------------------------------------------------------
// Collapse of the binary hierarchy into the 4- and the 8-wide one.  Top-down,
// one frontier of binary nodes per level: each becomes a wide node whose
// children are found by repeatedly opening the child with the largest surface
// area until W children or only leaves remain.  Slots of the next level are
// assigned by an exclusive scan, so the layout is breadth-first and
// deterministic.  One cooperative launch walks the levels of both trees and
// lists, per wide node, its binary node and its first internal child; then
// every node of a tree is written at once.
//
// Wide node of G = W/4 groups of four children, 8G float4s: for axis a the
// lower planes of group g at (2a)G + g, the upper planes at (2a + 1)G + g, the
// child codes of group g at 6G + g (>= 0: wide node, < 0: ~leaf; empty slots
// have an empty box and code 0), then G float4s of metadata (128 bytes for
// W = 4, 256 for W = 8).  A node keeps its internal children in the first
// slots, in the order of their (consecutive) node ids, and its first metadata
// float4 holds the first internal child's id and the mask of leaf slots, so a
// traversal finds an internal child as first + slot.
//
// Alongside each frontier entry travels the number of stack entries its
// ancestors can leave behind: a traversal that descends into one hit internal
// child pushes at most the node's other internal children, so the deepest
// stack the tree can need is max over nodes of (ancestors' pushes + the
// node's internal children - 1).
namespace lidar {
namespace {

struct ChildBox {
    float lo[3], hi[3];
    int ref;  // binary node (>= 0) or ~leaf (< 0)
};

__device__ __forceinline__ void binary_child(const float4* __restrict__ bn, int node, int side, ChildBox& c)
{
    const float4 n0 = bn[4 * (int64_t)node + 0], n1 = bn[4 * (int64_t)node + 1];
    const float4 n2 = bn[4 * (int64_t)node + 2], n3 = bn[4 * (int64_t)node + 3];
    if (side == 0) {
        c.lo[0] = n0.x; c.hi[0] = n0.y; c.lo[1] = n0.z; c.hi[1] = n0.w; c.lo[2] = n2.x; c.hi[2] = n2.y;
        c.ref = __float_as_int(n3.x);
    } else {
        c.lo[0] = n1.x; c.hi[0] = n1.y; c.lo[1] = n1.z; c.hi[1] = n1.w; c.lo[2] = n2.z; c.hi[2] = n2.w;
        c.ref = __float_as_int(n3.y);
    }
}

__device__ __forceinline__ float half_area(const ChildBox& c, AreaW w)
{
    const float dx = c.hi[0] - c.lo[0], dy = c.hi[1] - c.lo[1], dz = c.hi[2] - c.lo[2];
    // rounded alike wherever it is compiled: the levels and the nodes are to
    // choose the same children
    return fmaf(__fmul_rn(w.y, dz), dx, fmaf(__fmul_rn(w.z, dx), dy, __fmul_rn(__fmul_rn(w.x, dy), dz)));
}

// ---- SAH-optimal choice of a wide node's children (a dynamic program over the
// binary tree, in the manner of Ylitie, Karras and Laine, HPG 2017).  Expected
// cost of a tree: c_node x SA(N) summed over its wide nodes N plus c_tri x
// SA(t) over its triangle children t (surface areas relative to the root's).
// For binary node n and a budget of i child slots (i = 1..W):
//   D(n, i) = min over j of C(left, j) + C(right, i - j)   (n spread over i slots)
//   C(n, 1) = c_node SA(n) + D(n, W)                        (n one slot: a wide node)
//   C(n, i) = min(C(n, 1), D(n, i)),  i >= 2
// with C(t, i) = c_tri SA(t) for a triangle.  Per node the argmin split of
// D(n, i) and whether C(n, 1) won are kept; a wide node at n takes the slots
// D(n, W)'s split gives its two children, expanded while they win.
struct CollapseDP {
    const int* parent_node;   // [n_binary] parent of each internal node (-1: root)
    const int* parent_leaf;   // [n_leaves] parent of each triangle
    float* cost;              // [n_binary][W] C(n, i)
    uint8_t* split;           // [n_binary][W] argmin j of D(n, i) (i >= 2)
    uint16_t* single;         // [n_binary] bit i: C(n, 1) <= D(n, i)
    unsigned* visits;         // [n_binary] children finished, bottom-up
    float c_node, c_tri;
    AreaW w;                  // face weights of the area measure (also the largest-area rule's)
};

// (and, with `internal`, how many of each node's children are internal)
__global__ void k_parents(const float4* __restrict__ bn, int n_binary, int* parent_node, int* parent_leaf,
                          unsigned* internal)
{
    const int n = blockIdx.x * blockDim.x + threadIdx.x;
    if (n >= n_binary) return;
    const float4 n3 = bn[4 * (int64_t)n + 3];
    const int c[2] = {__float_as_int(n3.x), __float_as_int(n3.y)};
    if (internal) internal[n] = (c[0] >= 0 ? 1u : 0u) + (c[1] >= 0 ? 1u : 0u);
    for (int k = 0; k < 2; ++k) {
        // (a build that failed may have left any bits here)
        if (c[k] >= 0 && c[k] < n_binary) parent_node[c[k]] = n;
        else if (c[k] < 0 && ~c[k] <= n_binary) parent_leaf[~c[k]] = n;
    }
}

// one thread per triangle climbs towards the root; the second child to finish
// computes its parent's table, so every node is computed once, after both
// children.  A clustering that gave up leaves no tree (its status is set by
// then) but unwritten links: nothing is read then.
template <int W>
__global__ void k_collapse_dp(const float4* __restrict__ bn, int n_leaves, CollapseDP dp, int* status)
{
    if (*(volatile int*)status != ST_OK) return;
    const int leaf = blockIdx.x * blockDim.x + threadIdx.x;
    if (leaf >= n_leaves) return;
    int node = dp.parent_leaf[leaf];
    while (node >= 0) {
        __threadfence();
        // only the second arrival goes on (the other child is still running at
        // the first; links in a circle would bring more), so every climb ends
        if (atomicAdd(&dp.visits[node], 1u) != 1u) return;
        __threadfence();
        ChildBox cb[2];
        float cc[2][W];
        for (int side = 0; side < 2; ++side) {
            binary_child(bn, node, side, cb[side]);
            if (cb[side].ref >= n_leaves - 1) {
                raise_status(status, ST_BOUNDS);
                return;
            }
            if (cb[side].ref < 0) {
                const float v = dp.c_tri * half_area(cb[side], dp.w);
                for (int i = 0; i < W; ++i) cc[side][i] = v;
            } else {
                for (int i = 0; i < W; ++i) cc[side][i] = __ldcg(&dp.cost[(int64_t)cb[side].ref * W + i]);
            }
        }
        ChildBox u;
        for (int a = 0; a < 3; ++a) {
            u.lo[a] = fminf(cb[0].lo[a], cb[1].lo[a]);
            u.hi[a] = fmaxf(cb[0].hi[a], cb[1].hi[a]);
        }
        float D[W + 1];
        int J[W + 1];
        for (int i = 2; i <= W; ++i) {
            D[i] = INFINITY;
            J[i] = 1;
            for (int j = 1; j < i; ++j) {
                const float v = cc[0][j - 1] + cc[1][i - j - 1];
                if (v < D[i]) {
                    D[i] = v;
                    J[i] = j;
                }
            }
        }
        const float c1 = dp.c_node * half_area(u, dp.w) + D[W];
        unsigned mask = 0;
        float* out = dp.cost + (int64_t)node * W;
        uint8_t* sp = dp.split + (int64_t)node * W;
        out[0] = c1;
        sp[0] = 0;
        for (int i = 2; i <= W; ++i) {
            if (c1 <= D[i]) {
                out[i - 1] = c1;
                mask |= 1u << i;
            } else {
                out[i - 1] = D[i];
            }
            sp[i - 1] = (uint8_t)J[i];
        }
        dp.single[node] = (uint16_t)mask;
        node = dp.parent_node[node];
    }
}

// How much a child of `slots` slots wants to be opened (-2: not at all): of a
// node's children the first of the largest is, until there are W or none can be.
template <int W>
__device__ __forceinline__ float open_key(const ChildBox& c, int slots, const CollapseDP& dp, int use_dp)
{
    if (c.ref < 0) return -2.0f;
    if (use_dp) return slots >= 2 && !((dp.single[c.ref] >> slots) & 1u) ? 1.0f : -2.0f;
    const float v = half_area(c, dp.w);
    return v > -1.0f ? v : -2.0f;
}

// slots of binary node b's left child, of the `slots` that b has
template <int W>
__device__ __forceinline__ int left_slots(const CollapseDP& dp, int use_dp, int b, int slots)
{
    return use_dp ? dp.split[(int64_t)b * W + slots - 1] : 0;
}

// References of the children of the wide node at binary node b, by one thread;
// returns the number of internal ones.  The loops are unrolled, so that all is
// in registers: the levels of 1M triangles took 293 us with the children's
// boxes in local memory, 223 us so.
template <int W>
__device__ int gather_refs(const float4* __restrict__ bn, int b, const CollapseDP& dp, int use_dp, int ref[W], int& count)
{
    float key[W];
    int slots[W];
    ChildBox c;
    auto take = [&](int node, int side, int budget, int& r, float& k) {
        binary_child(bn, node, side, c);
        r = c.ref;
        k = open_key<W>(c, budget, dp, use_dp);
    };
    slots[0] = left_slots<W>(dp, use_dp, b, W);
    slots[1] = W - slots[0];
    take(b, 0, slots[0], ref[0], key[0]);
    take(b, 1, slots[1], ref[1], key[1]);
    count = 2;
#pragma unroll
    for (int at = 2; at < W; ++at) {
        float top = -1.0f;
        int open = -1, budget = 0;
#pragma unroll
        for (int k = 0; k < at; ++k)
            if (key[k] > top) {
                top = key[k];
                open = ref[k];
                budget = slots[k];
            }
        if (top == -1.0f) break;
        const int left = left_slots<W>(dp, use_dp, open, budget);
        int r;
        float key_left;
        take(open, 0, left, r, key_left);
        bool found = false;
#pragma unroll
        for (int k = 0; k < at; ++k)
            if (!found && key[k] == top) {
                found = true;
                ref[k] = r;
                key[k] = key_left;
                slots[k] = left;
            }
        slots[at] = budget - left;
        take(open, 1, slots[at], ref[at], key[at]);
        count = at + 1;
    }
    int internal = 0;
#pragma unroll
    for (int k = 0; k < W; ++k) internal += k < count && ref[k] >= 0;
    return internal;
}

// This lane's child of the wide node at binary node b, by the W lanes of a
// group (the same b in each; < 0: no node), the same ones in the same order.
// All 32 lanes call it; returns the number of children.
template <int W>
__device__ int gather_lanes(const float4* __restrict__ bn, int b, const CollapseDP& dp, int use_dp, ChildBox& c)
{
    constexpr unsigned kAll = 0xffffffffu;
    const int lane = threadIdx.x & (W - 1);
    int count = b >= 0 ? 2 : 0, slots = 0;
    float key = -2.0f;
    for (int a = 0; a < 3; ++a) {
        c.lo[a] = INFINITY;
        c.hi[a] = -INFINITY;
    }
    c.ref = -1;
    auto take = [&](int node, int side, int budget) {
        const int left = left_slots<W>(dp, use_dp, node, budget);
        slots = side ? budget - left : left;
        binary_child(bn, node, side, c);
        key = open_key<W>(c, slots, dp, use_dp);
    };
    if (lane < count) take(b, lane, W);
    for (;;) {
        float top = count < W ? key : -2.0f;
        int best = lane;
#pragma unroll
        for (int d = 1; d < W; d *= 2) {
            const float other = __shfl_xor_sync(kAll, top, d);
            const int at = __shfl_xor_sync(kAll, best, d);
            if (other > top || (other == top && at < best)) {
                top = other;
                best = at;
            }
        }
        const bool more = top > -1.0f;
        if (!__any_sync(kAll, more)) return count;
        const int open = __shfl_sync(kAll, c.ref, best, W);
        const int budget = __shfl_sync(kAll, slots, best, W);
        if (more && (lane == best || lane == count)) take(open, lane != best, budget);
        count += more;
    }
}

constexpr int kCollapseThreads = 256;

struct CollapseTree {
    CollapseDP dp;
    int* root;            // [slots] binary node of each wide node, breadth-first
    int* first;           // [slots] slot of its first internal child (0: none)
    int* pushes;          // [slots] stack entries its ancestors can leave behind
    int* kids;            // [level][W] internal children of the level being walked
    unsigned* total;      // per tile of a level: internal children
    int* state;           // the lone first block's level: nodes, first slot, levels
    MeetPlace* place;     // the meetings of this tree's blocks, zero before the launch
    WideInfo* info;       // stack_need zero before the launch
};

struct CollapseArgs {
    const float4* bn;
    int use_dp;
    CollapseTree tree[2];  // 4-wide, 8-wide
    BuildWait wait;
};

template <int W>
__device__ void collapse_levels(const CollapseArgs& a, const CollapseTree& c, unsigned block, unsigned blocks)
{
    constexpr int T = kCollapseThreads;
    const int tid = threadIdx.x;
    unsigned met = 0;
    int n = 1, base = 0, levels = 0, need = 0;
    // one level by blocks `me` of `of`: false when a meeting ran out
    auto level = [&](unsigned me, unsigned of) -> bool {
        const int tiles = (n + T - 1) / T;
        const int per = (tiles + (int)of - 1) / (int)of;
        const int t0 = min((int)me * per, tiles), t1 = min(t0 + per, tiles);
        const bool shared = tiles > 1 || of > 1;
        int ref[W], count = 0, internal = 0, below = 0;  // this thread's node of the last tile
        unsigned before = 0, sum = 0;
        for (int t = t0; t < t1; ++t) {
            const int i = t * T + tid;
            count = internal = 0;
            if (i < n) {
                const int slot = base + i;
                internal = gather_refs<W>(a.bn, slot ? __ldcg(&c.root[slot]) : 0, c.dp, a.use_dp, ref, count);
                below = (slot ? __ldcg(&c.pushes[slot]) : 0) + (internal > 0 ? internal - 1 : 0);
                need = max(need, below);
                if (per > 1) {
                    int m = 0;
#pragma unroll
                    for (int k = 0; k < W; ++k)
                        if (k < count && ref[k] >= 0) __stcg(&c.kids[(int64_t)i * W + m++], ref[k]);
                    __stcg(&c.first[slot], internal);
                }
            }
            before = block_prefix<T>((unsigned)internal, sum);
            if (shared && tid == 0) __stcg(&c.total[t], sum);
        }
        // internal children of the tiles before this block's, and of all
        unsigned at = 0, next = sum;
        if (shared) {
            if (!build_meet(c.place, of, met, a.wait)) return false;
            unsigned mine = 0, all = 0;
            for (int t = tid; t < tiles; t += T) {
                const unsigned v = __ldcg(&c.total[t]);
                all += v;
                if (t < t0) mine += v;
            }
            block_prefix<T>(mine, at);
            block_prefix<T>(all, next);
        }
        if (per == 1) {
            // the thread still holds its node's children (listed in memory in
            // between, and a lone block's sum too, a rebuild and cast took 317 us
            // at 770 triangles and 1,358 us at 1M; 296 and 1,338 us so)
            const int slot = base + t0 * T + tid;
            if (count > 0) {
                int off = base + n + (int)(at + before);
                __stcg(&c.first[slot], internal > 0 ? off : 0);
#pragma unroll
                for (int k = 0; k < W; ++k)
                    if (k < count && ref[k] >= 0) {
                        __stcg(&c.root[off], ref[k]);
                        __stcg(&c.pushes[off], below);
                        ++off;
                    }
            }
        } else {
            for (int t = t0; t < t1; ++t) {
                const int i = t * T + tid, slot = base + i;
                internal = i < n ? __ldcg(&c.first[slot]) : 0;
                const int off = base + n + (int)(at + block_prefix<T>((unsigned)internal, sum));
                at += sum;
                if (i >= n) continue;
                below = (slot ? __ldcg(&c.pushes[slot]) : 0) + (internal > 0 ? internal - 1 : 0);
                __stcg(&c.first[slot], internal > 0 ? off : 0);
                for (int k = 0; k < internal; ++k) {
                    __stcg(&c.root[off + k], __ldcg(&c.kids[(int64_t)i * W + k]));
                    __stcg(&c.pushes[off + k], below);
                }
            }
        }
        base += n;
        n = (int)next;
        ++levels;
        return build_meet(c.place, of, met, a.wait);
    };
    // the first levels fit one block, which walks them alone while the others wait once
    if (blocks > 1) {
        if (block == 0) {
            while (n > 0 && n <= T) level(0, 1);
            if (tid == 0) {
                __stcg(&c.state[0], n);
                __stcg(&c.state[1], base);
                __stcg(&c.state[2], levels);
            }
        }
        if (!build_meet(c.place, blocks, met, a.wait)) return;
        n = __ldcg(&c.state[0]);
        base = __ldcg(&c.state[1]);
        levels = __ldcg(&c.state[2]);
        while (n > T)
            if (!level(block, blocks)) return;
    }
    // so do the last ones
    if (block == 0)
        while (n > 0) level(0, 1);
    need = __reduce_max_sync(0xffffffffu, need);
    if ((tid & 31) == 0) atomicMax(&c.info->stack_need, need);
    if (block == 0 && tid == 0) {
        c.info->n_wide = base;
        c.info->levels = levels;
    }
}

// Even blocks walk the 4-wide tree, odd ones the 8-wide: the levels of the two
// hide each other's waits.  Bound by those: 1M triangles, both trees, 17 and 11
// levels, 2.6 ms with three launches and a host round trip a level and one
// block scanning it, 0.20 ms so.
__global__ void __launch_bounds__(kCollapseThreads) k_collapse_levels(const __grid_constant__ CollapseArgs a)
{
    // a build that failed left no tree to walk
    if (*(volatile int*)a.wait.status != ST_OK) return;
    if ((blockIdx.x & 1u) == 0) collapse_levels<4>(a, a.tree[0], blockIdx.x >> 1, gridDim.x >> 1);
    else collapse_levels<8>(a, a.tree[1], blockIdx.x >> 1, gridDim.x >> 1);
}

// Every node of a wide tree, a lane per child.  Bound by the loads of the
// opened nodes, one after another, and by the stores: with a thread per node,
// its children in local memory and 16-byte stores 128 or 256 bytes apart, 1M
// triangles took 108 us (8-wide) and 74 us (4-wide); so, 46 and 38 us.
template <int W>
__global__ void __launch_bounds__(kCollapseThreads) k_collapse_nodes(const float4* __restrict__ bn, int n,
                                                                     const int* __restrict__ root,
                                                                     const int* __restrict__ first,
                                                                     float4* __restrict__ nodes, const CollapseDP dp,
                                                                     int use_dp)
{
    const int lane = threadIdx.x & (W - 1), group = threadIdx.x & 31 & ~(W - 1);
    const int64_t i = ((int64_t)blockIdx.x * kCollapseThreads + threadIdx.x) / W;
    const bool live = i < n;
    ChildBox c;
    const int count = gather_lanes<W>(bn, live ? (i ? root[i] : 0) : -1, dp, use_dp, c);
    const unsigned inner = (__ballot_sync(0xffffffffu, c.ref >= 0) >> group) & ((1u << W) - 1u);
    if (!live) return;
    // internal children first, keeping their order (a stable partition)
    const unsigned below = (1u << lane) - 1u;
    const int n_inner = __popc(inner), rank = __popc(inner & below);
    const int next = first[i];
    const int k = lane >= count ? lane : (c.ref >= 0 ? rank : n_inner + lane - rank);
    const int code = lane >= count ? 0 : (c.ref >= 0 ? next + rank : c.ref);
    float* out = reinterpret_cast<float*>(nodes) + 8 * W * i + k;
    for (int a = 0; a < 3; ++a) {
        out[2 * a * W] = c.lo[a];
        out[(2 * a + 1) * W] = c.hi[a];
    }
    out[6 * W] = __int_as_float(code);
    const int leaf_mask = (int)(((1u << count) - 1u) & ~((1u << n_inner) - 1u));
    out[7 * W] = k == 0 ? __int_as_float(next) : (k == 1 ? __int_as_float(leaf_mask) : 0.0f);
}

}  // namespace

namespace {

// layout of the collapse's scratch (`base` may be NULL to size it)
struct CollapseScratch {
    CollapseArgs a{};
    MeetPlace* places;
    int *parent_node, *parent_leaf;
    size_t bytes;

    CollapseScratch(char* base, int64_t n_binary, int sah_dp)
    {
        const int64_t m = n_binary > 0 ? n_binary : 1;
        // a level's nodes have disjoint subtrees of two triangles or more
        const int64_t widest = (m + 1) / 2 + 1;
        size_t at = 0;
        auto get = [&](size_t b) {
            char* p = base + at;
            at += (b + 255) / 256 * 256;
            return p;
        };
        places = (MeetPlace*)get(2 * sizeof(MeetPlace) + 8 * sizeof(int));
        for (int k = 0; k < 2; ++k) {
            CollapseTree& t = a.tree[k];
            t.place = places + k;
            t.state = (int*)(places + 2) + 4 * k;
            t.root = (int*)get(m * sizeof(int));
            t.first = (int*)get(m * sizeof(int));
            t.pushes = (int*)get(m * sizeof(int));
            t.kids = (int*)get(widest * (k ? 8 : 4) * sizeof(int));
            t.total = (unsigned*)get((widest / kCollapseThreads + 2) * sizeof(unsigned));
        }
        parent_node = parent_leaf = nullptr;
        if (sah_dp) {
            // the dynamic program's tables; the costs and visits of one width give way to the other's
            parent_node = (int*)get(m * sizeof(int));
            parent_leaf = (int*)get((m + 1) * sizeof(int));
            float* cost = (float*)get(m * 8 * sizeof(float));
            unsigned* visits = (unsigned*)get(m * sizeof(unsigned));
            for (int k = 0; k < 2; ++k) {
                CollapseDP& dp = a.tree[k].dp;
                dp.parent_node = parent_node;
                dp.parent_leaf = parent_leaf;
                dp.cost = cost;
                dp.visits = visits;
                dp.split = (uint8_t*)get(m * (k ? 8 : 4));
                dp.single = (uint16_t*)get(m * sizeof(uint16_t));
            }
        }
        bytes = at;
    }
};

}  // namespace

size_t collapse_scratch_bytes(int64_t n_binary, int sah_dp)
{
    return CollapseScratch(nullptr, n_binary, sah_dp).bytes;
}

// Lists both wide trees' nodes (in scratch); info_dev[2] receives what they
// are (4-wide, 8-wide).
cudaError_t collapse_plan(cudaStream_t s, const float4* binary_nodes, int64_t n_binary, void* scratch,
                          size_t scratch_bytes, int sah_dp, float tri_cost, AreaW area_w, int* status, int num_sms,
                          int coop, uint64_t wait_ns, WideInfo info_dev[2])
{
    if (n_binary < 1) return cudaErrorInvalidValue;
    if (n_binary < 2) sah_dp = 0;  // a single triangle: nothing to choose
    CollapseScratch c((char*)scratch, n_binary, sah_dp);
    if (scratch_bytes < c.bytes) return cudaErrorInvalidValue;
    c.a.bn = binary_nodes;
    c.a.use_dp = sah_dp ? 1 : 0;
    c.a.wait = BuildWait{status, wait_ns};
    for (CollapseTree& t : c.a.tree) {
        t.dp.w = area_w;  // the largest-area rule reads it too
        t.dp.c_node = 1.0f;
        t.dp.c_tri = tri_cost;
    }
    c.a.tree[0].info = info_dev;
    c.a.tree[1].info = info_dev + 1;
    cudaError_t e = cudaMemsetAsync(c.places, 0, 2 * sizeof(MeetPlace), s);
    if (e == cudaSuccess) e = cudaMemsetAsync(info_dev, 0, 2 * sizeof(WideInfo), s);
    if (e != cudaSuccess) return e;
    if (sah_dp) {
        const int nb = (int)n_binary;
        // no parent (-1) but where k_parents finds a link
        e = cudaMemsetAsync(c.parent_node, 0xFF, (size_t)nb * sizeof(int), s);
        if (e == cudaSuccess) e = cudaMemsetAsync(c.parent_leaf, 0xFF, ((size_t)nb + 1) * sizeof(int), s);
        if (e != cudaSuccess) return e;
        k_parents<<<(nb + 255) / 256, 256, 0, s>>>(binary_nodes, nb, c.parent_node, c.parent_leaf, nullptr);
        for (int k = 0; k < 2; ++k) {
            const CollapseDP& dp = c.a.tree[k].dp;
            e = cudaMemsetAsync(dp.visits, 0, (size_t)nb * sizeof(unsigned), s);
            if (e != cudaSuccess) return e;
            if (k == 0) k_collapse_dp<4><<<(nb + 1 + 255) / 256, 256, 0, s>>>(binary_nodes, nb + 1, dp, status);
            else k_collapse_dp<8><<<(nb + 1 + 255) / 256, 256, 0, s>>>(binary_nodes, nb + 1, dp, status);
        }
        e = cudaGetLastError();
        if (e != cudaSuccess) return e;
    }
    // two blocks (one a tree, which meet nobody) for what one block's tiles hold
    // and one a tree and SM at most: a level's two meetings cost more with more
    // blocks than its widest tiles gain (1M triangles: 1,646 us for a rebuild and
    // cast, 1,661 with two, 1,702 with three)
    const int64_t want = std::min<int64_t>(2 * ((n_binary / 4 + kCollapseThreads - 1) / kCollapseThreads),
                                           2 * (int64_t)num_sms);
    const int grid =
        std::max(2, coop_blocks((const void*)k_collapse_levels, kCollapseThreads, 0, num_sms, coop, want) / 2 * 2);
    if (grid == 2) {
        k_collapse_levels<<<2, kCollapseThreads, 0, s>>>(c.a);
        e = cudaGetLastError();
    } else {
        void* args[] = {&c.a};
        e = cudaLaunchCooperativeKernel((const void*)k_collapse_levels, dim3(grid), dim3(kCollapseThreads), args, 0, s);
    }
    return e;
}

// Writes the nodes of the tree of `width` (4 or 8) that collapse_plan listed
// in the same scratch, with the same options.
cudaError_t collapse_write(cudaStream_t s, int width, const float4* binary_nodes, int64_t n_binary, float4* nodes,
                           int64_t n_wide, void* scratch, int sah_dp, AreaW area_w)
{
    if (n_wide <= 0) return cudaSuccess;
    if (n_binary < 2) sah_dp = 0;
    CollapseScratch c((char*)scratch, n_binary, sah_dp);
    CollapseTree& t = c.a.tree[width == 8];
    t.dp.w = area_w;
    const unsigned blocks = (unsigned)((n_wide * width + kCollapseThreads - 1) / kCollapseThreads);
    if (width == 8)
        k_collapse_nodes<8><<<blocks, kCollapseThreads, 0, s>>>(binary_nodes, (int)n_wide, t.root, t.first, nodes, t.dp,
                                                                sah_dp ? 1 : 0);
    else
        k_collapse_nodes<4><<<blocks, kCollapseThreads, 0, s>>>(binary_nodes, (int)n_wide, t.root, t.first, nodes, t.dp,
                                                                sah_dp ? 1 : 0);
    return cudaGetLastError();
}

}  // namespace lidar

// ---------------------------------------------------------------------------
// Treelet restructuring of the binary hierarchy (Karras and Aila, "Fast
// Parallel Construction of High-Quality Bounding Volume Hierarchies", HPG
// 2013), one warp per treelet.  Cost of a tree under the
// surface-area model: c_node x A(n) over its internal nodes plus c_tri x A(t)
// over its triangles (A: half the surface area of the box).  One round climbs
// the tree bottom-up (the second child to finish processes its parent, so a
// node is processed after its whole subtree).  At node n the thread forms a
// treelet: starting from n's two children it replaces the treelet leaf of
// largest area that is an internal node by that node's children, until there
// are kTreeletLeaves leaves or none is internal.  A dynamic program over the
// subsets S of the treelet's leaves gives the cheapest binary tree over them:
//   c({l}) = cost of leaf l's subtree,
//   c(S)   = c_node x A(S) + min over partitions S = P + Q of c(P) + c(Q).
// If that is cheaper than the treelet's current shape, its internal nodes
// (n first, so n's parent keeps pointing at it) are rewritten in the new
// shape with exact FP32 min/max child boxes.  Only the topology above the
// treelet's leaves changes, so the result is again a valid hierarchy over the
// same triangles.  Every decision depends only on the subtree below the
// node, so the result does not depend on the order threads run in.
namespace lidar {
namespace {

constexpr int kTreeletLeaves = 7;

struct TreeletArgs {
    int n_leaves;
    int n_binary;
    float4* nodes;            // binary nodes, rewritten in place
    int* parent;              // [n_binary], -1 at the root; kept up to date by the rewrites
    // A round visits the nodes below which something may change: all of them in
    // round 1, then those that the round before rewrote and their ancestors.
    uint8_t* on_path;         // [n_binary] the last round (from 2) that visits the node
    unsigned* expect;         // [n_binary] children the round visits
    unsigned* visits;         // [n_binary] of these, finished; zero at the start of a round
    float* cost;              // [n_binary] surface-area cost of each node's subtree
    // A treelet is a function of the nodes it opens and the costs of its leaves,
    // all at most kTreeletReach levels below its root, so one that was kept and
    // below which no node was rewritten and no cost moved (in its last bit) that
    // near is kept again without a look: mark[n] is the last round (1, 2, ...)
    // that rewrote node n; up[n] has, in its low four bits, the last round that
    // changed a node or a cost in n's subtree near enough for n's parent, and
    // above them how many levels below n (0: n itself) the nearest is.  (A change
    // a few levels down need not move the costs above it: they may be so much
    // larger that it is lost in their rounding.)
    uint8_t* mark;            // [n_binary]
    uint8_t* up;              // [n_binary]
    int round;
    unsigned long long* changed;  // treelets rewritten in the round
    int* status;              // ST_BOUNDS: a child reference out of range, or a climb longer than the bound
    float c_node, c_tri;
    AreaW w;                  // face weights of the area measure
};

// a chain of kTreeletLeaves - 1 internal nodes, the root the first, has its last leaves this far below
constexpr int kTreeletReach = kTreeletLeaves - 1;

// longest climb a valid hierarchy of up to 2^31 triangles can need is far
// below this; a longer one means a broken tree (a cycle), which ends the climb
constexpr int kTreeletMaxClimb = 4096;

struct TBox {
    float lo[3], hi[3];
};

__device__ __forceinline__ float tbox_area(const TBox& b, AreaW w)
{
    const float dx = b.hi[0] - b.lo[0], dy = b.hi[1] - b.lo[1], dz = b.hi[2] - b.lo[2];
    return w.z * dx * dy + w.x * dy * dz + w.y * dz * dx;
}

__device__ __forceinline__ void tbox_grow(TBox& a, const TBox& b)
{
    for (int k = 0; k < 3; ++k) {
        a.lo[k] = fminf(a.lo[k], b.lo[k]);
        a.hi[k] = fmaxf(a.hi[k], b.hi[k]);
    }
}

// child `side` of binary node `node` (read through L2: other threads of the
// round may have written it)
__device__ __forceinline__ void treelet_child(const float4* nodes, int node, int side, int& ref, TBox& b)
{
    const float4 n0 = __ldcg(&nodes[4 * (int64_t)node + 0]), n1 = __ldcg(&nodes[4 * (int64_t)node + 1]);
    const float4 n2 = __ldcg(&nodes[4 * (int64_t)node + 2]), n3 = __ldcg(&nodes[4 * (int64_t)node + 3]);
    if (side == 0) {
        b.lo[0] = n0.x; b.hi[0] = n0.y; b.lo[1] = n0.z; b.hi[1] = n0.w; b.lo[2] = n2.x; b.hi[2] = n2.y;
        ref = __float_as_int(n3.x);
    } else {
        b.lo[0] = n1.x; b.hi[0] = n1.y; b.lo[1] = n1.z; b.hi[1] = n1.w; b.lo[2] = n2.z; b.hi[2] = n2.w;
        ref = __float_as_int(n3.y);
    }
}

__device__ __forceinline__ bool ref_ok(const TreeletArgs& a, int ref)
{
    return ref >= 0 ? ref < a.n_binary : ~ref < a.n_leaves;
}

__device__ __forceinline__ float subtree_cost(const TreeletArgs& a, int ref, const TBox& b)
{
    return ref < 0 ? a.c_tri * tbox_area(b, a.w) : __ldcg(&a.cost[ref]);
}

// Subsets of a treelet's leaves by size (a bit mask each): the lanes of a warp
// take the subsets of one size together, which depend on smaller sizes only.
__device__ const unsigned char kSubsets2[21] = {3,  5,  6,  9,  10, 12, 17, 18, 20, 24, 33,
                                                34, 36, 40, 48, 65, 66, 68, 72, 80, 96};
__device__ const unsigned char kSubsets3[35] = {7,  11, 13, 14, 19, 21, 22, 25, 26, 28,  35, 37,
                                                38, 41, 42, 44, 49, 50, 52, 56, 67, 69,  70, 73,
                                                74, 76, 81, 82, 84, 88, 97, 98, 100, 104, 112};

// One warp's treelet in shared memory.
struct TreeletShared {
    float box[6][kTreeletLeaves + 1];  // lo.x, hi.x, lo.y, hi.y, lo.z, hi.z of the leaves
    float c[1 << kTreeletLeaves];      // c(S); before S is done, c_node x A(S)
    unsigned char split[1 << kTreeletLeaves];
    int ref[kTreeletLeaves + 1];       // the leaves
    int inner[kTreeletLeaves + 1];     // the treelet's internal nodes, the root first
    int out_s[kTreeletLeaves], out_id[kTreeletLeaves], out_ref[2][kTreeletLeaves];
};

// box of subset x of the treelet's leaves
__device__ __forceinline__ TBox subset_box(const TreeletShared& t, int x)
{
    TBox u;
    bool first = true;
    for (; x; x &= x - 1) {
        const int i = __ffs(x) - 1;
        TBox b;
        for (int k = 0; k < 3; ++k) {
            b.lo[k] = t.box[2 * k][i];
            b.hi[k] = t.box[2 * k + 1][i];
        }
        if (first) u = b;
        else tbox_grow(u, b);
        first = false;
    }
    return u;
}

// Cheapest partition of subset s (each once: the part with s's lowest leaf,
// low | q for the proper submasks q of the others, largest q first, the first
// of equal costs kept).  The lane tries q = v | fixed for the kTries submasks v
// of `varied`; a subset whose partitions are spread over several lanes gives
// each its own `fixed`.
template <int kTries>
__device__ __forceinline__ void best_partition(const TreeletShared& t, int s, int varied, int fixed, float& best,
                                               int& bq)
{
    const int low = s & -s, rest = s ^ low;
    best = INFINITY;
    bq = 0;
    int v = varied;
#pragma unroll
    for (int i = 0; i < kTries; ++i, v = (v - 1) & varied) {
        const int q = v | fixed;
        const float x = t.c[q | low] + t.c[s ^ (q | low)];
        if (x < best && q != rest) {
            best = x;
            bq = q;
        }
    }
}

// lanes xor-partnered over `width` lanes agree on the cheapest (largest q of equal costs)
__device__ __forceinline__ void merge_partition(float& best, int& bq, int width)
{
    for (int o = width / 2; o > 0; o >>= 1) {
        const float b2 = __shfl_xor_sync(0xffffffffu, best, o);
        const int q2 = __shfl_xor_sync(0xffffffffu, bq, o);
        if (b2 < best || (b2 == best && q2 > bq)) {
            best = b2;
            bq = q2;
        }
    }
}

// The treelet at `node`, by one warp (all lanes call it).  Lane i < 7 holds the
// treelet's leaf i while it grows; the areas of its 127 subsets are spread over
// the lanes, four each; the dynamic program runs size by size, one subset per
// lane up to five leaves, four lanes a subset at six, all lanes on the whole.
// 1: rewritten, or its cost changed; 0: all as it was; -1: a child reference out
// of range.
//
// A leaf that is an internal node has its own record in flight as soon as it
// joins the treelet, so that opening it later waits for no load.
__device__ int treelet_node(const TreeletArgs& a, int node, TreeletShared& t, int sub2, int sub3a, int sub3b)
{
    const int lane = threadIdx.x & 31;
    constexpr unsigned kAll = 0xffffffffu;
    float4 n0, n1, n2;       // this lane's leaf's record (the treelet's root at first)
    int left, right;
    auto fetch = [&](int r) {
        n0 = __ldcg(&a.nodes[4 * (int64_t)r + 0]);
        n1 = __ldcg(&a.nodes[4 * (int64_t)r + 1]);
        n2 = __ldcg(&a.nodes[4 * (int64_t)r + 2]);
        const int2 c = __ldcg(reinterpret_cast<const int2*>(&a.nodes[4 * (int64_t)r + 3]));
        left = c.x;
        right = c.y;
    };
    fetch(node);
    int ref = lane == 0 ? left : (lane == 1 ? right : -1);
    if (__any_sync(kAll, !ref_ok(a, ref))) return -1;
    TBox box;
    box.lo[0] = lane ? n1.x : n0.x; box.hi[0] = lane ? n1.y : n0.y;
    box.lo[1] = lane ? n1.z : n0.z; box.hi[1] = lane ? n1.w : n0.w;
    box.lo[2] = lane ? n2.z : n2.x; box.hi[2] = lane ? n2.w : n2.y;
    float root_area;
    {
        TBox whole;
        whole.lo[0] = fminf(n0.x, n1.x); whole.hi[0] = fmaxf(n0.y, n1.y);
        whole.lo[1] = fminf(n0.z, n1.z); whole.hi[1] = fmaxf(n0.w, n1.w);
        whole.lo[2] = fminf(n2.x, n2.z); whole.hi[2] = fmaxf(n2.y, n2.w);
        root_area = tbox_area(whole, a.w);
    }
    float area = tbox_area(box, a.w);
    float cost = a.c_tri * area;
    if (lane < 2 && ref >= 0) {
        fetch(ref);
        cost = __ldcg(&a.cost[ref]);
    }
    const float first_cost = cost;  // lanes 0 and 1: the root's children
    int k = 2, inner = node;        // lane j: the treelet's internal node j
    while (k < kTreeletLeaves) {
        // the internal leaf of largest area (ties to the lowest); areas are not
        // negative, so their bits order like the values
        const unsigned key = (lane < k && ref >= 0 && area > -1.0f) ? __float_as_uint(area) + 1u : 0u;
        const unsigned top = __reduce_max_sync(kAll, key);
        if (top == 0u) break;
        const int best = __ffs(__ballot_sync(kAll, key == top)) - 1;
        const int open = __shfl_sync(kAll, ref, best);
        if (lane == k - 1) inner = open;
        // side 0 stays in the opened leaf's lane, side 1 goes to lane k
        const float bx = __shfl_sync(kAll, n1.x, best), by = __shfl_sync(kAll, n1.y, best);
        const float bz = __shfl_sync(kAll, n1.z, best), bw = __shfl_sync(kAll, n1.w, best);
        const float cz = __shfl_sync(kAll, n2.z, best), cw = __shfl_sync(kAll, n2.w, best);
        const int rr = __shfl_sync(kAll, right, best);
        const bool mine = lane == best || lane == k;
        if (lane == best) {
            box.lo[0] = n0.x; box.hi[0] = n0.y; box.lo[1] = n0.z; box.hi[1] = n0.w; box.lo[2] = n2.x; box.hi[2] = n2.y;
            ref = left;
        }
        if (lane == k) {
            box.lo[0] = bx; box.hi[0] = by; box.lo[1] = bz; box.hi[1] = bw; box.lo[2] = cz; box.hi[2] = cw;
            ref = rr;
        }
        if (__any_sync(kAll, mine && !ref_ok(a, ref))) return -1;
        if (mine) {
            area = tbox_area(box, a.w);
            if (ref >= 0) {
                fetch(ref);
                cost = __ldcg(&a.cost[ref]);
            } else {
                cost = a.c_tri * area;
            }
        }
        ++k;
    }
    // the node's cost in its current shape
    const float c_now = a.c_node * root_area + __shfl_sync(kAll, first_cost, 0) + __shfl_sync(kAll, first_cost, 1);
    __syncwarp();  // the treelet before this one is done with the shared arrays
    if (lane < k) {
        for (int j = 0; j < 3; ++j) {
            t.box[2 * j][lane] = box.lo[j];
            t.box[2 * j + 1][lane] = box.hi[j];
        }
        t.ref[lane] = ref;
        if (lane < k - 1) t.inner[lane] = inner;
    }
    __syncwarp();
    // areas: lane l takes the subsets 4 l + {0, 1, 2, 3}
    const int full = (1 << k) - 1;
    if (4 * lane <= full) {
        TBox hi;
        for (int j = 0; j < 3; ++j) {
            hi.lo[j] = INFINITY;
            hi.hi[j] = -INFINITY;
        }
#pragma unroll
        for (int i = 2; i < kTreeletLeaves; ++i)
            if ((lane >> (i - 2)) & 1)
                for (int j = 0; j < 3; ++j) {
                    hi.lo[j] = fminf(hi.lo[j], t.box[2 * j][i]);
                    hi.hi[j] = fmaxf(hi.hi[j], t.box[2 * j + 1][i]);
                }
#pragma unroll
        for (int m = 0; m < 4; ++m) {
            TBox u = hi;
            for (int i = 0; i < 2; ++i)
                if ((m >> i) & 1)
                    for (int j = 0; j < 3; ++j) {
                        u.lo[j] = fminf(u.lo[j], t.box[2 * j][i]);
                        u.hi[j] = fmaxf(u.hi[j], t.box[2 * j + 1][i]);
                    }
            t.c[4 * lane + m] = a.c_node * tbox_area(u, a.w);
        }
    }
    __syncwarp();
    if (lane < k) t.c[1 << lane] = cost;
    __syncwarp();
    // up to five leaves: one subset per lane (those with leaves past k have none)
    auto one = [&](int s, auto tries) {
        if (s > full || s == 0) return;
        float best;
        int q;
        best_partition<decltype(tries)::value>(t, s, s & (s - 1), 0, best, q);
        t.c[s] += best;
        t.split[s] = (unsigned char)(q | (s & -s));
    };
    one(sub2, std::integral_constant<int, 2>());
    __syncwarp();
    one(sub3a, std::integral_constant<int, 4>());
    one(sub3b, std::integral_constant<int, 4>());
    __syncwarp();
    // subsets of four and five leaves are the complements of those of three and two
    if (k >= 4) {
        one(127 ^ sub3a, std::integral_constant<int, 8>());
        one(sub3b ? 127 ^ sub3b : 0, std::integral_constant<int, 8>());
        __syncwarp();
    }
    if (k >= 5) {
        one(sub2 ? 127 ^ sub2 : 0, std::integral_constant<int, 16>());
        __syncwarp();
    }
    if (k >= 6) {
        // six leaves: four lanes a subset, each its own choice of the two highest leaves
        const int s = lane < 28 ? 127 ^ (1 << (lane >> 2)) : 63;
        const int rest = s & (s - 1);
        const int b1 = 1 << (31 - __clz(rest)), b0 = 1 << (31 - __clz(rest ^ b1));
        float best;
        int q;
        best_partition<8>(t, s, rest ^ b1 ^ b0, ((lane & 1) ? b0 : 0) | ((lane & 2) ? b1 : 0), best, q);
        merge_partition(best, q, 4);
        __syncwarp();
        if (lane < 28 && (lane & 3) == 0 && s <= full) {
            t.c[s] += best;
            t.split[s] = (unsigned char)(q | (s & -s));
        }
        __syncwarp();
    }
    if (k == 7) {
        float best;
        int q;
        best_partition<2>(t, 127, 2, lane << 2, best, q);
        merge_partition(best, q, 32);
        __syncwarp();
        if (lane == 0) {
            t.c[127] += best;
            t.split[127] = (unsigned char)(q | 1);
        }
        __syncwarp();
    }
    // keep the current shape unless the optimum is clearly cheaper (it is
    // one of the shapes the program compares, so it is never dearer beyond
    // rounding)
    if (!(t.c[full] < c_now * (1.0f - 1e-5f))) {
        bool moved = false;
        if (lane == 0) {
            moved = __float_as_int(__ldcg(&a.cost[node])) != __float_as_int(c_now);
            a.cost[node] = c_now;
        }
        return __any_sync(kAll, moved) ? 1 : 0;
    }
    // rewrite: subset S at internal node id, its parts as leaves or the next
    // internal nodes of the treelet (one lane lays out the shape, then a lane
    // a node writes it)
    if (lane == 0) {
        // the stack of subsets to place, eight bits each, in one register; a
        // subset's internal node (of t.inner) goes along in the other
        unsigned long long st = (unsigned long long)full, at = 0;
        int next = 1;
        for (int j = 0; j < k - 1; ++j) {
            const int s = (int)(st & 0xFFu), id = (int)(at & 0xFFu);
            st >>= 8;
            at >>= 8;
            const int p = t.split[s];
            t.out_s[j] = s;
            t.out_id[j] = t.inner[id];
#pragma unroll
            for (int side = 0; side < 2; ++side) {
                const int x = side ? s ^ p : p;
                if ((x & (x - 1)) == 0) {
                    t.out_ref[side][j] = t.ref[__ffs(x) - 1];
                } else {
                    t.out_ref[side][j] = t.inner[next];
                    st = (st << 8) | (unsigned long long)x;
                    at = (at << 8) | (unsigned long long)next;
                    ++next;
                }
            }
        }
        atomicAdd(a.changed, 1ull);
    }
    __syncwarp();
    if (lane < k - 1) {
        const int s = t.out_s[lane], id = t.out_id[lane];
        const TBox L = subset_box(t, t.split[s]), R = subset_box(t, s ^ t.split[s]);
        a.nodes[4 * (int64_t)id + 0] = make_float4(L.lo[0], L.hi[0], L.lo[1], L.hi[1]);
        a.nodes[4 * (int64_t)id + 1] = make_float4(R.lo[0], R.hi[0], R.lo[1], R.hi[1]);
        a.nodes[4 * (int64_t)id + 2] = make_float4(L.lo[2], L.hi[2], R.lo[2], R.hi[2]);
        a.nodes[4 * (int64_t)id + 3] =
            make_float4(__int_as_float(t.out_ref[0][lane]), __int_as_float(t.out_ref[1][lane]), 0.0f, 0.0f);
        a.cost[id] = t.c[s];
        a.mark[id] = (uint8_t)a.round;
        for (int side = 0; side < 2; ++side)
            if (t.out_ref[side][lane] >= 0) a.parent[t.out_ref[side][lane]] = id;
    }
    return 1;
}

// One warp a block: warps end at very different times (most lanes stop after a
// few steps, a few climb to the root), and a block's slot is only free when its
// last warp ends.  16 a SM leaves 128 registers, without spills (0.65M
// triangles, eight rounds, the whole build and a cast: 5.54 ms; with spills,
// 18 and 20 a SM 6.0 ms, 24 and 28 6.4 and 6.5 ms; four-warp blocks, when the
// rest took longer, 11.4 ms against 11.0).
constexpr int kTreeletThreads = 32;
constexpr int kTreeletBlocks = 16;

// The nodes the round rewrote and all above them: the nodes the next one
// visits, and how many of each one's children are among them.
__global__ void __launch_bounds__(kBuildThreads) k_treelet_paths(TreeletArgs a)
{
    int n = blockIdx.x * blockDim.x + threadIdx.x;
    if (n >= a.n_binary || a.mark[n] != a.round - 1) return;
    for (int step = 0; n >= 0 && step < kTreeletMaxClimb; ++step) {
        // bytes have no atomics: the word that holds the node's
        unsigned* word = (unsigned*)(a.on_path + (n & ~3));
        const unsigned shift = 8u * (n & 3);
        unsigned seen = *(volatile unsigned*)word;
        while (((seen >> shift) & 0xFFu) != (unsigned)a.round) {
            const unsigned want = (seen & ~(0xFFu << shift)) | ((unsigned)a.round << shift);
            const unsigned was = atomicCAS(word, seen, want);
            if (was == seen) break;
            seen = was;
        }
        if (((seen >> shift) & 0xFFu) == (unsigned)a.round) return;  // the rest of the path is taken
        n = a.parent[n];
        if (n >= a.n_binary) {
            raise_status(a.status, ST_BOUNDS);
            return;
        }
        if (n >= 0) atomicAdd(&a.expect[n], 1u);
    }
}

// A lane per node: those none of whose children the round visits climb from
// there, each going on from a node when it is the last of the visited children
// to finish; the lanes whose node needs a look have the warp process the
// treelets one after another.
//
// What bounds it: the chain of each warp's treelets (issue ~40 %, ~1,000 warp
// instructions and ~7,000 cycles a treelet) in the first round, the climb (an
// arrival and two loads a level) in later ones, which look at few
// treelets.  Measured at 0.65M triangles (city, eight rounds): one thread a
// treelet with its program in local memory 9.4 ms a round; by a warp 1.2 ms;
// with the treelets whose subtree is unchanged kept unseen 1.2, 0.88, 0.64,
// 0.51, 0.41, 0.35, 0.31, 0.30 ms; climbing only where something was rewritten
// and with one acquire-release arrival a level 1.14, 0.83, 0.60, 0.42, 0.32,
// 0.30, 0.25, 0.24 ms.  (Looking kTreeletReach levels above every change, and
// not only while it still moves the costs, took the whole load from 5.21 to
// 5.31 ms, a round 1.14, 0.84, 0.61, 0.44, 0.34, 0.30, 0.25, 0.24 ms; it is what
// makes the rounds those of a full evaluation.)  A stride between a warp's nodes, fewer lanes or more
// nodes a warp all took longer: neighbours share the climb.
__global__ void __launch_bounds__(kTreeletThreads, kTreeletBlocks) k_treelet_round(TreeletArgs a)
{
    __shared__ TreeletShared s_t[kTreeletThreads / 32];
    TreeletShared& t = s_t[threadIdx.x >> 5];
    const int lane = threadIdx.x & 31;
    const int sub2 = lane < 21 ? kSubsets2[lane] : 0, sub3a = kSubsets3[lane], sub3b = lane < 3 ? kSubsets3[32 + lane] : 0;
    int node = blockIdx.x * blockDim.x + threadIdx.x;
    if (node >= a.n_binary || (a.round > 1 && a.on_path[node] != a.round) || a.expect[node] != 0u) node = -1;
    for (int step = 0;; ++step) {
        if (node >= a.n_binary || (node >= 0 && step >= kTreeletMaxClimb)) {
            raise_status(a.status, ST_BOUNDS);
            node = -1;
        }
        int2 c = make_int2(-1, -1);
        int parent = -1;
        bool look = false;           // the warp has to look at the treelet
        int levels = kTreeletReach;  // below the node is the nearest change of this round (or more)
        if (node >= 0) {
            const unsigned before = step > 0 ? arrive(&a.visits[node]) + 1u : 0u;
            const unsigned expect = a.expect[node];
            c = __ldcg(reinterpret_cast<const int2*>(&a.nodes[4 * (int64_t)node + 3]));
            parent = __ldcg(&a.parent[node]);
            look = a.round == 1 || __ldcg(&a.mark[node]) == a.round - 1;
            if (before != expect) node = -1;  // another child is still running
        }
        if (!__any_sync(0xffffffffu, node >= 0)) return;
        __syncwarp();  // what the arrivals acquired, the children's results, is the whole warp's
        if (node < 0) {
            look = false;
        } else if (!ref_ok(a, c.x) || !ref_ok(a, c.y)) {
            raise_status(a.status, ST_BOUNDS);
            look = false;
        } else if (c.x < 0 && c.y < 0) {
            // a pair of triangles has one shape: its lane notes the cost
            if (look) {
                int ref;
                TBox L, R;
                treelet_child(a.nodes, node, 0, ref, L);
                treelet_child(a.nodes, node, 1, ref, R);
                const float cost = subtree_cost(a, c.x, L), other = subtree_cost(a, c.y, R);
                tbox_grow(L, R);
                const float now = a.c_node * tbox_area(L, a.w) + cost + other;
                if (__float_as_int(__ldcg(&a.cost[node])) != __float_as_int(now)) levels = 0;
                a.cost[node] = now;
                look = false;
            }
        } else {
            auto nearest = [&](int child) {
                const int up = child >= 0 ? __ldcg(&a.up[child]) : 0;
                return (up & 15) == a.round ? (up >> 4) + 1 : kTreeletReach + 1;
            };
            levels = min(nearest(c.x), nearest(c.y));
            look = look || levels <= kTreeletReach;
        }
        for (unsigned todo = __ballot_sync(0xffffffffu, look); todo; todo &= todo - 1) {
            const int src = __ffs(todo) - 1;
            const int did = treelet_node(a, __shfl_sync(0xffffffffu, node, src), t, sub2, sub3a, sub3b);
            if (lane == src) {
                if (did < 0) raise_status(a.status, ST_BOUNDS);
                if (did > 0) levels = 0;
            }
        }
        if (node >= 0 && levels < kTreeletReach) a.up[node] = (uint8_t)(levels << 4 | a.round);
        __syncwarp();  // every lane's writes, before a lane's arrival releases them
        node = node >= 0 ? parent : -1;
    }
}

// Height of the root: the longest climb of a leaf (a leaf's climb reads one
// parent link a level, the upper ones from the caches, and needs no arrivals).
__global__ void __launch_bounds__(kBuildThreads) k_root_height(const int* __restrict__ parent_node,
                                                               const int* __restrict__ parent_leaf, int n_leaves,
                                                               int n_binary, int* max_height, int* status)
{
    const int leaf = blockIdx.x * blockDim.x + threadIdx.x;
    int h = 0;
    if (leaf < n_leaves)
        for (int p = parent_leaf[leaf]; p >= 0; p = parent_node[p]) {
            if (p >= n_binary || ++h > kTreeletMaxClimb) {
                raise_status(status, ST_BOUNDS);
                break;
            }
        }
    h = __reduce_max_sync(0xffffffffu, h);
    if ((threadIdx.x & 31) == 0) atomicMax(max_height, h);
}

__global__ void k_parents_reset(int* parent_node, int n_binary)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n_binary) parent_node[i] = -1;
}

}  // namespace

size_t treelet_scratch_bytes(int64_t n_tris)
{
    // parents of nodes and leaves, expected and finished children, costs, path, mark and up bytes
    return 5 * align256(n_tris * sizeof(int)) + 3 * align256(n_tris);
}

cudaError_t restructure_treelets(cudaStream_t s, int64_t n, float4* nodes, int* max_height_dev,
                                 int rounds, float tri_cost, void* scratch, size_t scratch_bytes,
                                 unsigned long long* treelets_dev, int* status, AreaW area_w)
{
    cudaError_t e = cudaMemsetAsync(treelets_dev, 0, sizeof(unsigned long long), s);
    if (e != cudaSuccess) return e;
    if (n < 3 || rounds <= 0) return cudaSuccess;
    if (scratch_bytes < treelet_scratch_bytes(n)) return cudaErrorInvalidValue;
    const int n_binary = (int)(n - 1);
    char* p = (char*)scratch;
    int* parent_node = (int*)p; p += align256(n * sizeof(int));
    int* parent_leaf = (int*)p; p += align256(n * sizeof(int));
    unsigned* expect = (unsigned*)p; p += align256(n * sizeof(int));
    unsigned* visits = (unsigned*)p; p += align256(n * sizeof(int));
    float* cost = (float*)p; p += align256(n * sizeof(float));
    uint8_t* on_path = (uint8_t*)p; p += align256(n);
    uint8_t* mark = (uint8_t*)p; p += align256(n);
    uint8_t* up = (uint8_t*)p; p += align256(n);
    const int nb_blocks = (n_binary + 255) / 256;
    TreeletArgs a{(int)n, n_binary, nodes, parent_node, on_path, expect, visits, cost, mark, up, 0, treelets_dev,
                  status, 1.0f, tri_cost, area_w};
    e = cudaMemsetAsync(on_path, 0, (size_t)(p - (char*)on_path), s);
    if (e == cudaSuccess) e = cudaMemsetAsync(expect, 0, (size_t)((char*)cost - (char*)expect), s);
    if (e != cudaSuccess) return e;
    k_parents_reset<<<nb_blocks, 256, 0, s>>>(parent_node, n_binary);
    k_parents<<<nb_blocks, 256, 0, s>>>(nodes, n_binary, parent_node, parent_leaf, expect);
    for (int r = 0; r < rounds; ++r) {
        a.round = r + 1;
        if (r > 0) {
            e = cudaMemsetAsync(expect, 0, (size_t)((char*)cost - (char*)expect), s);  // and visits
            if (e != cudaSuccess) return e;
            k_treelet_paths<<<nb_blocks, kBuildThreads, 0, s>>>(a);
        }
        k_treelet_round<<<(n_binary + kTreeletThreads - 1) / kTreeletThreads, kTreeletThreads, 0, s>>>(a);
    }
    // parents and root height of the final shape (every box a rewrite stored is
    // the exact union of the boxes below it)
    k_parents_reset<<<nb_blocks, 256, 0, s>>>(parent_node, n_binary);
    k_parents<<<nb_blocks, 256, 0, s>>>(nodes, n_binary, parent_node, parent_leaf, nullptr);
    e = cudaMemsetAsync(max_height_dev, 0, sizeof(int), s);
    if (e != cudaSuccess) return e;
    k_root_height<<<(int)((n + kBuildThreads - 1) / kBuildThreads), kBuildThreads, 0, s>>>(
        parent_node, parent_leaf, (int)n, n_binary, max_height_dev, status);
    return cudaGetLastError();
}

}  // namespace lidar
