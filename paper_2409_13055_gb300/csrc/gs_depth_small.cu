// gs_depth_small.cu -- the depth sort of small plans in one launch.
//
// The general depth sort (gs_sort.cu) is a chain of eleven launches (three per
// digit, two for the instance offsets); below some ten thousand pairs each of
// them moves next to nothing and the chain's length is its time, and the host's
// where a program launches call by call.  Here one cluster of 8 or 16 CTAs keeps the
// pairs' keys in its shared memory through a stable LSD radix sort: a pass ranks
// a CTA's keys by warp (match, per-warp counters), exchanges the CTAs' digit
// counts through distributed shared memory and writes each key straight to its
// place in the cluster.  It takes as many digits of at most kBits bits as the
// largest key less the smallest possible one (near_z) has: three for depths
// within 2^16 near_z.  The last step sums the tiles touched in depth order.  The
// buffers hold afterwards what the general sort leaves there, bit for bit.
// Bounded by the latency of its barriers and of the ranking, some 5 us a pass on
// 10k pairs; whole binning 58 -> 36 us there (43k instances), and a render launched
// call by call 118 -> 75 us (29 launches -> 9).
#include <cooperative_groups.h>

#include <atomic>

#include "gs_internal.cuh"

namespace cg = cooperative_groups;

namespace gs {
namespace {

constexpr int kThreads = 1024, kWarps = kThreads / 32;
constexpr int kBits = 9, kDigits = 1 << kBits;
constexpr unsigned kAll = 0xffffffffu;
constexpr uint32_t kCulled = 0xFFFFFFFFu;
// Shared memory of one CTA besides the dynamic part.
struct Fixed {
    uint32_t hist[kDigits];     // this CTA's digit counts (read by the others)
    uint32_t base[kDigits];     // where its keys of a digit start in the cluster
    uint32_t warp_tot[kWarps + 1];
    uint32_t sum, max_key;      // published to the others
};

// Exclusive scan over the CTA of one value per thread; total to every thread.
__device__ __forceinline__ uint32_t cta_scan(uint32_t x, uint32_t* wt, uint32_t& total) {
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    uint32_t inc = x;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(kAll, inc, o);
        if (lane >= o) inc += y;
    }
    __syncthreads();  // wt may still be read from the scan before
    if (lane == 31) wt[w] = inc;
    __syncthreads();
    if (w == 0) {
        const uint32_t t = wt[lane];
        uint32_t ti = t;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_up_sync(kAll, ti, o);
            if (lane >= o) ti += y;
        }
        wt[lane] = ti - t;
        if (lane == 31) wt[32] = ti;
    }
    __syncthreads();
    total = wt[32];
    return inc - x + wt[w];
}

struct SmallArgs {
    const uint32_t* __restrict__ dkey;
    const uint32_t* __restrict__ touched;
    uint32_t* __restrict__ depth_order;
    uint32_t* __restrict__ offs;
    DevCounters* ctr;
    uint32_t VN, cap, near_bits;
};

// Dynamic shared memory: values | keys | the warps' digit counts.
__host__ __device__ constexpr size_t sort_bytes(int items) {
    return (size_t)kThreads * items * 8 + (size_t)kWarps * kDigits * 2;
}

template <int CTAS, int ITEMS>
__global__ void __launch_bounds__(kThreads, 1) k_depth_small(SmallArgs a) {
    extern __shared__ uint32_t dyn[];
    __shared__ Fixed fx;
    cg::cluster_group cl = cg::this_cluster();
    const int rank = (int)cl.block_rank();
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    const unsigned lt = (1u << lane) - 1u;
    uint32_t* const sval = dyn;
    uint32_t* const skey = dyn + kThreads * ITEMS;
    uint16_t* const wcnt = reinterpret_cast<uint16_t*>(skey + kThreads * ITEMS);  // [warp][digit]
    grid_dep_begin();

    // 1. depth sort.  A thread's keys: kept in registers while a pass writes.
    uint32_t key[ITEMS], val[ITEMS];
    uint32_t first = (uint32_t)rank * (uint32_t)((a.VN + CTAS - 1) / CTAS);
    uint32_t count = min((a.VN + CTAS - 1) / CTAS, a.VN - min(first, a.VN));
    // the thread's items are idx(r), r < its = ceil(count / threads): a warp's
    // items are consecutive, 32 per step
    int its = (int)((count + kThreads - 1) / kThreads);
    uint32_t mx = 0u;
#pragma unroll
    for (int r = 0; r < ITEMS; ++r) {
        key[r] = kCulled;
        val[r] = 0u;
        const uint32_t i = (uint32_t)(w * its + r) * 32u + lane;
        if (r < its && i < count) {
            val[r] = first + i;
            const uint32_t k = a.dkey[first + i];
            if (k != kCulled) {
                key[r] = k - a.near_bits;
                mx = max(mx, key[r]);
            }
        }
    }
    if (tid == 0) fx.max_key = 0u;
    __syncthreads();
    mx = __reduce_max_sync(kAll, mx);
    if (lane == 0) atomicMax(&fx.max_key, mx);
    cl.sync();
    mx = 0u;
    for (int c = 0; c < CTAS; ++c) mx = max(mx, *cl.map_shared_rank(&fx.max_key, c));
    const int bits = 32 - __clz(mx | 1u);
    const int passes = (bits + kBits - 1) / kBits, width = (bits + passes - 1) / passes;
    const uint32_t mask = (1u << width) - 1u;
    uint32_t total = 0u, chunk = 1u;  // visible pairs; of them per CTA
    for (int pass = 0; pass < passes; ++pass) {
        const int shift = pass * width;
        for (int i = tid; i < kWarps * kDigits / 2; i += kThreads)
            reinterpret_cast<uint32_t*>(wcnt)[i] = 0u;
        if (pass > 0) {
#pragma unroll
            for (int r = 0; r < ITEMS; ++r) {
                const uint32_t i = (uint32_t)(w * its + r) * 32u + lane;
                key[r] = kCulled;
                if (r < its && i < count) {
                    key[r] = skey[i];
                    val[r] = sval[i];
                }
            }
        }
        __syncthreads();
        uint16_t* const mine = wcnt + w * kDigits;
        uint32_t rk[(ITEMS + 1) / 2];  // ranks within the warp, two per word
#pragma unroll
        for (int r = 0; r < ITEMS; ++r) {
            if ((r & 1) == 0) rk[r / 2] = 0u;
            if (r >= its) continue;
            const bool ok = key[r] != kCulled;
            const uint32_t d = ok ? (key[r] >> shift) & mask : 0x10000u;
            const unsigned peers = __match_any_sync(kAll, d);
            uint32_t x = 0u;
            if (ok) x = mine[d] + __popc(peers & lt);
            __syncwarp();
            if (ok && (peers & lt) == 0u) mine[d] = (uint16_t)(mine[d] + __popc(peers));
            __syncwarp();
            rk[r / 2] |= x << (16 * (r & 1));
        }
        __syncthreads();
        if (tid < kDigits) {
            uint32_t s = 0u;
            for (int k = 0; k < kWarps; ++k) {
                const uint32_t c = wcnt[k * kDigits + tid];
                wcnt[k * kDigits + tid] = (uint16_t)s;
                s += c;
            }
            fx.hist[tid] = s;
        }
        cl.sync();  // (also: every key is in registers)
        uint32_t lower = 0u, all = 0u;
        if (tid < kDigits) {
#pragma unroll
            for (int c = 0; c < CTAS; ++c) {
                const uint32_t h = *cl.map_shared_rank(&fx.hist[tid], c);
                if (c < rank) lower += h;
                all += h;
            }
        }
        const uint32_t start = cta_scan(all, fx.warp_tot, total);
        if (tid < kDigits) fx.base[tid] = start + lower;
        __syncthreads();
        chunk = max(1u, (total + CTAS - 1) / CTAS);
        const float inv = 1.0f / (float)chunk;
#pragma unroll
        for (int r = 0; r < ITEMS; ++r) {
            if (r < its && key[r] != kCulled) {
                const uint32_t d = (key[r] >> shift) & mask;
                const uint32_t pos = fx.base[d] + mine[d] + ((rk[r / 2] >> (16 * (r & 1))) & 0xffffu);
                uint32_t c = (uint32_t)((float)pos * inv);
                if (c * chunk > pos) --c;
                if ((c + 1) * chunk <= pos) ++c;
                const uint32_t i = pos - c * chunk;
                *cl.map_shared_rank(&skey[i], (int)c) = key[r];
                *cl.map_shared_rank(&sval[i], (int)c) = val[r];
            }
        }
        first = min((uint32_t)rank * chunk, total);
        count = min(chunk, total - first);
        its = (int)((count + kThreads - 1) / kThreads);
        cl.sync();
    }

    // the instances' offsets, a thread per entry: the CTA's sum first
    uint32_t cnt[ITEMS];
    uint32_t my_total = 0u;
#pragma unroll
    for (int r = 0; r < ITEMS; ++r) {
        const uint32_t i = (uint32_t)r * kThreads + tid;
        val[r] = i < count ? sval[i] : 0u;
        cnt[r] = i < count ? a.touched[val[r]] : 0u;
    }
#pragma unroll
    for (int r = 0; r < ITEMS; ++r) {
        if ((uint32_t)r * kThreads >= count) continue;
        uint32_t t;
        const uint32_t ex = cta_scan(cnt[r], fx.warp_tot, t);
        cnt[r] = my_total + ex;
        my_total += t;
    }
    if (tid == 0) fx.sum = my_total;
    cl.sync();
    unsigned long long raw = 0ull, before = 0ull;
    for (int c = 0; c < CTAS; ++c) {
        const uint32_t s = *cl.map_shared_rank(&fx.sum, c);
        if (c < rank) before += s;
        raw += s;
    }
#pragma unroll
    for (int r = 0; r < ITEMS; ++r) {
        const uint32_t i = (uint32_t)r * kThreads + tid;
        if (i < count) {
            a.depth_order[first + i] = val[r];
            a.offs[first + i] = (uint32_t)min(before + cnt[r], 0xFFFFFFFFull);
        }
    }
    if (rank == 0 && tid == 0) {
        a.ctr->n_raw = raw;
        a.ctr->vn = total;
        a.ctr->n_sorted = total;
        a.ctr->n_instances = (uint32_t)min(raw, (unsigned long long)a.cap);
        a.offs[total] = (uint32_t)min(raw, 0xFFFFFFFFull);
        if (raw > a.cap) atomicOr(&a.ctr->status, (uint32_t)GS_DEV_CAPACITY);
    }
    cl.sync();  // the sums are shared memory: a CTA stays until all have read them
}

constexpr int kItems8 = 4, kItems16 = 8;

template <int CTAS, int ITEMS>
cudaLaunchConfig_t cluster_config(cudaLaunchAttribute (&attr)[2], cudaStream_t st) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(CTAS);
    cfg.blockDim = dim3(kThreads);
    cfg.dynamicSmemBytes = sort_bytes(ITEMS);
    cfg.stream = st;
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = CTAS;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 2;
    return cfg;
}

template <int CTAS, int ITEMS>
bool prepare() {
    auto* kern = k_depth_small<CTAS, ITEMS>;
    return cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                (int)sort_bytes(ITEMS)) == cudaSuccess &&
           (CTAS <= 8 || cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed,
                                              1) == cudaSuccess);
}

// Whether this GPU can hold a cluster of 16 such CTAs at once (asked once per
// device; a cluster of 8 is always schedulable).
bool sixteen_fit() {
    static std::atomic<int> known[64];
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return false;
    int k = known[dev].load(std::memory_order_relaxed);
    if (k == 0) {
        cudaLaunchAttribute attr[2];
        cudaLaunchConfig_t cfg = cluster_config<16, kItems16>(attr, nullptr);
        cfg.numAttrs = 1;
        int clusters = 0;
        const bool ok = prepare<16, kItems16>() &&
                        cudaOccupancyMaxActiveClusters(&clusters, k_depth_small<16, kItems16>,
                                                       &cfg) == cudaSuccess &&
                        clusters > 0;
        if (!ok) (void)cudaGetLastError();
        k = ok ? 1 : 2;
        known[dev].store(k, std::memory_order_relaxed);
    }
    return k == 1;
}

template <int CTAS, int ITEMS>
gs_status launch(const SmallArgs& a, cudaStream_t st) {
    if (!prepare<CTAS, ITEMS>()) return GS_ERR_CUDA;
    cudaLaunchAttribute attr[2];
    const cudaLaunchConfig_t cfg = cluster_config<CTAS, ITEMS>(attr, st);
    (void)cudaLaunchKernelEx(&cfg, k_depth_small<CTAS, ITEMS>, a);
    return launch_status();
}

}  // namespace

// At most 8 x 4096 pairs (8 CTAs) or 16 x 8192 (16).
bool depth_small_fits(const Plan* p, int32_t n) {
    const int64_t VN = (int64_t)p->vt.n_views * n;
    return VN <= (int64_t)8 * kThreads * kItems8 ||
           (VN <= (int64_t)16 * kThreads * kItems16 && sixteen_fit());
}

gs_status launch_depth_small(const Plan* p, int32_t n, void* ws, cudaStream_t st) {
    SmallArgs a;
    a.dkey = buf<uint32_t>(p, ws, B_DKEY_A);
    a.touched = buf<uint32_t>(p, ws, GS_BUF_TOUCHED);
    a.depth_order = buf<uint32_t>(p, ws, GS_BUF_DEPTH_ORDER);
    a.offs = buf<uint32_t>(p, ws, B_OFFSETS);
    a.ctr = buf<DevCounters>(p, ws, GS_BUF_COUNTERS);
    a.VN = (uint32_t)p->vt.n_views * (uint32_t)n;
    a.cap = (uint32_t)p->inst_capacity;
    const float near_z = p->cfg.near_z;
    __builtin_memcpy(&a.near_bits, &near_z, sizeof(near_z));
    return a.VN <= 8u * kThreads * kItems8 ? launch<8, kItems8>(a, st)
                                           : launch<16, kItems16>(a, st);
}

}  // namespace gs
