// gs_tiles.cu -- A3-A4 for plans of up to kCountTiles tiles: the emission of the
// (Gaussian, tile) instances in depth order and their stable sort by tile, as a
// counting sort over all tiles at once.
//
// The radix passes over the tile id (gs_sort.cu) move every instance once per
// digit, three launches each, and the ranges and the tile order take three more.
// Here a CTA owns a run of the emission and counts its instances of every tile in
// shared memory, so one pass places them:
//
//   k_emit_count   emits the CTA's run and writes its row of the count matrix;
//   k_tile_starts  turns the matrix's columns into starts within the tile and
//                  adds the list lengths' buckets;
//   k_place        adds the tiles' starts, counts the run again by placing warp
//                  and moves each instance to its place: a warp takes its part of
//                  the run in order, 32 instances at a time, so the sort is stable.
//                  It also writes the ranges and the heavy-first tile order.
//
// The run is cut by instances, not by Gaussians (the near ones have many times
// the tiles of the far ones).  One CTA per SM: the counters are 4 B per tile, and
// 2 B per tile and placing warp.
#include "gs_internal.cuh"

namespace gs {
namespace {

constexpr unsigned kAll = 0xffffffffu;
constexpr int kThreads = 1024, kWarps = kThreads / 32;

// Exclusive scan over the CTA (kThreads threads) of one value per thread.
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

// The part of the emission that CTA b of g takes: a multiple of 32 instances each.
__device__ __forceinline__ void cta_run(uint32_t n, uint32_t b, uint32_t g, uint32_t& lo,
                                        uint32_t& hi) {
    const uint32_t per = ((n + g - 1) / g + 31u) & ~31u;
    lo = min(b * per, n);
    hi = min(lo + per, n);
}

// Order bucket of a list length, longest first: the leading one and the next
// three bits.
__device__ __forceinline__ int len_bucket(uint32_t len) {
    if (len == 0u) return kOrderBuckets - 1;
    const int lz = __clz(len);
    const uint32_t next = lz >= 31 ? 0u : ((len << (lz + 1)) >> 29);
    return lz * kOrderSub + (int)(7u - next);
}

constexpr int kEntries = kThreads;     // entries of a round, one per thread
constexpr uint32_t kBatch = 8192;      // instances gathered before they are written out
constexpr uint32_t kLarge = 48;        // tiles from which an entry's warp lists it together
struct EmitShared {
    uint32_t key[kBatch + kBatch / 32], val[kBatch + kBatch / 32];
    uint32_t span[kEntries * kSpanRows];  // see span_word
    uint32_t first;  // the entry that holds the run's first instance
    uint32_t stop;   // the round's end
};
__device__ __forceinline__ int batch_slot(uint32_t q) { return (int)(q + (q >> 5)); }

// Row r of entry e's spans: the rows of 32 entries interleaved so that threads
// walking their own entries meet no bank conflict.
__device__ __forceinline__ uint32_t* span_word(uint32_t* span, int e, uint32_t r) {
    return span + ((e >> 5) * kSpanRows + (int)r) * 32 + (e & 31);
}

// An entry as its thread loads it, a round ahead.
struct Entry {
    uint32_t vg, off, end;
    uint2 rect;
    uint4 s0;
};

__global__ void __launch_bounds__(kThreads, 1)
k_emit_count(const uint32_t* __restrict__ order, const uint32_t* __restrict__ off,
             const uint2* __restrict__ rects, const DevCounters* __restrict__ ctr, int n,
             ViewTable vt, uint32_t* __restrict__ ikeys, uint32_t* __restrict__ ivals,
             uint32_t* __restrict__ gid_of, const uint32_t* __restrict__ spans,
             const uint32_t* __restrict__ pool, int tiles, uint32_t* __restrict__ matrix,
             uint32_t* __restrict__ order_scratch) {
    extern __shared__ uint2 dyn2[];
    EmitShared& sh = *reinterpret_cast<EmitShared*>(dyn2);
    uint32_t* const hist = reinterpret_cast<uint32_t*>(&sh + 1);
    const int tid = threadIdx.x, lane = tid & 31;
    for (int t = tid; t < tiles; t += kThreads) hist[t] = 0u;
    grid_dep_begin();
    // the tile order's bucket counts and cursors start at zero
    if (blockIdx.x == 0)
        for (int i = tid; i < 2 * kOrderBuckets; i += kThreads) order_scratch[i] = 0u;
    uint32_t lo, hi;
    cta_run(ctr->n_instances, blockIdx.x, gridDim.x, lo, hi);
    const uint32_t entries = ctr->vn;
    if (tid < 32 && lo < hi) {
        // the last entry with off[e] <= lo: 32 probes per step
        uint32_t a = 0u, b = entries;  // off[a] <= lo < off[b]
        while (b - a > 1u) {
            const uint32_t step = max(1u, (b - a + 31u) / 32u);
            const uint32_t e = a + step * (uint32_t)lane;
            const unsigned m = __ballot_sync(kAll, e < b && off[e] <= lo);
            a += step * (uint32_t)(31 - __clz(m));  // (lane 0 always answers yes)
            b = min(b, a + step);
        }
        if (lane == 0) sh.first = a;
    }
    __syncthreads();
    // the entry of this thread in the round that starts at e0 (off = end: none)
    auto load = [&](uint32_t e0) {
        Entry x = {0u, hi, hi, make_uint2(0u, 0u), make_uint4(0u, 0u, 0u, 0u)};
        const uint32_t e = e0 + (uint32_t)tid;
        if (e < entries) {
            x.vg = order[e];
            x.off = min(off[e], hi);
            x.end = min(off[e + 1], hi);
            x.rect = rects[x.vg];
            if (vt.tight_rect)
                x.s0 = *reinterpret_cast<const uint4*>(spans + (size_t)x.vg * kSpanRows);
        }
        return x;
    };
    uint32_t e0 = lo < hi ? sh.first : 0u, base = lo;
    Entry next = load(e0);
    while (base < hi && e0 < entries) {
        const Entry me = next;
        const uint32_t nrows = (me.rect.y >> 16) - (me.rect.x >> 16);
        const uint32_t x0 = me.rect.x & 0xFFFF, x1 = me.rect.y & 0xFFFF;
        const bool tall = nrows > (uint32_t)kSpanRows;
        // the rows' spans, or the rect's width in every row
        const bool has_spans = vt.tight_rect && !(tall && me.s0.x == kSpanNoPool);
        const uint32_t whole = x0 | (x1 << 16);
        if (has_spans && !tall) {
            const uint4* src = reinterpret_cast<const uint4*>(spans + (size_t)me.vg * kSpanRows);
            uint4 s[4];
            s[0] = me.s0;
#pragma unroll
            for (int k = 1; k < 4; ++k)
                s[k] = nrows > 4u * k ? src[k] : make_uint4(0u, 0u, 0u, 0u);
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                if (nrows <= 4u * k) break;
                *span_word(sh.span, tid, 4 * k) = s[k].x;
                *span_word(sh.span, tid, 4 * k + 1) = s[k].y;
                *span_word(sh.span, tid, 4 * k + 2) = s[k].z;
                *span_word(sh.span, tid, 4 * k + 3) = s[k].w;
            }
        }
        const ViewGeom& geo = vt.v[me.vg / (uint32_t)n];
        const uint32_t tiles_x = (uint32_t)geo.tiles_x;
        const uint32_t tile0 = (uint32_t)geo.tile_offset + (me.rect.x >> 16) * tiles_x;
        if (tid == kThreads - 1) sh.stop = me.end;  // (entries past the last one end at hi)
        e0 += kEntries;
        next = load(e0);  // on its way while this round is listed
        // this thread's place in its entry: instance p, row r, column x (the run may
        // start inside the first entry)
        const bool large = me.end - me.off >= kLarge || tall;
        auto span_of = [&](uint32_t row) {
            return has_spans ? *span_word(sh.span, tid, row) : whole;
        };
        uint32_t p = me.off, r = 0u, sp = whole, x = x0;
        if (!large && p < me.end) {
            uint32_t k = lo > p ? min(lo, me.end) - p : 0u;  // instances before the run
            p += k;
            sp = span_of(0u);
            while (r + 1u < nrows && k >= (sp >> 16) - (sp & 0xFFFF)) {
                k -= (sp >> 16) - (sp & 0xFFFF);
                sp = span_of(++r);
            }
            x = (sp & 0xFFFF) + k;
        }
        __syncthreads();
        const uint32_t stop = sh.stop;
        for (; base < stop; base += kBatch) {
            const uint32_t b_end = min(base + kBatch, stop);
            if (!large) {
                const uint32_t to = min(me.end, b_end);
                while (p < to) {
                    // (a count that disagreed would land past the row; stay inside
                    // the rect)
                    const int q = batch_slot(p - base);
                    sh.key[q] = tile0 + r * tiles_x + min(x, x1 - 1u);
                    sh.val[q] = me.vg;
                    ++p;
                    ++x;
                    while (x >= (sp >> 16) && r + 1u < nrows) {  // the next row with a tile
                        sp = span_of(++r);
                        x = sp & 0xFFFF;
                    }
                }
            }
            // large entries: their warp, row by row, a lane per column
            unsigned todo = __ballot_sync(kAll, large && me.off < b_end && me.end > base);
            while (todo) {
                const int src = __ffs(todo) - 1;
                todo &= todo - 1u;
                uint32_t q0 = __shfl_sync(kAll, me.off, src);
                const uint32_t e_vg = __shfl_sync(kAll, me.vg, src);
                const uint32_t e_end = min(__shfl_sync(kAll, me.end, src), b_end);
                const uint32_t e_tile = __shfl_sync(kAll, tile0, src);
                const uint32_t e_tx = __shfl_sync(kAll, tiles_x, src);
                const uint32_t e_rows = __shfl_sync(kAll, nrows, src);
                const uint32_t e_x = __shfl_sync(kAll, whole, src);
                const uint32_t e_pool = __shfl_sync(kAll, me.s0.x, src);
                const bool e_spans = __shfl_sync(kAll, (int)has_spans, src) != 0;
                const bool e_tall = e_rows > (uint32_t)kSpanRows;
                for (uint32_t row0 = 0u; row0 < e_rows && q0 < e_end; row0 += 32u) {
                    uint32_t mine = e_x;  // the span of row row0 + lane
                    if (e_spans && row0 + lane < e_rows)
                        mine = e_tall ? pool[e_pool + row0 + lane]
                                      : *span_word(sh.span, (tid & ~31) + src, lane);
                    const uint32_t rows_here = min(32u, e_rows - row0);
                    for (uint32_t k = 0u; k < rows_here && q0 < e_end; ++k) {
                        const uint32_t s = __shfl_sync(kAll, mine, (int)k);
                        const uint32_t b = s & 0xFFFF, w = (s >> 16) - b;
                        for (uint32_t c = lane; c < w; c += 32u) {
                            const uint32_t at = q0 + c;
                            if (at >= base && at < e_end) {
                                const int q = batch_slot(at - base);
                                sh.key[q] = e_tile + (row0 + k) * e_tx +
                                            min(b + c, (e_x >> 16) - 1u);
                                sh.val[q] = e_vg;
                            }
                        }
                        q0 += w;
                    }
                }
            }
            __syncthreads();
            for (uint32_t q = tid; q < b_end - base; q += kThreads) {
                const uint32_t pos = base + q, key = sh.key[batch_slot(q)];
                const uint32_t vg = sh.val[batch_slot(q)];
                ikeys[pos] = key;
                if (gid_of) gid_of[pos] = vg;  // (its value is the emission position)
                else ivals[pos] = vg;
                atomicAdd(&hist[key], 1u);
            }
            __syncthreads();
        }
        base = stop;
        __syncthreads();  // stop and the spans are written again
    }
    __syncthreads();
    uint32_t* row = matrix + (size_t)blockIdx.x * tiles;
    for (int t = tid; t < tiles; t += kThreads) row[t] = hist[t];
}

// Columns of the count matrix: 32 tiles per CTA, the rows in kSegs segments.
constexpr int kSegs = 16, kSegRows = kCountRows / kSegs;
__global__ void __launch_bounds__(32 * kSegs)
k_tile_starts(uint32_t* __restrict__ matrix, int rows, int tiles, uint32_t* __restrict__ lengths,
              uint32_t* __restrict__ buckets) {
    __shared__ uint32_t part[kSegs][32];
    grid_dep_begin();
    const int lane = threadIdx.x & 31, seg = threadIdx.x >> 5, t = blockIdx.x * 32 + lane;
    uint32_t x[kSegRows], s = 0u;
#pragma unroll
    for (int k = 0; k < kSegRows; ++k) {
        const int r = seg * kSegRows + k;
        x[k] = t < tiles && r < rows ? matrix[(size_t)r * tiles + t] : 0u;
        s += x[k];
    }
    part[seg][lane] = s;
    __syncthreads();
    uint32_t run = 0u, len = 0u;
    for (int k = 0; k < kSegs; ++k) {
        const uint32_t y = part[k][lane];
        if (k < seg) run += y;
        len += y;
    }
    if (t >= tiles) return;
#pragma unroll
    for (int k = 0; k < kSegRows; ++k) {
        const int r = seg * kSegRows + k;
        if (r < rows) matrix[(size_t)r * tiles + t] = run;
        run += x[k];
    }
    if (seg == 0) {
        lengths[t] = len;
        atomicAdd(&buckets[len_bucket(len)], 1u);
    }
}

__global__ void __launch_bounds__(kThreads, 1)
k_place(const uint32_t* __restrict__ ikeys, const uint32_t* __restrict__ ivals, int positions,
        const DevCounters* __restrict__ ctr, int tiles, int rows,
        const uint32_t* __restrict__ matrix, const uint32_t* __restrict__ lengths,
        uint32_t* __restrict__ buckets, uint32_t* __restrict__ keys, uint32_t* __restrict__ vals,
        uint2* __restrict__ ranges, uint32_t* __restrict__ order) {
    extern __shared__ uint32_t dyn[];
    __shared__ uint32_t wt[kWarps + 1], bucket0[kOrderBuckets];
    uint32_t* const start = dyn;  // [tiles]: where this CTA's instances of the tile go
    uint32_t* const cnt = dyn + (tiles + 1) / 2 * 2;  // [rows] 16-bit counters per placing warp
    const int words = (tiles + 3) / 4 * 2;             // 32-bit words per row
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    const unsigned lt = (1u << lane) - 1u;
    for (int i = tid; i < rows * words; i += kThreads) cnt[i] = 0u;
    grid_dep_begin();
    uint32_t total;
    {
        const uint32_t s = cta_scan(tid < kOrderBuckets ? buckets[tid] : 0u, wt, total);
        if (tid < kOrderBuckets) bucket0[tid] = s;
    }
    // the tiles' starts: lengths to shared memory, a thread's consecutive tiles
    // summed, one scan over the CTA
    const int each = ((tiles + kThreads - 1) / kThreads) | 1;  // (odd: free of bank conflicts)
    const uint32_t* mine = matrix + (size_t)blockIdx.x * tiles;
    for (int t0 = tid; t0 < tiles; t0 += 8 * kThreads) {
        uint32_t x[8];
#pragma unroll
        for (int k = 0; k < 8; ++k)
            x[k] = t0 + k * kThreads < tiles ? lengths[t0 + k * kThreads] : 0u;
#pragma unroll
        for (int k = 0; k < 8; ++k)
            if (t0 + k * kThreads < tiles) start[t0 + k * kThreads] = x[k];
    }
    __syncthreads();
    {
        const int a = min(tid * each, tiles), b = min(a + each, tiles);
        uint32_t s = 0u;
        for (int t = a; t < b; ++t) s += start[t];
        s = cta_scan(s, wt, total);
        for (int t = a; t < b; ++t) {
            const uint32_t len = start[t];
            start[t] = s;
            s += len;
        }
    }
    __syncthreads();
    // the ranges, the order and the sorted keys of this CTA's slice of the tiles
    const int slice = (tiles + gridDim.x - 1) / gridDim.x;
    const int own0 = min((int)blockIdx.x * slice, tiles), own1 = min(own0 + slice, tiles);
    for (int t = own0 + tid; t < own1; t += kThreads) {
        const uint32_t len = lengths[t], b = start[t];
        ranges[t] = len ? make_uint2(b, b + len) : make_uint2(0u, 0u);
        const int k = len_bucket(len);
        order[bucket0[k] + atomicAdd(&buckets[kOrderBuckets + k], 1u)] = (uint32_t)t;
    }
    const uint32_t n_inst = ctr->n_instances;
    for (int t = own0 + w; t < own1; t += kWarps) {
        const uint32_t b = start[t], e = t + 1 < tiles ? start[t + 1] : n_inst;
        for (uint32_t p = b + lane; p < e; p += 32u) keys[p] = (uint32_t)t;
    }
    __syncthreads();
    for (int t0 = tid; t0 < tiles; t0 += 8 * kThreads) {
        uint32_t x[8];
#pragma unroll
        for (int k = 0; k < 8; ++k)
            x[k] = t0 + k * kThreads < tiles ? mine[t0 + k * kThreads] : 0u;
#pragma unroll
        for (int k = 0; k < 8; ++k)
            if (t0 + k * kThreads < tiles) start[t0 + k * kThreads] += x[k];
    }
    // this CTA's run again, by placing warp
    uint32_t lo, hi;
    cta_run(n_inst, blockIdx.x, gridDim.x, lo, hi);
    const uint32_t per = max(32u, ((hi - lo + rows - 1) / rows + 31u) & ~31u);
    __syncthreads();
    for (uint32_t p0 = lo + tid; p0 < hi; p0 += 8u * kThreads) {
        uint32_t k[8];
#pragma unroll
        for (int j = 0; j < 8; ++j)
            k[j] = p0 + j * kThreads < hi ? ikeys[p0 + j * kThreads] : 0u;
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            const uint32_t p = p0 + j * kThreads;
            if (p < hi)
                atomicAdd(&cnt[(p - lo) / per * words + (k[j] >> 1)], 1u << (16 * (k[j] & 1)));
        }
    }
    __syncthreads();
    // counts -> exclusive over the CTA's warps, two tiles at a time
    for (int i = tid; i < words; i += kThreads) {
        uint32_t s = 0u;
        for (int r0 = 0; r0 < rows; r0 += 8) {
            uint32_t x[8];
#pragma unroll
            for (int r = 0; r < 8; ++r) x[r] = r0 + r < rows ? cnt[(r0 + r) * words + i] : 0u;
#pragma unroll
            for (int r = 0; r < 8; ++r) {
                if (r0 + r < rows) cnt[(r0 + r) * words + i] = s;
                s += x[r];
            }
        }
    }
    __syncthreads();
    if (w < rows) {
        uint16_t* const cur = reinterpret_cast<uint16_t*>(cnt + (size_t)w * words);
        const uint32_t b = min(lo + (uint32_t)w * per, hi), e = min(b + per, hi);
        auto get = [&](uint32_t p) {
            return p < e ? make_uint2(ikeys[p], positions ? p : ivals[p])
                         : make_uint2(kAll, 0u);
        };
        constexpr int kAhead = 6;  // steps of 32 instances in flight
        uint2 ahead[kAhead];
#pragma unroll
        for (int k = 0; k < kAhead; ++k) ahead[k] = get(b + 32u * k + lane);
        for (uint32_t p0 = b; p0 < e; p0 += 32u * kAhead) {
#pragma unroll
            for (int k = 0; k < kAhead; ++k) {
                const uint2 x = ahead[k];
                const uint32_t p = p0 + 32u * k + lane;
                ahead[k] = get(p + 32u * kAhead);
                const unsigned peers = __match_any_sync(kAll, x.x);
                const bool ok = p < e;
                uint32_t pos = 0u, c = 0u;
                if (ok) {
                    c = cur[x.x];
                    pos = start[x.x] + c + __popc(peers & lt);
                }
                __syncwarp();
                if (ok && (peers & lt) == 0u) cur[x.x] = (uint16_t)(c + __popc(peers));
                __syncwarp();
                if (ok) vals[pos] = x.y;
            }
        }
    }
}

size_t emit_smem(int tiles) { return sizeof(EmitShared) + (size_t)tiles * 4; }
size_t place_smem(int tiles, int rows) {
    return (size_t)((tiles + 1) / 2 * 2) * 4 + (size_t)rows * ((tiles + 3) / 4 * 2) * 4;
}
constexpr size_t kSmemMost = 226 * 1024 - 2048;  // dynamic, beside the static arrays

// Placing warps: as many as have room for their counters.
int placing_rows(int tiles) {
    int r = kWarps;
    while (r > 1 && place_smem(tiles, r) > kSmemMost) r = r > 8 ? r / 2 : r - 1;
    return place_smem(tiles, r) <= kSmemMost ? r : 0;
}

}  // namespace

// Plans whose tiles' counters fit shared memory and whose capacity is at most
// 2^20 instances: the counting sort is then two to three launches instead of ten.
// Larger ones are ahead with the radix passes, whose writes are runs of a digit
// (one CTA per SM and a 4-byte write per instance here): 3.1M instances over 12750
// tiles 175 us for the whole binning against 159, 150k over 1200 tiles 51 against
// 60, 43k over 300 tiles 36 against 58.
bool tiles_fit(const Plan* p) {
    return sm_count() > 0 && p->inst_capacity <= (int64_t(1) << 20) &&
           p->inst_capacity / sm_count() < 65000 &&  // (a run's counts of a tile are 16 bits)
           p->total_tiles <= kCountTiles && p->len[B_TILE_COUNTS] != 0 &&
           emit_smem(p->total_tiles) <= kSmemMost && placing_rows(p->total_tiles) > 0;
}

gs_status launch_tiles(const Plan* p, int32_t n, void* ws, cudaStream_t st) {
    const bool odd = (p->tile_passes & 1) != 0;  // where readers look for the sorted instances
    const bool det = p->cfg.deterministic != 0;
    uint32_t* ek = buf<uint32_t>(p, ws, odd ? (int)GS_BUF_TILE_KEYS : (int)B_IKEY_B);
    uint32_t* ev = buf<uint32_t>(p, ws, odd ? (int)GS_BUF_TILE_VALUES : (int)B_IVAL_B);
    uint32_t* keys = buf<uint32_t>(p, ws, odd ? (int)B_IKEY_B : (int)GS_BUF_TILE_KEYS);
    uint32_t* vals = buf<uint32_t>(p, ws, odd ? (int)B_IVAL_B : (int)GS_BUF_TILE_VALUES);
    uint32_t* matrix = buf<uint32_t>(p, ws, B_TILE_COUNTS);
    uint32_t* lengths = matrix + (size_t)kCountRows * p->total_tiles;
    uint32_t* order = buf<uint32_t>(p, ws, B_TILE_ORDER);
    uint32_t* buckets = order + p->total_tiles;  // counts | cursors
    const DevCounters* ctr = buf<DevCounters>(p, ws, GS_BUF_COUNTERS);
    const int tiles = p->total_tiles, rows = placing_rows(tiles);
    const int g = sm_count() < kCountRows ? sm_count() : kCountRows;
    const size_t se = emit_smem(tiles), sp = place_smem(tiles, rows);
    if (cudaFuncSetAttribute(k_emit_count, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)se) !=
            cudaSuccess ||
        cudaFuncSetAttribute(k_place, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sp) !=
            cudaSuccess)
        return GS_ERR_CUDA;
    launch_pdl(k_emit_count, g, kThreads, se, st, buf<uint32_t>(p, ws, GS_BUF_DEPTH_ORDER),
               buf<uint32_t>(p, ws, B_OFFSETS), buf<uint2>(p, ws, GS_BUF_RECT), ctr, n, p->vt, ek,
               ev, det ? buf<uint32_t>(p, ws, B_GID_OF) : nullptr, buf<uint32_t>(p, ws, B_SPANS),
               cbuf<uint32_t>(p, ws, B_SPAN_POOL), tiles, matrix, buckets);
    launch_pdl(k_tile_starts, (tiles + 31) / 32, 32 * kSegs, 0, st, matrix, g, tiles, lengths,
               buckets);
    launch_pdl(k_place, g, kThreads, sp, st, ek, ev, det ? 1 : 0, ctr, tiles, rows, matrix,
               lengths, buckets, keys, vals, buf<uint2>(p, ws, GS_BUF_RANGES), order);
    return launch_status();
}

}  // namespace gs
