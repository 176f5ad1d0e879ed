// gs_blocks.cu -- A5 forward compositing and A7 pixel adjoint over 8x8 pixel
// blocks, for tiles that are whole 8x8 blocks.
//
// A warp owns one 8x8 block of a tile: lane l holds the two pixels of row l / 4
// at columns 2 (l % 4) and the next one.  It walks its tile's list on its own,
// so nothing in these kernels waits for another warp.
//
//  * Staging.  32 list entries at a time, one per lane: the lane's record
//    arrives by cp.async, is turned into tile-local coordinates and, where the
//    tile is more than the block or its list is a square rect's, tested
//    against the block (the smallest value of the Gaussian's quadratic form
//    over the block's rectangle).  The Gaussians that can reach the block are
//    packed into the warp's stage two by two: {x, x', y, y'}, {-a/2, -a'/2, -b, -b'},
//    {-c/2, -c'/2, -o, -o'}, so that one packed FP32 operation (.f32x2) evaluates
//    both at a pixel with no register shuffled into pairs.
//  * The forward blends front to back, the adjoint walks back to front; both
//    evaluate alpha with the same rounded operations as gs_render.cu and take
//    the same decisions.
//  * The adjoint's sums over the block.  Per blended Gaussian the 64 pixels'
//    dL/dpower and blend weights go to shared memory as one row of a window; over
//    eight rows a lane then sums the pixel pairs of one column of one row, and four
//    lanes add up.  Products and sums are FP32, about the Gaussian's mean and in
//    the order of the shuffles of gs_render.cu: an 8x8 tile's sums are the same
//    bits as that kernel's.
//
// What bounds them: instruction issue and the ALU and heavy FMA pipes, two
// cycles per instruction each (packed FP32 runs on the heavy pipe alone), and
// for small launches the longest list, which one warp walks.  At 1M Gaussians,
// 1200x680, 8x8 tiles (2.0M walked (block, Gaussian) pairs), against the kernels
// of gs_render.cu at their best launch shape: forward 182 -> 128 us, adjoint 319 ->
// 240 us.  Sixteen views of a 500k map: 1003 -> 629 and 1593 -> 1332 us.  200k
// Gaussians, 640x480, 16x16 tiles: 68 -> 37 and 177 -> 70 us (there the block test
// and the four warps per tile count as well).
//
// The sums on mma.sync (TF32, each operand in two parts) take 233 us at 1M and
// 77 at 200k, and two parts hold 22 bits of 24: every product came out low by 2e-7
// on average, four times the rounding of the FP32 sums in the gradients of the SH
// coefficients.  Tried and not kept: 32 slots per stage for a sixth CTA per SM (256
// us against 241 then).  In the forward, two pairs evaluated before a vote: 137 ->
// 131 us.
#include "gs_render.cuh"

namespace gs {
namespace {

constexpr int kBlock = 8;      // pixels along each side of a block
constexpr int kWarps = 4;      // warps (blocks) per CTA
constexpr int kChunk = 32;     // list entries staged at a time, one per lane
constexpr int kStep = 2;       // pairs of Gaussians the forward evaluates before a vote
constexpr unsigned kAll = 0xffffffffu;

// e^p = 2^(p log2 e) by the hardware's base-2 exponential (ex2.approx.ftz): the
// results below 2^-126 that it flushes to zero are far below 1/255.
constexpr float kLog2e = 1.4426950408889634f;
__device__ __forceinline__ float ex2_approx(float x) {
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
__device__ __forceinline__ float2 dup(float x) { return make_float2(x, x); }

// A Gaussian that does not count at a pixel is multiplied by zero there.  Where a
// colour of the map or a dL/dC of the block is wild(), the ODD variants select
// instead.  (The projection says whether a colour is: looked for in every chunk, the
// adjoint of 16 views of 500k took 1386 us against 1332.)
__device__ __forceinline__ float2 where(float2 n, float2 x, float2 y) {
    return make_float2(n.x != 0.0f ? x.x : y.x, n.y != 0.0f ? x.y : y.y);
}

// A warp's staged Gaussians.  par: pairs of slots; col: the colour, each
// channel twice, and the slot's tag (the list position in the forward, the
// list value in the adjoint).
template <int SLOTS>
struct Stage {
    float4 par[SLOTS / 2][3];
    float4 col[SLOTS][2];
};

// Whether the Gaussian's alpha can reach 1/255 in the pixels [x0, x0 + 7] x
// [y0, y0 + 7]: q(d) = a dx^2 + 2 b dx dy + c dy^2 against 2 ln(255 o).  The
// smallest q over a rectangle that does not hold the mean lies on one of the
// two edges that face it.  The level is widened by what rounding can do: 1% +
// 0.02 for the logarithm and the exponential, and for the form's terms, which
// cancel along a needle, 2e-6 of the largest sum of their magnitudes in the block
// (a pixel's power and q here are each off by at most six roundings of 2^-24 of it).
__device__ __forceinline__ bool meets_block(float lx, float ly, float a, float b, float c,
                                            float o, float x0, float y0) {
    const float xe = fminf(fmaxf(lx, x0), x0 + 7.0f) - lx;
    const float ye = fminf(fmaxf(ly, y0), y0 + 7.0f) - ly;
    const float dy = fminf(fmaxf(__fdividef(-b * xe, c), y0 - ly), y0 + 7.0f - ly);
    const float dx = fminf(fmaxf(__fdividef(-b * ye, a), x0 - lx), x0 + 7.0f - lx);
    const float q1 = fmaf(a * xe, xe, fmaf(2.0f * b * xe, dy, c * dy * dy));
    const float q2 = fmaf(a * dx, dx, fmaf(2.0f * b * dx, ye, c * ye * ye));
    const float X = fabsf(x0 + 3.5f - lx) + 3.5f, Y = fabsf(y0 + 3.5f - ly) + 3.5f;
    const float most = fmaf(a * X, X, fmaf(2.0f * fabsf(b) * X, Y, c * Y * Y));
    const float level = fmaf(2e-6f, most, 2.02f * __logf(255.0f * o) + 0.02f);
    return !(fminf(q1, q2) > level);
}

// One chunk of a list on its way through a warp's raw buffer into its stage.
// RING chunks are in flight.
template <int SLOTS, int RING>
struct Feeder {
    float4* raw;  // RING x kChunk x 3
    Stage<SLOTS>* st;
    const uint32_t* __restrict__ ivals;
    const uint32_t* __restrict__ gid_of;
    const float4* __restrict__ rec;
    uint32_t next;         // this lane's list value of the next chunk to issue
    uint32_t tag[RING];    // ... and of the chunks in flight
    int issued;            // chunks issued so far

    // pos(c): this lane's position in the list in chunk c, or -1
    template <class Pos>
    __device__ __forceinline__ void load_next(const Pos& pos) {
        const int p = pos(issued);
        next = p >= 0 ? __ldg(ivals + p) : 0u;
    }
    template <class Pos>
    __device__ __forceinline__ void issue(const Pos& pos, int slot, int lane) {
        const int p = pos(issued);
#pragma unroll
        for (int k = 0; k < RING; ++k)
            if (slot == k) tag[k] = next;
        if (p >= 0) {
            const uint32_t vg = gid_of ? __ldg(gid_of + next) : next;
            const float4* src = rec + (size_t)vg * 3;
            float4* dst = raw + (slot * kChunk + lane) * 3;
            cp_async16(dst, src);
            cp_async16(dst + 1, src + 1);
            cp_async16(dst + 2, src + 2);
        }
        cp_async_commit();
        ++issued;
        load_next(pos);
    }
    template <class Pos>
    __device__ __forceinline__ void start(const Pos& pos, int lane) {
        issued = 0;
        load_next(pos);
#pragma unroll
        for (int i = 0; i < RING; ++i) issue(pos, i, lane);
    }
    // Stages chunk c behind the ns slots in use; returns the lanes whose entry
    // was kept.  LISTPOS: the tag is the list position instead of the value.
    template <int CH, bool CULL, bool LISTPOS, class Pos>
    __device__ __forceinline__ unsigned stage(const Pos& pos, int c, int ns, int lane, float tx0,
                                              float ty0, float bx, float by, int list_base) {
        asm volatile("cp.async.wait_group %0;\n" ::"n"(RING - 1) : "memory");
        __syncwarp();
        const int slot = RING == 1 ? 0 : (c & (RING - 1));
        const int p = pos(c);
        float4 m, q, col = make_float4(0.f, 0.f, 0.f, 0.f);
        bool keep = p >= 0;
        if (keep) {
            const float4* src = raw + (slot * kChunk + lane) * 3;
            m = src[0];
            q = src[1];
            col = src[2];
            m.x = __fadd_rn(__fsub_rn(m.x, tx0), m.z);
            m.y = __fadd_rn(__fsub_rn(m.y, ty0), m.w);
            if (CULL) keep = meets_block(m.x, m.y, q.x, q.y, q.z, q.w, bx, by);
        }
        uint32_t t = tag[0];
#pragma unroll
        for (int k = 1; k < RING; ++k) t = slot == k ? tag[k] : t;
        const unsigned mask = __ballot_sync(kAll, keep);
        issue(pos, slot, lane);
        if (keep) {
            const int s = ns + __popc(mask & ((1u << lane) - 1u));
            float* f = reinterpret_cast<float*>(&st->par[s >> 1][0]) + (s & 1);
            f[0] = m.x;
            f[2] = m.y;
            f[4] = -0.5f * q.x;
            f[6] = -q.y;
            f[8] = -0.5f * q.z;
            f[10] = -q.w;
            const float word = __uint_as_float(LISTPOS ? (uint32_t)(p - list_base) : t);
            if (CH == 3) {
                st->col[s][0] = make_float4(col.x, col.x, col.y, col.y);
                st->col[s][1] = make_float4(col.z, col.z, word, 0.0f);
            } else {
                const float g = (col.x + col.y + col.z) * (1.0f / 3.0f);
                st->col[s][0] = make_float4(g, g, word, 0.0f);
            }
        }
        return mask;
    }
    // The slots from ns to the next multiple of M never reach a pixel.
    template <int M>
    __device__ __forceinline__ void pad(int ns, int lane) {
        const int top = (ns + M - 1) & ~(M - 1);
        for (int s = ns; s < top; ++s) {
            if (lane < 6) reinterpret_cast<float*>(&st->par[s >> 1][0])[2 * lane + (s & 1)] = 0.0f;
            if (lane < 8) reinterpret_cast<float*>(&st->col[s][0])[lane] = 0.0f;
        }
    }
    // Whether a staged Gaussian may need what most do not: it can reach alpha =
    // 0.99 (o >= 0.99), or its conic is so close to singular that rounding could
    // make its power positive.  With b^2 <= (1 - e) a c the exact power is at
    // most -e/4 (a dx^2 + c dy^2) and its rounding error below 4e-7 times the
    // same sum: e = 1e-5.
    __device__ __forceinline__ bool hard(int ns, int lane) const {
        bool h = false;
#pragma unroll
        for (int k = 0; k < SLOTS / 64; ++k) {
            const int p = lane + 32 * k;
            if (2 * p < ns) {
                const float4 B = st->par[p][1], D = st->par[p][2];
                h = h || !(D.z > -kAlphaMax && D.w > -kAlphaMax &&
                           B.z * B.z <= 3.99996f * B.x * D.x &&
                           B.w * B.w <= 3.99996f * B.y * D.y);
            }
        }
        return __any_sync(kAll, h);
    }
};

// -o e^power of two Gaussians (the halves) at one pixel, and their powers.
struct PairAlpha {
    float2 pw, noG;
};
// hcdd, ha: -c dy^2 / 2 and -a / 2 (halving is exact, so the power -(a dx^2 + c
// dy^2) / 2 - b dx dy is rounded as gauss_power rounds it).
__device__ __forceinline__ PairAlpha pair_alpha(float2 dx, float2 dy, float2 hcdd, float2 ha,
                                                float2 nb, float2 no) {
    PairAlpha r;
    const float2 q = fma2(ha, mul2(dx, dx), hcdd), t = mul2(nb, mul2(dx, dy));
    // (scalar sums: a packed product whose only use is a packed sum is fused
    // with it, which rounds once instead of twice)
    r.pw = make_float2(__fadd_rn(q.x, t.x), __fadd_rn(q.y, t.y));
    r.noG = mul2(no, make_float2(ex2_approx(r.pw.x * kLog2e), ex2_approx(r.pw.y * kLog2e)));
    return r;
}
// ... with alpha clamped at 0.99 and no weight at a positive power, for the
// batches that Feeder::hard names (the others reach neither).
__device__ __forceinline__ float2 tame(const PairAlpha& e) {
    return make_float2(e.pw.x <= 0.0f ? fmaxf(-kAlphaMax, e.noG.x) : 0.0f,
                       e.pw.y <= 0.0f ? fmaxf(-kAlphaMax, e.noG.y) : 0.0f);
}

// ---------------------------------------------------------------------------
// Forward.
// ---------------------------------------------------------------------------

template <int CH>
struct FwdPixels {
    float2 T, C[CH];  // transmittance, negated once the pixel is done; minus the colour
    int l0, l1;       // slot of the last blended Gaussian of this batch, or -1
};

// Blends one Gaussian (n = -alpha where it counts at the pixel, else 0) at both
// pixels without a branch: alpha zero leaves a pixel as it is; the Gaussian
// that would take T below 1e-4 is not added and negates T, after which nothing
// passes the test of Tn.  ODD: the colour may be wild.
template <int CH, bool ODD>
__device__ __forceinline__ void blend_one(FwdPixels<CH>& s, float2 na, const float4* col,
                                          int slot) {
    const float2 Tn = mul2(s.T, make_float2(1.0f + na.x, 1.0f + na.y));
    const bool a0 = Tn.x >= kTMin, a1 = Tn.y >= kTMin;
    const float2 w = mul2(na, s.T);
    const float2 nw = make_float2(a0 ? w.x : 0.0f, a1 ? w.y : 0.0f);
    const float4 c01 = col[0];
    auto add = [&](float2 c, float2& C) {
        const float2 x = fma2(nw, c, C);
        C = ODD ? where(nw, x, C) : x;
    };
    add(make_float2(c01.x, c01.y), s.C[0]);
    if constexpr (CH == 3) {
        add(make_float2(c01.z, c01.w), s.C[1]);
        add(*reinterpret_cast<const float2*>(col + 1), s.C[2]);
    }
    s.l0 = nw.x < 0.0f ? slot : s.l0;
    s.l1 = nw.y < 0.0f ? slot : s.l1;
    s.T.x = a0 ? Tn.x : -fabsf(s.T.x);
    s.T.y = a1 ? Tn.y : -fabsf(s.T.y);
}

// Blends a staged batch.  HARD: alphas are clamped and positive powers skipped.
// ODD: some colour is wild.
template <int CH, bool HARD, bool ODD, int SLOTS>
__device__ __forceinline__ void blend_batch(FwdPixels<CH>& s, const Stage<SLOTS>& st, int ns,
                                            float2 nx0, float2 nx1, float2 ny) {
    constexpr int kS = ODD ? 1 : kStep;
    auto evaluate = [&](int p, float2& n0, float2& n1) {
        const float4 A = st.par[p][0], B = st.par[p][1], D = st.par[p][2];
        const float2 dy = add2(make_float2(A.z, A.w), ny);
        const float2 cdd = mul2(make_float2(D.x, D.y), mul2(dy, dy));
        const float2 gx = make_float2(A.x, A.y), a = make_float2(B.x, B.y),
                     nb = make_float2(B.z, B.w), no = make_float2(D.z, D.w);
        const PairAlpha e0 = pair_alpha(add2(gx, nx0), dy, cdd, a, nb, no);
        const PairAlpha e1 = pair_alpha(add2(gx, nx1), dy, cdd, a, nb, no);
        n0 = HARD ? tame(e0) : e0.noG;
        n1 = HARD ? tame(e1) : e1.noG;
    };
    for (int p = 0; 2 * p < ns; p += kS) {
        float2 n0[kS], n1[kS];
        bool mine0 = false, mine1 = false;
#pragma unroll
        for (int k = 0; k < kS; ++k) {
            evaluate(p + k, n0[k], n1[k]);
            mine0 = mine0 || fminf(n0[k].x, n0[k].y) <= -kAlphaMin;
            mine1 = mine1 || fminf(n1[k].x, n1[k].y) <= -kAlphaMin;
        }
        // one vote for the step: that a pixel still accumulating blends any
        if (!__any_sync(kAll, (mine0 && s.T.x > 0.0f) || (mine1 && s.T.y > 0.0f))) {
            if (!__any_sync(kAll, fmaxf(s.T.x, s.T.y) > 0.0f)) return;
            continue;
        }
#pragma unroll
        for (int k = 0; k < kS; ++k) {
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const float a0 = h ? n0[k].y : n0[k].x, a1 = h ? n1[k].y : n1[k].x;
                const float2 na = make_float2(a0 <= -kAlphaMin ? a0 : 0.0f,
                                              a1 <= -kAlphaMin ? a1 : 0.0f);
                const int slot = 2 * (p + k) + h;
                blend_one<CH, ODD>(s, na, st.col[slot], slot);
            }
        }
    }
}

template <int CH, bool CULL, int SLOTS, int RING>
__device__ __forceinline__ void fwd_block(const ViewTable& vt, const TileCtx& tc, int bx, int by,
                                          Feeder<SLOTS, RING>& fd, bool odd, float bg0, float bg1,
                                          float bg2, float* __restrict__ images,
                                          float* __restrict__ final_T,
                                          int32_t* __restrict__ last_idx) {
    const int lane = threadIdx.x & 31;
    const int lx = bx + 2 * (lane & 3), ly = by + (lane >> 2);
    const int px = tc.tx0 + lx, py = tc.ty0 + ly;
    const float2 nx0 = dup(-(float)lx), nx1 = dup(-(float)(lx + 1)), ny = dup(-(float)ly);
    const bool in0 = py < tc.height && px < tc.width, in1 = py < tc.height && px + 1 < tc.width;
    FwdPixels<CH> s;
    s.T = make_float2(in0 ? 1.0f : -1.0f, in1 ? 1.0f : -1.0f);
#pragma unroll
    for (int c = 0; c < CH; ++c) s.C[c] = dup(0.0f);
    int last0 = 0, last1 = 0;
    const int total = (int)(tc.end - tc.begin), begin = (int)tc.begin;
    const int chunks = (total + kChunk - 1) / kChunk;
    auto pos = [&](int c) {
        const int i = c * kChunk + lane;
        return i < total ? begin + i : -1;
    };
    fd.start(pos, lane);
    int c = 0;
    bool alive = __any_sync(kAll, in0 || in1);
    while (c < chunks && alive) {
        int ns = 0;
        do {
            ns += __popc(fd.template stage<CH, CULL, true>(pos, c, ns, lane, (float)tc.tx0,
                                                           (float)tc.ty0, (float)bx, (float)by,
                                                           begin));
            ++c;
        } while (ns <= SLOTS - kChunk && c < chunks);
        fd.template pad<2 * kStep>(ns, lane);
        __syncwarp();
        s.l0 = s.l1 = -1;
        if (odd)
            blend_batch<CH, true, true>(s, *fd.st, ns, nx0, nx1, ny);
        else if (fd.hard(ns, lane))
            blend_batch<CH, true, false>(s, *fd.st, ns, nx0, nx1, ny);
        else
            blend_batch<CH, false, false>(s, *fd.st, ns, nx0, nx1, ny);
        constexpr int kTag = CH == 3 ? 6 : 2;
        if (s.l0 >= 0)
            last0 = __float_as_int(reinterpret_cast<const float*>(fd.st->col[s.l0])[kTag]) + 1;
        if (s.l1 >= 0)
            last1 = __float_as_int(reinterpret_cast<const float*>(fd.st->col[s.l1])[kTag]) + 1;
        alive = __any_sync(kAll, fmaxf(s.T.x, s.T.y) > 0.0f);
    }
    cp_async_wait_all();  // nothing may still be landing in shared memory
    __syncwarp();
    if (!in0) return;
    s.T = make_float2(fabsf(s.T.x), fabsf(s.T.y));
    const int64_t plane = (int64_t)tc.width * tc.height;
    const int64_t pix = (int64_t)py * tc.width + px;
    const float bgc[3] = {bg0, bg1, bg2};
    const float bgg = (bg0 + bg1 + bg2) * (1.0f / 3.0f);
#pragma unroll
    for (int ch = 0; ch < CH; ++ch) {
        float* o = images + tc.val_base + ch * plane + pix;
        const float b = CH == 3 ? bgc[ch] : bgg;
        o[0] = fmaf(s.T.x, b, -s.C[ch].x);
        if (in1) o[1] = fmaf(s.T.y, b, -s.C[ch].y);
    }
    final_T[tc.pix_base + pix] = s.T.x;
    last_idx[tc.pix_base + pix] = last0;
    if (in1) {
        final_T[tc.pix_base + pix + 1] = s.T.y;
        last_idx[tc.pix_base + pix + 1] = last1;
    }
}

// A warp's next block: a slot of the heavy-first tile order times the tile's
// blocks, from the launch's queue counter.
__device__ __forceinline__ int next_slot(uint32_t* queue) {
    int s = 0;
    if ((threadIdx.x & 31) == 0) s = (int)atomicAdd(queue, 1u);
    return __shfl_sync(kAll, s, 0);
}

constexpr int kSlots = 2 * kChunk;
// Chunks in flight: where the block test may leave a chunk little to do, the
// copies of several have to overlap (two to four: 43 -> 41 us forward and 86 -> 80
// adjoint at 200k Gaussians with 16x16 tiles).
template <bool CULL>
constexpr int kRing = CULL ? 4 : 1;

template <bool CULL>
struct FwdShared {
    Stage<kSlots> st;
    float4 raw[kRing<CULL> * kChunk * 3];
};

template <bool CULL>
__global__ void __launch_bounds__(32 * kWarps, CULL ? 5 : 8)
k_blocks_fwd(ViewTable vt, const uint32_t* __restrict__ ranges,
             const uint32_t* __restrict__ order, const uint32_t* __restrict__ ivals,
             const uint32_t* __restrict__ gid_of, const float4* __restrict__ rec, int log2_bx,
             int log2_blocks, int total_blocks, uint32_t* queue,
             const DevCounters* __restrict__ ctr, float bg0, float bg1, float bg2,
             float* __restrict__ images, float* __restrict__ final_T,
             int32_t* __restrict__ last_idx) {
    __shared__ FwdShared<CULL> sh[kWarps];
    FwdShared<CULL>& my = sh[threadIdx.x >> 5];
    Feeder<kSlots, kRing<CULL>> fd;
    fd.raw = my.raw;
    fd.st = &my.st;
    fd.ivals = ivals;
    fd.gid_of = gid_of;
    fd.rec = rec;
    const bool wild_map = ctr->wild_colour != 0u;
    for (;;) {
        const int slot = next_slot(queue);
        if (slot >= total_blocks) break;
        const TileCtx tc = tile_ctx(vt, ranges, (int)order[slot >> log2_blocks]);
        const int sub = slot & ((1 << log2_blocks) - 1);
        const int bx = (sub & ((1 << log2_bx) - 1)) * kBlock, by = (sub >> log2_bx) * kBlock;
        if (tc.tx0 + bx >= tc.width || tc.ty0 + by >= tc.height) continue;
        if (tc.channels == 3)
            fwd_block<3, CULL>(vt, tc, bx, by, fd, wild_map, bg0, bg1, bg2, images, final_T,
                               last_idx);
        else
            fwd_block<1, CULL>(vt, tc, bx, by, fd, wild_map, bg0, bg1, bg2, images, final_T,
                               last_idx);
    }
}

// ---------------------------------------------------------------------------
// Adjoint.
// ---------------------------------------------------------------------------

// Rows of the window in shared memory: Gaussian r's lane e (its two pixels)
// holds {dp, dp', w, w'} (both negated) at row_slot(r, e); the order within a row makes
// the reads below free of bank conflicts.
constexpr int kRows = 8;
__device__ __forceinline__ int row_slot(int r, int e) { return r * 32 + (e ^ ((r & 1) << 2)); }
// ... and {|h_x|, |h_y|} of the density statistic.
__device__ __forceinline__ int abs_slot(int r, int e) { return r * 32 + (e ^ ((r & 3) << 2)); }

template <bool CULL, bool ABS>
struct BwdShared {
    float4 win[kRows * 32];
    float2 habs[ABS ? kRows * 32 : 2];
    float4 g01[32];  // dL/dC of the lanes' two pixels, channels 0 and 1
    float2 g2[32];   // ... and the last channel
    Stage<kSlots> st;
    float4 raw[kRing<CULL> * kChunk * 3];
};

struct BwdOut {
    float* __restrict__ grad2d;
    float* __restrict__ absgrad;
    float* __restrict__ partial;
};

// One sum of flush_window over the lanes of a row: x holds the pairs' sums of
// rows {0, 1} + {4, 5}, y those of {2, 3} + {6, 7}; then the row's four lanes.
__device__ __forceinline__ float block_sum(float2 x, float2 y) {
    const float2 z = add2(x, y);
    float t = __fadd_rn(z.x, z.y);
    t = __fadd_rn(t, __shfl_xor_sync(kAll, t, 2));
    return __fadd_rn(t, __shfl_xor_sync(kAll, t, 1));
}
// (scalar sums: see pair_alpha)
__device__ __forceinline__ float2 sum2(float2 a, float2 b) {
    return make_float2(__fadd_rn(a.x, b.x), __fadd_rn(a.y, b.y));
}

// Sums the window's rows over the block and sends the gradients of the
// Gaussians of its first `rows` rows on their way.  slot0: the stage slot of row
// 0.  Lane (r, c) = (lane / 4, lane % 4) takes row r's pixel pairs of column c,
// whose dL/dC are g01 and g2.  Every product and sum is FP32, about the Gaussian's
// mean, in the order in which a shuffle over the lanes 16, 8, 4, 2 and 1 apart adds
// them.  ODD: colours or dL/dC may be wild().
template <int CH, bool ABS, bool ODD, int SLOTS>
__device__ __forceinline__ void flush_window(const float4* win, const float2* habs,
                                             const float4* g01, const float2* g2,
                                             int slot0, const Stage<SLOTS>& st, int rows, int bx,
                                             int by, const BwdOut& out) {
    const int lane = threadIdx.x & 31, r = lane >> 2, c = lane & 3;
    __syncwarp();
    const int slot = slot0 + r;
    const float* f = reinterpret_cast<const float*>(&st.par[slot >> 1][0]) + (slot & 1);
    const float gx = f[0], gy = f[2];
    const float2 dx = add2(dup(gx), make_float2(-(float)(bx + 2 * c), -(float)(bx + 2 * c + 1)));
    // the six moments (negated) and the colour weights of the pixel rows y, y + 1
    auto two_rows = [&](int y, float2 (&m)[6], float2 (&k)[CH]) {
        const float4 q0 = win[row_slot(r, 4 * y + c)], q1 = win[row_slot(r, 4 * y + 4 + c)];
        const float2 t0 = mul2(make_float2(q0.x, q0.y), dx), t1 = mul2(make_float2(q1.x, q1.y), dx);
        const float2 u0 = mul2(t0, dx), u1 = mul2(t1, dx);
        const float2 dy = add2(dup(gy), make_float2(-(float)(by + y), -(float)(by + y + 1)));
        m[0] = make_float2(__fadd_rn(q0.x, q0.y), __fadd_rn(q1.x, q1.y));
        m[1] = make_float2(__fadd_rn(t0.x, t0.y), __fadd_rn(t1.x, t1.y));
        m[2] = mul2(dy, m[0]);
        m[3] = make_float2(__fadd_rn(u0.x, u0.y), __fadd_rn(u1.x, u1.y));
        m[4] = mul2(dy, m[1]);
        m[5] = mul2(dy, m[2]);
        const float2 w0 = make_float2(q0.z, q0.w), w1 = make_float2(q1.z, q1.w);
        auto weigh = [](float2 w, float2 g) {
            const float2 x = mul2(w, g);
            return ODD ? where(w, x, dup(0.0f)) : x;
        };
        if constexpr (CH == 3) {
            const float4 a0 = g01[4 * y + c], a1 = g01[4 * y + 4 + c];
            const float2 x0 = weigh(w0, make_float2(a0.x, a0.y)),
                         x1 = weigh(w1, make_float2(a1.x, a1.y));
            const float2 y0 = weigh(w0, make_float2(a0.z, a0.w)),
                         y1 = weigh(w1, make_float2(a1.z, a1.w));
            k[0] = make_float2(__fadd_rn(x0.x, x0.y), __fadd_rn(x1.x, x1.y));
            k[1] = make_float2(__fadd_rn(y0.x, y0.y), __fadd_rn(y1.x, y1.y));
        }
        const float2 z0 = weigh(w0, g2[4 * y + c]), z1 = weigh(w1, g2[4 * y + 4 + c]);
        k[CH - 1] = make_float2(__fadd_rn(z0.x, z0.y), __fadd_rn(z1.x, z1.y));
    };
    float2 m[2][6], k[2][CH];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        float2 m4[6], k4[CH];
        two_rows(2 * h, m[h], k[h]);
        two_rows(2 * h + 4, m4, k4);
#pragma unroll
        for (int i = 0; i < 6; ++i) m[h][i] = sum2(m[h][i], m4[i]);
#pragma unroll
        for (int i = 0; i < CH; ++i) k[h][i] = sum2(k[h][i], k4[i]);
    }
    float n[6], col[CH], hx = 0.0f, hy = 0.0f;
#pragma unroll
    for (int i = 0; i < 6; ++i) n[i] = block_sum(m[0][i], m[1][i]);
#pragma unroll
    for (int i = 0; i < CH; ++i) col[i] = -block_sum(k[0][i], k[1][i]);
    if constexpr (ABS) {
        float2 p[2][2];
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int y = 2 * h;
            const float2 a = habs[abs_slot(r, 4 * y + c)], b = habs[abs_slot(r, 4 * y + 4 + c)],
                         d = habs[abs_slot(r, 4 * y + 16 + c)],
                         e = habs[abs_slot(r, 4 * y + 20 + c)];
            p[h][0] = sum2(make_float2(a.x, b.x), make_float2(d.x, e.x));
            p[h][1] = sum2(make_float2(a.y, b.y), make_float2(d.y, e.y));
        }
        hx = block_sum(p[0][0], p[1][0]);
        hy = block_sum(p[0][1], p[1][1]);
    }
    __syncwarp();  // the window may be written again
    if (r >= rows) return;
    const float nb = f[6], no = f[10], na = 2.0f * f[4], nc = 2.0f * f[8];
    constexpr int kTag = CH == 3 ? 6 : 2;
    const uint32_t id =
        __float_as_uint(reinterpret_cast<const float*>(st.col[slot])[kTag]);
    // lane c writes components c, 4 + c (c < 2) and 6 + c (c < CH)
    const float v0 = c == 0   ? fmaf(-na, n[1], __fmul_rn(-nb, n[2]))
                     : c == 1 ? fmaf(-nb, n[1], __fmul_rn(-nc, n[2]))
                     : c == 2 ? 0.5f * n[3]
                              : n[4];
    const float v1 = c == 0 ? 0.5f * n[5] : (n[0] != 0.0f ? n[0] / no : 0.0f);
    float v2 = col[0];
    if constexpr (CH == 3) v2 = c == 0 ? col[0] : c == 1 ? col[1] : col[2];
    if (out.partial) {
        float* o = out.partial + (size_t)id * 11;
        o[c] = v0;
        if (c < 2) o[4 + c] = v1;
        if (c < CH) o[6 + c] = v2;
        if (ABS && c == 3) {
            o[9] = hx;
            o[10] = hy;
        }
    } else {
        float* o = out.grad2d + (size_t)id * kGrad2d;
        if (v0 != 0.0f) atomicAdd(o + c, v0);
        if (c < 2 && v1 != 0.0f) atomicAdd(o + 4 + c, v1);
        if (c < CH && v2 != 0.0f) atomicAdd(o + 6 + c, v2);
        if (ABS && c == 3) {
            float* h = out.absgrad + (size_t)id * 2;
            if (hx != 0.0f) atomicAdd(h, hx);
            if (hy != 0.0f) atomicAdd(h + 1, hy);
        }
    }
}

template <int CH>
struct BwdPixels {
    float2 T, nS, g[CH];  // T behind the current Gaussian; -dL/dC . (colour behind); dL/dC
};

// One Gaussian's adjoint at the lane's two pixels into a row of the window
// (win, habs: the lane's places in it).  na: -alpha where the Gaussian counts
// at the pixel, else 0, which leaves the pixel's state as it is; nG: -o G where
// alpha = o G, 0 where alpha is clamped (and passes no gradient).  ODD: the colour or
// dL/dC may be wild.
template <int CH, bool ABS, bool ODD>
__device__ __forceinline__ void adjoint_one_block(BwdPixels<CH>& s, float2 na, float2 nG,
                                                  const float4* col, float4* win, float2* habs,
                                                  float ha, float nb, float hc, float dx0,
                                                  float dx1, float dy) {
    const float2 inv = make_float2(rcp_approx(1.0f + na.x), rcp_approx(1.0f + na.y));
    s.T = mul2(s.T, inv);
    const float2 nw = mul2(na, s.T);
    const float4 c01 = col[0];
    float2 gc = mul2(s.g[0], make_float2(c01.x, c01.y));
    if constexpr (CH == 3) {
        const float2 c2 = *reinterpret_cast<const float2*>(col + 1);
        gc = fma2(s.g[1], make_float2(c01.z, c01.w), gc);
        gc = fma2(s.g[2], c2, gc);
    }
    const float2 dal = fma2(s.T, gc, mul2(inv, s.nS));
    const float2 nS = fma2(nw, gc, s.nS);
    s.nS = ODD ? where(na, nS, s.nS) : nS;
    float2 ndp = mul2(nG, dal);
    if (ODD) ndp = where(nG, ndp, dup(0.0f));
    *win = make_float4(ndp.x, ndp.y, nw.x, nw.y);
    if constexpr (ABS) {
        // each pixel's own contribution to dL/dmean2d, by magnitude
        const float a = -2.0f * ha, c = -2.0f * hc;
        const float hx = fabsf(ndp.x * fmaf(a, dx0, -nb * dy)) + fabsf(ndp.y * fmaf(a, dx1, -nb * dy));
        const float hy = fabsf(ndp.x * fmaf(-nb, dx0, c * dy)) + fabsf(ndp.y * fmaf(-nb, dx1, c * dy));
        *habs = make_float2(hx, hy);
    }
}

// The adjoint of a staged batch, eight slots (a window) at a time.  Every slot
// takes its row: nearly all reach a pixel of the block, and a row of zeros costs
// less than finding out.  HARD: alphas are clamped and positive powers skipped; ODD:
// colours or dL/dC may be wild.
template <int CH, bool ABS, bool HARD, bool ODD, int SLOTS>
__device__ __forceinline__ void adjoint_batch(
    BwdPixels<CH>& s, const Stage<SLOTS>& st, int ns, int from0, int from1, int checked,
    float2 nx0, float2 nx1, float2 ny, float4* win, float2* habs, const float4* g01,
    const float2* g2, int bx, int by, const BwdOut& out) {
    const int lane = threadIdx.x & 31;
    for (int g = 0; g < ns; g += kRows) {
#pragma unroll(ODD ? 1 : kRows / 2)
        for (int k = 0; k < kRows / 2; ++k) {
            const int slot = g + 2 * k;
            const float4 A = st.par[slot >> 1][0], B = st.par[slot >> 1][1],
                         D = st.par[slot >> 1][2];
            const float2 dy = add2(make_float2(A.z, A.w), ny);
            const float2 cdd = mul2(make_float2(D.x, D.y), mul2(dy, dy));
            const float2 gx = make_float2(A.x, A.y), a = make_float2(B.x, B.y),
                         nb = make_float2(B.z, B.w), no = make_float2(D.z, D.w);
            const float2 dx0 = add2(gx, nx0), dx1 = add2(gx, nx1);
            const PairAlpha e0 = pair_alpha(dx0, dy, cdd, a, nb, no);
            const PairAlpha e1 = pair_alpha(dx1, dy, cdd, a, nb, no);
            const float2 n0 = HARD ? tame(e0) : e0.noG, n1 = HARD ? tame(e1) : e1.noG;
            bool hA0 = n0.x <= -kAlphaMin, hA1 = n1.x <= -kAlphaMin;
            bool hB0 = n0.y <= -kAlphaMin, hB1 = n1.y <= -kAlphaMin;
            if (slot < checked) {  // beyond some pixel's part of the list
                hA0 = hA0 && slot >= from0;
                hA1 = hA1 && slot >= from1;
                hB0 = hB0 && slot + 1 >= from0;
                hB1 = hB1 && slot + 1 >= from1;
            }
            const float2 naA = make_float2(hA0 ? n0.x : 0.0f, hA1 ? n1.x : 0.0f);
            const float2 naB = make_float2(hB0 ? n0.y : 0.0f, hB1 ? n1.y : 0.0f);
            float2 nGA = naA, nGB = naB;
            if (HARD) {
                nGA = make_float2(e0.noG.x > -kAlphaMax ? naA.x : 0.0f,
                                  e1.noG.x > -kAlphaMax ? naA.y : 0.0f);
                nGB = make_float2(e0.noG.y > -kAlphaMax ? naB.x : 0.0f,
                                  e1.noG.y > -kAlphaMax ? naB.y : 0.0f);
            }
            adjoint_one_block<CH, ABS, ODD>(
                s, naA, nGA, st.col[slot], win + row_slot(2 * k, lane),
                habs + abs_slot(2 * k, lane), a.x,
                nb.x, D.x, dx0.x, dx1.x, dy.x);
            adjoint_one_block<CH, ABS, ODD>(
                s, naB, nGB, st.col[slot + 1], win + row_slot(2 * k + 1, lane),
                habs + abs_slot(2 * k + 1, lane), a.y,
                nb.y, D.y, dx0.y, dx1.y, dy.y);
        }
        flush_window<CH, ABS, ODD>(win, habs, g01, g2, g, st, min(ns - g, kRows), bx, by, out);
    }
}

template <int CH, bool CULL, bool ABS, int SLOTS, int RING>
__device__ __forceinline__ void bwd_block(const TileCtx& tc, int bx, int by,
                                          Feeder<SLOTS, RING>& fd, float4* win, float2* habs,
                                          float4* g01, float2* g2, bool wild_map, float bg0,
                                          float bg1, float bg2,
                                          const float* __restrict__ final_T,
                                          const int32_t* __restrict__ last_idx,
                                          const float* __restrict__ dL, const BwdOut& out) {
    const int lane = threadIdx.x & 31;
    const int lx = bx + 2 * (lane & 3), ly = by + (lane >> 2);
    const int px = tc.tx0 + lx, py = tc.ty0 + ly;
    const bool in0 = py < tc.height && px < tc.width, in1 = py < tc.height && px + 1 < tc.width;
    const int64_t plane = (int64_t)tc.width * tc.height;
    const int64_t pix = (int64_t)py * tc.width + px;
    int last0 = 0, last1 = 0;
    if (in0) last0 = last_idx[tc.pix_base + pix];
    if (in1) last1 = last_idx[tc.pix_base + pix + 1];
    const int top = (int)__reduce_max_sync(kAll, (unsigned)max(last0, last1));
    if (top == 0) return;
    const int begin = (int)tc.begin;
    const int chunks = (top + kChunk - 1) / kChunk;
    // chunk c, lane i: the list from its last blended entry on, backwards
    auto pos = [&](int c) {
        const int i = top - 1 - (c * kChunk + lane);
        return i >= 0 ? begin + i : -1;
    };
    fd.start(pos, lane);
    BwdPixels<CH> s;
    s.T = make_float2(in0 ? final_T[tc.pix_base + pix] : 1.0f,
                      in1 ? final_T[tc.pix_base + pix + 1] : 1.0f);
    const float bgc[3] = {bg0, bg1, bg2};
    const float bgg = (bg0 + bg1 + bg2) * (1.0f / 3.0f);
    float2 gb2 = dup(0.0f);
    bool big = false;
#pragma unroll
    for (int ch = 0; ch < CH; ++ch) {
        const float* d = dL + tc.val_base + ch * plane + pix;
        s.g[ch] = make_float2(in0 ? d[0] : 0.0f, in1 ? d[1] : 0.0f);
        big = big || wild(s.g[ch].x) || wild(s.g[ch].y);
        gb2 = fma2(s.g[ch], dup(CH == 3 ? bgc[ch] : bgg), gb2);
    }
    const bool odd = __any_sync(kAll, big) || wild_map;
    s.nS = mul2(s.T, make_float2(-gb2.x, -gb2.y));  // minus the background seen through T_final
    // for flush_window (as registers of the lanes that need them: 251 us at 1M
    // against 239)
    if constexpr (CH == 3) g01[lane] = make_float4(s.g[0].x, s.g[0].y, s.g[1].x, s.g[1].y);
    g2[lane] = s.g[CH - 1];
    __syncwarp();
    const float2 nx0 = dup(-(float)lx), nx1 = dup(-(float)(lx + 1)), ny = dup(-(float)ly);
    for (int c = 0; c < chunks;) {
        // from0, from1: the first slot of this batch within the pixel's part of the list
        int ns = 0, from0 = 0, from1 = 0;
        do {
            const unsigned mask = fd.template stage<CH, CULL, false>(
                pos, c, ns, lane, (float)tc.tx0, (float)tc.ty0, (float)bx, (float)by, begin);
            const int hi = top - c * kChunk;  // entries behind the pixel's last: hi - last
            const int d0 = min(max(hi - last0, 0), 32), d1 = min(max(hi - last1, 0), 32);
            from0 += __popc(mask & (unsigned)((1ull << d0) - 1ull));
            from1 += __popc(mask & (unsigned)((1ull << d1) - 1ull));
            ns += __popc(mask);
            ++c;
        } while (ns <= SLOTS - kChunk && c < chunks);
        fd.template pad<kRows>(ns, lane);
        __syncwarp();
        // slots before this one may lie beyond some pixel's part of the list
        const int checked = (int)__reduce_max_sync(kAll, (unsigned)max(from0, from1));
        if (odd)
            adjoint_batch<CH, ABS, true, true>(s, *fd.st, ns, from0, from1, checked, nx0, nx1, ny,
                                               win, habs, g01, g2, bx, by, out);
        else if (fd.hard(ns, lane))
            adjoint_batch<CH, ABS, true, false>(s, *fd.st, ns, from0, from1, checked, nx0, nx1, ny,
                                                win, habs, g01, g2, bx, by, out);
        else
            adjoint_batch<CH, ABS, false, false>(s, *fd.st, ns, from0, from1, checked, nx0, nx1, ny,
                                                 win, habs, g01, g2, bx, by, out);
        __syncwarp();  // the stage has been read
    }
    cp_async_wait_all();
    __syncwarp();
}


template <bool CULL, bool ABS>
__global__ void __launch_bounds__(32 * kWarps, CULL ? 4 : 5)
k_blocks_bwd(ViewTable vt, const uint32_t* __restrict__ ranges,
             const uint32_t* __restrict__ order, const uint32_t* __restrict__ ivals,
             const uint32_t* __restrict__ gid_of, const float4* __restrict__ rec, int log2_bx,
             int log2_blocks, int total_blocks, uint32_t* queue,
             const DevCounters* __restrict__ ctr, float bg0, float bg1, float bg2,
             const float* __restrict__ final_T, const int32_t* __restrict__ last_idx,
             const float* __restrict__ dL, BwdOut out) {
    extern __shared__ float4 smem[];
    BwdShared<CULL, ABS>& my = reinterpret_cast<BwdShared<CULL, ABS>*>(smem)[threadIdx.x >> 5];
    Feeder<kSlots, kRing<CULL>> fd;
    fd.raw = my.raw;
    fd.st = &my.st;
    fd.ivals = ivals;
    fd.gid_of = gid_of;
    fd.rec = rec;
    const bool wild_map = ctr->wild_colour != 0u;
    for (;;) {
        const int slot = next_slot(queue);
        if (slot >= total_blocks) break;
        const TileCtx tc = tile_ctx(vt, ranges, (int)order[slot >> log2_blocks]);
        const int sub = slot & ((1 << log2_blocks) - 1);
        const int bx = (sub & ((1 << log2_bx) - 1)) * kBlock, by = (sub >> log2_bx) * kBlock;
        if (tc.channels == 3)
            bwd_block<3, CULL, ABS>(tc, bx, by, fd, my.win, my.habs, my.g01, my.g2, wild_map, bg0,
                                    bg1, bg2, final_T, last_idx, dL, out);
        else
            bwd_block<1, CULL, ABS>(tc, bx, by, fd, my.win, my.habs, my.g01, my.g2, wild_map, bg0,
                                    bg1, bg2, final_T, last_idx, dL, out);
    }
}

// CTAs of a launch over `total` blocks: the resident ones, but no more than
// leave each warp per_warp2 / 2 blocks (and at least two per SM).  A warp's
// share of its SM shrinks with every other warp there, and a launch is not over
// before its longest list, which one warp walks alone: where there are few
// blocks, fewer warps that run faster end sooner.  Forward (8 halves),
// at 8 / 5 / 3 / 2 CTAs per SM: 113640 blocks 628 / 673 / 823 / 1056 us, 12750
// blocks 140 / 132 / 136 / 160, 4800 blocks 38 / 38 / 33 / 33.  Adjoint (6 halves)
// at 5 / 3 / 2: 113640 blocks 1333 / 1591 / 2027, 12750 blocks 240 / 272 / 336, 4800
// blocks 71 / 67 / 62; by 5 / 6 / 8 halves: 4800 blocks 65 / 61 / 61 us, 6120 blocks 87 /
// 82 / 92, 8100 blocks 103 / 96 / 101, 4800 blocks of 16x16 tiles 75 / 70 / 70.
int launch_ctas(const void* kern, size_t smem, int total, int per_warp2) {
    const int resident = persistent_blocks(kern, 32 * kWarps, smem, kWarps, total);
    const int sms = sm_count();
    if (resident < 0 || sms <= 0) return -1;
    const int per_sm = max(2, (int)(2ll * total / ((long long)sms * kWarps * per_warp2)));
    return per_sm < resident / sms ? per_sm * sms : resident;
}

int ilog2(int x) {
    int l = 0;
    while ((1 << (l + 1)) <= x) ++l;
    return l;
}

}  // namespace

// The block kernels take every tile that is whole 8x8 blocks; with a
// deterministic adjoint only the 8x8 tile itself, whose (Gaussian, tile)
// pairs one warp sums (the larger tiles' pairs would be split over warps).
bool blocks_fit(const Plan* p) {
    if (p->cfg.tile_w % kBlock || p->cfg.tile_h % kBlock) return false;
    return !p->cfg.deterministic || (p->cfg.tile_w == kBlock && p->cfg.tile_h == kBlock);
}

gs_status launch_blocks_fwd(const Plan* p, const uint32_t* vals, void* ws, float* images,
                            float* final_T, int32_t* last_idx, cudaStream_t st) {
    const int log2_bx = ilog2(p->cfg.tile_w / kBlock);
    const int log2_blocks = log2_bx + ilog2(p->cfg.tile_h / kBlock);
    const bool cull = log2_blocks > 0 || !p->vt.tight_rect;
    const int total = p->total_tiles << log2_blocks;
    auto* kern = cull ? k_blocks_fwd<true> : k_blocks_fwd<false>;
    const int blocks = launch_ctas((const void*)kern, 0, total, 8);
    if (blocks < 0) return GS_ERR_CUDA;
    uint32_t* queue = buf<uint32_t>(p, ws, B_TILE_QUEUE);
    if (cudaMemsetAsync(queue, 0, sizeof(uint32_t), st) != cudaSuccess) return GS_ERR_CUDA;
    kern<<<blocks, 32 * kWarps, 0, st>>>(
        p->vt, cbuf<uint32_t>(p, ws, GS_BUF_RANGES), cbuf<uint32_t>(p, ws, B_TILE_ORDER), vals,
        p->cfg.deterministic ? cbuf<uint32_t>(p, ws, B_GID_OF) : nullptr,
        cbuf<float4>(p, ws, GS_BUF_PROJ), log2_bx, log2_blocks, total, queue,
        cbuf<DevCounters>(p, ws, GS_BUF_COUNTERS), p->cfg.bg[0], p->cfg.bg[1], p->cfg.bg[2],
        images, final_T, last_idx);
    return launch_status();
}

gs_status launch_blocks_bwd(const Plan* p, const uint32_t* vals, void* ws, const float* final_T,
                            const int32_t* last_idx, const float* dL, cudaStream_t st) {
    const int log2_bx = ilog2(p->cfg.tile_w / kBlock);
    const int log2_blocks = log2_bx + ilog2(p->cfg.tile_h / kBlock);
    const bool cull = log2_blocks > 0 || !p->vt.tight_rect;
    const bool abs_stats = p->cfg.density_stats != 0;
    const int total = p->total_tiles << log2_blocks;
    auto* kern = cull ? (abs_stats ? k_blocks_bwd<true, true> : k_blocks_bwd<true, false>)
                      : (abs_stats ? k_blocks_bwd<false, true> : k_blocks_bwd<false, false>);
    const size_t per_warp =
        cull ? (abs_stats ? sizeof(BwdShared<true, true>) : sizeof(BwdShared<true, false>))
             : (abs_stats ? sizeof(BwdShared<false, true>) : sizeof(BwdShared<false, false>));
    const size_t smem = kWarps * per_warp;
    if (smem > 48 * 1024 &&
        cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) !=
            cudaSuccess)
        return GS_ERR_CUDA;
    const int blocks = launch_ctas((const void*)kern, smem, total, 6);
    if (blocks < 0) return GS_ERR_CUDA;
    uint32_t* queue = buf<uint32_t>(p, ws, B_TILE_QUEUE) + 1;
    if (cudaMemsetAsync(queue, 0, sizeof(uint32_t), st) != cudaSuccess) return GS_ERR_CUDA;
    BwdOut out;
    out.grad2d = buf<float>(p, ws, GS_BUF_GRAD2D);
    out.absgrad = abs_stats ? buf<float>(p, ws, GS_BUF_ABSGRAD) : nullptr;
    out.partial = p->cfg.deterministic ? buf<float>(p, ws, B_PARTIAL) : nullptr;
    kern<<<blocks, 32 * kWarps, smem, st>>>(
        p->vt, cbuf<uint32_t>(p, ws, GS_BUF_RANGES), cbuf<uint32_t>(p, ws, B_TILE_ORDER), vals,
        p->cfg.deterministic ? cbuf<uint32_t>(p, ws, B_GID_OF) : nullptr,
        cbuf<float4>(p, ws, GS_BUF_PROJ), log2_bx, log2_blocks, total, queue,
        cbuf<DevCounters>(p, ws, GS_BUF_COUNTERS), p->cfg.bg[0], p->cfg.bg[1], p->cfg.bg[2],
        final_T, last_idx, dL, out);
    return launch_status();
}

}  // namespace gs
