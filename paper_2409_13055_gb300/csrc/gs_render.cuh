// gs_render.cuh -- what the two families of render kernels share: gs_blocks.cu
// (a warp per 8x8 pixel block) and gs_render.cu (a team per tile, any shape).
#pragma once

#include "gs_internal.cuh"

namespace gs {

__device__ __forceinline__ void cp_async16(void* smem, const void* gmem) {
    const unsigned s = (unsigned)__cvta_generic_to_shared(smem);
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(s), "l"(gmem) : "memory");
}
__device__ __forceinline__ void cp_async_commit() {
    asm volatile("cp.async.commit_group;\n" ::: "memory");
}
__device__ __forceinline__ void cp_async_wait_all() {
    asm volatile("cp.async.wait_group 0;\n" ::: "memory");
}
__device__ __forceinline__ void cp_async_wait_one() {
    asm volatile("cp.async.wait_group 1;\n" ::: "memory");
}

struct TileCtx {
    int view, tile_local, tx0, ty0, width, height, channels;
    int64_t pix_base, val_base;
    uint32_t begin, end;
};

__device__ __forceinline__ TileCtx tile_ctx(const ViewTable& vt, const uint32_t* ranges,
                                            int tile) {
    TileCtx c;
    c.view = view_of_tile(vt, tile);
    const ViewGeom& g = vt.v[c.view];
    c.tile_local = tile - g.tile_offset;
    c.tx0 = (c.tile_local % g.tiles_x) * vt.tile_w;
    c.ty0 = (c.tile_local / g.tiles_x) * vt.tile_h;
    c.width = g.width;
    c.height = g.height;
    c.channels = g.channels;
    c.pix_base = g.pixel_offset;
    c.val_base = g.value_offset;
    c.begin = ranges[2 * tile];
    c.end = ranges[2 * tile + 1];
    return c;
}

// Reciprocal by the hardware approximation (PTX rcp.approx.ftz.f32, within
// about one ulp); the argument 1 - alpha lies in [0.01, 1].
__device__ __forceinline__ float rcp_approx(float x) {
    float y;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

// CTAs of a persistent launch: the resident CTAs of the whole GPU, no more
// than there are teams' worth of tiles (gs_render.cu).
int persistent_blocks(const void* kern, int threads, size_t smem, int tiles_per_block,
                      int total_tiles);

// The block kernels (gs_blocks.cu): whether they take a plan, and their launches.
bool blocks_fit(const Plan* p);
gs_status launch_blocks_fwd(const Plan* p, const uint32_t* vals, void* ws, float* images,
                            float* final_T, int32_t* last_idx, cudaStream_t st);
gs_status launch_blocks_bwd(const Plan* p, const uint32_t* vals, void* ws, const float* final_T,
                            const int32_t* last_idx, const float* dL, cudaStream_t st);

}  // namespace gs
