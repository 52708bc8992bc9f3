// internal.h -- launchers the host runtime calls (not part of the C ABI).
#pragma once
#include <cuda_runtime.h>

#include "device.cuh"

namespace curast {

struct LaunchShape {
    int stage1_blocks_per_sm[2][3];   // [instanced][variant: 0 plain meshes, 1 compressed ones,
                                      //  2 single-pair cull with vertex windows (not instanced)]
    int stage1x_blocks_per_sm;        // exact kernel of stage 1
    int stage2_blocks_per_sm;
    int stage3_blocks_per_sm;
    int stage3t_blocks_per_sm[4];     // binned stage 3 per tile side 2^4 .. 2^7
    int num_sms;
};

cudaError_t query_launch_shape(LaunchShape *out, int device);

cudaError_t launch_clear(uint64_t *vis, uint64_t n, cudaStream_t s);

// The start of a frame (k_begin): n16 16-byte words of tables copied from
// pinned host memory, counters and tile counts zeroed, buffers cleared.
constexpr int kBeginViews = 8;
struct BeginArgs {
    const uint4 *src;
    uint4 *dst;
    uint64_t n16;
    Counters *ctr;
    uint32_t *tile_cnt;
    uint32_t n_tiles;
    int n_vis;
    unsigned long long *stamps;
    uint64_t *vis[kBeginViews];
    uint64_t n[kBeginViews];
};
cudaError_t launch_begin(const BeginArgs &a, cudaStream_t s);
// A stage kernel, launched ahead of its predecessor's end where the frame
// allows it (begin_stage waits).
template <class... P, class... A>
inline cudaError_t launch_stage(bool pdl, void (*k)(P...), int blocks, int threads, size_t smem, cudaStream_t s, A... args) {
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.gridDim = dim3((unsigned)blocks);
    cfg.blockDim = dim3((unsigned)threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cfg.attrs = at;
    cfg.numAttrs = pdl ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, k, args...);
}

// Stage 1 of round r: the cull kernel, then the exact kernel over the round's
// bitmap.  near = false launches the cull without its near-plane test (valid
// when no pair's mesh bounds reach the near plane).
cudaError_t launch_stage1(const FrameDev &f, bool instanced, int variant, uint32_t r, int blocks, bool near,
                          cudaStream_t s);
cudaError_t launch_stage1_exact(const FrameDev &f, bool comp, uint32_t r, int blocks, cudaStream_t s);
cudaError_t launch_stage2(const FrameDev &f, int blocks, cudaStream_t s);
cudaError_t launch_stage3(const FrameDev &f, int blocks, cudaStream_t s);
// Binned stage 3: scan of the per-tile part counts, scatter of the parts into
// tile order, then one block per tile with the tile's words in shared memory.
cudaError_t launch_stage3_binned(const FrameDev &f, int scatter_blocks, int tile_blocks, cudaStream_t s);
// scratch: 256 * 6 floats; out6: xmin ymin zmin xmax ymax zmax
cudaError_t launch_aabb(const float *pos, uint64_t V, float *scratch, float *out6, cudaStream_t s);
// Section 4.6 encoding (compress.cu)
cudaError_t launch_minmax_u32(const uint32_t *v, uint64_t n, unsigned *out2, cudaStream_t s);
cudaError_t launch_pack_indices(const uint32_t *idx, uint64_t n, uint32_t imin, uint32_t bits, uint32_t *words,
                                uint64_t nwords, cudaStream_t s);
// grid flags of the 128-triangle groups of a mesh: ceil(ceil(T / 128) / 32) words
cudaError_t launch_grid_flags(const uint32_t *idx, uint64_t T, uint64_t V, uint32_t *flags, uint64_t nwords,
                              cudaStream_t s);
cudaError_t launch_quantize_positions(const float *pos, uint64_t V, const double lo[3], const double size[3],
                                      uint16_t *q, cudaStream_t s);
cudaError_t launch_count_diff(const uint64_t *a, const uint64_t *b, uint64_t n, unsigned long long *out,
                              cudaStream_t s);

struct InstDev {                // an instance of the screen passes
    uint64_t base;              // global id of its triangle 0
    uint32_t mesh, pad;
};

// The instances of a scene of at most kFew, by value: no upload before the
// kernel, and no chain of loads in it from a pixel's id to the buffers of its
// mesh.  Sixteen whole mesh records are what 4 KB of kernel parameters hold;
// more (the toolkit allows 32 KB), or leaner records, were not tried.  One
// 16.8 M-triangle terrain at 3840 x 2160 in 8, 16, 17, 32 and 64 instances, us a
// call: resolve 148 152 161 163 159, super-sampled 145 148 163 166 163, textured
// 163 165 173 178 177.
constexpr int kFew = 16;
struct FewInst {
    uint64_t base[kFew + 1];    // of instances past the last one: the total
    uint32_t mesh_id[kFew];
    float mv[kFew][12];
    MeshDev mesh[kFew];
};

struct ShadeArgs {
    const uint64_t *vis;
    int W, H;
    float fx, fy;
    const float *inst_mv;       // n_inst x 12
    const InstDev *inst;        // n_inst + 1, the last one's base is the total
    const MeshDev *meshes;
    int n_inst;
    int rows;                   // pixel rows a thread walks (set by the launchers)
    uint64_t tris;              // triangles of all instances
    // resolve
    float *rgba_f32;
    uint8_t *rgba8;
    int ss;                     // super-sampled resolve: samples per pixel axis
    uint8_t *level;             // textured resolve: the mip level per pixel (255: none), or null
    // interpolate
    uint32_t mesh;
    const float *pos;           // overrides the mesh's positions when non-null
    const float *attr;
    int C;
    float *out;
    const float *grad_out;
    float *grad_attr;
    float *grad_pos;
    FewInst few;                // n_inst <= kFew (inst_mv and inst are not read then)
};
static_assert(sizeof(ShadeArgs) + 16 <= 4096, "kernel parameters");

cudaError_t launch_resolve(ShadeArgs &a, cudaStream_t s);
// a.W, a.H: the super-sampled buffer (ss W x ss H); W, H: the output
cudaError_t launch_resolve_ss(const ShadeArgs &a, int W, int H, cudaStream_t s);
// resolve with textures and the 4-ray mip-level choice (Section 4.4)
cudaError_t launch_resolve_textured(ShadeArgs &a, cudaStream_t s);
cudaError_t launch_interpolate(ShadeArgs &a, cudaStream_t s);
cudaError_t launch_interpolate_backward(const ShadeArgs &a, cudaStream_t s);

}  // namespace curast
