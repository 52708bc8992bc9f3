// shade.cu -- resolve pass (Section 4.4) and the differentiable interpolation
// step (forward and backward) on a fixed visibility buffer.
//
// The screen passes are chains of dependent gathers (visibility word,
// instance, indices, positions and attributes) with FP32 arithmetic of a fixed
// order behind them.  A thread therefore walks a short column of pixels: their
// words are loaded together, the instance under one pixel is tried for the
// next before the table is searched, and two pixels' gathers are in flight at
// a time.  What depends on the column or the row alone (the ray's first two
// coordinates, two IEEE divisions each) is computed once a block.
#include "internal.h"

namespace curast {

namespace sh {
constexpr int kRows = 4;                 // most rows a thread walks
constexpr int kTile = 8 * kRows;         // a block's pixel rows at that, and its columns
}

__device__ __forceinline__ float interp3(float b0, float b1, float b2, float c0, float c1, float c2) {
    return __fadd_rn(__fadd_rn(__fmul_rn(b0, c0), __fmul_rn(b1, c1)), __fmul_rn(b2, c2));
}

// The instance a thread's last pixel showed: its ids [lo, hi), number, mesh.
struct Under {
    uint64_t lo = 1, hi = 0;
    int inst = -1;
    const MeshDev *mesh = nullptr;          // (not FEW)
};

// Section 4.4: the mesh instance owning a global id is found by binary
// search of the exclusive prefix sum (last instance with base <= id), unless
// it is the one under the previous pixel.  False for an empty pixel and for an
// id past the last instance's triangles.  FEW: the tables are parameters.
template <bool FEW>
__device__ __forceinline__ bool find_instance(const ShadeArgs &a, uint64_t key, Under &u) {
    if (key == kEmpty) return false;
    const uint64_t id = key & kIdMask;
    if (id < u.lo || id >= u.hi) {
        if (FEW) {
            if (a.n_inst == 0 || id < a.few.base[0]) return false;
            int i = 0;
            while (i + 1 < a.n_inst && a.few.base[i + 1] <= id) ++i;
            u.inst = i;
            u.lo = a.few.base[i];
            u.hi = a.few.base[i + 1];
            return id < u.hi;
        }
        int lo = 0, hi = a.n_inst;   // first index with base > id
        while (lo < hi) {
            const int mid = (lo + hi) >> 1;
            if (a.inst[mid].base <= id) lo = mid + 1; else hi = mid;
        }
        if (lo == 0) return false;
        u.inst = lo - 1;
        u.lo = a.inst[lo - 1].base;
        u.hi = a.inst[lo].base;
        u.mesh = a.meshes + a.inst[lo - 1].mesh;
    }
    return id < u.hi;
}

template <bool FEW>
__device__ __forceinline__ const MeshDev &mesh_of(const ShadeArgs &a, const Under &u) {
    return FEW ? a.few.mesh[u.inst] : *u.mesh;
}

template <bool FEW>
__device__ __forceinline__ void model_view_of(const ShadeArgs &a, int inst, float (&mv)[12]) {
#pragma unroll
    for (int q = 0; q < 12; ++q) mv[q] = FEW ? a.few.mv[inst][q] : __ldg(a.inst_mv + 12 * (size_t)inst + q);
}

// Vertex indices of the pixel's triangle; false when one is out of range.
__device__ __forceinline__ bool pixel_indices(const MeshDev &m, const Under &u, uint64_t key, uint32_t (&vi)[3]) {
    const uint64_t k = 3 * ((key & kIdMask) - u.lo);
    const uint32_t *idx = m.idx;
    if (!m.cidx) {
#pragma unroll
        for (int c = 0; c < 3; ++c) vi[c] = __ldg(idx + k + c);
    } else {
#pragma unroll
        for (int c = 0; c < 3; ++c) vi[c] = mesh_index(m, k + c);
    }
    const uint64_t V = m.V;
    return vi[0] < V && vi[1] < V && vi[2] < V;
}

// Object-space positions of the three vertices (pos: the caller's, or null).
__device__ __forceinline__ void pixel_positions(const MeshDev &m, const float *pos, const uint32_t (&vi)[3], float (&p)[9]) {
    const float *src = pos ? pos : m.pos;
    if (src) {
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            const float *q = src + 3 * (size_t)vi[c];
            p[3 * c] = __ldg(q); p[3 * c + 1] = __ldg(q + 1); p[3 * c + 2] = __ldg(q + 2);
        }
    } else {
#pragma unroll
        for (int c = 0; c < 3; ++c) mesh_vertex(m, vi[c], p[3 * c], p[3 * c + 1], p[3 * c + 2]);
    }
}

// The plane of a triangle for barycentrics of ray hits (Moeller-Trumbore
// form, unclamped): e1 = v1 - v0, e2 = v2 - v0, p = r x e2, det = e1.p,
// u = (-v0).p / det, q = (-v0) x e1, w = r.q / det, b = (1 - u - w, u, w).
// r = (rx, ry, -1): its products by -1 are exact negations.
struct Plane { float3 e1, e2, tv, qv; };

__device__ __forceinline__ Plane plane_of(const float *mv, const float (&p)[9]) {
    const float3 v0 = view_space(mv, p), v1 = view_space(mv, p + 3), v2 = view_space(mv, p + 6);
    Plane P;
    P.e1 = sub3(v1, v0);
    P.e2 = sub3(v2, v0);
    P.tv = make_float3(-v0.x, -v0.y, -v0.z);
    P.qv = cross3(P.tv, P.e1);
    return P;
}

__device__ __forceinline__ void ray_bary(const Plane &P, float rx, float ry, float &b0, float &b1, float &b2) {
    const float3 pv = make_float3(__fadd_rn(__fmul_rn(ry, P.e2.z), P.e2.y), __fsub_rn(-P.e2.x, __fmul_rn(rx, P.e2.z)),
                                  __fsub_rn(__fmul_rn(rx, P.e2.y), __fmul_rn(ry, P.e2.x)));
    const float det = dot3(P.e1, pv);
    b1 = __fdiv_rn(dot3(P.tv, pv), det);
    b2 = __fdiv_rn(__fsub_rn(__fadd_rn(__fmul_rn(rx, P.qv.x), __fmul_rn(ry, P.qv.y)), P.qv.z), det);
    b0 = __fsub_rn(__fsub_rn(1.0f, b1), b2);
}

// c / 255 for a byte c, correctly rounded (equal to the IEEE division for all
// 256 bytes, checked): the product by the nearest float of 1/255, its
// remainder exact by FMA, and one correction (Markstein 1990) -- three
// operations for the division's ten or more, twelve times a pixel.
__device__ __forceinline__ float byte_unit(uint32_t rgba, int ch) {
    const float f = __fsub_rn(__uint_as_float(__byte_perm(rgba, 0x4B000000u, 0x7540u | (unsigned)ch)), 8388608.0f);
    const float r = 0x1.010102p-8f, q = __fmul_rn(f, r);
    return __fmaf_rn(__fmaf_rn(-q, 255.0f, f), r, q);
}

// Vertex colours byte / 255 interpolated.
__device__ __forceinline__ void blend_rgba(float b0, float b1, float b2, const uint32_t (&q)[3], float (&c)[4]) {
#pragma unroll
    for (int ch = 0; ch < 4; ++ch)
        c[ch] = interp3(b0, b1, b2, byte_unit(q[0], ch), byte_unit(q[1], ch), byte_unit(q[2], ch));
}

// The FP32 colour and its bytes, rint(clamp(c, 0, 1) 255): 2^23 plus a number
// up to 255 holds it rounded to the nearest integer in its low byte.
__device__ __forceinline__ void store_rgba(const ShadeArgs &a, size_t pix, const float (&c)[4]) {
    if (a.rgba_f32) reinterpret_cast<float4 *>(a.rgba_f32)[pix] = make_float4(c[0], c[1], c[2], c[3]);
    if (a.rgba8) {
        uint32_t q[4];
#pragma unroll
        for (int ch = 0; ch < 4; ++ch)
            q[ch] = __float_as_uint(__fadd_rn(__fmul_rn(fminf(fmaxf(c[ch], 0.0f), 1.0f), 255.0f), 8388608.0f));
        reinterpret_cast<uint32_t *>(a.rgba8)[pix] =
            __byte_perm(__byte_perm(q[0], q[1], 0x0040), __byte_perm(q[2], q[3], 0x0040), 0x5410);
    }
}

// The ray coordinates of the columns x0 .. x0 + nx - 1 and rows y0 .. y0 + ny - 1
// of a W x H image, by the first threads of the block.
__device__ __forceinline__ void ray_tables(float *rx, float *ry, int x0, int nx, int y0, int ny, int W, int H,
                                           const ShadeArgs &a) {
    const int t = threadIdx.x;
    if (t < nx) rx[t] = ray_axis(x0 + t, W, a.fx);
    else if (t - nx < ny) ry[t - nx] = ray_axis(y0 + t - nx, H, a.fy);
    __syncthreads();
}

// ---------------------------------------------------------------- resolve --
// Colours of the samples (x, y0 + k), k < n <= 2, of a W-wide buffer:
// barycentrics of the pixel-centre ray; 0 where the sample is empty or the
// mesh has no colours.
template <bool FEW>
__device__ __forceinline__ void resolve_pair(const ShadeArgs &a, const uint64_t (&key)[2], float rx, const float *ry,
                                             Under &u, float (&c)[2][4]) {
    uint32_t vi[2][3], q[2][3];
    float p[2][9];
    int inst[2];
    bool ok[2];
#pragma unroll
    for (int k = 0; k < 2; ++k) {
        ok[k] = find_instance<FEW>(a, key[k], u) && mesh_of<FEW>(a, u).rgba;
        if (ok[k]) ok[k] = pixel_indices(mesh_of<FEW>(a, u), u, key[k], vi[k]);
        if (ok[k]) {
            const MeshDev &m = mesh_of<FEW>(a, u);
            inst[k] = u.inst;
            pixel_positions(m, nullptr, vi[k], p[k]);
            const uint32_t *rgba = reinterpret_cast<const uint32_t *>(m.rgba);
#pragma unroll
            for (int v = 0; v < 3; ++v) q[k][v] = __ldg(rgba + vi[k][v]);
        }
    }
#pragma unroll
    for (int k = 0; k < 2; ++k) {
        c[k][0] = c[k][1] = c[k][2] = c[k][3] = 0.0f;
        if (ok[k]) {
            float mv[12], b0, b1, b2;
            model_view_of<FEW>(a, inst[k], mv);
            ray_bary(plane_of(mv, p[k]), rx, ry[k], b0, b1, b2);
            blend_rgba(b0, b1, b2, q[k], c[k]);
        }
    }
}

template <bool FEW>
__global__ void __launch_bounds__(256, 4) k_resolve(const __grid_constant__ ShadeArgs a) {
    using namespace sh;
    __shared__ float rx[32], ry[kTile + 1];
    const int lane = threadIdx.x & 31, rows = a.rows;
    const int bx = blockIdx.x * 32, by = blockIdx.y * 8 * rows;
    ray_tables(rx, ry, bx, 32, by, 8 * rows, a.W, a.H, a);
    const int x = bx + lane, ly = (threadIdx.x >> 5) * rows;
    const int n = x < a.W ? min(rows, a.H - (by + ly)) : 0;
    if (n <= 0) return;
    const size_t pix0 = (size_t)(by + ly) * a.W + x;
    uint64_t key[kRows];
#pragma unroll
    for (int k = 0; k < kRows; ++k) key[k] = k < n ? a.vis[pix0 + (size_t)k * a.W] : kEmpty;
    Under u;
#pragma unroll
    for (int k = 0; k < kRows; k += 2) {
        if (k >= n) break;
        const uint64_t two[2] = {key[k], key[k + 1]};
        float c[2][4];
        resolve_pair<FEW>(a, two, rx[lane], ry + ly + k, u, c);
        store_rgba(a, pix0 + (size_t)k * a.W, c[0]);
        if (k + 1 < n) store_rgba(a, pix0 + (size_t)(k + 1) * a.W, c[1]);
    }
}

// Super-sampled resolve: the visibility buffer holds (ss W) x (ss H)
// samples (the same view rendered at ss times the resolution per axis);
// output pixel (x, y) is the box filter of its ss x ss samples -- their
// colours summed row by row, y outer and x inner, then divided by ss^2.  A
// block resolves a square of samples as k_resolve does, (32 / ss) outputs a
// side, keeps their colours in shared memory, and sums each output's there.
template <bool FEW>
__global__ void __launch_bounds__(256, 4) k_resolve_ss(const __grid_constant__ ShadeArgs a, int W, int H) {
    using namespace sh;
    __shared__ float rx[32], ry[kTile + 1];
    __shared__ float4 col[kTile][32];
    const int ss = a.ss, side = 32 / ss;             // outputs a side of the block
    const int lane = threadIdx.x & 31;
    const int bx = blockIdx.x * side * ss, by = blockIdx.y * side * ss, n_s = side * ss;
    ray_tables(rx, ry, bx, 32, by, kTile, a.W, a.H, a);
    const int x = bx + lane, ly = (threadIdx.x >> 5) * kRows;
    const int n = lane < n_s && x < a.W ? min(min(kRows, n_s - ly), a.H - (by + ly)) : 0;
    uint64_t key[kRows];
#pragma unroll
    for (int k = 0; k < kRows; ++k) key[k] = k < n ? a.vis[(size_t)(by + ly + k) * a.W + x] : kEmpty;
    Under u;
#pragma unroll
    for (int k = 0; k < kRows; k += 2) {
        if (k >= n) break;
        const uint64_t two[2] = {key[k], key[k + 1]};
        float c[2][4];
        resolve_pair<FEW>(a, two, rx[lane], ry + ly + k, u, c);
        col[ly + k][lane] = make_float4(c[0][0], c[0][1], c[0][2], c[0][3]);
        col[ly + k + 1][lane] = make_float4(c[1][0], c[1][1], c[1][2], c[1][3]);
    }
    __syncthreads();
    const float den = __int2float_rn(ss * ss);
    for (int o = threadIdx.x; o < side * side; o += 256) {
        const int oy = o / side, ox = o - oy * side;
        const int X = blockIdx.x * side + ox, Y = blockIdx.y * side + oy;
        if (X >= W || Y >= H) continue;
        float sum[4] = {0.0f, 0.0f, 0.0f, 0.0f};
        for (int sy = 0; sy < ss; ++sy)
            for (int sx = 0; sx < ss; ++sx) {
                const float4 c = col[oy * ss + sy][ox * ss + sx];
                sum[0] = __fadd_rn(sum[0], c.x);
                sum[1] = __fadd_rn(sum[1], c.y);
                sum[2] = __fadd_rn(sum[2], c.z);
                sum[3] = __fadd_rn(sum[3], c.w);
            }
#pragma unroll
        for (int ch = 0; ch < 4; ++ch) sum[ch] = __fdiv_rn(sum[ch], den);
        store_rgba(a, (size_t)Y * W + X, sum);
    }
}

// ------------------------------------------------------- textured resolve --
// Section 4.4 "Shading and Mip Mapping": rays through the centres of the
// pixel and of its right (x + 1), top (y + 1) and top-right neighbours meet
// the plane of the pixel's triangle; their barycentrics (unclamped: points
// off the triangle extrapolate) interpolate the vertex uv; the footprint is
// the larger side of the four samples' uv bounding box in level-0 texels,
// F = max(du, dv) 2^L, and the level is floor(log2 F) -- read off the
// float's exponent -- clamped to 0..L (0 when F < 1).  The colour is the
// nearest texel of that level at the pixel's own uv (column floor(u s), row
// floor(v s), s the level's side, clamped to it), c = byte / 255.  Pixels of
// meshes without a texture take the vertex colours of k_resolve.
template <bool FEW>
__global__ void __launch_bounds__(256) k_resolve_tex(const __grid_constant__ ShadeArgs a) {
    using namespace sh;
    __shared__ float rx[33], ry[kTile + 1];
    const int lane = threadIdx.x & 31, rows = a.rows;
    const int bx = blockIdx.x * 32, by = blockIdx.y * 8 * rows;
    ray_tables(rx, ry, bx, 33, by, 8 * rows + 1, a.W, a.H, a);
    const int x = bx + lane, ly = (threadIdx.x >> 5) * rows;
    const int n = x < a.W ? min(rows, a.H - (by + ly)) : 0;
    if (n <= 0) return;
    const size_t pix0 = (size_t)(by + ly) * a.W + x;
    uint64_t key[kRows];
#pragma unroll
    for (int k = 0; k < kRows; ++k) key[k] = k < n ? a.vis[pix0 + (size_t)k * a.W] : kEmpty;
    Under u;
#pragma unroll
    for (int k = 0; k < kRows; ++k) {
        if (k >= n) break;
        float c[4] = {0.0f, 0.0f, 0.0f, 0.0f};
        int lev = 255;
        uint32_t vi[3];
        bool shown = find_instance<FEW>(a, key[k], u);
        if (shown) {
            const MeshDev &m = mesh_of<FEW>(a, u);
            shown = (m.uv || m.rgba) && pixel_indices(m, u, key[k], vi);
        }
        if (shown) {
            const MeshDev &m = mesh_of<FEW>(a, u);
            float p[9], mv[12];
            pixel_positions(m, nullptr, vi, p);
            const float2 *uv = reinterpret_cast<const float2 *>(m.uv);
            model_view_of<FEW>(a, u.inst, mv);
            if (uv) {
                const float2 t0 = __ldg(uv + vi[0]), t1 = __ldg(uv + vi[1]), t2 = __ldg(uv + vi[2]);
                const Plane P = plane_of(mv, p);
                float us[4], vs[4];
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    float b0, b1, b2;
                    ray_bary(P, rx[lane + (q & 1)], ry[ly + k + (q >> 1)], b0, b1, b2);
                    us[q] = interp3(b0, b1, b2, t0.x, t1.x, t2.x);
                    vs[q] = interp3(b0, b1, b2, t0.y, t1.y, t2.y);
                }
                const float du = __fsub_rn(fmaxf(fmaxf(us[0], us[1]), fmaxf(us[2], us[3])),
                                           fminf(fminf(us[0], us[1]), fminf(us[2], us[3])));
                const float dv = __fsub_rn(fmaxf(fmaxf(vs[0], vs[1]), fmaxf(vs[2], vs[3])),
                                           fminf(fminf(vs[0], vs[1]), fminf(vs[2], vs[3])));
                const int L = m.tex_log2;
                const float F = __fmul_rn(fmaxf(du, dv), __int2float_rn(1 << L));
                lev = 0;
                if (F >= 1.0f) lev = isfinite(F) ? (int)((__float_as_uint(F) >> 23) & 0xFFu) - 127 : L;
                lev = min(lev, L);
                // level lev follows the finer levels' sum of (2^(L - l))^2 texels, l < lev:
                // (4^(L + 1) - 4^(L + 1 - lev)) / 3
                const uint64_t off = ((1ull << (2 * L + 2)) - (1ull << (2 * (L - lev) + 2))) / 3;
                const int side = 1 << (L - lev);
                const float fs = __int2float_rn(side);
                float cu = floorf(__fmul_rn(us[0], fs)), cv = floorf(__fmul_rn(vs[0], fs));
                if (!(cu >= 0.0f)) cu = 0.0f;
                if (cu > __fsub_rn(fs, 1.0f)) cu = __fsub_rn(fs, 1.0f);
                if (!(cv >= 0.0f)) cv = 0.0f;
                if (cv > __fsub_rn(fs, 1.0f)) cv = __fsub_rn(fs, 1.0f);
                const uint64_t texel = off + (uint64_t)(uint32_t)cv * (uint64_t)side + (uint64_t)(uint32_t)cu;
                const uint32_t q = __ldg(reinterpret_cast<const uint32_t *>(m.tex) + texel);
#pragma unroll
                for (int ch = 0; ch < 4; ++ch) c[ch] = byte_unit(q, ch);
            } else {
                const uint32_t *rgba = reinterpret_cast<const uint32_t *>(m.rgba);
                const uint32_t q[3] = {__ldg(rgba + vi[0]), __ldg(rgba + vi[1]), __ldg(rgba + vi[2])};
                float b0, b1, b2;
                ray_bary(plane_of(mv, p), rx[lane], ry[ly + k], b0, b1, b2);
                blend_rgba(b0, b1, b2, q, c);
            }
        }
        const size_t pix = pix0 + (size_t)k * a.W;
        if (a.level) a.level[pix] = (uint8_t)lev;
        store_rgba(a, pix, c);
    }
}

// ------------------------------------------------------- interpolate fwd --
// The pixel's triangle when it belongs to an instance of the interpolated
// mesh: its vertex indices and positions.
template <bool FEW>
__device__ __forceinline__ bool interp_pixel(const ShadeArgs &a, uint64_t key, Under &u, uint32_t (&vi)[3], float (&p)[9]) {
    if (!find_instance<FEW>(a, key, u)) return false;
    if (FEW ? a.few.mesh_id[u.inst] != a.mesh : u.mesh != a.meshes + a.mesh) return false;
    if (!pixel_indices(mesh_of<FEW>(a, u), u, key, vi)) return false;
    pixel_positions(mesh_of<FEW>(a, u), a.pos, vi, p);
    return true;
}

// CN: the number of channels where it is a usual one, 0: a.C of them.
template <int CN, bool FEW>
__global__ void __launch_bounds__(256) k_interp_fwd(const __grid_constant__ ShadeArgs a) {
    using namespace sh;
    __shared__ float rx[32], ry[kTile + 1];
    const int C = CN ? CN : a.C, lane = threadIdx.x & 31, rows = a.rows;
    const int bx = blockIdx.x * 32, by = blockIdx.y * 8 * rows;
    ray_tables(rx, ry, bx, 32, by, 8 * rows, a.W, a.H, a);
    const int x = bx + lane, ly = (threadIdx.x >> 5) * rows;
    const int n = x < a.W ? min(rows, a.H - (by + ly)) : 0;
    if (n <= 0) return;
    const size_t pix0 = (size_t)(by + ly) * a.W + x;
    uint64_t key[kRows];
#pragma unroll
    for (int k = 0; k < kRows; ++k) key[k] = k < n ? a.vis[pix0 + (size_t)k * a.W] : kEmpty;
    Under u;
#pragma unroll
    for (int k = 0; k < kRows; ++k) {
        if (k >= n) break;
        float *o = a.out + (size_t)C * (pix0 + (size_t)k * a.W);
        uint32_t vi[3];
        float p[9];
        if (interp_pixel<FEW>(a, key[k], u, vi, p)) {
            float mv[12];
            model_view_of<FEW>(a, u.inst, mv);
            const float *c0 = a.attr + (size_t)C * vi[0], *c1 = a.attr + (size_t)C * vi[1], *c2 = a.attr + (size_t)C * vi[2];
            float b0, b1, b2;
            if (CN) {                                // (the attributes' loads go out with the positions')
                float t[3][CN ? CN : 1];
#pragma unroll
                for (int ch = 0; ch < CN; ++ch) t[0][ch] = __ldg(c0 + ch), t[1][ch] = __ldg(c1 + ch), t[2][ch] = __ldg(c2 + ch);
                ray_bary(plane_of(mv, p), rx[lane], ry[ly + k], b0, b1, b2);
#pragma unroll
                for (int ch = 0; ch < CN; ++ch) o[ch] = interp3(b0, b1, b2, t[0][ch], t[1][ch], t[2][ch]);
            } else {
                ray_bary(plane_of(mv, p), rx[lane], ry[ly + k], b0, b1, b2);
                for (int ch = 0; ch < C; ++ch) o[ch] = interp3(b0, b1, b2, __ldg(c0 + ch), __ldg(c1 + ch), __ldg(c2 + ch));
            }
        } else {
            for (int ch = 0; ch < C; ++ch) o[ch] = 0.0f;
        }
    }
}

// ------------------------------------------------------- interpolate bwd --
constexpr int kMaxC = 16;

// Double-float numbers (hi + lo, |lo| <= ulp(hi) / 2) for the two
// quantities whose cancellation the backward cannot afford: the view-space
// vertex v0 and the pixel ray r.  Error-free product by FMA, error-free sum
// (Knuth's two-sum), and a sum of two double-floats.
struct DF { float hi, lo; };
__device__ __forceinline__ DF two_prod(float a, float b) {
    const float p = __fmul_rn(a, b);
    return {p, __fmaf_rn(a, b, -p)};
}
__device__ __forceinline__ DF two_sum(float a, float b) {
    const float s = __fadd_rn(a, b), bb = __fsub_rn(s, a);
    return {s, __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb))};
}
__device__ __forceinline__ DF df_add(DF x, DF y) {
    const DF s = two_sum(x.hi, y.hi);
    const float lo = __fadd_rn(s.lo, __fadd_rn(x.lo, y.lo));
    const float hi = __fadd_rn(s.hi, lo);
    return {hi, __fsub_rn(lo, __fsub_rn(hi, s.hi))};
}
// x / d for a double-float x and a float d, as a double-float: the first
// quotient rounded, its remainder exact by FMA, the remainder's quotient.
__device__ __forceinline__ DF df_div(DF x, float d) {
    const float q = __fdiv_rn(x.hi, d);
    const float rem = __fadd_rn(__fmaf_rn(-q, d, x.hi), x.lo);
    return two_sum(q, __fdiv_rn(rem, d));
}

// One coordinate of the pixel-centre ray, ((2 i + 1) / n - 1) / f, as a
// double-float (2 i + 1 and n are exact floats below 2^24).
__device__ __forceinline__ DF ray_coord(int i, int n, float f) {
    DF t = df_div({__int2float_rn(2 * i + 1), 0.0f}, __int2float_rn(n));
    t = df_add(t, {-1.0f, 0.0f});
    return df_div(t, f);
}

// a b - c d for double-floats: the hi products error-free, their difference
// as a double-float, the cross terms in FP32 (they are ulp-sized).
__device__ __forceinline__ float df_cross1(DF a, DF b, DF c, DF d) {
    const DF p = two_prod(a.hi, b.hi), q = two_prod(c.hi, d.hi);
    const DF t = df_add(p, {-q.hi, -q.lo});
    const float x = __fsub_rn(__fadd_rn(__fmul_rn(a.hi, b.lo), __fmul_rn(a.lo, b.hi)),
                              __fadd_rn(__fmul_rn(c.hi, d.lo), __fmul_rn(c.lo, d.hi)));
    return __fadd_rn(t.hi, __fadd_rn(t.lo, x));
}

// Gradient of I = sum_k b_k c_k with the visibility held fixed.  With
// D_k = r . (v_{k+1} x v_{k+2}) and S = sum_k D_k the barycentrics are
// b_k = D_k / S, so for g = dL/dI, gamma_k = g . c_k and gbar = sum b_k gamma_k:
//   dL/dc_k = g b_k,
//   dL/dv_j = [ (gamma_{j-1} - gbar) (v_{j+1} x r) + (gamma_{j+1} - gbar) (r x v_{j-1}) ] / S,
//   dL/dp_j = M^T dL/dv_j   (M = the 3x3 part of the instance's model-view).
// A pixel's ray passes ~100x closer to its triangle than the triangle lies
// to the camera, so written naively these cancel in FP32.  Everything is
// expressed instead through the ray's moment about v0, m = v0 x r, and the
// edges E_1 = e1 = v1 - v0, E_2 = e2 = v2 - v0 (E_0 = 0):
//   D_1 = e2 . m,  D_2 = -(e1 . m),  S = r . (e1 x e2),  D_0 = S - D_1 - D_2,
//   v_{j+1} x r = m + E_{j+1} x r,  r x v_{j-1} = -(m + E_{j-1} x r),
// which are all well conditioned once m is: m alone carries the
// cancellation, and is computed from v0 and r held as double-floats (v0 from
// the FP32 model-view and position with error-free products, r by
// double-float division) with a compensated cross product.  The edges come from the model-space
// differences rotated by M.  Everything else is plain FP32.
//
// The sums: a pixel adds n = 9 + 3 C numbers, three vertices' positions and
// attributes.  The lanes leave theirs in shared memory, the pixels of one
// triangle form a group, and the warp walks (group, number) pairs 32 at a
// time: a lane sums the group's number over its pixels and adds it once.
// Consecutive numbers are consecutive in memory, so a warp's additions fall
// into a third of the sectors that an addition per pixel and number, each lane
// at a vertex of its own, falls into -- and no lane searches the warp for
// equal vertices 18 times over.  A warp's pixels are an 8 x 4 patch: more of
// them share a triangle than in a row of 32.
constexpr int kBwdWarps = 8;

struct BwdGroup { uint32_t members, v[3]; };

struct BwdShared {                                   // of a block, beside the numbers
    BwdGroup groups[kBwdWarps][32];
    uint32_t dest[9 + 3 * kMaxC];                    // number: vertex | offset in the row << 2 | attribute << 31
    DF rx[32], ry[8];
};

template <bool FEW>
__global__ void __launch_bounds__(32 * kBwdWarps) k_interp_bwd(const __grid_constant__ ShadeArgs a) {
    extern __shared__ float bwd_vals[];              // [warp][lane][n | 1]
    __shared__ BwdShared blk;
    const int C = a.C, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int np = a.grad_pos ? 9 : 0, n = np + (a.grad_attr ? 3 * C : 0);
    const int bx = blockIdx.x * 32, by = blockIdx.y * 8;
    if (threadIdx.x < 32) blk.rx[lane] = ray_coord(bx + lane, a.W, a.fx);
    else if (threadIdx.x < 40) blk.ry[threadIdx.x - 32] = ray_coord(by + threadIdx.x - 32, a.H, a.fy);
    else if (threadIdx.x >= 64 && threadIdx.x < 64 + n) {
        const int c = threadIdx.x - 64, q = c - np;
        blk.dest[c] = c < np ? (uint32_t)(c / 3) | (uint32_t)(c % 3) << 2 : (uint32_t)(q / C) | (uint32_t)(q % C) << 2 | 1u << 31;
    }
    __syncthreads();
    const int lx = (warp & 3) * 8 + (lane & 7), ly = (warp >> 2) * 4 + (lane >> 3);
    const int x = bx + lx, y = by + ly;
    float *vals = bwd_vals + (size_t)(32 * warp + lane) * (n | 1);
    Under u;
    uint32_t vi[3] = {0, 0, 0};
    float p[9];
    uint64_t key = kEmpty;
    bool hit = false;
    const size_t pix = (size_t)y * a.W + x;
    if (x < a.W && y < a.H) {
        key = a.vis[pix];
        hit = interp_pixel<FEW>(a, key, u, vi, p);
    }
    if (hit) {
        float mv[12];
        model_view_of<FEW>(a, u.inst, mv);
        // v0 as double-floats, row by row
        DF v0[3];
#pragma unroll
        for (int r = 0; r < 3; ++r) {
            DF acc = two_prod(mv[4 * r], p[0]);
            acc = df_add(acc, two_prod(mv[4 * r + 1], p[1]));
            acc = df_add(acc, two_prod(mv[4 * r + 2], p[2]));
            v0[r] = df_add(acc, {mv[4 * r + 3], 0.0f});
        }
        // the pixel-centre ray as double-floats
        const DF dx = blk.rx[lx], dy = blk.ry[ly];
        const DF dz = {-1.0f, 0.0f};
        const float3 r = make_float3(dx.hi, dy.hi, -1.0f);
        // m = v0 x r
        const float3 mm = make_float3(df_cross1(v0[1], dz, v0[2], dy), df_cross1(v0[2], dx, v0[0], dz),
                                      df_cross1(v0[0], dy, v0[1], dx));
        // edges: model-space differences through M
        float3 E[3];
        E[0] = make_float3(0.0f, 0.0f, 0.0f);
#pragma unroll
        for (int k = 1; k < 3; ++k) {
            const float d0 = __fsub_rn(p[3 * k], p[0]), d1 = __fsub_rn(p[3 * k + 1], p[1]), d2 = __fsub_rn(p[3 * k + 2], p[2]);
            E[k] = make_float3(__fadd_rn(__fadd_rn(__fmul_rn(mv[0], d0), __fmul_rn(mv[1], d1)), __fmul_rn(mv[2], d2)),
                               __fadd_rn(__fadd_rn(__fmul_rn(mv[4], d0), __fmul_rn(mv[5], d1)), __fmul_rn(mv[6], d2)),
                               __fadd_rn(__fadd_rn(__fmul_rn(mv[8], d0), __fmul_rn(mv[9], d1)), __fmul_rn(mv[10], d2)));
        }
        const float S = dot3(r, cross3(E[1], E[2]));
        float D[3], b[3];
        D[1] = dot3(E[2], mm);
        D[2] = -dot3(E[1], mm);
        D[0] = __fsub_rn(__fsub_rn(S, D[1]), D[2]);
        const float invS = __frcp_rn(S);
#pragma unroll
        for (int k = 0; k < 3; ++k) b[k] = __fmul_rn(D[k], invS);
        float gam[3] = {0.0f, 0.0f, 0.0f};
        for (int ch = 0; ch < C; ++ch) {
            const float g = __ldg(a.grad_out + (size_t)C * pix + ch);
#pragma unroll
            for (int k = 0; k < 3; ++k) {
                gam[k] = __fmaf_rn(g, __ldg(a.attr + (size_t)C * vi[k] + ch), gam[k]);
                if (a.grad_attr) vals[np + k * C + ch] = __fmul_rn(g, b[k]);
            }
        }
        if (np) {
            const float gbar = __fmaf_rn(b[0], gam[0], __fmaf_rn(b[1], gam[1], __fmul_rn(b[2], gam[2])));
#pragma unroll
            for (int j = 0; j < 3; ++j) {
                const int jm = (j + 2) % 3, jp = (j + 1) % 3;
                const float w1 = __fmul_rn(__fsub_rn(gam[jm], gbar), invS), w2 = __fmul_rn(__fsub_rn(gam[jp], gbar), invS);
                const float3 cp = cross3(E[jp], r), cm = cross3(E[jm], r);
                const float wd = __fsub_rn(w1, w2);
                const float3 d = make_float3(__fmaf_rn(wd, mm.x, __fsub_rn(__fmul_rn(w1, cp.x), __fmul_rn(w2, cm.x))),
                                             __fmaf_rn(wd, mm.y, __fsub_rn(__fmul_rn(w1, cp.y), __fmul_rn(w2, cm.y))),
                                             __fmaf_rn(wd, mm.z, __fsub_rn(__fmul_rn(w1, cp.z), __fmul_rn(w2, cm.z))));
#pragma unroll
                for (int ax = 0; ax < 3; ++ax)
                    vals[3 * j + ax] = __fmaf_rn(mv[ax], d.x, __fmaf_rn(mv[4 + ax], d.y, __fmul_rn(mv[8 + ax], d.z)));
            }
        }
    }
    // the groups: pixels of one triangle
    const unsigned hits = __ballot_sync(0xffffffffu, hit);
    if (hits == 0 || n == 0) return;
    const unsigned same = __match_any_sync(0xffffffffu, (unsigned long long)(hit ? key & kIdMask : kEmpty)) & hits;
    const bool leads = hit && (same & ((1u << lane) - 1u)) == 0;
    const unsigned leaders = __ballot_sync(0xffffffffu, leads);
    if (leads) blk.groups[warp][__popc(leaders & ((1u << lane) - 1u))] = BwdGroup{same, {vi[0], vi[1], vi[2]}};
    __syncwarp();
    const float *all = bwd_vals + (size_t)32 * warp * (n | 1);
    const int total = __popc(leaders) * n;
    const int dg = 32 / n, dc = 32 - dg * n;         // a step of 32 numbers: dg groups and dc numbers
    int g = lane / n, c = lane - g * n;
    for (int i = lane; i < total; i += 32) {
        const BwdGroup &gr = blk.groups[warp][g];
        uint32_t m = gr.members;
        float sum = all[(__ffs(m) - 1) * (n | 1) + c];
        for (m &= m - 1; m; m &= m - 1) sum = __fadd_rn(sum, all[(__ffs(m) - 1) * (n | 1) + c]);
        const uint32_t d = blk.dest[c], off = (d >> 2) & 31u;
        const size_t v = gr.v[d & 3u];
        atomicAdd(d >> 31 ? a.grad_attr + (size_t)C * v + off : a.grad_pos + 3 * v + off, sum);
        g += dg;
        c += dc;
        if (c >= n) c -= n, ++g;
    }
}

// -------------------------------------------------------------- launchers --
// Rows a thread walks.  More rows share the column's tables and the instance
// found; small images want the blocks instead.  Resolve at 3840 x 2160 with 1,
// 2, 4 rows: 213, 146, 134 us; at 1920 x 1080: 47.0, 42.5, 43.7; at 300 x 200:
// 4.3, 4.9, 7.2 (one row a thread and every ray for itself: 174, 46, 5.0).
// (With the instances as parameters: 3840 x 2160 with 4 rows 123, 1920 x 1080
// with 2 rows 37.)  Where many triangles fall to a pixel, the gathers of a
// column share nothing and four rows only spread a block's addresses: with 36
// triangles a pixel at 3840 x 2160 4, 2, 1 rows took 334, 311, 320 us, with 121
// 516, 492, 488, with 259 642, 615, 597 (one row a thread and every ray for
// itself: 340, 496, 602).  Nothing here tells a close view of such a scene,
// which likes four rows (12 triangles a pixel, close: 126, 148, 185; 219 so).
static int rows_of(const ShadeArgs &a) {
    const uint64_t px = (uint64_t)a.W * (uint64_t)a.H;
    return px >= 4000000 ? (a.tris < 64 * px ? 4 : 1) : px >= 300000 ? 2 : 1;
}

static dim3 pixel_grid(int W, int H, int rows) { return dim3((unsigned)((W + 31) / 32), (unsigned)((H + 8 * rows - 1) / (8 * rows))); }

cudaError_t launch_resolve_ss(const ShadeArgs &a, int W, int H, cudaStream_t s) {
    const int side = 32 / a.ss;
    const dim3 grid((unsigned)((W + side - 1) / side), (unsigned)((H + side - 1) / side));
    if (a.n_inst <= kFew) k_resolve_ss<true><<<grid, 256, 0, s>>>(a, W, H);
    else k_resolve_ss<false><<<grid, 256, 0, s>>>(a, W, H);
    return cudaGetLastError();
}

cudaError_t launch_resolve(ShadeArgs &a, cudaStream_t s) {
    a.rows = rows_of(a);
    const dim3 grid = pixel_grid(a.W, a.H, a.rows);
    if (a.n_inst <= kFew) k_resolve<true><<<grid, 256, 0, s>>>(a);
    else k_resolve<false><<<grid, 256, 0, s>>>(a);
    return cudaGetLastError();
}

cudaError_t launch_resolve_textured(ShadeArgs &a, cudaStream_t s) {
    a.rows = rows_of(a);
    const dim3 grid = pixel_grid(a.W, a.H, a.rows);
    if (a.n_inst <= kFew) k_resolve_tex<true><<<grid, 256, 0, s>>>(a);
    else k_resolve_tex<false><<<grid, 256, 0, s>>>(a);
    return cudaGetLastError();
}

template <bool FEW>
static void interp_fwd(const ShadeArgs &a, dim3 grid, cudaStream_t s) {
    if (a.C == 1) k_interp_fwd<1, FEW><<<grid, 256, 0, s>>>(a);
    else if (a.C == 3) k_interp_fwd<3, FEW><<<grid, 256, 0, s>>>(a);
    else if (a.C == 4) k_interp_fwd<4, FEW><<<grid, 256, 0, s>>>(a);
    else k_interp_fwd<0, FEW><<<grid, 256, 0, s>>>(a);
}

cudaError_t launch_interpolate(ShadeArgs &a, cudaStream_t s) {
    a.rows = rows_of(a);
    const dim3 grid = pixel_grid(a.W, a.H, a.rows);
    if (a.n_inst <= kFew) interp_fwd<true>(a, grid, s);
    else interp_fwd<false>(a, grid, s);
    return cudaGetLastError();
}

cudaError_t launch_interpolate_backward(const ShadeArgs &a, cudaStream_t s) {
    const int n = (a.grad_pos ? 9 : 0) + (a.grad_attr ? 3 * a.C : 0);
    const size_t smem = (size_t)32 * kBwdWarps * (n | 1) * sizeof(float);
    void (*k)(ShadeArgs) = a.n_inst <= kFew ? k_interp_bwd<true> : k_interp_bwd<false>;
    if (smem + sizeof(BwdShared) > 48 * 1024) {      // (what a launch may have without asking counts both)
        const cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
    }
    k<<<pixel_grid(a.W, a.H, 1), 32 * kBwdWarps, smem, s>>>(a);
    return cudaGetLastError();
}

}  // namespace curast
