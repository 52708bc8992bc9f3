// stage2.cuh -- stage 2 (Section 4.2), included by raster.cu.
//
// A warp takes up to 32 queued triangles at a time.  Each lane sets one up:
// transform, clip (Sutherland-Hodgman, near plane and guard band) where it
// reaches beyond a plane, snap, visible pixel range.  Most of the clipped
// ones end there with no pixel on the screen; whole triangles of at most
// 1024 pixels go through the small triangles' pixel loop together; the warp
// works through the rest one by one, rasterizing sub-triangles of at most
// s2_max pixels itself and splitting larger ones along tile boundaries into
// stage-3 parts.  A queue shorter than the warps gives each triangle several
// of them, which share its pixels or tiles.
#pragma once

namespace s2 {
constexpr int kWarps = 4;
constexpr unsigned long long kGrabPx = 2048;
constexpr unsigned kMaxShare = 16;

// The share of a triangle that a warp has: the k-th of n.
struct Share { uint32_t k, n; };
}

// A part that queue 2 has no room for, by one lane.  (Out of line: the kernel
// waits for its instructions where the queue is short.)
template <bool RAY>
__device__ __noinline__ void part_in_place(const FrameDev *f, const SubTri *s, uint32_t pidx, const ViewDev *vw, int x0, int x1,
                                           int y0, int y1) {
    if (RAY) {
        RayTri R;
        if (ray_tri_of(*f, pidx, s->id, R)) ray_range(R, x0, x1, y0, y1, 0, 1, *vw, s->id);
    } else {
        raster_range(*s, x0, x1, y0, y1, 0, 1, vw->vis, vw->W);
    }
}

// The warp's share of the tiles of [x0, x1] x [y0, y1] as stage-3 parts, with
// one reservation of queue 2.  RAY: the whole triangle is ray cast, s holds its id alone.  Parts
// past the queue's capacity are rasterized in place.  Returns their number.
template <bool RAY>
__device__ __forceinline__ uint32_t append_parts(const FrameDev &f, const SubTri &s, uint32_t pidx, uint32_t view,
                                                 const ViewDev &vw, int x0, int x1, int y0, int y1, int lane,
                                                 s2::Share sh) {
    const int tl = (int)f.tile_log2, ts = 1 << tl;
    const int tx0 = x0 >> tl, ty0 = y0 >> tl, ntx = (x1 >> tl) - tx0 + 1;
    const int all = ntx * ((y1 >> tl) - ty0 + 1);
    const int each = (all + (int)sh.n - 1) / (int)sh.n, first = each * (int)sh.k, nt = min(each, all - first);
    if (nt <= 0) return 0;
    unsigned long long base = 0;
    if (lane == 0) base = atomicAdd(&f.ctr->q2_count, (unsigned long long)nt);
    base = __shfl_sync(0xffffffffu, base, 0);
    // the entry but for its tile, as the four 16-byte words it is stored in
    static_assert(sizeof(Q2Entry) == 64, "a part is four 16-byte words");
    uint4 w0, w1, w2;
    if (RAY) {
        w0 = make_uint4((uint32_t)x0, (uint32_t)x1, 0u, (uint32_t)y0);
        w1 = make_uint4((uint32_t)y1, 0u, 0u, 0u);
        w2 = make_uint4(0u, view, (uint32_t)s.id, (uint32_t)(s.id >> 32));
    } else {
        w0 = make_uint4((uint32_t)s.X[0], (uint32_t)s.X[1], (uint32_t)s.X[2], (uint32_t)s.Y[0]);
        w1 = make_uint4((uint32_t)s.Y[1], (uint32_t)s.Y[2], __float_as_uint(s.iz[0]), __float_as_uint(s.iz[1]));
        w2 = make_uint4(__float_as_uint(s.iz[2]), view, (uint32_t)s.id, (uint32_t)(s.id >> 32));
    }
    int tx = (first + lane) % ntx, ty = ty0 + (first + lane) / ntx;   // stepped by 32 tiles: sy rows and sx columns
    const int sx = 32 % ntx, sy = 32 / ntx;
    for (int k = lane; k < nt; k += 32) {
        const uint32_t ex = (uint32_t)(tx0 + tx), ey = (uint32_t)ty;
        tx += sx;
        ty += sy;
        if (tx >= ntx) tx -= ntx, ++ty;
        if (base + k < f.q2_cap) {
            uint4 *e = reinterpret_cast<uint4 *>(f.q2 + base + k);
            e[0] = w0; e[1] = w1; e[2] = w2;
            e[3] = make_uint4(ex, ey, RAY ? pidx : 0u, RAY ? 1u : 0u);
            if (f.s3_bin) atomicAdd(&f.tile_cnt[vw.tile0 + ey * vw.ntx + ex], 1u);
        } else {
            atomicAdd(&f.ctr->overflow2, 1ull);
            const int rx0 = max(x0, (int)ex * ts), rx1 = min(x1, (int)ex * ts + ts - 1);
            const int ry0 = max(y0, (int)ey * ts), ry1 = min(y1, (int)ey * ts + ts - 1);
            const SubTri t = s;
            part_in_place<RAY>(&f, &t, pidx, &vw, rx0, rx1, ry0, ry1);
        }
    }
    return (uint32_t)nt;
}

// One sub-triangle by the whole warp.
__device__ __forceinline__ void stage2_subtri(const FrameDev &f, SubTri &s, uint32_t view, const ViewDev &vw, int lane,
                                              s2::Share sh, unsigned long long &n_s2, unsigned long long &n_parts) {
    if (!setup_subtri(s, vw.W, vw.H)) return;
    const int64_t cnt = (int64_t)(s.x1 - s.x0 + 1) * (int64_t)(s.y1 - s.y0 + 1);
    if (cnt <= (int64_t)f.s2_max) {
        raster_range(s, s.x0, s.x1, s.y0, s.y1, lane + 32 * (int)sh.k, 32 * (int)sh.n, vw.vis, vw.W);
        n_s2 += sh.k == 0;
    } else {
        n_parts += append_parts<false>(f, s, 0u, view, vw, s.x0, s.x1, s.y0, s.y1, lane, sh);
    }
}

// A queued triangle as the polygon of its screen vertices (X, Y, iz)[0 .. np),
// by the whole warp.
__device__ __forceinline__ void stage2_poly(const FrameDev &f, const int *X, const int *Y, const float *iz, int np,
                                            uint64_t id, uint32_t pair, uint32_t view, const ViewDev &vw, int lane,
                                            s2::Share sh, unsigned long long &n_s2, unsigned long long &n_parts) {
    SubTri s;
    s.id = id;
    if (f.s3_ray) {
        // the paper's stage 3: a triangle whose visible bbox holds more
        // than s2_max pixel centres is ray cast over that range, in tiles
        int x0, x1, y0, y1;
        const int64_t cnt = poly_range(X, Y, np, vw.W, vw.H, x0, x1, y0, y1);
        if (cnt == 0) return;
        if (cnt > (int64_t)f.s2_max) {
            n_parts += append_parts<true>(f, s, pair, view, vw, x0, x1, y0, y1, lane, sh);
            return;
        }
    }
    // sub-triangles dealt out to the shares, or all of them to each
    const uint32_t m = (uint32_t)np - 2, each = sh.n / m;
    int j = 1, end = np - 1;
    if (each > 0) {
        if (sh.k / each >= m) return;
        j += (int)(sh.k / each);
        end = j + 1;
        sh = {sh.k % each, each};
    }
    for (; j < end; ++j) {
        s.X[0] = X[0]; s.X[1] = X[j]; s.X[2] = X[j + 1];
        s.Y[0] = Y[0]; s.Y[1] = Y[j]; s.Y[2] = Y[j + 1];
        s.iz[0] = iz[0]; s.iz[1] = iz[j]; s.iz[2] = iz[j + 1];
        stage2_subtri(f, s, view, vw, lane, sh, n_s2, n_parts);
    }
}

// Whether a triangle beyond some plane covers anything: false when its
// clipped polygon holds no pixel centre of the screen.
__device__ __noinline__ bool clipped_visible(const CV *c, const ViewDev *vw) {
    CV poly[kMaxPoly];
    const int np = clip_polygon(c, vw->nearv, poly);
    if (np < 3) return false;
    int X[kMaxPoly], Y[kMaxPoly];
    float iz;
    for (int k = 0; k < np; ++k) snap(poly[k], vw->hw, vw->hh, X[k], Y[k], iz);
    int x0, x1, y0, y1;
    return poly_range(X, Y, np, vw->W, vw->H, x0, x1, y0, y1) > 0;
}

// per: triangles a warp takes at once.  Big triangles are dealt out finely,
// kGrabPx pixels a grab by the queue's average, or the last warps to get some
// would work long after the others; a short queue is dealt out singly, so that
// all warps share it.  (A 100 M-triangle view whose queue is half clipped
// triangles without a pixel and half small ones handed over: 67 us singly,
// 35 us in sevens.)  A warp's first grab is its own by its number, so that the
// ones without any leave at once: one atomic of each of 2432 warps on one
// counter is 4 us.  A queue of fewer triangles than half the warps gives each
// to several, up to kMaxShare: the triangles in it are then as a rule the large
// ones, and a single warp would write thousands of parts (twelve triangles
// that fill 3840 x 2160: 23 us, 8 now).
__global__ void __launch_bounds__(32 * s2::kWarps) k_stage2(const __grid_constant__ FrameDev f) {
    using namespace s2;
    __shared__ s1::SmallBatch<1> sw[kWarps];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    s1::SmallBatch<1> &S = sw[warp];
    begin_stage(f, kStampStage2);
    const unsigned long long total = *((volatile unsigned long long *)&f.ctr->q1_count);
    const unsigned long long n = total < f.q1_cap ? total : f.q1_cap;
    const unsigned long long nw = (unsigned long long)gridDim.x * kWarps;
    const uint32_t fair = max((uint32_t)min(n, 64 * nw) / (uint32_t)(2 * nw), n < nw ? 1u : 4u);
    const float light = __fdividef((float)kGrabPx * __ull2float_rn(total),
                                   __ull2float_rn(*((volatile unsigned long long *)&f.ctr->q1_px)) + 1.0f);
    const uint32_t per = max(1u, min(32u, min(fair, (uint32_t)light)));
    const uint32_t share = 2 * n <= nw ? min(kMaxShare, (uint32_t)nw / ((uint32_t)n + 1)) : 1u;   // per is 1 then
    unsigned long long n_s2 = 0, n_parts = 0;
    unsigned long long unit = (unsigned long long)warp * gridDim.x + blockIdx.x;   // neighbours on different SMs
    for (;;) {
        const unsigned long long i0 = share > 1 ? (uint32_t)unit / share : unit * per;
        const Share sh = {share > 1 ? (uint32_t)unit % share : 0u, share};
        if (i0 >= n) break;
        const uint32_t g = (uint32_t)min((unsigned long long)per, n - i0);
        uint32_t npx = 0, view = 0;
        bool whole = false, clip = false;             // for the warp: unclipped, clipped
        if (lane < g) {
            const Q1Entry e = f.q1[i0 + lane];
            const PairDev &pr = f.pairs[e.pair];
            view = pr.view;
            const ViewDev &vw = f.views[view];
            CV c[3];
            load_clip(f, f.meshes[pr.mesh], e.pair, e.id - pr.base, vw, c);
            if ((outcode(c[0], vw.nearv) | outcode(c[1], vw.nearv) | outcode(c[2], vw.nearv)) == 0) {
                // inside every plane: Sutherland-Hodgman would return it unchanged
                int X[3], Y[3];
                float iz[3];
#pragma unroll
                for (int k = 0; k < 3; ++k) snap(c[k], vw.hw, vw.hh, X[k], Y[k], iz[k]);
                int x0, x1, y0, y1;
                const int64_t cnt = poly_range(X, Y, 3, vw.W, vw.H, x0, x1, y0, y1);
                const int ex = max(X[0], max(X[1], X[2])) - min(X[0], min(X[1], X[2]));
                const int ey = max(Y[0], max(Y[1], Y[2])) - min(Y[0], min(Y[1], Y[2]));
                if (cnt > 1024 || max(ex, ey) >= (1 << 14) || (!e.small && cnt > (int64_t)f.s2_max)) {
                    whole = true;
                    S.t[lane][0] = make_uint4((uint32_t)X[0], (uint32_t)X[1], (uint32_t)X[2], (uint32_t)Y[0]);
                    S.t[lane][1] = make_uint4((uint32_t)Y[1], (uint32_t)Y[2], __float_as_uint(iz[0]), __float_as_uint(iz[1]));
                    S.t[lane][2] = make_uint4(__float_as_uint(iz[2]), 0u, 0u, 0u);
                } else if (cnt > 0) {
                    const int A = (X[1] - X[0]) * (Y[2] - Y[0]) - (X[2] - X[0]) * (Y[1] - Y[0]);
                    if (A > 0)
                        npx = put_small(S.t[lane], X, Y, iz, A, e.id, view, x0, y0, (uint32_t)(x1 - x0 + 1),
                                          (uint32_t)(y1 - y0 + 1));
                }
            } else {
                clip = per == 1 || clipped_visible(c, &vw);
#pragma unroll
                for (int k = 0; k < 3; ++k)
                    S.t[lane][k] = make_uint4(__float_as_uint(c[k].x), __float_as_uint(c[k].y), __float_as_uint(c[k].w), 0u);
            }
        }
        if (sh.k != 0) npx = 0;                       // whole in the first share
        S.npx[lane] = npx;
        __syncwarp();
        small_raster<1>(f, S, lane, nullptr);
        n_s2 += __popc(__ballot_sync(0xffffffffu, npx != 0));
        const unsigned clipped = __ballot_sync(0xffffffffu, clip);
        for (unsigned m = __ballot_sync(0xffffffffu, whole) | clipped; m; m &= m - 1) {
            const int l = __ffs(m) - 1;
            const Q1Entry e = f.q1[i0 + l];
            const uint32_t v = f.pairs[e.pair].view;
            const ViewDev &vw = f.views[v];
            const uint4 ta = S.t[l][0], tb = S.t[l][1], tc = S.t[l][2];
            int X[kMaxPoly], Y[kMaxPoly], np = 3;
            float iz[kMaxPoly];
            if (clipped >> l & 1u) {
                const CV c[3] = {{__uint_as_float(ta.x), __uint_as_float(ta.y), __uint_as_float(ta.z)},
                                 {__uint_as_float(tb.x), __uint_as_float(tb.y), __uint_as_float(tb.z)},
                                 {__uint_as_float(tc.x), __uint_as_float(tc.y), __uint_as_float(tc.z)}};
                CV poly[kMaxPoly];
                np = clip_polygon(c, vw.nearv, poly);
                if (np < 3) continue;
                for (int k = 0; k < np; ++k) snap(poly[k], vw.hw, vw.hh, X[k], Y[k], iz[k]);
            } else {
                X[0] = (int)ta.x; X[1] = (int)ta.y; X[2] = (int)ta.z;
                Y[0] = (int)ta.w; Y[1] = (int)tb.x; Y[2] = (int)tb.y;
                iz[0] = __uint_as_float(tb.z); iz[1] = __uint_as_float(tb.w); iz[2] = __uint_as_float(tc.x);
            }
            stage2_poly(f, X, Y, iz, np, e.id, e.pair, v, vw, lane, sh, n_s2, n_parts);
        }
        __syncwarp();
        if (share > 1) break;                         // units for all warps at most: n share <= nw
        if (lane == 0) unit = nw + atomicAdd(&f.ctr->q1_next, 1ull);
        unit = __shfl_sync(0xffffffffu, unit, 0);
    }
    if (f.stats && lane == 0) {
        stat_add(f, kStatS2, n_s2);
        stat_add(f, kStatParts, n_parts);
    }
}
