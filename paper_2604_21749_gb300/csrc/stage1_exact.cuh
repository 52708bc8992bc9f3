// stage1_exact.cuh -- the exact part of stage 1 (Section 4.1), included by raster.cu.
//
// A warp takes the survivors that the cull left in the round's bitmap, up to
// 32 * kExactK at a time, and works in three steps that meet in the warp's
// shared memory, so that no step holds registers for another:
//   gather     every lane loads the indices and positions of its kExactK
//              survivors before any arithmetic;
//   set up     one survivor a lane: transform, cull, snap, classify; a small
//              triangle leaves its snapped vertices, 1/depths and pixel range;
//   rasterize  the pixel ranges of the whole batch laid end to end, 32 pixels
//              a step, one a lane, whatever triangles they belong to.
// A lane that walked its own triangle's pixels alone would keep the warp for
// the largest range of the 32, with the division and the atomic issued at
// nearly every step for a lane or two.
#pragma once

namespace s1 {
constexpr int kExactWarps = 20;                      // one block an SM, 96 registers a thread
constexpr int kExactK = 3;                           // survivors a lane gathers together
constexpr int kBatch = 32 * kExactK;
constexpr uint32_t kUnits = 13;                      // units dealt out of one block of the bitmap
constexpr uint32_t kUnitSurvivors = 128;             // survivors of a unit, about
constexpr int kDenseBits = 12;                       // words with as many survivors are unpacked by the whole warp
constexpr uint32_t kSegPx = 1024;                    // pixels whose triangle starts are marked at once

// A small triangle ready for the pixel loop is three 16-byte words (eight lanes'
// 16-byte loads of neighbouring records touch every bank once):
//   e0, e1, A, c0     edge functions 0 and 1 at the centre of pixel (x0, y0); the sum of all three;
//   c1, iz[3]         c0, c1: edges 0 (vertex 1 to 2) and 1 (2 to 0) as dx + 65536 dy, in subpixels.  The
//                     sign is that of dy, or of dx where dy is 0: negative for a top-left edge.
//                     iz: 1/depth of the vertices
//   id, idh, at, sh   the global id's low word; its 4 high bits | view << 8; x0 | y0 << 16 of the pixel
//                     range; its width w | ceil(2^20 / w) << 11

// Up to 32 K small triangles of one warp, K a lane, and the pixel loop's marks.
template <int K>
struct SmallBatch {
    uint4 t[32 * K][3];        // the record of each slot
    uint32_t npx[32 * K];      // pixels of its range (0: nothing to rasterize)
    uint32_t list[32 * K];     // triangles with pixels: first pixel of the batch | slot << 20
    uint32_t starts[kSegPx / 32];   // bit i: pixel i of the segment is a triangle's first
};

struct ExactWarp : SmallBatch<kExactK> {             // (t first holds the nine gathered floats)
    uint2 e[kBatch];           // (triangle, pair)
};
}  // namespace s1

__device__ __forceinline__ uint32_t fastdiv(uint32_t n, uint32_t m, uint32_t sh) {   // (fastdiv_consts)
    const uint32_t t = __umulhi(n, m);
    return (t + ((n - t) >> 1)) >> sh;
}

// The record of a front-facing triangle with both extents below 2^14
// subpixels, doubled area A and a range of at most 1024 pixels, w a row and h
// a column, from (x0, y0) on; returns its pixels.
__device__ __forceinline__ uint32_t put_small(uint4 (&t)[3], const int (&X)[3], const int (&Y)[3], const float (&iz)[3],
                                              int A, uint64_t id, uint32_t view, int x0, int y0, uint32_t w, uint32_t h) {
    // m = ceil(2^20 / w): the approximate quotient is off by less than 1/w, so its floor is the true one or,
    // where w divides 2^20, perhaps one less
    uint32_t m = (uint32_t)(1048576.0f * rcp_approx((float)w));
    m += m * w < (1u << 20) ? 1u : 0u;
    // edge k runs from vertex k+1 to vertex k+2; (px, py) is the first pixel's centre
    const int px = 256 * x0 + 128, py = 256 * y0 + 128;
    const int dx0 = X[2] - X[1], dy0 = Y[2] - Y[1], dx1 = X[0] - X[2], dy1 = Y[0] - Y[2];
    const int e0 = dx0 * (py - Y[1]) - dy0 * (px - X[1]), e1 = dx1 * (py - Y[2]) - dy1 * (px - X[2]);
    t[0] = make_uint4((uint32_t)e0, (uint32_t)e1, (uint32_t)A, (uint32_t)(dx0 + 65536 * dy0));
    t[1] = make_uint4((uint32_t)(dx1 + 65536 * dy1), __float_as_uint(iz[0]), __float_as_uint(iz[1]), __float_as_uint(iz[2]));
    t[2] = make_uint4((uint32_t)id, (uint32_t)(id >> 32) | view << 8, (uint32_t)x0 | (uint32_t)y0 << 16, w | m << 11);
    return w * h;
}

// Set-up of the survivor in `slot`: its class, and for a small triangle its
// record in the warp's shared memory, with its number of pixels (else 0).
// Same decisions and values as outcode, snap and setup_subtri give; what is
// left out cannot change them:
//   - inside every plane is decided from w >= near, |x| <= 128 w, |y| <= 128 w,
//     which have the signs of the five plane values (a sum of two finite
//     floats rounds to zero only when it is zero; NaN fails both forms; an
//     infinite 128 w takes the outcodes);
//   - snap's clamp: inside the guard band |X| < 129 * 8192 * 256 < 2^29, once
//     1/w is finite; vertices with w < 2^-120 (wmin) send the triangle to
//     stage 2;
//   - its two multiplications by H/2 and 256 as one by 128 H (a scaling by a
//     power of two is exact).
template <bool RAY>
__device__ __forceinline__ void exact_setup(const FrameDev &f, s1::ExactWarp &S, int slot, bool live) {
    uint32_t npx = 0, px = 0;                      // px: pixels of a triangle for stage 2
    bool queue = false;
    uint64_t id = 0;
    uint2 e = make_uint2(0u, 0u);
    const MeshDev *mesh = f.meshes;
    unsigned st = kStatCount;
    if (live) {
        e = S.e[slot];
        const PairDev &pr = f.pairs[e.y];
        const float4 *pw = reinterpret_cast<const float4 *>(&pr);
        const float4 r0 = pw[0], r1 = pw[1], r2 = pw[2], cam = pw[3];
        const float4 pa = reinterpret_cast<const float4 *>(S.t[slot])[0], pb = reinterpret_cast<const float4 *>(S.t[slot])[1];
        const float p[9] = {pa.x, pa.y, pa.z, pa.w, pb.x, pb.y, pb.z, pb.w, __uint_as_float(S.t[slot][2].x)};
        // (scalar: the assembler contracts packed mul.rn.f32x2 / add.rn.f32x2 pairs into FMAs)
        const float mv[12] = {r0.x, r0.y, r0.z, r0.w, r1.x, r1.y, r1.z, r1.w, r2.x, r2.y, r2.z, r2.w};
        CV c[3];
#pragma unroll
        for (int k = 0; k < 3; ++k) c[k] = to_clip(mv, p[3 * k], p[3 * k + 1], p[3 * k + 2], cam.x, cam.y);
        id = pr.base + e.x;
        mesh = f.meshes + pr.mesh;
        bool inside = true;
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            const float gw = __fmul_rn(kGuard, c[k].w);
            inside &= (c[k].w >= cam.w) & (gw < INFINITY) & (fabsf(c[k].x) <= gw) & (fabsf(c[k].y) <= gw);
        }
        if (!inside) {
            // beyond one clip plane, or to be clipped by stage 2
            queue = (outcode(c[0], cam.z) & outcode(c[1], cam.z) & outcode(c[2], cam.z)) == 0;
            if (!queue) st = kStatClip;
        } else {
            const float4 scr = pw[4];                // sx, sy, W, H
            int X[3], Y[3];
            float iz[3];
#pragma unroll
            for (int k = 0; k < 3; ++k) {
                iz[k] = __frcp_rn(c[k].w);
                X[k] = __float2int_rn(__fmul_rn(__fadd_rn(__fmul_rn(c[k].x, iz[k]), 1.0f), scr.x));
                Y[k] = __float2int_rn(__fmul_rn(__fadd_rn(__fmul_rn(c[k].y, iz[k]), 1.0f), scr.y));
            }
            const int minX = min(X[0], min(X[1], X[2])), maxX = max(X[0], max(X[1], X[2]));
            const int minY = min(Y[0], min(Y[1], Y[2])), maxY = max(Y[0], max(Y[1], Y[2]));
            const bool big = max(maxX - minX, maxY - minY) >= (1 << 14);
            const int ux = X[1] - X[0], uy = Y[1] - Y[0], wx = X[2] - X[0], wy = Y[2] - Y[0];
            const int A = ux * wy - wx * uy;         // (of no use where big)
            const bool front = big ? (int64_t)ux * wy - (int64_t)wx * uy > 0 : A > 0;
            int x0, x1, y0, y1;
            centre_range(minX, maxX, __float_as_int(scr.z), x0, x1);
            centre_range(minY, maxY, __float_as_int(scr.w), y0, y1);
            if (!front) {
                st = kStatBack;
            } else if (x0 > x1 || y0 > y1) {
                st = kStatTiny;
            } else {
                const uint32_t w = (uint32_t)(x1 - x0 + 1), h = (uint32_t)(y1 - y0 + 1);
                queue = big || w * h > f.s1_max;
                if (queue) px = w * h;
                else npx = put_small(S.t[slot], X, Y, iz, A, id, pr.view, x0, y0, w, h);
            }
        }
    }
    S.npx[slot] = npx;
    q1_append<RAY>(f, queue, px, id, e.y, mesh, e.x);
    if (f.stats && live) {
        stat_add(f, kStatIn, 1);
        if (st != kStatCount) stat_add(f, st, 1);
        if (npx) stat_add(f, kStatS1, 1);
    }
}

// The pixels p0 .. p1 - 1 of a batch, 32 a step.  npx / at0: as in
// small_raster; first: triangles that start before p0, less one.
template <int K>
__device__ __forceinline__ void small_span(const FrameDev &f, s1::SmallBatch<K> &S, const uint32_t (&npx)[K], uint32_t at0,
                                           uint32_t p0, uint32_t p1, int first, int lane) {
    using namespace s1;
    const uint32_t upto = 0xffffffffu >> (31 - lane);
    for (uint32_t sb = p0; sb < p1; sb += kSegPx) {
        const uint32_t nwin = (min(p1 - sb, kSegPx) + 31) / 32;
        for (uint32_t w = lane; w < nwin; w += 32) S.starts[w] = 0;
        __syncwarp();
        uint32_t at = at0;
#pragma unroll
        for (int u = 0; u < K; ++u)
            if (npx[u]) {
                const uint32_t i = (at & 0xFFFFFu) - sb;
                if (i < 32 * nwin) atomicOr(&S.starts[i >> 5], 1u << (i & 31));
                at += npx[u] + (1u << 20);
            }
        __syncwarp();
        for (uint32_t w = 0; w < nwin; ++w) {
            const uint32_t word = S.starts[w], i = sb + 32 * w + lane;
            const int o = first + __popc(word & upto);
            first += __popc(word);
            if (i >= p1) continue;
            const uint32_t L = S.list[o], k = i - (L & 0xFFFFFu);
            const uint4 *t = S.t[L >> 20];
            const uint4 ta = t[0], tb = t[1], tc = t[2];
            const uint32_t dy = (k * (tc.w >> 11)) >> 20, dx = k - dy * (tc.w & 2047u);
            // one column changes E_k by -256 dy_k and one row by 256 dx_k
            const int X0 = (int)(ta.w << 16) >> 8, X1 = (int)(tb.x << 16) >> 8;
            const int e0 = (int)ta.x + (int)dy * X0 - (int)dx * (((int)ta.w - (X0 >> 8)) >> 8);
            const int e1 = (int)ta.y + (int)dy * X1 - (int)dx * (((int)tb.x - (X1 >> 8)) >> 8);
            const int e2 = (int)ta.z - e0 - e1;
            // less 1 where the edge is not top-left: the signs decide; edge 2 is minus the sum of the others
            if (((e0 - 1 - ((int)ta.w >> 31)) | (e1 - 1 - ((int)tb.x >> 31)) |
                 (e2 - 1 - (-((int)ta.w + (int)tb.x) >> 31))) < 0) continue;
            const float s = __fadd_rn(__fadd_rn(__fmul_rn(__int2float_rn(e0), __uint_as_float(tb.y)),
                                                __fmul_rn(__int2float_rn(e1), __uint_as_float(tb.z))),
                                      __fmul_rn(__int2float_rn(e2), __uint_as_float(tb.w)));
            const float depth = __fdiv_rn(__int2float_rn((int)ta.z), s);
            const ViewDev &vw = f.views[tc.y >> 8];
            const uint64_t key = (uint64_t)(__float_as_uint(depth) >> 3) << 36 | (uint64_t)(tc.y & 15u) << 32 | tc.x;
            depth_min(vw.vis, (size_t)((tc.z >> 16) + dy) * (size_t)vw.W + ((tc.z & 0xFFFFu) + dx), key);
        }
        __syncwarp();
    }
}

// Rasterizes the small triangles of a batch: slot s holds npx[s] pixels.  The
// ranges are laid end to end in the order (lane, u); the triangle of pixel i
// is the last one to start at or before i, found by counting the marked starts
// up to it.  A range is walked row by row: pixel k of a range of width w is
// (k mod w, k / w), the division as a multiplication by m = ceil(2^20 / w),
// exact for k, w <= 1024 (k (m w - 2^20) < 2^20).  The edge functions are
// int32: both extents are below 2^14 subpixels, so |E| < 2^30 at every visited
// sample, and E2 = A - E0 - E1 exactly.  (A lane a 2 x 2 quad, its covered
// pixels one by one, needs fewer steps but was no faster: 923 us against 905
// on the billion-triangle frame, 620 against 621 on compressed terrain.)
// give(want, slot): where the batch holds more than 2 kSegPx pixels, hands
// over the triangles that start past pixel kSegPx, the lanes' `want`ed ones
// in lane order, and returns false to those it has no room for (the last
// ones); nullptr keeps them all.
template <int K, class Give>
__device__ __forceinline__ void small_raster(const FrameDev &f, s1::SmallBatch<K> &S, int lane, Give give) {
    using namespace s1;
    uint32_t npx[K], own = 0;                      // own: pixels | triangles << 20
#pragma unroll
    for (int u = 0; u < K; ++u) npx[u] = S.npx[lane + 32 * u];
#pragma unroll
    for (int u = 0; u < K; ++u) own += npx[u] ? npx[u] + (1u << 20) : 0u;
    uint32_t incl = own;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t v = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += v;
    }
    const uint32_t all = __shfl_sync(0xffffffffu, incl, 31), P = all & 0xFFFFFu;
    if (P == 0) return;
    const uint32_t at0 = incl - own;
    uint32_t at = at0;
#pragma unroll
    for (int u = 0; u < K; ++u)
        if (npx[u]) {
            S.list[at >> 20] = (at & 0xFFFFFu) | (uint32_t)(lane + 32 * u) << 20;
            at += npx[u] + (1u << 20);
        }
    uint32_t pa = P, pb = P;                         // pixels pa .. pb - 1 are handed over
    int fb = 0;
    if constexpr (!std::is_same<Give, std::nullptr_t>::value) {
        if (P > 2 * kSegPx) {
            __syncwarp();
            const int nt = (int)(all >> 20);
            int g0 = 0;                              // the first triangle to start at or past kSegPx
            for (int b = 0; b < nt; b += 32)
                g0 += __popc(__ballot_sync(0xffffffffu, b + lane < nt && (S.list[min(b + lane, nt - 1)] & 0xFFFFFu) < kSegPx));
            int kept = nt;                           // triangles from here on found no room
            for (int b = g0; b < nt && kept == nt; b += 32) {
                const bool want = b + lane < nt;
                const bool ok = give(want, (int)(S.list[want ? b + lane : nt - 1] >> 20));
                const unsigned bad = __ballot_sync(0xffffffffu, want && !ok);
                if (bad) kept = b + __ffs(bad) - 1;
            }
            if (g0 < nt) pa = S.list[g0] & 0xFFFFFu;
            if (kept < nt) pb = S.list[kept] & 0xFFFFFu;
            fb = kept - 1;
        }
    }
    small_span(f, S, npx, at0, 0u, pa, -1, lane);
    if (pb < P) small_span(f, S, npx, at0, pb, P, fb, lane);
}

size_t exact_smem_bytes() { return sizeof(s1::ExactWarp) * s1::kExactWarps; }

// The exact kernel, round r, one block of 20 warps an SM.  Warps take the
// bitmap in units of 1 .. 128 words, a word, two or four for each lane:
// survivors come in clusters where the view looks closely, and a fixed deal of
// 32-word chunks to warps left some SMs with twice the average (the full-HD
// view of a 4.2 M-triangle mesh: 179 us, 108 now).  A unit in a cluster
// holds some 128 survivors: with 64 the fetches cost more than the balance gains (75 M
// triangles compressed: 671 us against 621), with 512 single units last too
// long (the full-HD view 147 us, a clustered 100 M-triangle view 537 against
// 397); sparse frames reach 128 words first.  Units of more than eight words
// are runs of eight kUnits runs apart, so that a cluster spreads over several.
// The SM's share of the units is taken from a counter in shared memory, the
// last of them from one in global memory, which evens the SMs out: one global
// address takes an atomic add every 1.8 ns, too slow for every unit (32-word
// units of the billion-triangle frame: 1.75 ms against 0.90).  The words of
// the next unit are in flight while a batch runs.  COMP: the round's meshes
// are compressed (one kernel for both tested it per triangle, 1% of the frame).
template <bool RAY, bool COMP>
__global__ void __launch_bounds__(32 * s1::kExactWarps, 1)
    k_stage1_exact(const __grid_constant__ FrameDev f, uint32_t r) {
    using namespace s1;
    extern __shared__ __align__(128) unsigned char exact_smem[];
    __shared__ uint32_t s_taken;                    // units the SM has taken of its share
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    ExactWarp &S = reinterpret_cast<ExactWarp *>(exact_smem)[warp];
    __shared__ uint32_t s_sample;                   // survivors at the places sampled | places with any << 20
    if (threadIdx.x == 0) s_taken = s_sample = 0;
    __syncthreads();
    begin_stage(f, kStampCount);
    if (f.stamps && blockIdx.x == 0 && threadIdx.x == 0 && r + 1 == f.hdr->n_rounds) f.stamps[kStampExact] = now_ns();
    const RoundDev rd = f.rounds[r];
    const uint64_t nwords = rd.w1 - rd.w0;
    const int n_segs = (int)f.hdr->n_segs;
    const uint32_t G = kConsumerWarps * f.tpt;
    const uint64_t per_item = (uint64_t)kConsumers * f.tpt;
    const uint32_t nw = gridDim.x * kExactWarps;
    // 2^lw words a unit.  Every block estimates the survivors and their density where there are any from the
    // same 640 places (the cull would pay 3% for counting them): a unit of kUnitSurvivors at that density,
    // fewer where an SM would get less than 16 such units, but 16 words where there are twelve of that for
    // every warp, and not so small that the fetches over empty stretches pile up.  Frames with few words need
    // no estimate.  All blocks have to arrive at the same split: the cull before this kernel wrote the words
    // while it was already resident, so they are read from L2, never through the constant-data path.
    uint64_t per_unit = nwords / nw;
    if (nwords >= 8ull * nw) {
        const uint64_t q = nwords / 4 * threadIdx.x / blockDim.x;
        const uint4 v = __ldcg(reinterpret_cast<const uint4 *>(f.bits) + q);
        const uint32_t n = __popc(v.x) + __popc(v.y) + __popc(v.z) + __popc(v.w);
        const uint32_t sum = __reduce_add_sync(0xffffffffu, n) | (uint32_t)__popc(__ballot_sync(0xffffffffu, n != 0)) << 20;
        if (lane == 0 && sum) atomicAdd(&s_sample, sum);
        __syncthreads();
        const uint32_t bits = max(s_sample & 0xFFFFFu, 1u), places = s_sample >> 20;
        const uint64_t survivors = bits * (nwords / (4 * blockDim.x));
        const uint64_t hold = min((uint64_t)kUnitSurvivors, survivors / (16 * gridDim.x));
        per_unit = max(max(hold * 4 * places / bits, min((uint64_t)16, nwords / (12 * (uint64_t)nw))), nwords / (128 * (uint64_t)nw));
    }
    int lw = 0;
    while (lw < 7 && per_unit >> (lw + 1) != 0) ++lw;
    const int wide = max(lw - 5, 0);                // 2^wide words a lane
    const uint32_t per_block = lw > 3 ? kUnits : 1u;
    const uint32_t block = per_block << lw;         // words
    const uint32_t nunits = (uint32_t)((nwords + block - 1) / block) * per_block;   // (a unit is 128 words if many)
    const uint32_t at = (uint32_t)lane << wide;     // the lane's place in its unit
    const uint64_t lane0 = at >> lw != 0 ? nwords : (uint64_t)(at >> 3) * 8 * kUnits + (at & 7u);
    // the SM's share of all units but the last, at most 1/8 of them, then whatever is left of those
    const uint32_t shared_out = nunits - min(nunits / 8, 2 * nw);
    auto grab = [&]() -> uint32_t {
        const uint32_t u = blockIdx.x + atomicAdd(&s_taken, 1u) * gridDim.x;
        return u < shared_out ? u : shared_out + atomicAdd(&f.ctr->xwork[r], 1u);
    };
    uint32_t next = lane == 0 ? grab() : 0u;        // lane 0: the unit after the one being fetched
    uint64_t word = 0;                              // the lane's first word of the unit
    bool more = true;
    // moves to the next unit and issues its load
    auto fetch = [&]() -> uint4 {
        const uint32_t unit = __shfl_sync(0xffffffffu, next, 0);
        more = unit < nunits;
        if (lane == 0 && more) next = grab();
        const uint32_t b = lw > 3 ? unit / kUnits : unit;
        word = lane0 + (uint64_t)b * block + (lw > 3 ? 8 * (unit - b * kUnits) : 0u);
        uint4 w = make_uint4(0u, 0u, 0u, 0u);
        if (more && word < nwords) {                // (a round's words are a multiple of 8)
            if (wide == 0) {
                w.x = __ldcs(f.bits + word);
            } else if (wide == 1) {
                const uint2 v = __ldcs(reinterpret_cast<const uint2 *>(f.bits + word));
                w.x = v.x; w.y = v.y;
            } else {
                w = __ldcs(reinterpret_cast<const uint4 *>(f.bits + word));
            }
        }
        return w;
    };
    uint4 w_next = fetch();
    uint32_t m = 0, m1 = 0, m2 = 0, m3 = 0;         // bits of the lane's words not yet batched
    uint32_t t0 = 0, pair = 0;                      // the triangle of bit 0 of m, and its pair
    int seg = 0;                                    // segment of the lane's last run so far
    const unsigned lt_mask = (1u << lane) - 1u;
    while (true) {
        int n = 0;                                  // survivors in the batch (warp-uniform)
        while (n < kBatch) {
            if (__ballot_sync(0xffffffffu, m != 0) == 0) {
                if (__ballot_sync(0xffffffffu, (m1 | m2 | m3) != 0)) {
                    m = m1; m1 = m2; m2 = m3; m3 = 0;   // the next word of the runs
                    t0 += 32;
                    continue;
                }
                if (!more) break;
                m = w_next.x; m1 = w_next.y; m2 = w_next.z; m3 = w_next.w;   // the next unit
                const uint64_t at = rd.w0 + word;
                w_next = fetch();
                if (m | m1 | m2 | m3) {
                    // the run's segment: strides doubled forward, then halved (20,000 meshes of one instance
                    // each walked one by one: exact kernel 14.8 ms, 0.20 so)
                    int stride = 1;
                    for (; seg + stride < n_segs && f.segs[seg + stride].word0 <= at; stride <<= 1) seg += stride;
                    while (stride > 1) {
                        stride >>= 1;
                        if (seg + stride < n_segs && f.segs[seg + stride].word0 <= at) seg += stride;
                    }
                    const SegDev &sg = f.segs[seg];
                    const uint64_t local = at - sg.word0;
                    const uint32_t per = sg.npairs * G;         // words per item (<= 64 * 32)
                    uint64_t jb;
                    uint32_t pi, g;
                    if (sg.npairs == 1 && local < (1ull << 32)) {   // one pair: item and group
                        jb = fastdiv((uint32_t)local, f.g_m, f.g_s);
                        g = (uint32_t)local - (uint32_t)jb * G;
                        pi = 0;
                    } else {
                        jb = local < (1ull << 32) ? (uint64_t)((uint32_t)local / per) : local / per;
                        const uint32_t rem = (uint32_t)(local - jb * per);
                        pi = rem / G;
                        g = rem - pi * G;
                    }
                    t0 = (uint32_t)(jb * per_item) + 32u * g;
                    pair = sg.pair0 + pi;
                }
                continue;
            }
            const int cnt = __popc(m);
            const unsigned dense = __ballot_sync(0xffffffffu, cnt >= kDenseBits);
            if (dense) {
                // dense words: a word's bits a lane each, words that surely fit first, then as many bits as fit
                unsigned left = dense;
                for (; left != 0 && n + 32 <= kBatch; left &= left - 1) {
                    const int l = __ffs(left) - 1;
                    const uint32_t bits = __shfl_sync(0xffffffffu, m, l), wt = __shfl_sync(0xffffffffu, t0, l),
                                   wp = __shfl_sync(0xffffffffu, pair, l);
                    if ((bits >> lane) & 1u) S.e[n + __popc(bits & lt_mask)] = make_uint2(wt + lane, wp);
                    n += __popc(bits);
                }
                if (((dense ^ left) >> lane) & 1u) m = 0;
                if (left != 0 && n < kBatch) {
                    const int l = __ffs(left) - 1;
                    const uint32_t bits = __shfl_sync(0xffffffffu, m, l), wt = __shfl_sync(0xffffffffu, t0, l),
                                   wp = __shfl_sync(0xffffffffu, pair, l);
                    const bool set = (bits >> lane) & 1u;
                    const int to = n + __popc(bits & lt_mask);
                    if (set && to < kBatch) S.e[to] = make_uint2(wt + lane, wp);
                    const unsigned rest = __ballot_sync(0xffffffffu, set && to >= kBatch);
                    if (lane == l) m = rest;
                    n = min(n + __popc(bits), kBatch);
                }
                continue;
            }
            // sparse words: every lane appends its first bits, as many as fit
            int incl = cnt;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int v = __shfl_up_sync(0xffffffffu, incl, o);
                if (lane >= o) incl += v;
            }
            const int total = __shfl_sync(0xffffffffu, incl, 31);
            int to = n + incl - cnt;
            while (m && to < kBatch) {
                const int bit = __ffs(m) - 1;
                m &= m - 1u;
                S.e[to++] = make_uint2(t0 + (uint32_t)bit, pair);
            }
            n = min(n + total, kBatch);
        }
        if (n == 0) break;
        __syncwarp();
        if (f.stats && lane == 0) stat_add(f, kStatFast, (unsigned long long)n);
        {
            Tri9 p[kExactK];
#pragma unroll
            for (int u = 0; u < kExactK; ++u) {
                const bool live = lane + 32 * u < n;
                exact_gather<COMP>(f, S.e[live ? lane + 32 * u : 0], live, p[u]);
            }
#pragma unroll
            for (int u = 0; u < kExactK; ++u) {
                float4 *t = reinterpret_cast<float4 *>(S.t[lane + 32 * u]);
                t[0] = make_float4(p[u].v[0], p[u].v[1], p[u].v[2], p[u].v[3]);
                t[1] = make_float4(p[u].v[4], p[u].v[5], p[u].v[6], p[u].v[7]);
                S.t[lane + 32 * u][2].x = __float_as_uint(p[u].v[8]);
            }
        }
#pragma unroll 1
        for (int u = 0; u < kExactK; ++u)           // (a lane reads and writes its own slots only)
            exact_setup<RAY>(f, S, lane + 32 * u, lane + 32 * u < n);
        __syncwarp();
        // a batch of heavy triangles (a near surface, up to 128 pixels each) would keep its warp long after
        // the others: of a batch of more than 2 kSegPx pixels, the triangles that start past pixel kSegPx go
        // to stage 2, which deals them out finely.  Exact kernel + stage 2, us, of a close 4K view of a 100 M-
        // triangle scan and of the full-HD view: none handed over 439 + 29, 110 + 11; kSegPx 2048 351 + 38,
        // 111 + 12; 1024 303 + 67, 108 + 12; 512 305 + 115, 94 + 17
        small_raster<kExactK>(f, S, lane, [&](bool want, int slot) -> bool {
            unsigned long long base = 0;
            const unsigned all = __ballot_sync(0xffffffffu, want);
            if (lane == 0) base = atomicAdd(&f.ctr->q1_count, (unsigned long long)__popc(all));
            const uint32_t px = __reduce_add_sync(0xffffffffu, want ? S.npx[slot] : 0u);
            if (lane == 0) atomicAdd(&f.ctr->q1_px, (unsigned long long)px);
            base = __shfl_sync(0xffffffffu, base, 0) + __popc(all & lt_mask);
            if (f.stats && lane == 0) stat_add(f, kStatS1, 0ull - (unsigned long long)__popc(all));   // now stage 2's
            if (!want) return false;
            if (base >= f.q1_cap) {
                atomicAdd(&f.ctr->overflow1, 1ull);
                return false;
            }
            const uint2 e = S.e[slot];
            f.q1[base] = Q1Entry{f.pairs[e.y].base + e.x, e.y, 1u};
            return true;
        });
        __syncwarp();
    }
}
