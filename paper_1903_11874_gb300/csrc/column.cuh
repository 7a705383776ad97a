// Column form of the circular cone beam (device code).
//
// Source and detector rows are such that every ray of one detector column u
// lies over the same line of the xy plane: the source's z is the same for all
// rays and a pixel's xy position does not depend on its row v. A ray is then
// (2D line of (view, u)) x (z slope of row v), and the chord of ray (u, v) in
// voxel (x, y, z) is the overlap of two parameter intervals: the one in which
// the line of u crosses the cell (x, y), and the one in which the slope of v
// lies between the planes z and z + 1. Both come from products:
//   plane x = i:  ((i - nx/2) - X) * (1/dx),  X = x offset of the line at tau = 0
//   row j of height slope j ds:  z - zs = j ds (tau + tc)
// tau is the ray parameter (0 at the source, 1 at the detector) less tc = the
// rotation axis's, so that FP32 carries distances from the middle of the volume
// (<= ~180 voxels of a 256^3 volume) and not from the source (~1000).
#pragma once

#include "siddon_device.cuh"

namespace bsgd {

// Inverse slope of a line parallel to the planes: so that a plane
// below gives a huge negative and one above a huge positive time.
constexpr float kFlat = 1e30f;
// floor by an addition rounded down: 1.5 * 2^23 + f keeps the integer part in
// its low mantissa bits for |f| < 2^22
constexpr float kMagic = 12582912.f;
constexpr int kMagicBits = 0x4B400000;
// chord interval of the line R with the cell whose low corner is (x, y), both
// relative to the volume's centre
__device__ __forceinline__ void cell_interval(const ColRay &R, float x, float y, float &t0, float &t1) {
    const float xa = ((x - R.xh) - R.xl) * R.ix, xb = ((x + 1.f - R.xh) - R.xl) * R.ix;
    const float ya = ((y - R.yh) - R.yl) * R.iy, yb = ((y + 1.f - R.yh) - R.yl) * R.iy;
    t0 = fmaxf(fminf(xa, xb), fminf(ya, yb));
    t1 = fminf(fmaxf(xa, xb), fmaxf(ya, yb));
}

__device__ __forceinline__ ColRay load_ray(const ColRay *p) {
    const float4 *q = reinterpret_cast<const float4 *>(p);
    const float4 a = __ldg(q), b = __ldg(q + 1);
    return ColRay{a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w};
}

// Squared length of a line's xy part (mm), and the factor of a row's weight: the
// ray's length over the rise of the row (the level row: of row 1).
__device__ __forceinline__ float column_length2(const DeviceGeom &G, const ColRay &C) {
    const float lx = C.dx * G.hx, ly = C.dy * G.hy;
    return fmaf(lx, lx, ly * ly);
}
__device__ __forceinline__ float column_weight(const DeviceGeom &G, float len2, int v) {
    const float j = (float)v - 0.5f * (float)(G.nv - 1);
    const float lz = j * G.vstep * G.hz;
    return sqrtf(fmaf(lz, lz, len2)) / (G.vstep * (j != 0.f ? fabsf(j) : 1.f));
}

// Detector columns whose lines may cross the unit cell centred at (px, py)
// (voxel units from the volume's low corner): the shadow of the centre, widened
// by a bound on the shadow of the half diagonal and by G.umargin, which holds the
// rounding of the lines and of the shadow. cell_interval decides.
// t: ray parameter at the centre (divergent beams).
template <bool kParallel = false>
__device__ __forceinline__ int2 cell_columns(const DeviceGeom &G, int a, float px, float py, float *t = nullptr) {
    const float4 *p = reinterpret_cast<const float4 *>(G.rays + a);
    const float4 A = __ldg(p), B = __ldg(p + 1), C = __ldg(p + 2);   // p0 | pu c0 | cu
    const float rx = px - A.x, ry = py - A.y;
    const float ax = B.z - A.x, ay = B.w - A.y, cx = C.y, cy = C.z;
    const float hn = 0.5f * (fabsf(ax) + fabsf(ay));
    const float N = fmaf(rx, ay, -ry * ax);
    float fu, w;
    if (kParallel) {   // every line along (ax, ay), (cx, cy) apart
        const float D = fmaf(cx, ay, -cy * ax);
        fu = __fdividef(N, D);
        w = __fdividef(hn, fabsf(D)) + G.umargin;
    } else {
        const float D = fmaf(rx, cy, -ry * cx);
        if (t) *t = __fdividef(D, fmaf(ax, cy, -ay * cx));
        const float hd = 0.5f * (fabsf(cx) + fabsf(cy));
        const float room = fabsf(D) - hd;
        if (!(room > 0.f)) return make_int2(0, G.nu - 1);
        fu = __fdividef(-N, D);
        w = __fdividef(fmaf(fabsf(fu), hd, hn), room) + G.umargin;
    }
    const float uc = fu + 0.5f * (float)(G.nu - 1);
    const float lo = fminf(fmaxf(ceilf(uc - w), 0.f), (float)G.nu);
    const float hi = fmaxf(fminf(floorf(uc + w), (float)(G.nu - 1)), -1.f);
    return make_int2((int)lo, (int)hi);
}

// ---------------------------------------------------------------------------
// Back projection as a gather. A warp owns a column (one (x, y); a voxel per
// lane, 32 planes at a time). Its lanes first find candidates, lanes over views:
// the detector columns u whose shadow the cell is in. Of 32 candidates at a
// time, lanes over candidates, they work out the crossing (the interval [t0, t1]
// of u's line in the cell); then every lane runs down the list of crossings and
// adds weight x overlap over the detector rows that can meet its voxel inside
// the interval, two rows at a time. No atomics, no clearing of the target, no
// barrier, and the same sum in every run.
//
// 45 views into 256^3 voxels (1.06 G updates): 2.16 ms as the scatter of the
// incremental walk (an L2 sector operation for half of its updates), 1.03 ms
// gathered; into one 32-plane slab (172 M updates) 0.437 and 0.198 ms. What
// bounds it: issue slots and L1. A crossing of one chunk takes 25 instructions
// for the 45 or so updates of its 32 lanes (161 M warp instructions for the
// slab, a third of them for finding the crossings; issue active 67 %, L1 76 % of
// peak, 7.7 sectors per load of weights). Weights carry 1 / (j ds) so that no
// table of inverse slopes is read per row (2.07 ms with one: its loads and 16
// more instructions); a list per column for all chunks instead of one per chunk:
// 1.55 ms; rows padded so that no window needs clamping: 1.17; lists filled to 32
// across views, one pair of rows per pass over the list: 1.03. 64 registers and
// 4 CTAs of 8 warps per SM; 5 CTAs (48 registers) 1.04, 6 (spills) 1.12. 4 x 2
// columns per CTA share weight rows in L1 in either direction of the rays (80 %
// of sectors hit; 8 x 1: 71 %).
//
// Row j (counted from the source's height) is at height j t ds (ds: slope per
// row), so its overlap with the voxel [kin, kout] (heights from the source's,
// |.| growing along the ray) is, for a rise of less than a voxel per interval,
//   ov = min(j dt ds, j t1 ds - kin, kout - j t0 ds),   chord = ov / (j ds).
// The first term carries the whole interval without cancellation; 1 / (j ds)
// is part of the stored weight (row 0, which never rises, is added apart).
constexpr int kGatherWarps = 8, kGatherRows = 2;   // warps of a CTA, and the rows of y they take
constexpr int kGatherAcross = kGatherWarps / kGatherRows;
constexpr int kGatherChunks = 8;   // chunks of 32 planes that a warp takes with one list

// A warp's shared memory: crossings of a chunk, candidates, sums per chunk.
struct GatherWarp {
    float4 work[32];
    uint2 cand[64];
    int half[64];
    float sums[kGatherChunks][32];
};

// The crossing of line `ray` with the cell: {row of weights, t0 ds, (t1 - t0) ds,
// -}; false if the line misses the cell.
__device__ __forceinline__ bool crossing(const DeviceGeom &G, uint2 ray, float x, float y, float4 &out) {
    const ColRay R = load_ray(G.cray + ray.x);
    float t0, t1;
    cell_interval(R, x, y, t0, t1);
    out.x = __uint_as_float(ray.y * (uint32_t)G.nvp);
    out.y = (t0 + G.tc) * G.vstep;
    out.z = (t1 - t0) * G.vstep;
    return t1 > t0;
}

// A lane's voxel: heights of its faces from the source's, and its side.
struct GatherVoxel {
    float klo, kin, kout, sign, vs;   // vs = -sign * centre row
    float vlow;                       // rows of the window's low end = klo * rows per voxel + vlow
    bool astride, centre;
    // slack: rows by which the window's low end may lie lower than at the end of
    // the interval that the crossing gives (planes below the source's height, in
    // a chunk that has both)
    __device__ __forceinline__ GatherVoxel(const DeviceGeom &G, int z, float slack) {
        const float vc = 0.5f * (float)(G.nv - 1);
        klo = (float)z - G.zs;
        const float khi = klo + 1.f;
        const bool lower = khi <= 0.f;
        astride = klo < 0.f && khi > 0.f;
        centre = klo <= 0.f && khi > 0.f && vc == floorf(vc);
        sign = lower ? -1.f : 1.f;
        kin = lower ? -khi : fmaxf(klo, 0.f);
        kout = lower ? -klo : khi;
        vs = -sign * vc;
        vlow = vc - 1e-2f - (klo < 0.f ? slack : 0.f);
    }
};

// Adds two rows of one crossing to a voxel: A = {row 0 of the weights less the
// magic bits, t0 ds, dt ds, rows per voxel of height at the window's low end},
// `skip` rows above the window's first. The rows of weights are padded by what a
// chunk of planes can reach past the detector's edges.
// kMiddle: the chunk holds a voxel that needs the middle's form. kNear: it lies on
// both sides of the source's height, too, and takes no slack (gather_column): below
// that height, a window's low end is where the ray enters the cell, and A.w is of
// where it leaves it, so that its rows per voxel are worked out again.
template <bool kMiddle, bool kNear = false>
__device__ __forceinline__ void gather_pair(const GatherVoxel &V, float skip, const float4 &A,
                                            const float *__restrict__ w, float &acc) {
    const float t1 = A.y + A.z;
    // first row above the window's low end: floor + 1
    const float c = kNear && V.klo < 0.f ? __fdividef(1.f, A.y) : A.w;
    const float S = __fadd_rd(fmaf(V.klo, c, V.vlow), kMagic + 1.f + skip);
    const float *__restrict__ row = w + (__float_as_uint(A.x) + __float_as_uint(S));
    const float w0 = __ldg(row), w1 = __ldg(row + 1);
    float j0 = fmaf(V.sign, S - kMagic, V.vs), j1 = j0 + V.sign, k0 = V.kout, k1 = V.kout;
    if (kMiddle && V.astride) {   // rows leave through either face
        k0 = j0 < 0.f ? -V.klo : V.kout;
        k1 = j1 < 0.f ? -V.klo : V.kout;
        j0 = fabsf(j0);
        j1 = fabsf(j1);
    }
    const float o0 = fminf(fminf(j0 * A.z, fmaf(j0, t1, -V.kin)), fmaf(-j0, A.y, k0));
    const float o1 = fminf(fminf(j1 * A.z, fmaf(j1, t1, -V.kin)), fmaf(-j1, A.y, k1));
    if (o0 > 0.f) acc = fmaf(o0, w0, acc);
    if (o1 > 0.f) acc = fmaf(o1, w1, acc);
}

// Whether a chunk holds a voxel that needs the middle's form: the source's height
// lies inside it, or a level row of rays in its lower face.
__device__ __forceinline__ bool gather_middle(const DeviceGeom &G, float ka, float kb) {
    return kb > 0.f && ka <= 0.f && ((G.nv & 1) || G.zs != floorf(G.zs));
}

// Rows that a chunk of planes with faces ka, kb (heights) can meet in a
// crossing: false if they are all off the detector. c: rows per voxel of height
// where the window's low end lies (a chunk on both sides of the source's height:
// of its upper planes); extra: pairs of rows after the first.
// half: 1 / 2 for the rows below / from nv / 2 only (a drawn detector cell).
__device__ __forceinline__ bool gather_window(const DeviceGeom &G, const float4 &A, float ka, float kb,
                                              float slack, int half, float &c, int &extra) {
    const float c_in = __fdividef(1.f, A.y), c_out = __fdividef(1.f, A.y + A.z);
    c = kb > 0.f ? c_out : c_in;
    // an open interval of this width holds floor + 1 rows at most
    const float kmax = fmaxf(1.f, fmaxf(fabsf(ka), fabsf(kb)));
    const float width = fmaf(kmax, c_in - c_out, c_out) + 0.03f + slack;
    extra = (int)fminf(width, 1e6f) >> 1;
    const float vc = 0.5f * (float)(G.nv - 1);
    const float top = vc + kb * (kb > 0.f ? c_in : c_out), bottom = vc + ka * (ka < 0.f ? c_in : c_out);
    const float first = half == 2 ? (float)(G.nv >> 1) : 0.f;
    const float last = (float)((half == 1 ? (G.nv >> 1) : G.nv) - 1);
    return top > first - 0.02f && bottom < last + 0.02f;
}

// Column (x, y) over `n_slots` views, planes [z0, z1) (at most kGatherChunks
// chunks of 32). The sum of plane z0 + 32 q + lane is left at sums[q][lane].
// view(slot, cell): the view (-1: none); sets its slot among the weights and its
// drawn detector cell (-1: all).
// A chunk on both sides of the source's height has its windows widened by G.vslack, a
// bound for the cell nearest to the source, which costs a pair of rows per two rows of
// it, everywhere. kNear, taken above a row: planes below that height find their windows
// by themselves. 128^2 x 32 from 60 views with the source 20 voxels from the volume (17
// rows) 133 us against 413, x 48 with 60 voxels (2.4 rows) 167 against 184; where the
// bound is small the reciprocal costs 2 to 4 %, and a choice inside the loop 30 %.
template <bool kNear, class View>
__device__ __forceinline__ void gather_column(const DeviceGeom &G, int n_slots, View &&view,
                                              const float *__restrict__ w, int x, int y, int z0, int z1,
                                              int n_cells, GatherWarp &M) {
    const int lane = threadIdx.x & 31, chunks = (z1 - z0 + 31) >> 5;
    const unsigned below = (1u << lane) - 1u;
    const float fx = (float)x - 0.5f * (float)G.nx, fy = (float)y - 0.5f * (float)G.ny;
    const float ka = (float)z0 - G.zs, kb = (float)z1 - G.zs, vc = 0.5f * (float)(G.nv - 1);
    for (int q = 0; q < chunks; ++q) M.sums[q][lane] = 0.f;

    // the first m <= 32 candidates
    auto process = [&](int m) {
        __syncwarp();
        float4 E = make_float4(0.f, 1.f, 0.f, 0.f);
        const int half = lane < m ? M.half[lane] : 0;
        const bool have = lane < m && crossing(G, M.cand[lane], fx, fy, E);
        for (int q = 0; q < chunks; ++q) {
            const int zb = z0 + 32 * q, planes = min(32, z1 - zb);
            const float ka = (float)zb - G.zs, kb = ka + (float)planes;
            const bool both = ka < 0.f && kb > 0.f;
            const float slack = !kNear && both ? G.vslack : 0.f;
            int extra = 0;
            bool hit = have && gather_window(G, E, ka, kb, slack, half, E.w, extra);
            unsigned m = __ballot_sync(0xffffffffu, hit);
            if (!m) continue;
            const bool middle = gather_middle(G, ka, kb) || (kNear && both);
            const GatherVoxel V(G, zb + min(lane, planes - 1), slack);
            float acc = M.sums[q][lane];
            for (float skip = 0.f; m; skip += 2.f) {
                if (hit)
                    M.work[__popc(m & below)] = make_float4(
                        __uint_as_float(__float_as_uint(E.x) - (uint32_t)(kMagicBits - G.vpad)), E.y, E.z, E.w);
                __syncwarp();
                const int n = __popc(m);
                if (middle) {
                    for (int e = 0; e < n; ++e) {
                        const float4 A = M.work[e];
                        gather_pair<true, kNear>(V, skip, A, w, acc);
                        if (V.centre && skip == 0.f)   // the level row, stored as row 1 of its side
                            acc = fmaf(A.z, __ldg(w + (__float_as_uint(A.x) + (uint32_t)(kMagicBits + (G.nv >> 1)))), acc);
                    }
                } else {
#pragma unroll 4
                    for (int e = 0; e < n; ++e) gather_pair<false>(V, skip, M.work[e], w, acc);
                }
                __syncwarp();
                hit = hit && --extra >= 0;   // rows closer than half a voxel: the next pair
                m = __ballot_sync(0xffffffffu, hit);
            }
            M.sums[q][lane] = acc;
        }
    };

    int n = 0;
    for (int b = 0; b < n_slots; b += 32) {
        int cell = -1, slot = b + lane, kd = 0;
        const int a = slot < n_slots ? view(slot, cell) : -1;
        int2 ur = make_int2(0, -1);
        if (a >= 0) {
            float t;
            ur = cell_columns(G, a, (float)x + 0.5f, (float)y + 0.5f, &t);
            // nothing to do where all planes lie past the detector's rows (by the
            // rows at the cell's centre and a bound on their change across it)
            const float c = __fdividef(1.f, t * G.vstep), more = G.vslack * (1.f / 32.f);
            const float top = fmaf(kb, c, fmaf(fabsf(kb), more, vc)), bottom = fmaf(ka, c, fmaf(-fabsf(ka), more, vc));
            if (top < -0.5f || bottom > (float)G.nv - 0.5f) ur.y = -1;
        }
        if (cell >= 0) {
            if (cell & 1) ur.x = max(ur.x, G.nu / 2);
            else ur.y = min(ur.y, G.nu / 2 - 1);
            if (n_cells == 4) kd = (cell >> 1) ? 2 : 1;
        }
        for (;;) {
            const bool has = ur.x <= ur.y;
            const unsigned m = __ballot_sync(0xffffffffu, has);
            if (!m) break;
            if (has) {
                const int k = n + __popc(m & below);
                M.cand[k] = make_uint2((uint32_t)a * (uint32_t)G.nu + ur.x, (uint32_t)slot * (uint32_t)G.nu + ur.x);
                M.half[k] = kd;
                ++ur.x;
            }
            n += __popc(m);
            if (n < 32) continue;
            process(32);
            n -= 32;
            if (lane < n) {   // the rest moves up
                M.cand[lane] = M.cand[32 + lane];
                M.half[lane] = M.half[32 + lane];
            }
            __syncwarp();
        }
    }
    if (n) process(n);
    __syncwarp();
}

}  // namespace bsgd
