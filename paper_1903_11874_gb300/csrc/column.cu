// Column form of the circular cone beam: its tables and the back projection
// that gathers (column.cuh).
#include <algorithm>
#include <cmath>

#include "column.cuh"

namespace bsgd {

namespace {

// Lines of every (view, detector column), from the FP32 ray table (the same rays
// as the incremental walk's), in FP64.
__global__ void column_tables_kernel(const DeviceGeom G, ColRay *__restrict__ cray, float2 *__restrict__ slice) {
    const int64_t n = (int64_t)G.n_views * G.nu;
    for (int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; k < n;
         k += (int64_t)gridDim.x * blockDim.x) {
        const ViewRay &R = G.rays[k / G.nu];
        const float fu = (float)(int)(k % G.nu) - 0.5f * (float)(G.nu - 1);
        const float x0 = fmaf(fu, R.pu[0], R.p0[0]), y0 = fmaf(fu, R.pu[1], R.p0[1]);
        const float dx = fmaf(fu, R.cu[0], R.c0[0]) - x0, dy = fmaf(fu, R.cu[1], R.c0[1]) - y0;
        const double X = (double)x0 + (double)G.tc * dx - 0.5 * G.nx;
        const double Y = (double)y0 + (double)G.tc * dy - 0.5 * G.ny;
        ColRay c;
        c.xh = (float)X;
        c.yh = (float)Y;
        c.xl = (float)(X - c.xh);
        c.yl = (float)(Y - c.yh);
        c.dx = dx;
        c.dy = dy;
        c.ix = dx != 0.f ? (float)(1.0 / dx) : kFlat;
        c.iy = dy != 0.f ? (float)(1.0 / dy) : kFlat;
        // a line lying in a face belongs to the cell on its + side
        if (dx == 0.f) c.xl += 1e-9f;
        if (dy == 0.f) c.yl += 1e-9f;
        if (cray) cray[k] = c;
        if (slice) {
            slice[k] = make_float2(c.xh, c.xl);
            slice[n + k] = make_float2(c.yh, c.yl);
            slice[2 * n + k] = make_float2(c.ix, c.iy);
            reinterpret_cast<float *>(slice + 3 * n)[k] = sqrtf(column_length2(G, c));
        }
    }
}

// View slots of a plain back projection: of its row blocks in turn, or, where they
// are all of the geometry's, the views in order, whose lines lie side by side (the
// top slab of 256^3 from 360 views in 8 interleaved blocks 988 us block by block,
// 855 in order).
__host__ __device__ __forceinline__ int gather_slots(const DeviceGeom &G, const RowSel &R) {
    return R.n == G.M ? G.n_views : R.n * G.max_views;
}
__device__ __forceinline__ int gather_view(const DeviceGeom &G, const RowSel &R, int slot) {
    return R.n == G.M ? slot : sel_view(G, R, slot);
}

// w[slot][u][vpad + v] = scale * r[a][v][u] * |d| / (|j| ds): the ray's length
// and the rise of its row j = v - (nv - 1) / 2 (the level row: j = 1), through a
// 32 x 33 shared tile so that both sides are coalesced. Rows of nvp elements.
template <typename T>
__global__ void __launch_bounds__(256) column_weights_kernel(const DeviceGeom G, const RowSel R, int j0, int j1,
                                                             const T *__restrict__ r, float scale,
                                                             float *__restrict__ w) {
    __shared__ float s[32][33];
    const int a = gather_view(G, R, blockIdx.y);
    if (a < 0) return;
    const int lane = threadIdx.x & 31, row = threadIdx.x >> 5;
    const int tu = (G.nu + 31) / 32;
    const int u0 = (blockIdx.x % tu) * 32, v0 = (int)(blockIdx.x / tu) * 32 - G.vpad;
    // rays outside the slab's band meet none of its voxels: their weights are not
    // read as data; the padding, whose rows could, is always written
    const Band b = band_of(G, a, j0, j1);
    if (v0 >= 0 && v0 + 32 <= G.nv && (u0 > b.u1 || u0 + 31 < b.u0 || v0 > b.v1 || v0 + 31 < b.v0)) return;
    const ColRay C = load_ray(G.cray + (size_t)a * G.nu + min(u0 + lane, G.nu - 1));
    const float len = column_length2(G, C);
#pragma unroll
    for (int k = row; k < 32; k += 8) {
        const int v = v0 + k, u = u0 + lane;
        float val = 0.f;
        if (v >= 0 && v < G.nv && u < G.nu)
            val = ldf(r + ((int64_t)a * G.nv + v) * G.nu + u) * scale * column_weight(G, len, v);
        s[k][lane] = val;
    }
    __syncthreads();
#pragma unroll
    for (int k = row; k < 32; k += 8) {
        const int u = u0 + k, v = v0 + lane;
        if (u < G.nu && v + G.vpad < G.nvp) w[((size_t)blockIdx.y * G.nu + u) * G.nvp + v + G.vpad] = s[lane][k];
    }
}

// The columns of a CTA: kGatherAcross along x, kGatherRows along y, one per warp.
// out(index, value) for every voxel of planes [z0, z1), along x.
template <bool kNear, class View, class Out>
__device__ __forceinline__ void gather_cta(const DeviceGeom &G, int n_slots, View &&view, const float *__restrict__ w,
                                           int z0, int z1, int n_cells, Out &&out) {
    __shared__ GatherWarp warps[kGatherWarps];
    const int tiles = (G.nx + kGatherAcross - 1) / kGatherAcross;
    const int x0 = blockIdx.x % tiles * kGatherAcross, y0 = blockIdx.x / tiles * kGatherRows;
    const int warp = threadIdx.x >> 5, x = x0 + warp % kGatherAcross, y = y0 + warp / kGatherAcross;
    if (x < G.nx && y < G.ny) gather_column<kNear>(G, n_slots, view, w, x, y, z0, z1, n_cells, warps[warp]);
    __syncthreads();
    for (int k = threadIdx.x; k < (z1 - z0) * kGatherWarps; k += blockDim.x) {
        const int c = k % kGatherWarps, z = k / kGatherWarps, xx = x0 + c % kGatherAcross, yy = y0 + c / kGatherAcross;
        if (xx < G.nx && yy < G.ny)
            out(((int64_t)(z0 + z) * G.ny + yy) * G.nx + xx, warps[c].sums[z >> 5][z & 31]);
    }
}

// x = (or +=) the plain back projection of planes [z0, z1), kGatherChunks chunks
// of 32 per CTA (grid y).
template <bool kNear>
__global__ void __launch_bounds__(32 * kGatherWarps, 4)
    bp_gather_kernel(const DeviceGeom G, const RowSel R, int z0, int z1, const float *__restrict__ w,
                     float *__restrict__ x, int add) {
    auto view = [&](int &slot, int &) { return gather_view(G, R, slot); };
    const int zb = z0 + (int)blockIdx.y * 32 * kGatherChunks;
    gather_cta<kNear>(G, gather_slots(G, R), view, w, zb, min(z1, zb + 32 * kGatherChunks), 1,
               [&](int64_t k, float v) { x[k] = add ? x[k] + v : v; });
}

// g_J += (A_R^J)^T w over the drawn pairs of column block J (blockIdx.z of the
// iteration's blocks).
template <bool kNear>
__global__ void __launch_bounds__(32 * kGatherWarps, 4) solve_gather_kernel(const DeviceGeom G, const SolveDev S) {
    __shared__ int s_pairs[kMaxPairs];
    const Work &W = *S.work;
    if ((int)blockIdx.z >= W.n_cols) return;
    const int j = W.cols[blockIdx.z];
    if (S.owned && !S.owned[j]) return;   // another process owns block j
    const int z1 = G.plane_start[j + 1], zb = G.plane_start[j] + (int)blockIdx.y * 32 * kGatherChunks;
    if (zb >= z1) return;
    int np = 0;   // pairs of this block (the same in every thread)
    for (int p = 0; p < W.n_pairs; ++p)
        if (W.pair_j[p] == j) {
            if (threadIdx.x == 0) s_pairs[np] = p;
            ++np;
        }
    __syncthreads();
    auto view = [&](int &slot, int &cell) {   // slot: of the pairs' views, then of the weights
        const int k = np > 1 ? slot / G.max_views : 0, s = slot - k * G.max_views, p = s_pairs[k];
        slot = p * G.max_views + s;
        if (S.n_cells > 1) cell = S.cells[slot];
        return G.block_views[W.pair_i[p] * G.max_views + s];
    };
    gather_cta<kNear>(G, np * G.max_views, view, S.w, zb, min(z1, zb + 32 * kGatherChunks), S.n_cells,
               [&](int64_t k, float v) { S.g[k] += v; });
}

// The weights of pair blockIdx.z at view slot blockIdx.y, over a 32 x 32 tile of
// its band: r - r~^j for the rays that take part (r~^j = r), 0 for the others.
template <typename T>
__global__ void __launch_bounds__(256) column_change_kernel(const DeviceGeom G, const SolveDev S) {
    __shared__ float s[32][33];
    const Work &W = *S.work;
    const int p = blockIdx.z, slot = blockIdx.y;
    if (p >= W.n_pairs) return;
    const int i = W.pair_i[p], j = W.pair_j[p];
    if (S.owned && !S.owned[j]) return;   // another process owns block j
    if (slot >= G.block_nviews[i]) return;
    const int a = G.block_views[i * G.max_views + slot];
    const Band b = G.bands[(size_t)a * (G.N + 1) + j];
    if (b.u0 > b.u1 || b.v0 > b.v1) return;
    const int tu = (b.u1 - b.u0 + 32) / 32;
    const int u0 = b.u0 + (int)(blockIdx.x % tu) * 32, v0 = b.v0 + (int)(blockIdx.x / tu) * 32;
    if (v0 > b.v1) return;
    Band c = b;   // the rays of the drawn cell
    if (S.n_cells > 1) cell_rect(G.nu, G.nv, S.n_cells, S.cells[p * G.max_views + slot], c);
    const T *r = reinterpret_cast<const T *>(S.r);
    T *rt = reinterpret_cast<T *>(S.rt);
    const int lane = threadIdx.x & 31, row = threadIdx.x >> 5;
    const ColRay C = load_ray(G.cray + (size_t)a * G.nu + min(u0 + lane, G.nu - 1));
    const float len = column_length2(G, C);
#pragma unroll
    for (int k = row; k < 32; k += 8) {
        const int u = u0 + lane, v = v0 + k;
        float dw = 0.f;
        if (u >= c.u0 && u <= c.u1 && v >= c.v0 && v <= c.v1) {
            bool in;
            const int64_t kt = zslot(G, j, a, u, v, in);
            const float rv = ldv(r + ((int64_t)a * G.nv + v) * G.nu + u);
            dw = (rv - ldv(rt + kt)) * column_weight(G, len, v);
            stf(rt + kt, rv);
        }
        s[k][lane] = dw;
    }
    __syncthreads();
#pragma unroll
    for (int k = row; k < 32; k += 8) {
        const int u = u0 + k, v = v0 + lane;
        if (u <= b.u1 && v <= b.v1)
            S.w[(((int64_t)p * G.max_views + slot) * G.nu + u) * G.nvp + G.vpad + v] = s[lane][k];
    }
}

// Adds view a of a 2D kind to pixel (xx, y), whose low corner is (fx, fy) from
// the image's centre.
template <bool kParallel, typename T>
__device__ __forceinline__ void slice_view(const DeviceGeom &G, int a, int xx, int y, float fx, float fy,
                                           const T *__restrict__ r, float scale, float &acc) {
    const int2 ur = cell_columns<kParallel>(G, a, (float)xx + 0.5f, (float)y + 0.5f);
    for (int u = ur.x; u <= ur.y; ++u) {
        const int i = a * G.nu + u;
        const float2 X = __ldg(G.sx + i), Y = __ldg(G.sy + i), I = __ldg(G.si + i);
        const float wl = ldf(r + i) * scale * __ldg(G.slen + i);
        float t0, t1;
        cell_interval(ColRay{X.x, X.y, I.x, 0.f, Y.x, Y.y, I.y, 0.f}, fx, fy, t0, t1);
        if (t1 > t0) acc = fmaf(t1 - t0, wl, acc);
    }
}

// Back projection of a 2D kind into rows [y0, y1) of the image, as a gather: a
// CTA takes 32 pixels of a row, its 8 warps every 8th view each, whichever row
// block it is of; a thread tests the detector columns whose shadow its pixel is
// in (one to three) and adds weight x chord. 256^2 pixels from 360 fan views of 384
// bins (30 M updates): 193 us as a scatter, whose atomics meet on 65536 addresses,
// 127 us gathered (168 us with the lines as 32-byte records: a warp's load then
// spans ten 128-byte lines). What bounds it: issue slots, half of them for finding
// the columns, and lanes that wait for the ones with three columns.
// kViews: all of the geometry's in order; the listed blocks', listed on chip 256 at a
// time; or block by block, read in place, where a block's views fill the warps (blocks
// of 64 views or more: 512^2 from three of 90, 351 us, listed 359). Small blocks leave
// warps idle: 64^2 from 90 blocks of one view 94 us block by block, 11 in order, 23
// scattered; 512^2 from 80 blocks of 9 views 1171, 894, 977; 15 of 360 blocks of one
// view into 256^2 31, listed 18, scattered 35. 32 registers, so that 8 CTAs are
// resident (36: 4 % slower, 1024^2 from one view 39 us for 29); the blocks' form has
// them by itself, and loses 2 % where it is told to.
enum SliceViews { kSliceAll, kSliceListed, kSliceBlocks };

template <bool kParallel, SliceViews kViews, typename T>
__device__ __forceinline__ void slice_body(const DeviceGeom &G, const RowSel &R, int y0, const T *__restrict__ r,
                                           float scale, float *__restrict__ x, int add) {
    __shared__ float s[8][32];
    const int tiles = (G.nx + 31) / 32, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int xx = (int)(blockIdx.x % tiles) * 32 + lane, y = y0 + (int)(blockIdx.x / tiles);
    const float fx = (float)xx - 0.5f * (float)G.nx, fy = (float)y - 0.5f * (float)G.ny;
    float acc = 0.f;
    if (kViews == kSliceListed) {
        __shared__ int s_views[256];
        const int slots = R.n * G.max_views;
        for (int b = 0; b < slots; b += 256) {
            if (b) __syncthreads();
            s_views[threadIdx.x] = sel_view(G, R, b + threadIdx.x);
            __syncthreads();
            for (int q = warp; q < min(256, slots - b); q += 8)
                if (s_views[q] >= 0)   // (a block with fewer views than the largest)
                    slice_view<kParallel>(G, s_views[q], xx, y, fx, fy, r, scale, acc);
        }
    } else if (kViews == kSliceAll) {
        for (int a = warp; a < G.n_views; a += 8) slice_view<kParallel>(G, a, xx, y, fx, fy, r, scale, acc);
    } else {
        for (int k = 0; k < R.n; ++k) {
            const int *views = G.block_views + R.ids[k] * G.max_views;
            const int n = G.block_nviews[R.ids[k]];
            for (int q = warp; q < n; q += 8) slice_view<kParallel>(G, views[q], xx, y, fx, fy, r, scale, acc);
        }
    }
    s[warp][lane] = acc;
    __syncthreads();
    if (warp > 0 || xx >= G.nx) return;
#pragma unroll
    for (int q = 1; q < 8; ++q) acc += s[q][lane];
    float *p = x + (int64_t)y * G.nx + xx;
    *p = add ? *p + acc : acc;
}

template <bool kParallel, SliceViews kViews, typename T>
__global__ void __launch_bounds__(256, 8) bp_slice_kernel(const DeviceGeom G, const RowSel R, int y0,
                                                          const T *__restrict__ r, float scale,
                                                          float *__restrict__ x, int add) {
    slice_body<kParallel, kViews>(G, R, y0, r, scale, x, add);
}

template <bool kParallel, typename T>
__global__ void __launch_bounds__(256) bp_slice_blocks_kernel(const DeviceGeom G, const RowSel R, int y0,
                                                              const T *__restrict__ r, float scale,
                                                              float *__restrict__ x, int add) {
    slice_body<kParallel, kSliceBlocks>(G, R, y0, r, scale, x, add);
}

}  // namespace

// Lanes that the gather spends per ray that meets a voxel of its column: chunks
// of 32 planes that `planes` do not fill, and rows further apart than a voxel,
// cost as much as full ones, while the scatter follows the rays there are.
static double gather_waste(const bsgd_geometry *g, int planes) {
    const bsgd_geometry_desc &d = g->desc;
    return (planes + 31) / 32 * 32.0 / planes * (d.dv * d.dso / d.dsd / d.dz);
}

// Planes of [z0, z1) that a view's detector covers, on the mean over the depth of
// the volume along the view.
static double covered_planes(const bsgd_geometry *g, int z0, int z1) {
    const bsgd_geometry_desc &d = g->desc;
    const double depth = 0.5 * (d.nx * d.dx + d.ny * d.dy), mid = 0.5 * d.nz;
    double sum = 0.0;
    for (int k = 0; k < 8; ++k) {
        const double s = ((k + 0.5) / 8.0 - 0.5) * depth;
        const double reach = 0.5 * d.nv * d.dv * (d.dso - s) / d.dsd / d.dz;   // planes from the middle
        sum += std::max(0.0, std::min(z1 - mid, reach) - std::max(z0 - mid, -reach));
    }
    return sum / 8.0;
}

// Whether the back projection of `views` views into planes [z0, z1) gathers. A
// warp runs through all views of its column (0.43 us each, whatever the other
// warps do), so small slabs seen from many views scatter instead: 64 x 64 x 32
// from 360 views 151 us scattered, 164 gathered; 64^3 from 90 views 114 and 66
// us; 48 x 48 x 32 from 24 views 35 and 23 us; 32^3 from 90 views 35 and 39 us.
// Full chunks gather 2.1 times as fast as they scatter at a waste of 0.8, 1.2
// times at 1.4.
// The padding of the weights measures a source that all but touches the volume
// (rows per voxel that change across a cell by many rows, times the planes), where
// a lane runs through the rows of the chunk's outermost plane; us scattered /
// gathered with the padding per voxel of a view's weights in brackets: 128^3 from
// 60 views, source 5.5 voxels away [0.29] 731 / 462, 3.5 [0.62] 726 / 630, 2.5 [1.1]
// 756 / 818; 256^3 from 45, 4 voxels [0.40] 3771 / 3285, 3 [0.69] 3799 / 4298; a
// 32-plane slab of it, 9 voxels [0.77] 769 / 585, 5 [2.1] 804 / 1243.
// A list costs a warp the same however few planes its rays then reach: 256^2 from 45
// views, rows 0.5 / 0.8 voxel apart, 12 planes 248 / 307 and 184 / 193, 16 planes 313
// / 309 and 218 / 195, 20 planes 376 / 312 and 265 / 196; slabs at the end of a
// volume that the detector covers in part (covered planes in brackets): 512^2 x 32
// from 45 views [5.1] 303 / 334, [7.8] 405 / 376, 128^2 x 32 from 360 [8.1] 398 / 441,
// [9.6] 451 / 446, 256^2 x 32 from 360 [3.0] 417 / 641, [10.1] 989 / 877.
bool column_bp_pays(const bsgd_geometry *g, int z0, int z1, int views) {
    const int planes = z1 - z0;
    const int64_t plane = (int64_t)g->desc.nx * g->desc.ny, voxels = plane * planes;
    if (g->dg.nvp == 0 || planes < 16 || voxels < (views <= 32 ? 64000 : 160000)) return false;
    const double pad = (double)g->desc.nu * 2.0 * g->dg.vpad;
    return pad <= 0.64 * (double)(plane * g->desc.nz) && pad <= 1.2 * (double)voxels && gather_waste(g, planes) <= 1.7 &&
           covered_planes(g, z0, z1) >= 9.0;
}

// Lines of a 2D kind (arrays, DeviceGeom::sx) or of a cone (records).
bsgd_status column_tables(bsgd_geometry *g, void *tables) {
    DeviceGeom &dg = g->dg;
    const int64_t n = (int64_t)g->desc.n_views * g->desc.nu;
    const bool slice = g->desc.kind != BSGD_CONE3D;
    ColRay *cray = slice ? nullptr : (ColRay *)tables;
    float2 *lines = slice ? (float2 *)tables : nullptr;
    const int gb = (int)std::max<int64_t>(1, std::min<int64_t>((n + 127) / 128, 152 * 16));
    column_tables_kernel<<<gb, 128>>>(dg, cray, lines);
    BSGD_CUDA(cudaGetLastError());
    BSGD_CUDA(cudaStreamSynchronize(0));
    dg.cray = cray;
    if (slice) {
        dg.sx = lines;
        dg.sy = lines + n;
        dg.si = lines + 2 * n;
        dg.slen = reinterpret_cast<float *>(lines + 3 * n);
    }
    return BSGD_OK;
}

size_t column_plan(bsgd_geometry *g) {
    const bsgd_geometry_desc &d = g->desc;
    DeviceGeom &dg = g->dg;
    const size_t rays = (size_t)d.n_views * d.nu;
    // a line's ends, and the products of the lengths that give a shadow, round to
    // 2^-24 of the ray's length each: eight of these in detector columns (with
    // 0.01 alone, a fan from 1e6 voxels away lost 3e-4 of the sum)
    const double length = d.kind == BSGD_PAR2D ? std::hypot(d.nx * d.dx, d.ny * d.dy) + 2.0 : d.dsd;
    const double rounding = std::ldexp(8.0, -24) * length / std::min(d.dx, d.dy) / (d.du / std::max(d.dx, d.dy));
    dg.umargin = (float)(0.01 + rounding);
    if (d.kind != BSGD_CONE3D) {
        dg.tc = d.kind == BSGD_PAR2D ? 0.5f : (float)(d.dso / d.dsd);
        return 28 * rays;
    }
    if (d.nz < 2 || d.nv < 2) return 0;
    // FP32 holds the place along a ray where it crosses a plane to 2^-24 of its
    // length: up to a hundredth of a voxel, which a row of rays that lies along a
    // face loses (1e-4 of its sum at 6e5 voxels, where the walk loses 2e-6); and
    // rays that round to half a column or more could meet voxels outside the bands,
    // where no weights are laid out
    if (std::ldexp(length / std::min(d.dx, d.dy), -24) > 0.01 || rounding > 1.0) return 0;
    // rows are found by an addition that holds them in 22 bits, and to 0.01 by FP32
    // from the detector's middle
    const double near = d.dso - 0.5 * std::hypot(d.nx * d.dx, d.ny * d.dy);
    if (d.nv > (1 << 14) || d.dz * d.dsd / (near * d.dv) > 1e3) return 0;
    // a ray rises less than a voxel while it crosses a column
    const double rise = 0.5 * (d.nv - 1) * d.dv / d.dz / d.dsd;   // voxels per mm along the axis
    if (std::sqrt(2.0) * std::max(d.dx, d.dy) * rise > 0.95) return 0;
    dg.tc = (float)(d.dso / d.dsd);
    dg.zs = g->rays[0].p0[2];
    dg.vstep = g->rays[0].cv[2];
    // rows that 32 planes can span past the first or last row that meets one of
    // them: at the volume's near edge, with the change of a row's height in a cell
    const double rows = d.dz * d.dsd / (near * d.dv);
    const double change = rows * std::sqrt(2.0) * std::max(d.dx, d.dy) / near;   // rows per voxel of height
    dg.vslack = (float)(32.0 * change * 1.01);
    const double pad = std::ceil(33.0 * rows + (2.0 * d.nz + 32.0) * change) + 8.0;
    if (pad > 1e6) return 0;   // a source in the volume's corner: past any use, and past int
    dg.vpad = (int)pad;
    dg.nvp = (d.nv + 2 * dg.vpad + 7) / 8 * 8;
    return sizeof(ColRay) * rays;
}

size_t column_weights_len(const bsgd_geometry *g, int n_rb) {
    // rows of weights are addressed by 32-bit offsets
    const size_t n = (size_t)n_rb * g->max_views * g->desc.nu * g->dg.nvp;
    return n < (1ull << 32) ? n : 0;
}

// Whether a gathering state takes FP, residual and weights as passes of their own
// and not as one: the one holds up to four blocks' rays through its walks (63
// registers against 40, 8 CTAs per SM against 12), but sets a pixel up once and
// skips the pass over the bands, which shows where cells leave few rays to walk. us
// per iteration one / apart, 256^2 x 32 from 45 views, 2, 3, 4 blocks: whole views
// 735 / 720, 1146 / 1047, 1494 / 1349, geometric cells 485 / 502, 746 / 721, 972 /
// 921, uniform cells 377 / 411, 566 / 579, 735 / 732; from 11 views, whole views 295
// / 298, 438 / 423, 566 / 536; 128^2 x 32 from 90 views, 2, 3, 4 blocks, whole views
// 392 / 406, 592 / 576, 772 / 734, geometric cells 252 / 282, 374 / 390, 482 / 488.
bool column_solve_apart(const bsgd_geometry *g, int kM, int kN, int cells) {
    const int64_t work = (int64_t)g->desc.nx * g->desc.ny * (g->desc.nz / g->N) * kN * g->max_views * kM;
    return kN >= 3 && (cells == BSGD_CELLS_NONE || (cells == BSGD_CELLS_GEOMETRIC && work >= 250000000));
}

int column_blocks_within(const bsgd_geometry *g, int n_rb, size_t floats) {
    int n = std::min(n_rb, 64);
    while (n > 0 && (column_weights_len(g, n) == 0 || column_weights_len(g, n) > floats)) --n;
    return n;
}

// Whether a chunk on both sides of the source's height would be widened by more than
// a row (gather_column).
static bool gather_near(const bsgd_geometry *g) { return g->dg.vslack > 1.f; }

static dim3 gather_grid(const bsgd_geometry *g, int planes, int z) {
    const int across = (g->desc.nx + kGatherAcross - 1) / kGatherAcross, rows = (g->desc.ny + kGatherRows - 1) / kGatherRows;
    return dim3((unsigned)(across * rows), (planes + 32 * kGatherChunks - 1) / (32 * kGatherChunks), z);
}

bsgd_status launch_bp_column(const bsgd_geometry *g, const PlainLaunch &L, const void *r,
                             bsgd_dtype rt, float *x, float scale, int accumulate, float *w,
                             cudaStream_t st, int per) {
    const int z0 = g->plane_start[L.j0], z1 = g->plane_start[L.j1];
    const dim3 grid = gather_grid(g, z1 - z0, 1);
    for (int k = 0; k < L.n_rb; k += per) {
        RowSel R{};
        R.n = std::min(per, L.n_rb - k);
        for (int t = 0; t < R.n; ++t) R.ids[t] = L.row_ids[k + t];
        const dim3 wg((unsigned)((g->desc.nu + 31) / 32 * ((g->dg.nvp + 31) / 32)), gather_slots(g->dg, R));
        if (rt == BSGD_F32) column_weights_kernel<float><<<wg, 256, 0, st>>>(g->dg, R, L.j0, L.j1, (const float *)r, scale, w);
        else if (rt == BSGD_BF16) column_weights_kernel<__nv_bfloat16><<<wg, 256, 0, st>>>(g->dg, R, L.j0, L.j1, (const __nv_bfloat16 *)r, scale, w);
        else column_weights_kernel<__half><<<wg, 256, 0, st>>>(g->dg, R, L.j0, L.j1, (const __half *)r, scale, w);
        if (gather_near(g)) bp_gather_kernel<true><<<grid, 32 * kGatherWarps, 0, st>>>(g->dg, R, z0, z1, w, x, accumulate || k > 0);
        else bp_gather_kernel<false><<<grid, 32 * kGatherWarps, 0, st>>>(g->dg, R, z0, z1, w, x, accumulate || k > 0);
        BSGD_CUDA(cudaGetLastError());
    }
    return BSGD_OK;
}

// Floats of the weights of a solver that draws kM row blocks and kN column blocks
// per iteration, 0 where its BP scatters beside the FP in one pass instead. That
// pass sets a ray up once for both, so the gather needs full warps (slabs of 28
// planes or more) and enough columns and views to pay for a pass of its own:
// us per iteration scattered / gathered (FP32, 8 or 4 row blocks), one block:
// 256^2 x 32 from 45 views 432 / 390, 192^2 x 32 from 22 160 / 148, 96^2 x 32
// from 45 83 / 81, 256^2 x 32 from 11 162 / 169, 256^2 x 16 from 45 258 / 312;
// two blocks: 256^2 x 32 from 45 887 / 758, 128^2 x 32 from 11 120 / 90, 96^2 x
// 12 from 22 70 / 68. At a waste of 1.58 (205 x 170 x 40 from 59 views, rows a
// voxel apart) 284 / 333.
// With detector cells one block's pass traces a fraction of the rays that the
// gather lists: 160^2 x 32 from 45 views 90 / 109, 256^2 x 32 258 / 260.
size_t column_solve_len(const bsgd_geometry *g, int kM, int kN, bool cells) {
    if (g->dg.nvp == 0 || (cells && kN == 1)) return 0;
    const int planes = g->desc.nz / g->N;   // of the thinnest slab
    const int64_t work = (int64_t)g->desc.nx * g->desc.ny * planes * kN * g->max_views * kM;
    if (planes < 28 || work < (kN > 1 ? 10000000 : 25000000) ||
        gather_waste(g, (g->desc.nz + g->N - 1) / g->N) > 1.12)
        return 0;
    return column_weights_len(g, kM * kN);
}

// Whether the back projection of a 2D kind into `rows` image rows gathers: us
// scattered / gathered, 64^2 from 90 views 15.4 / 10.7, 128^2 from 60 17.4 /
// 10.5, 100 x 17 of a strip from 180 20.1 / 20.1, 512^2 from 720 977 / 894.
// At strips of some 2000 pixels the two are level.
bool slice_bp_pays(const bsgd_geometry *g, int rows, int views) {
    return g->dg.sx && (int64_t)g->desc.nx * rows >= 4096 && views >= 1;
}

bsgd_status launch_bp_slice(const bsgd_geometry *g, const PlainLaunch &L, const void *r, bsgd_dtype rt,
                            float *x, float scale, int accumulate, cudaStream_t st) {
    const int y0 = g->plane_start[L.j0], y1 = g->plane_start[L.j1];
    const unsigned grid = (unsigned)((g->desc.nx + 31) / 32) * (y1 - y0);
    // all blocks: one launch, whose view order does not read the list
    const bool all = L.n_rb == g->M;
    for (int k = 0; k < L.n_rb; k += all ? L.n_rb : 64) {
        RowSel R{};
        R.n = std::min(64, L.n_rb - k);
        for (int t = 0; t < R.n; ++t) R.ids[t] = L.row_ids[k + t];
        const int add = accumulate || k > 0;
#define SLICE_KIND(KERNEL, ...)                                                                                \
    if (g->desc.kind == BSGD_PAR2D)                                                                            \
        KERNEL<true, __VA_ARGS__><<<grid, 256, 0, st>>>(g->dg, R, y0, rr, scale, x, add);                      \
    else KERNEL<false, __VA_ARGS__><<<grid, 256, 0, st>>>(g->dg, R, y0, rr, scale, x, add);
#define SLICE_GO(T)                                                                                            \
    const T *rr = (const T *)r;                                                                                \
    if (all) { SLICE_KIND(bp_slice_kernel, kSliceAll, T) }                                                     \
    else if (R.n > 1 && g->max_views < 64) { SLICE_KIND(bp_slice_kernel, kSliceListed, T) }                    \
    else { SLICE_KIND(bp_slice_blocks_kernel, T) }
        if (rt == BSGD_F32) { SLICE_GO(float) }
        else if (rt == BSGD_BF16) { SLICE_GO(__nv_bfloat16) }
        else { SLICE_GO(__half) }
#undef SLICE_GO
#undef SLICE_KIND
        BSGD_CUDA(cudaGetLastError());
    }
    return BSGD_OK;
}

bsgd_status launch_column_change(const bsgd_geometry *g, const SolveDev &S, bsgd_dtype st_t,
                                 int max_pairs, cudaStream_t st) {
    const dim3 grid((unsigned)((g->desc.nu + 31) / 32 * ((g->desc.nv + 31) / 32)), g->max_views, max_pairs);
    if (st_t == BSGD_F32) column_change_kernel<float><<<grid, 256, 0, st>>>(g->dg, S);
    else if (st_t == BSGD_BF16) column_change_kernel<__nv_bfloat16><<<grid, 256, 0, st>>>(g->dg, S);
    else column_change_kernel<__half><<<grid, 256, 0, st>>>(g->dg, S);
    BSGD_CUDA(cudaGetLastError());
    return BSGD_OK;
}

bsgd_status launch_column_solve(const bsgd_geometry *g, const SolveDev &S, int max_cols, cudaStream_t st) {
    int planes = 1;
    for (int j = 0; j < g->N; ++j) planes = std::max(planes, g->plane_start[j + 1] - g->plane_start[j]);
    const dim3 grid = gather_grid(g, planes, max_cols);
    if (gather_near(g)) solve_gather_kernel<true><<<grid, 32 * kGatherWarps, 0, st>>>(g->dg, S);
    else solve_gather_kernel<false><<<grid, 32 * kGatherWarps, 0, st>>>(g->dg, S);
    BSGD_CUDA(cudaGetLastError());
    return BSGD_OK;
}

}  // namespace bsgd
