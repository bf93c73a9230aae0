// lbm_region.cuh -- enumeration of the node region around a body and
// lattice-neighbour helpers shared by the geometry and boundary-node kernels.
#pragma once

#include "lbm_dev.cuh"

namespace lbm {

struct RegionCell {
    int x, y, z;
    long long cell;
};

// The shell rlo <= |x - X| <= rhi around a body, geom_rows rows (y, z) of its
// region at a time.  Only the shell holds work (a seventh of the region of a
// sphere of radius 9), so a chunk's rows are cut to it first: one lane of warp
// 0 per row takes the one or two stretches of the row that the shell covers
// (slightly wide: the callers test each cell's distance themselves), a scan
// numbers their cells, and every thread of the block then finds its cell e by
// a search over the 32 row prefixes -- full warps of cells that all do the
// work, instead of warps in which a few lanes of the box do, and blocks for
// every 32 rows instead of every 4096 cells (a disc's whole region was one
// block).  Bound by the latency of dependent loads and FP64 operations.
// Measured alone, before -> after: the 135x1073 FP64 disc's geom_a + b + c
// 169 -> 22 us, the two moving spheres of a 151x97x84 box's fgeom1 + fgeom2l
// 89 -> 31 us, two cylinders' 26 -> 14 us.  Cells are numbered in ascending cell order, also across a
// periodic seam.
struct ShellChunk {
    Frame F;
    int lo[3], s0, split;   // region origin; its first x (wrapped) and the offset past the x seam
    int pre[GEOM_ROWS + 1]; // cells before each row
    int a0[GEOM_ROWS], a1[GEOM_ROWS], b0[GEOM_ROWS], b1[GEOM_ROWS]; // stretches of x offsets
    int y[GEOM_ROWS], z[GEOM_ROWS];
};

// Opens chunk `chunk` of body B's region for the pose P + at (at = 3: wrapped
// pose of t, 9: of t+1); called by the whole block, syncs it; returns the
// number of cells.
__device__ __forceinline__ int shell_open(const Params &p, const BodyDev &B, const double *P, int at, int chunk,
                                          float rlo, float rhi, ShellChunk &c) {
    __syncthreads(); // the last chunk is done with
    if (threadIdx.x < 32) {
        const int lane = threadIdx.x;
        if (lane == 0) make_frame(P + at, c.F);
        if (lane < 3) c.lo[lane] = region_lo_axis(p, B, P, REGION_MARGIN, lane);
        __syncwarp();
        const int e0 = B.ext[0], e1 = B.ext[1], rows = e1 * B.ext[2];
        const int n = p.nx, lo = c.lo[0];
        const bool full = p.per[0] && e0 >= n;
        const int s0 = full || !p.per[0] ? 0 : ((lo % n) + n) % n;
        const int split = !p.per[0] || full || s0 + e0 <= n ? e0 : n - s0;
        const int rpc = geom_rows(p.nz);
        const int r = lane < rpc ? chunk * rpc + lane : rows;
        const int kz = r / e1, ky = r - kz * e1;
        int a0 = 0, a1 = 0, b0 = 0, b1 = 0;
        int y = -1, z = -1;
        if (r < rows) {
            y = region_axis(ky, c.lo[1], e1, p.ny, p.per[1]);
            z = region_axis(kz, c.lo[2], B.ext[2], p.nz, p.per[2]);
        }
        if (y >= 0 && z >= 0) {
            const float dy = frame_axis(y - c.F.xi[1], c.F.fr[1], p.ny, p.per[1]);
            const float dz = B.shape == 1 ? frame_axis(z - c.F.xi[2], c.F.fr[2], p.nz, p.per[2]) : 0.0f;
            const float r2 = dy * dy + dz * dz, ro = rhi + 0.05f, ri = rlo - 0.05f;
            const float h2 = ro * ro - r2, g2 = ri > 0.0f ? ri * ri - r2 : -1.0f;
            if (full) { // the row may meet the shell across the seam: all of it
                if (h2 >= 0.0f) a1 = n;
            } else if (h2 >= 0.0f) {
                const float mid = (float)(P[at - 3] - (double)lo), h = sqrtf(h2);
                a0 = max(0, (int)ceilf(mid - h - 0.05f));
                a1 = min(e0, (int)floorf(mid + h + 0.05f) + 1);
                if (!p.per[0]) {
                    a0 = max(a0, -lo);
                    a1 = min(a1, n - lo);
                }
                const float g = g2 > 0.0f ? sqrtf(g2) - 0.05f : 0.0f;
                const int end = (int)floorf(mid - g) + 1, beg = (int)ceilf(mid + g);
                if (g > 0.0f && beg > end) { // a hole in the middle
                    b0 = max(a0, beg);
                    b1 = max(b0, a1);
                    a1 = min(a1, end);
                }
                a1 = max(a0, a1);
            }
        }
        c.y[lane] = y;
        c.z[lane] = z;
        c.a0[lane] = a0;
        c.a1[lane] = a1;
        c.b0[lane] = b0;
        c.b1[lane] = b1;
        const int cnt = (a1 - a0) + (b1 - b0);
        int inc = cnt;
        for (int o = 1; o < 32; o <<= 1) {
            const int v = __shfl_up_sync(0xffffffffu, inc, o);
            if (lane >= o) inc += v;
        }
        c.pre[lane] = inc - cnt;
        if (lane == 31) c.pre[GEOM_ROWS] = inc;
        if (lane == 0) {
            c.s0 = s0;
            c.split = split;
        }
    }
    __syncthreads();
    return c.pre[GEOM_ROWS];
}

// cell e (0 <= e < shell_open's count) of the open chunk
__device__ __forceinline__ RegionCell shell_cell(const Params &p, const ShellChunk &c, int e) {
    int r = 0;
#pragma unroll
    for (int k = GEOM_ROWS / 2; k > 0; k >>= 1)
        if (c.pre[r + k] <= e) r += k;
    int j = e - c.pre[r];
    const int a0 = c.a0[r], a1 = c.a1[r], b0 = c.b0[r], b1 = c.b1[r], sp = c.split;
    // offsets past the seam come first: their wrapped x are the smaller ones
    const int pa = max(a0, sp), pb = max(b0, sp);
    const int na = max(0, a1 - pa), nb = max(0, b1 - pb);
    int o;
    if (j < na) o = pa + j;
    else if (j < na + nb) o = pb + (j - na);
    else {
        j -= na + nb;
        const int qa = max(0, min(a1, sp) - a0);
        o = j < qa ? a0 + j : b0 + (j - qa);
    }
    RegionCell rc;
    if (!p.per[0]) {
        rc.x = c.lo[0] + o;
    } else {
        rc.x = c.s0 + o;
        if (rc.x >= p.nx) rc.x -= p.nx;
    }
    rc.y = c.y[r];
    rc.z = c.z[r];
    rc.cell = cell_of(p, rc.x, rc.y, rc.z);
    return rc;
}

// neighbour x - k c_i; -1 if it falls outside a non-periodic axis
template <class L>
__device__ __forceinline__ long long nbr(const Params &p, int x, int y, int z, int i, int k) {
    int q[3] = {x - k * L::cx(i), y - k * L::cy(i), z - k * L::cz(i)};
    const int n[3] = {p.nx, p.ny, p.nz};
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        if (q[a] >= 0 && q[a] < n[a]) continue;
        if (!p.per[a]) return -1;
        while (q[a] < 0) q[a] += n[a]; // |k c_i| <= 2: at most two turns
        while (q[a] >= n[a]) q[a] -= n[a];
    }
    return cell_of(p, q[0], q[1], q[2]);
}

// nbr<L>(p, x, y, z, i, 1) for a node one cell or more inside every face of
// the lattice (no wrap): the cell index minus c_i's offset
template <class L>
__device__ __forceinline__ long long nbr1_inner(long long cell, long long sy, long long sz, int i) {
    return cell - ((long long)L::cx(i) + (L::cy(i) == 0 ? 0ll : (L::cy(i) > 0 ? sy : -sy)) +
                   (L::cz(i) == 0 ? 0ll : (L::cz(i) > 0 ? sz : -sz)));
}

__device__ __forceinline__ bool inner1(const Params &p, int x, int y, int z) {
    return x >= 1 && x <= p.nx - 2 && y >= 1 && y <= p.ny - 2 && (p.nz == 1 || (z >= 1 && z <= p.nz - 2));
}

__device__ __forceinline__ bool edge_node(const Params &p, int x, int y, int z) {
    return (!p.per[0] && (x == 0 || x == p.nx - 1)) || (!p.per[1] && (y == 0 || y == p.ny - 1)) ||
           (!p.per[2] && (z == 0 || z == p.nz - 1));
}

// distance of a cell from the axis or centre of a body (FP32 frame)
__device__ __forceinline__ float frame_dist(const Params &p, const BodyDev &B, const Frame &F, const RegionCell &rc) {
    float d[3];
    frame_disp_f(p, F, rc.x, rc.y, rc.z, d);
    return sqrtf(d[0] * d[0] + d[1] * d[1] + (B.shape == 1 ? d[2] * d[2] : 0.0f));
}

} // namespace lbm
