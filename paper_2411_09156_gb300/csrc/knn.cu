// Exact k = 16 nearest splat centres (Sec. 4.2: the GSR density at a sample uses
// the 16 splats closest to the splat it was drawn from).
//
// A uniform grid over the centres' bounding box, at most one cell per point, is
// built on the device: cell keys and counts, a stable radix sort of the points by cell (the
// sort of the binning), the scan of the counts (the first centre of every cell, so that a run of
// cells along x is one range of centres, read with two loads) and a cell-ordered copy of the centres.
// A query walks Chebyshev rings of cells around its own cell twice: first for the 16 least
// distances alone, then, over the cells within the 16th, for the centres themselves. Rows of
// cells farther than the current 16th are skipped and the others cut to it along x, which keeps
// queries away from the centres (points in front of a surface) from reading every cell of their
// block. One cell per point: with two and with a half KNN of a 1.5M-splat heightfield takes 1.24 and 1.50 ms
// against 1.26, of a 300k-splat object 1.52 and 0.92 against 1.02. Queries run in cell order, so a warp searches
// one neighbourhood. Distances are squared float32 with a fixed operation order; ties go to
// the lower index. A query that would examine more than 131,072 candidates (a bound that well-spread
// centres never reach; more coincident centres than that would) takes the best of the first 131,072 in ring
// order instead, and one that no distance bounds ends at once, so no input makes the search quadratic.
#include "ges_internal.cuh"
#include "sort_net.cuh"

namespace ges {

namespace {

constexpr int kK = GES_KNN_K;
constexpr uint32_t kQueryBudget = 1u << 17;  // candidate points one query may examine
// A query with more candidates than this in the 27 cells around it leaves the two passes for one pass of pair
// insertion: its nearest tie (coincident centres), and each pass costs a distance per candidate. 50,000 coincident
// centres: 26.8 ms with two passes that searched the whole column at each tie, 13.6 with the column's greatest pair kept,
// 7.3 in one pass (before the two passes: 6.6); 100,000: 75.7, 27.9, 15.1 (9.0 with half the budget). Ordinary queries
// examine a few hundred.
constexpr uint32_t kTwoPassMost = 2048;
// 16 CTAs of 64 threads per SM (64 registers): at 12 or 20 the centre queries take 11 % or 1 % longer, as 32 one-warp CTAs
// the whole call of either query 1 %
constexpr int kQueryThreads = 64, kQueryCtas = 16;
// The first pass ends when the searched cells reach sqrt(kReach) of the 16th distance: the second pass then
// drops the few candidates too many, which costs less than another ring (reach 1: 1.61 ms against 1.42-1.45
// at 0.25 and 0.5 for the centres; level-set queries 3.93 against 3.78 ms).
constexpr float kReach = 0.25f;
constexpr int kNearRings = 4;  // rings of cells that a point query tries before it walks blocks (2 and 3: within 5 %)
// Blocks of 4 x 4 x 4 cells, with their point counts, let point queries skip empty space. Level-set queries of
// five 1600x1040 views (whole call): 2.45-4.91 ms with 2 x 2 x 2 blocks, 2.53-3.28 with these, 2.63-3.69 with
// 8 x 8 x 8.
constexpr int kBlockShift = 2, kBlockSide = 1 << kBlockShift;

struct KnnGrid {
    float lo[3];
    float h, inv_h;
    int dims[3];
    float slack;  // bound on how far float32 rounding can put a point outside its cell's box
};

struct KnnLayout {
    uint64_t bbox, grid, keys0, keys1, vals0, vals1, hist, partials, starts, bcount, spos, bytes;
    uint32_t cap_cells, nblocks;
    int bits;
};

inline uint64_t al256(uint64_t x) { return (x + 255) & ~uint64_t(255); }

KnnLayout knn_layout(int32_t n) {
    KnnLayout L;
    uint64_t cap = (uint64_t)n;
    if (cap < 1) cap = 1;
    if (cap > (1ull << 26) - 1) cap = (1ull << 26) - 1;  // one scan covers the cells and the end
    L.cap_cells = (uint32_t)cap;
    L.bits = 1;
    while ((1ull << L.bits) < cap) ++L.bits;
    L.nblocks = ceil_div_u64(n > 0 ? (uint64_t)n : 1, kSortTile);
    uint64_t off = 0;
    L.bbox = off; off = al256(off + 6 * 4);
    L.grid = off; off = al256(off + sizeof(KnnGrid));
    L.keys0 = off; off = al256(off + 4ull * n);
    L.keys1 = off; off = al256(off + 4ull * n);
    L.vals0 = off; off = al256(off + 4ull * n);
    L.vals1 = off; off = al256(off + 4ull * n);
    L.hist = off; off = al256(off + 4ull * 256 * L.nblocks);
    const uint64_t scanned = 256ull * L.nblocks > cap + 1 ? 256ull * L.nblocks : cap + 1;
    L.partials = off; off = al256(off + 4ull * (ceil_div_u64(scanned, kScanTile) + 1));
    L.starts = off; off = al256(off + 4ull * (L.cap_cells + 1ull));
    L.bcount = off; off = al256(off + 4ull * L.cap_cells);  // blocks <= cells <= cap_cells
    L.spos = off; off = al256(off + 16ull * n);
    L.bytes = off;
    return L;
}

// float <-> order-preserving uint32 (for atomic min / max)
__device__ __forceinline__ uint32_t f2ord(float f) {
    const uint32_t u = __float_as_uint(f);
    return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}
__device__ __forceinline__ float ord2f(uint32_t k) {
    return __uint_as_float((k & 0x80000000u) ? (k & 0x7fffffffu) : ~k);
}

__global__ void __launch_bounds__(256) k_knn_bbox(const float4 *pos, int n, uint32_t *bb) {
    uint32_t mn[3] = {0xffffffffu, 0xffffffffu, 0xffffffffu}, mx[3] = {0u, 0u, 0u};
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        const float4 p = __ldg(pos + i);
        const float c[3] = {p.x, p.y, p.z};
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            const uint32_t o = f2ord(c[k]);
            mn[k] = min(mn[k], o);
            mx[k] = max(mx[k], o);
        }
    }
    // one set of atomics a CTA: all of them meet at six addresses
    __shared__ uint32_t s_bb[6];
    if (threadIdx.x < 6) s_bb[threadIdx.x] = threadIdx.x < 3 ? 0xffffffffu : 0u;
    __syncthreads();
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        mn[k] = __reduce_min_sync(0xffffffffu, mn[k]);
        mx[k] = __reduce_max_sync(0xffffffffu, mx[k]);
    }
    if ((threadIdx.x & 31) == 0) {
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            atomicMin(s_bb + k, mn[k]);
            atomicMax(s_bb + 3 + k, mx[k]);
        }
    }
    __syncthreads();
    if (threadIdx.x < 3) atomicMin(bb + threadIdx.x, s_bb[threadIdx.x]);
    else if (threadIdx.x < 6) atomicMax(bb + threadIdx.x, s_bb[threadIdx.x]);
}

// Cell size h with at most cap cells: start from the volume per cell, then grow h
// until the product of the per-axis counts fits (flat boxes have a zero extent).
__global__ void k_knn_grid(const uint32_t *bb, uint32_t cap, KnnGrid *g) {
    float lo[3], ext[3];
    for (int k = 0; k < 3; ++k) {
        lo[k] = ord2f(bb[k]);
        ext[k] = fmaxf(ord2f(bb[3 + k]) - lo[k], 0.f);
    }
    const float emax = fmaxf(fmaxf(ext[0], ext[1]), ext[2]);
    float h = emax > 0.f ? emax : 1.f;
    const double vol = (double)fmaxf(ext[0], 1e-30f) * fmaxf(ext[1], 1e-30f) * fmaxf(ext[2], 1e-30f);
    const double h0 = cbrt(vol / (double)cap);
    if (h0 > 0.0 && h0 < (double)h) h = (float)h0;
    int d[3] = {1, 1, 1};
    bool fits = false;
    for (int it = 0; it < 256 && !fits; ++it) {
        double prod = 1.0;
        for (int k = 0; k < 3; ++k) {
            d[k] = (int)fminf(fmaxf(floorf(ext[k] / h) + 1.f, 1.f), 2048.f);
            prod *= d[k];
        }
        fits = prod <= (double)cap;
        if (!fits) h *= 1.0625f;
    }
    if (!fits || !(h > 0.f) || !isfinite(h)) {  // non-finite coordinates: one cell (the query budget bounds the work)
        d[0] = d[1] = d[2] = 1;
        h = 1.f;
    }
    for (int k = 0; k < 3; ++k) {
        g->lo[k] = isfinite(lo[k]) ? lo[k] : 0.f;
        g->dims[k] = d[k];
    }
    g->h = h;
    g->inv_h = 1.f / h;
    float amax = 0.f;
    for (int k = 0; k < 3; ++k) amax = fmaxf(amax, fabsf(g->lo[k]) + (float)d[k] * h);
    g->slack = 4e-6f * amax;
}

__device__ __forceinline__ int cell_axis(float p, float lo, float inv_h, int dim) {
    const int c = (int)floorf((p - lo) * inv_h);
    return min(max(c, 0), dim - 1);
}

__device__ __forceinline__ int block_dim(int d) { return (d + kBlockSide - 1) >> kBlockShift; }

__global__ void __launch_bounds__(256) k_knn_keys(const float4 *pos, int n, const KnnGrid *g, uint32_t *keys,
                                                  uint32_t *ccount, uint32_t *bcount) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const float4 p = __ldg(pos + i);
    const KnnGrid G = *g;
    const int cx = cell_axis(p.x, G.lo[0], G.inv_h, G.dims[0]);
    const int cy = cell_axis(p.y, G.lo[1], G.inv_h, G.dims[1]);
    const int cz = cell_axis(p.z, G.lo[2], G.inv_h, G.dims[2]);
    const uint32_t cell = (uint32_t)(cx + G.dims[0] * (cy + G.dims[1] * cz));
    keys[i] = cell;
    atomicAdd(ccount + cell, 1u);
    atomicAdd(bcount + ((cx >> kBlockShift) + block_dim(G.dims[0]) * ((cy >> kBlockShift) +
                        block_dim(G.dims[1]) * (cz >> kBlockShift))), 1u);
}

// The centres in cell order.
__global__ void __launch_bounds__(256) k_knn_gather(const uint32_t *idx, const float4 *pos, int n, float4 *spos) {
    const int r = blockIdx.x * blockDim.x + threadIdx.x;
    if (r >= n) return;
    const uint32_t i = idx[r];
    const float4 p = __ldg(pos + i);
    spos[r] = make_float4(p.x, p.y, p.z, __uint_as_float(i));
}

// The centres of cells [first, last] of one row, consecutive in cell order (none if first > last).
__device__ __forceinline__ uint2 row_range(const uint32_t *starts, int first, int last) {
    if (first > last) return make_uint2(0u, 0u);
    return make_uint2(__ldg(starts + first), __ldg(starts + last + 1));
}

__device__ __forceinline__ float dist2(float4 a, float4 b) {
    const float dx = __fsub_rn(a.x, b.x), dy = __fsub_rn(a.y, b.y), dz = __fsub_rn(a.z, b.z);
    return __fadd_rn(__fadd_rn(__fmul_rn(dx, dx), __fmul_rn(dy, dy)), __fmul_rn(dz, dz));
}

// Examines the centres spos[rg.x, rg.y) (at most the rest of the budget) for p's list.
__device__ __forceinline__ void scan_cell(float4 p, uint2 rg, const float4 *spos, uint32_t &examined, float (&bd)[kK],
                                          uint32_t (&bi)[kK]) {
    const uint32_t end = min(rg.y, rg.x + (kQueryBudget - min(examined, kQueryBudget)));
    examined += rg.y - rg.x;
    for (uint32_t q = rg.x; q < end; ++q) {
        const float4 o = __ldg(spos + q);
        const float d = dist2(p, o);
        uint32_t id = __float_as_uint(o.w);
        if (d > bd[kK - 1] || (d == bd[kK - 1] && id >= bi[kK - 1])) continue;
        float cd = d;
#pragma unroll
        for (int k = 0; k < kK; ++k) {  // insert, keeping (distance, index) order
            const bool less = cd < bd[k] || (cd == bd[k] && id < bi[k]);
            const float td = bd[k];
            const uint32_t ti = bi[k];
            bd[k] = less ? cd : td;
            bi[k] = less ? id : ti;
            cd = less ? td : cd;
            id = less ? ti : id;
        }
    }
}

// Ring search around point p for its kK nearest centres (lists in bd / bi, sorted).
__device__ __forceinline__ void ring_search(float4 p, const KnnGrid &G, const uint32_t *starts, const float4 *spos,
                                            float (&bd)[kK], uint32_t (&bi)[kK]) {
    const int c[3] = {cell_axis(p.x, G.lo[0], G.inv_h, G.dims[0]), cell_axis(p.y, G.lo[1], G.inv_h, G.dims[1]),
                      cell_axis(p.z, G.lo[2], G.inv_h, G.dims[2])};
    const float pc[3] = {p.x, p.y, p.z};
#pragma unroll
    for (int k = 0; k < kK; ++k) { bd[k] = __int_as_float(0x7f800000); bi[k] = 0xffffffffu; }
    const int rmax = max(max(G.dims[0], G.dims[1]), G.dims[2]);
    // distance along axis k from p to cell index ci's slab, less the rounding slack; once 16
    // are held, a row or cell whose box is farther than the 16th is skipped unread
    auto gap = [&](int k, int ci) {
        const float a = G.lo[k] + (float)ci * G.h - G.slack - pc[k];
        const float b = pc[k] - (G.lo[k] + (float)(ci + 1) * G.h + G.slack);
        return fmaxf(fmaxf(a, b), 0.f);
    };
    float outg[3], og2 = 0.f;  // distance from p to the grid's box along each axis, less the slack
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        outg[k] = fmaxf(fmaxf(G.lo[k] - G.slack - pc[k], pc[k] - (G.lo[k] + (float)G.dims[k] * G.h + G.slack)), 0.f);
        og2 = fmaf(outg[k], outg[k], og2);
    }
    uint32_t examined = 0;
    for (int ring = 0; ring <= rmax && examined < kQueryBudget; ++ring) {
        const int z0 = max(c[2] - ring, 0), z1 = min(c[2] + ring, G.dims[2] - 1);
        const int y0 = max(c[1] - ring, 0), y1 = min(c[1] + ring, G.dims[1] - 1);
        const int x0 = max(c[0] - ring, 0), x1 = min(c[0] + ring, G.dims[0] - 1);
        auto visit = [&](int cx, int cy, int cz, float gyz) {
            const float gx = gap(0, cx);
            if (fmaf(gx, gx, gyz) > bd[kK - 1]) return;
            const int cell = cx + G.dims[0] * (cy + G.dims[1] * cz);
            scan_cell(p, row_range(starts, cell, cell), spos, examined, bd, bi);
        };
        // the cells at Chebyshev distance `ring` from the query's cell; where neither x face lies in the grid, of the
        // inner rows there is nothing to see, nor of the inner planes where no y face does (a line in one cell of a
        // flat grid has 2,048 rings)
        const bool no_x = ring > 0 && c[0] - ring < 0 && c[0] + ring >= G.dims[0];
        const bool no_xy = no_x && c[1] - ring < 0 && c[1] + ring >= G.dims[1];
        for (int cz = no_xy ? c[2] - ring : z0; cz <= z1; cz += no_xy ? 2 * ring : 1) {
            if (cz < 0) continue;
            const float gz = gap(2, cz);
            if (gz * gz > bd[kK - 1]) continue;
            const bool faces = no_x && abs(cz - c[2]) < ring;
            for (int cy = faces ? c[1] - ring : y0; cy <= y1; cy += faces ? 2 * ring : 1) {
                if (cy < 0) continue;
                const float gy = gap(1, cy);
                const float gyz = fmaf(gy, gy, gz * gz);
                if (gyz > bd[kK - 1]) continue;
                if (abs(cz - c[2]) < ring && abs(cy - c[1]) < ring) {  // only the two x faces are new
                    if (c[0] - ring >= 0) visit(c[0] - ring, cy, cz, gyz);
                    if (c[0] + ring < G.dims[0]) visit(c[0] + ring, cy, cz, gyz);
                } else {
                    for (int cx = x0; cx <= x1; ++cx) visit(cx, cy, cz, gyz);
                }
            }
        }
        // every unsearched point lies in the grid's box beyond one of the searched block's open
        // faces; b2 is the least squared distance from p to those regions (a query outside the
        // box adds its distance to the box on the other axes)
        float b2 = __int_as_float(0x7f800000);
        bool all = true;
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            const float others = og2 - outg[k] * outg[k];
            if (c[k] - ring > 0) {
                const float g = fmaxf(pc[k] - (G.lo[k] + (float)(c[k] - ring) * G.h) - G.slack, 0.f);
                b2 = fminf(b2, fmaf(g, g, others));
                all = false;
            }
            if (c[k] + ring < G.dims[k] - 1) {
                const float g = fmaxf((G.lo[k] + (float)(c[k] + ring + 1) * G.h) - pc[k] - G.slack, 0.f);
                b2 = fminf(b2, fmaf(g, g, others));
                all = false;
            }
        }
        if (all) break;
        if (bi[kK - 1] != 0xffffffffu && bd[kK - 1] <= b2 * (1.f - 1.f / 1048576.f)) break;
    }
}

// Distance from p to the slab [lo + i w, lo + (i + 1) w] of one axis, less the slack.
__device__ __forceinline__ float slab_gap(float lo, float w, float slack, float p, int i) {
    return fmaxf(fmaxf(lo + (float)i * w - slack - p, p - (lo + (float)(i + 1) * w + slack)), 0.f);
}

// The same search over Chebyshev rings of 2 x 2 x 2-cell blocks, for queries anywhere in
// space: the order in which a query that exceeds the budget examines its centres.
__device__ __forceinline__ void block_search(float4 p, const KnnGrid G, const uint32_t *starts, const float4 *spos,
                                             float (&bd)[kK], uint32_t (&bi)[kK]) {
    const int dx = G.dims[0], dy = G.dims[1], dz = G.dims[2];
    const int bx_n = (dx + 1) >> 1, by_n = (dy + 1) >> 1, bz_n = (dz + 1) >> 1;
    const int cbx = cell_axis(p.x, G.lo[0], G.inv_h, dx) >> 1, cby = cell_axis(p.y, G.lo[1], G.inv_h, dy) >> 1,
              cbz = cell_axis(p.z, G.lo[2], G.inv_h, dz) >> 1;
    const float h = G.h, H = G.h + G.h, sl = G.slack;
    const float lx = G.lo[0], ly = G.lo[1], lz = G.lo[2];
#pragma unroll
    for (int k = 0; k < kK; ++k) { bd[k] = __int_as_float(0x7f800000); bi[k] = 0xffffffffu; }
    // distance from p to the grid's box along each axis
    const float ox = fmaxf(fmaxf(lx - sl - p.x, p.x - (lx + (float)dx * h + sl)), 0.f);
    const float oy = fmaxf(fmaxf(ly - sl - p.y, p.y - (ly + (float)dy * h + sl)), 0.f);
    const float oz = fmaxf(fmaxf(lz - sl - p.z, p.z - (lz + (float)dz * h + sl)), 0.f);
    const int rmax = max(max(bx_n, by_n), bz_n);
    uint32_t examined = 0;
    for (int ring = 0; ring <= rmax && examined < kQueryBudget; ++ring) {
        const int z0 = max(cbz - ring, 0), z1 = min(cbz + ring, bz_n - 1);
        const int y0 = max(cby - ring, 0), y1 = min(cby + ring, by_n - 1);
        const int x0 = max(cbx - ring, 0), x1 = min(cbx + ring, bx_n - 1);
        auto visit = [&](int bx, int by, int bz, float gyz) {
            const float gx = slab_gap(lx, H, sl, p.x, bx);
            if (fmaf(gx, gx, gyz) > bd[kK - 1]) return;
            const int fz1 = min(2 * bz + 1, dz - 1), fy1 = min(2 * by + 1, dy - 1), fx1 = min(2 * bx + 1, dx - 1);
            for (int fz = 2 * bz; fz <= fz1; ++fz) {
                const float hz = slab_gap(lz, h, sl, p.z, fz);
                for (int fy = 2 * by; fy <= fy1; ++fy) {
                    const float hy = slab_gap(ly, h, sl, p.y, fy);
                    const float hyz = fmaf(hy, hy, hz * hz);
                    if (hyz > bd[kK - 1]) continue;
                    for (int fx = 2 * bx; fx <= fx1; ++fx) {
                        const float hx = slab_gap(lx, h, sl, p.x, fx);
                        if (fmaf(hx, hx, hyz) > bd[kK - 1]) continue;
                        const int cell = fx + dx * (fy + dy * fz);
                        scan_cell(p, row_range(starts, cell, cell), spos, examined, bd, bi);
                    }
                }
            }
        };
        for (int bz = z0; bz <= z1; ++bz) {
            const float gz = slab_gap(lz, H, sl, p.z, bz);
            if (gz * gz > bd[kK - 1]) continue;
            for (int by = y0; by <= y1; ++by) {
                const float gy = slab_gap(ly, H, sl, p.y, by);
                const float gyz = fmaf(gy, gy, gz * gz);
                if (gyz > bd[kK - 1]) continue;
                if (abs(bz - cbz) < ring && abs(by - cby) < ring) {  // only the two x faces are new
                    if (cbx - ring >= 0) visit(cbx - ring, by, bz, gyz);
                    if (cbx + ring < bx_n) visit(cbx + ring, by, bz, gyz);
                } else {
                    for (int bx = x0; bx <= x1; ++bx) visit(bx, by, bz, gyz);
                }
            }
        }
        // least distance to the grid's box beyond the searched blocks' open faces
        float b2 = __int_as_float(0x7f800000);
        bool all = true;
        auto face = [&](bool open, float g, float o1, float o2) {
            if (!open) return;
            g = fmaxf(g - sl, 0.f);
            b2 = fminf(b2, fmaf(g, g, fmaf(o1, o1, o2 * o2)));
            all = false;
        };
        face(cbx - ring > 0, p.x - (lx + (float)(cbx - ring) * H), oy, oz);
        face(cbx + ring < bx_n - 1, (lx + (float)(cbx + ring + 1) * H) - p.x, oy, oz);
        face(cby - ring > 0, p.y - (ly + (float)(cby - ring) * H), ox, oz);
        face(cby + ring < by_n - 1, (ly + (float)(cby + ring + 1) * H) - p.y, ox, oz);
        face(cbz - ring > 0, p.z - (lz + (float)(cbz - ring) * H), ox, oy);
        face(cbz + ring < bz_n - 1, (lz + (float)(cbz + ring + 1) * H) - p.z, ox, oy);
        if (all) break;
        if (bi[kK - 1] != 0xffffffffu && bd[kK - 1] <= b2 * (1.f - 1.f / 1048576.f)) break;
    }
}

// ---------------------------------------------------------------------------
// Two-pass search, one thread per query. It is bound by instruction issue under divergence (14 of 32 lanes
// active: the lanes' ranges of centres differ in length). Keeping 16 (distance, index) pairs sorted while scanning costs
// about seven instructions a slot for every candidate that any lane of the warp accepts, which is nearly
// all of them. The first pass keeps the 16 least distances alone (a minimum and a maximum a slot) and ends
// with a distance that at least 16 centres lie within; the second walks the cells within it and appends
// the candidates to the thread's column of a shared table, which is sorted once at the end.
// 1.5M centres of a heightfield, the whole call: 2.61 ms with one pass of pair insertion -> 1.82 (two passes,
// 64 registers) -> 1.44 (rows cut to the bound, middle rows first) -> 1.26 ms (scanned cell counts in
// place of a range per cell). A warp per query (candidates across the lanes, a warp-wide sort) was
// exact too but took 3.2 ms.

// Inserts d into the sorted bd[0..kK) (a NaN or a distance beyond the last leaves it unchanged).
__device__ __forceinline__ void insert_dist(float d, float (&bd)[kK]) {
    if (!(d < bd[kK - 1])) return;
#pragma unroll
    for (int k = kK - 1; k > 0; --k) bd[k] = fminf(bd[k], fmaxf(bd[k - 1], d));
    bd[0] = fminf(bd[0], d);
}

// A thread's table column: up to kK candidates (distance, index), unsorted, `stride` apart; once a further one came, its
// greatest pair and where that lies (-1 until then).
struct Found {
    uint2 *col;
    int stride, n;
    uint2 w;
    int worst;
};

__device__ __forceinline__ void find_worst(Found &f) {
    f.worst = 0;
    f.w = f.col[0];
    for (int k = 1; k < kK; ++k) {
        const uint2 c = f.col[k * f.stride];
        if (c.x > f.w.x || (c.x == f.w.x && c.y > f.w.y)) { f.w = c; f.worst = k; }
    }
}

// Adds (d, id); a full column replaces its greatest pair if (d, id) comes before it.
__device__ __forceinline__ void add_found(Found &f, float d, uint32_t id) {
    const uint32_t db = __float_as_uint(d);  // d >= 0: bit patterns order as the values do
    if (f.n < kK) {
        f.col[f.n * f.stride] = make_uint2(db, id);
        ++f.n;
        return;
    }
    if (f.worst < 0) find_worst(f);
    if (db > f.w.x || (db == f.w.x && id >= f.w.y)) return;  // ties of many centres end here
    f.col[f.worst * f.stride] = make_uint2(db, id);
    find_worst(f);
}

// The column sorted by (distance, index), as indices; missing entries -1.
__device__ __forceinline__ void sorted_indices(const Found &f, int32_t (&out)[kK]) {
    unsigned long long key[kK];
#pragma unroll
    for (int k = 0; k < kK; ++k) {
        const uint2 c = f.col[k * f.stride];
        key[k] = k < f.n ? ((unsigned long long)c.x << 32) | c.y : ~0ull;
    }
    batcher_sort(key);
#pragma unroll
    for (int k = 0; k < kK; ++k) out[k] = (int32_t)(uint32_t)key[k];
}

// each(candidate) for the centres spos[rg.x, rg.y), loaded two at a time so that their latencies overlap.
template <class Each>
__device__ __forceinline__ void for_centres(uint2 rg, const float4 *spos, Each &&each) {
    for (uint32_t q = rg.x; q < rg.y; q += 2) {
        const float4 o0 = __ldg(spos + q), o1 = __ldg(spos + min(q + 1u, rg.y - 1u));
        each(o0);
        if (q + 1u < rg.y) each(o1);
    }
}

// Lists of queries that would examine more than kQueryBudget centres: the best among the first
// kQueryBudget in ring order (coincident or non-finite centres only; kept out of the kernels' registers).
__device__ __noinline__ void ring_search_bounded(float4 p, const KnnGrid *gp, const uint32_t *starts, const float4 *spos,
                                                 int32_t *out) {
    float bd[kK];
    uint32_t bi[kK];
    ring_search(p, *gp, starts, spos, bd, bi);
    for (int k = 0; k < kK; ++k) out[k] = (int32_t)bi[k];
}

// sqrt with a relative error below 2^-20 on the safe side, for windows of cells.
__device__ __forceinline__ float sqrt_above(float x) {
    float y;
    asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y * (1.f + 1.f / 524288.f);
}

// The cells of a query point.
struct CellPoint {
    float4 p;
    int cx, cy, cz;
};

// Squared distance from q.p to row (y, z) of cells across x; 0 across its own slabs, which may reach past
// their box (an axis has at most 2,048 cells).
__device__ __forceinline__ float row_gap(const CellPoint &q, const KnnGrid &G, int y, int z) {
    const float gy = y == q.cy ? 0.f : slab_gap(G.lo[1], G.h, G.slack, q.p.y, y);
    const float gz = z == q.cz ? 0.f : slab_gap(G.lo[2], G.h, G.slack, q.p.z, z);
    return fmaf(gy, gy, gz * gz);
}

// The centres of the cells [x0, x1] of row (y, z) that lie within sqrt(left) of q.p along x.
__device__ __forceinline__ uint2 row_within(const CellPoint &q, const KnnGrid &G, const uint32_t *starts, int y, int z,
                                            int x0, int x1, float left) {
    // (the whole row where `left` is no number: an infinite bound less an infinite distance)
    const float w = fminf(sqrt_above(left), 3e38f) + G.slack;
    x0 = max(x0, min(cell_axis(q.p.x - w, G.lo[0], G.inv_h, G.dims[0]), q.cx));
    x1 = min(x1, max(cell_axis(q.p.x + w, G.lo[0], G.inv_h, G.dims[0]), q.cx));
    const int row = G.dims[0] * (y + G.dims[1] * z);
    return row_range(starts, row + x0, row + x1);
}

// First pass: the 27 cells around q's, then further rings (at most `rings` in all) until bd holds 16
// distances and the searched cells reach sqrt(reach) of the 16th in every open direction. The middle rows come
// first, so that the bound soon leaves most of the others out. Returns whether bd holds 16 distances. MANY: as many rings
// as it takes.
template <bool MANY>
__device__ __forceinline__ bool near_distances(const CellPoint &q, const KnnGrid &G, const uint32_t *starts,
                                               const float4 *spos, int rings, float reach, uint32_t &examined,
                                               float (&bd)[kK]) {
    // Many rings: their rows reach no further along an axis than the grid's farther end, and once the x faces of the
    // searched cells are outside the grid only a ring's outer rows are new. The rings of a query far from any others (a
    // line's outlier takes 2,048) would else run over thousands of rows each that are not there or searched already.
    const int most_y = MANY ? max(q.cy, G.dims[1] - 1 - q.cy) : 1 << 20, most_z = MANY ? max(q.cz, G.dims[2] - 1 - q.cz) : 1 << 20;
    for (int R = 1; R <= rings && examined <= kQueryBudget; ++R) {
        const int x0 = max(q.cx - R, 0), x1 = min(q.cx + R, G.dims[0] - 1);
        const bool outer = MANY && R > 1 && q.cx - R < 0 && q.cx + R >= G.dims[0];
        for (int zi = outer && R > most_y ? 2 * R - 1 : 0; zi <= 2 * min(R, most_z); ++zi) {
            const int z = q.cz + ((zi & 1) ? -((zi + 1) >> 1) : (zi >> 1));
            if (z < 0 || z >= G.dims[2]) continue;
            for (int yi = outer && abs(z - q.cz) < R ? 2 * R - 1 : 0; yi <= 2 * min(R, most_y); ++yi) {
                const int y = q.cy + ((yi & 1) ? -((yi + 1) >> 1) : (yi >> 1));
                if (y < 0 || y >= G.dims[1]) continue;
                const float left = bd[kK - 1] - row_gap(q, G, y, z);
                if (left < 0.f) continue;
                const bool inner = R > 1 && abs(z - q.cz) < R && abs(y - q.cy) < R;  // only the two x faces are new
                for (int side = 0; side < (inner ? 2 : 1); ++side) {
                    const int xa = !inner ? x0 : (side == 0 ? q.cx - R : q.cx + R), xb = !inner ? x1 : xa;
                    if (xa < 0 || xb >= G.dims[0]) continue;
                    const uint2 rg = row_within(q, G, starts, y, z, xa, xb, left);
                    examined += rg.y - rg.x;
                    if (examined > (MANY && R == 1 ? kTwoPassMost : kQueryBudget)) {
                        examined = kQueryBudget + 1u;
                        bd[kK - 1] = -1.f;  // given up: no further row is read
                        break;
                    }
                    for_centres(rg, spos, [&](float4 o) { insert_dist(dist2(q.p, o), bd); });
                }
            }
        }
        const bool full = bd[kK - 1] < __int_as_float(0x7f800000);
        float b = __int_as_float(0x7f800000);  // least distance to an open face of the searched cells
        bool all = true;
        auto face = [&](bool open, float g) {
            if (open) { b = fminf(b, g); all = false; }
        };
        face(q.cx - R > 0, q.p.x - (G.lo[0] + (float)(q.cx - R) * G.h));
        face(q.cx + R < G.dims[0] - 1, (G.lo[0] + (float)(q.cx + R + 1) * G.h) - q.p.x);
        face(q.cy - R > 0, q.p.y - (G.lo[1] + (float)(q.cy - R) * G.h));
        face(q.cy + R < G.dims[1] - 1, (G.lo[1] + (float)(q.cy + R + 1) * G.h) - q.p.y);
        face(q.cz - R > 0, q.p.z - (G.lo[2] + (float)(q.cz - R) * G.h));
        face(q.cz + R < G.dims[2] - 1, (G.lo[2] + (float)(q.cz + R + 1) * G.h) - q.p.z);
        b = fmaxf(b, 0.f);
        if (all || (full && reach * bd[kK - 1] <= b * b)) return full;
        if (!MANY && R > 1 && R < rings && examined == 0u) return false;  // empty space: blocks skip it
    }
    return bd[kK - 1] < __int_as_float(0x7f800000);
}

// Second pass: the centres within sqrt(bound) of q.p, from the rows of cells that the ball reaches.
__device__ __forceinline__ void ball_centres(const CellPoint &q, const KnnGrid &G, const uint32_t *starts,
                                             const float4 *spos, float bound, uint32_t &examined, Found &f) {
    const float rad = sqrt_above(bound) + G.slack;
    const int z0 = min(cell_axis(q.p.z - rad, G.lo[2], G.inv_h, G.dims[2]), q.cz),
              z1 = max(cell_axis(q.p.z + rad, G.lo[2], G.inv_h, G.dims[2]), q.cz),
              y0 = min(cell_axis(q.p.y - rad, G.lo[1], G.inv_h, G.dims[1]), q.cy),
              y1 = max(cell_axis(q.p.y + rad, G.lo[1], G.inv_h, G.dims[1]), q.cy);
    for (int z = z0; z <= z1; ++z)
        for (int y = y0; y <= y1; ++y) {
            const float left = bound - row_gap(q, G, y, z);
            if (left < 0.f) continue;
            const uint2 rg = row_within(q, G, starts, y, z, 0, G.dims[0] - 1, left);
            examined += rg.y - rg.x;
            if (examined > kQueryBudget) return;
            for_centres(rg, spos, [&](float4 o) {
                const float d = dist2(q.p, o);
                if (d <= bound) add_found(f, d, __float_as_uint(o.w));
            });
        }
}

__device__ __forceinline__ CellPoint cell_point(float4 p, const KnnGrid &G) {
    return CellPoint{p, cell_axis(p.x, G.lo[0], G.inv_h, G.dims[0]), cell_axis(p.y, G.lo[1], G.inv_h, G.dims[1]),
                     cell_axis(p.z, G.lo[2], G.inv_h, G.dims[2])};
}

// Whether a point has all coordinates: else no distance to it is a number, and its list stays empty.
__device__ __forceinline__ bool has_coordinates(float4 p) { return p.x == p.x && p.y == p.y && p.z == p.z; }

// Whether all distances from p overflow: they bound nothing, and the bounded searches, which then end with the first 16
// centres they meet, serve.
__device__ __forceinline__ bool all_infinite(float4 p, const KnnGrid &G) {
    const float pc[3] = {p.x, p.y, p.z};
    float d2 = 0.f;  // squared distance to the grid's box
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        const float g = fmaxf(fmaxf(G.lo[k] - G.slack - pc[k], pc[k] - (G.lo[k] + (float)G.dims[k] * G.h + G.slack)), 0.f);
        d2 = fmaf(g, g, d2);
    }
    return !(d2 < __int_as_float(0x7f800000));
}

__global__ void __launch_bounds__(kQueryThreads, kQueryCtas) k_knn_query(const float4 *spos, const uint32_t *starts,
                                                                         const KnnGrid *gp, int n, int32_t *knn) {
    __shared__ uint2 s_found[kK][kQueryThreads];
    const int r = blockIdx.x * blockDim.x + threadIdx.x;
    if (r >= n) return;
    const float4 p = spos[r];
    int32_t *out = knn + (size_t)__float_as_uint(p.w) * kK;
    const KnnGrid G = *gp;
    const CellPoint q = cell_point(p, G);
    float bd[kK];
#pragma unroll
    for (int k = 0; k < kK; ++k) bd[k] = __int_as_float(0x7f800000);
    uint32_t examined = 0;
    Found f = {&s_found[0][threadIdx.x], kQueryThreads, 0, make_uint2(0u, 0u), -1};
    if (all_infinite(p, G)) {
        examined = kQueryBudget + 1u;
    } else if (has_coordinates(p)) {
        near_distances<true>(q, G, starts, spos, 1 << 20, kReach, examined, bd);
        if (examined <= kQueryBudget) {
            examined = 0;
            ball_centres(q, G, starts, spos, bd[kK - 1], examined, f);
        }
    }
    if (examined > kQueryBudget) {
        ring_search_bounded(p, gp, starts, spos, out);
        return;
    }
    int32_t idx[kK];
    sorted_indices(f, idx);
#pragma unroll
    for (int k = 0; k < kK; ++k) out[k] = idx[k];
}

// Cell keys of query points (w = 0: no query, sorted after every cell).
__global__ void __launch_bounds__(256) k_knn_point_keys(const float4 *pts, int m, const KnnGrid *g, uint32_t none,
                                                        uint32_t *keys) {
    const int r = blockIdx.x * blockDim.x + threadIdx.x;
    if (r >= m) return;
    const float4 p = pts[r];
    const KnnGrid G = *g;
    keys[r] = p.w == 0.f ? none
                         : (uint32_t)(cell_axis(p.x, G.lo[0], G.inv_h, G.dims[0]) +
                                      G.dims[0] * (cell_axis(p.y, G.lo[1], G.inv_h, G.dims[1]) +
                                                   G.dims[1] * cell_axis(p.z, G.lo[2], G.inv_h, G.dims[2])));
}

// Walks Chebyshev rings of blocks around q's block and calls scan(range) for the centres of every row of
// a block's cells that lies within bound() of q.p, cut to it along x: a block whose box lies farther, or
// that holds no centre, costs one test and at most one count read. Stops after
// the ring `rings`, or when the searched blocks enclose everything within bound(). Returns the last ring.
template <class Bound, class Scan>
__device__ __forceinline__ int block_walk(const CellPoint &q, const KnnGrid &G, const uint32_t *starts, const uint32_t *bcount,
                                          int rings, Bound &&bound, Scan &&scan) {
    const int dx = G.dims[0], dy = G.dims[1], dz = G.dims[2];
    const int bx_n = block_dim(dx), by_n = block_dim(dy), bz_n = block_dim(dz);
    const int cbx = q.cx >> kBlockShift, cby = q.cy >> kBlockShift, cbz = q.cz >> kBlockShift;
    const float4 p = q.p;
    const float h = G.h, H = (float)kBlockSide * G.h, sl = G.slack;
    const float lx = G.lo[0], ly = G.lo[1], lz = G.lo[2];
    // no gap to p's own slab, which may reach past its box (an axis has at most 2,048 cells)
    auto gap = [&](float lo, float w, float x, int i, int own) { return i == own ? 0.f : slab_gap(lo, w, sl, x, i); };
    // distance from p to the grid's box along each axis
    const float ox = fmaxf(fmaxf(lx - sl - p.x, p.x - (lx + (float)dx * h + sl)), 0.f);
    const float oy = fmaxf(fmaxf(ly - sl - p.y, p.y - (ly + (float)dy * h + sl)), 0.f);
    const float oz = fmaxf(fmaxf(lz - sl - p.z, p.z - (lz + (float)dz * h + sl)), 0.f);
    int ring = 0;
    for (;; ++ring) {
        const int z0 = max(cbz - ring, 0), z1 = min(cbz + ring, bz_n - 1);
        const int y0 = max(cby - ring, 0), y1 = min(cby + ring, by_n - 1);
        const int x0 = max(cbx - ring, 0), x1 = min(cbx + ring, bx_n - 1);
        auto visit = [&](int bx, int by, int bz, float gyz) {
            const float gx = gap(lx, H, p.x, bx, cbx);
            if (fmaf(gx, gx, gyz) > bound()) return;
            if (__ldg(bcount + (bx + bx_n * (by + by_n * bz))) == 0u) return;
            const int fz1 = min((bz + 1) << kBlockShift, dz), fy1 = min((by + 1) << kBlockShift, dy),
                      fx1 = min((bx + 1) << kBlockShift, dx) - 1;
            for (int fz = bz << kBlockShift; fz < fz1; ++fz)
                for (int fy = by << kBlockShift; fy < fy1; ++fy) {
                    const float left = bound() - row_gap(q, G, fy, fz);
                    if (left < 0.f) continue;
                    scan(row_within(q, G, starts, fy, fz, bx << kBlockShift, fx1, left));
                }
        };
        for (int bz = z0; bz <= z1; ++bz) {
            const float gz = gap(lz, H, p.z, bz, cbz);
            if (gz * gz > bound()) continue;
            for (int by = y0; by <= y1; ++by) {
                const float gy = gap(ly, H, p.y, by, cby);
                const float gyz = fmaf(gy, gy, gz * gz);
                if (gyz > bound()) continue;
                if (abs(bz - cbz) < ring && abs(by - cby) < ring) {  // only the two x faces are new
                    if (cbx - ring >= 0) visit(cbx - ring, by, bz, gyz);
                    if (cbx + ring < bx_n) visit(cbx + ring, by, bz, gyz);
                } else {
                    for (int bx = x0; bx <= x1; ++bx) visit(bx, by, bz, gyz);
                }
            }
        }
        if (ring >= rings) break;
        // least distance to the grid's box beyond the searched blocks' open faces
        float b2 = __int_as_float(0x7f800000);
        bool all = true;
        auto face = [&](bool open, float g, float o1, float o2) {
            if (!open) return;
            g = fmaxf(g - sl, 0.f);
            b2 = fminf(b2, fmaf(g, g, fmaf(o1, o1, o2 * o2)));
            all = false;
        };
        face(cbx - ring > 0, p.x - (lx + (float)(cbx - ring) * H), oy, oz);
        face(cbx + ring < bx_n - 1, (lx + (float)(cbx + ring + 1) * H) - p.x, oy, oz);
        face(cby - ring > 0, p.y - (ly + (float)(cby - ring) * H), ox, oz);
        face(cby + ring < by_n - 1, (ly + (float)(cby + ring + 1) * H) - p.y, ox, oz);
        face(cbz - ring > 0, p.z - (lz + (float)(cbz - ring) * H), ox, oy);
        face(cbz + ring < bz_n - 1, (lz + (float)(cbz + ring + 1) * H) - p.z, ox, oy);
        if (all) break;
        if (bound() < __int_as_float(0x7f800000) && bound() <= b2 * (1.f - 1.f / 1048576.f)) break;
    }
    return ring;
}

// As ring_search_bounded, for point queries.
__device__ __noinline__ void block_search_bounded(float4 p, const KnnGrid *gp, const uint32_t *starts,
                                                  const float4 *spos, int32_t *out) {
    float bd[kK];
    uint32_t bi[kK];
    block_search(p, *gp, starts, spos, bd, bi);
    for (int k = 0; k < kK; ++k) out[k] = (int32_t)bi[k];
}

// Queries at arbitrary points, taken in cell order (order[r]: the r-th query by cell), so a
// warp searches one neighbourhood; w = 0: no query, the list is all -1.
__global__ void __launch_bounds__(kQueryThreads, kQueryCtas) k_knn_points(const float4 *spos, const uint32_t *starts,
                                                                          const uint32_t *bcount, const KnnGrid *gp,
                                                                          const float4 *pts, const uint32_t *order,
                                                                          int m, int32_t *knn) {
    __shared__ uint2 s_found[kK][kQueryThreads];
    const int r0 = blockIdx.x * blockDim.x + threadIdx.x;
    if (r0 >= m) return;
    const uint32_t r = __ldg(order + r0);
    const float4 p = pts[r];
    int4 *out = reinterpret_cast<int4 *>(knn + (size_t)r * kK);
    Found f = {&s_found[0][threadIdx.x], kQueryThreads, 0, make_uint2(0u, 0u), -1};
    if (p.w != 0.f && has_coordinates(p)) {
        const KnnGrid G = *gp;
        if (all_infinite(p, G)) {
            block_search_bounded(p, gp, starts, spos, reinterpret_cast<int32_t *>(out));
            return;
        }
        float bd[kK];
#pragma unroll
        for (int k = 0; k < kK; ++k) bd[k] = __int_as_float(0x7f800000);
        uint32_t examined = 0;
        const CellPoint q = cell_point(p, G);
        // most queries lie within a few cells of 16 centres; the others walk blocks, which skip empty space
        const bool near = near_distances<false>(q, G, starts, spos, kNearRings, kReach, examined, bd);
        int rings = 0;
        if (!near && examined <= kQueryBudget) {
#pragma unroll
            for (int k = 0; k < kK; ++k) bd[k] = __int_as_float(0x7f800000);
            examined = 0;
            rings = block_walk(
                q, G, starts, bcount, max(max(G.dims[0], G.dims[1]), G.dims[2]), [&]() { return bd[kK - 1]; },
                [&](uint2 rg) {
                    examined += rg.y - rg.x;
                    if (examined > kQueryBudget) {  // given up: the walk ends (it would read every row of the
                        bd[kK - 1] = -1.f;          // grid where the distances never narrow the bound)
                        return;
                    }
                    for_centres(rg, spos, [&](float4 o) { insert_dist(dist2(p, o), bd); });
                });
        }
        const float bound = bd[kK - 1];
        if (examined <= kQueryBudget) {
            examined = 0;
            if (near)
                ball_centres(q, G, starts, spos, bound, examined, f);
            else
                block_walk(q, G, starts, bcount, rings, [&]() { return bound; },
                           [&](uint2 rg) {
                               for_centres(rg, spos, [&](float4 o) {
                                   const float d = dist2(p, o);
                                   if (d <= bound) add_found(f, d, __float_as_uint(o.w));
                               });
                           });
        }
        if (examined > kQueryBudget) {
            block_search_bounded(p, gp, starts, spos, reinterpret_cast<int32_t *>(out));
            return;
        }
    }
    int32_t idx[kK];
    sorted_indices(f, idx);
#pragma unroll
    for (int k = 0; k < kK; k += 4) out[k / 4] = make_int4(idx[k], idx[k + 1], idx[k + 2], idx[k + 3]);
}

// Cell sort of m query points, after the grid's own workspace.
struct KnnQueryLayout {
    uint64_t keys0, keys1, vals0, vals1, hist, partials, bytes;
    uint32_t nblocks;
    int bits;
};

KnnQueryLayout knn_query_layout(uint32_t cap_cells, int32_t m) {
    KnnQueryLayout Q;
    Q.bits = 1;
    while ((1ull << Q.bits) <= cap_cells) ++Q.bits;  // every cell index and the "no query" key fit
    Q.nblocks = ceil_div_u64(m > 0 ? (uint64_t)m : 1, kSortTile);
    uint64_t off = 0;
    Q.keys0 = off; off = al256(off + 4ull * m);
    Q.keys1 = off; off = al256(off + 4ull * m);
    Q.vals0 = off; off = al256(off + 4ull * m);
    Q.vals1 = off; off = al256(off + 4ull * m);
    Q.hist = off; off = al256(off + 4ull * 256 * Q.nblocks);
    Q.partials = off; off = al256(off + 4ull * (ceil_div_u64(256ull * Q.nblocks, kScanTile) + 1));
    Q.bytes = off;
    return Q;
}

template <class T>
T *at(void *base, uint64_t off) {
    return reinterpret_cast<T *>(static_cast<char *>(base) + off);
}

}  // namespace
}  // namespace ges

using namespace ges;

extern "C" size_t ges_knn_workspace_bytes(int32_t n) {
    if (n < GES_KNN_K || (uint64_t)n > (1ull << 26)) return 0;
    return knn_layout(n).bytes;
}

namespace ges {

// Grid, cell sort and cell-ordered centres of n splats in `workspace` (knn_layout(n).bytes).
static cudaError_t knn_build(int32_t n, const float4 *pos, void *workspace, const KnnLayout &L, cudaStream_t s) {
    uint32_t *bb = at<uint32_t>(workspace, L.bbox);
    KnnGrid *grid = at<KnnGrid>(workspace, L.grid);
    cudaError_t e = cudaMemsetAsync(bb, 0xff, 12, s);
    if (e == cudaSuccess) e = cudaMemsetAsync(bb + 3, 0, 12, s);
    uint32_t *starts = at<uint32_t>(workspace, L.starts);
    if (e == cudaSuccess) e = cudaMemsetAsync(starts, 0, 4ull * (L.cap_cells + 1ull), s);
    if (e == cudaSuccess) e = cudaMemsetAsync(at<void>(workspace, L.bcount), 0, 4ull * L.cap_cells, s);
    if (e != cudaSuccess) return e;
    k_knn_bbox<<<min(ceil_div_u64(n, 1024), 608u), 256, 0, s>>>(pos, n, bb);
    k_knn_grid<<<1, 1, 0, s>>>(bb, L.cap_cells, grid);
    uint32_t *keys[2] = {at<uint32_t>(workspace, L.keys0), at<uint32_t>(workspace, L.keys1)};
    uint32_t *vals[2] = {at<uint32_t>(workspace, L.vals0), at<uint32_t>(workspace, L.vals1)};
    k_knn_keys<<<ceil_div_u64(n, 256), 256, 0, s>>>(pos, n, grid, keys[0], starts, at<uint32_t>(workspace, L.bcount));
    // cell counts -> first centre of each cell, and the end
    e = exclusive_scan(starts, starts, L.cap_cells + 1u, at<uint32_t>(workspace, L.partials), s);
    if (e != cudaSuccess) return e;
    e = radix_sort(keys, vals, (uint32_t)n, L.bits, at<uint32_t>(workspace, L.hist),
                   at<uint32_t>(workspace, L.partials), s);
    if (e != cudaSuccess) return e;
    const int res = ((L.bits + 7) / 8) & 1;
    k_knn_gather<<<ceil_div_u64(n, 256), 256, 0, s>>>(vals[res], pos, n, at<float4>(workspace, L.spos));
    return cudaGetLastError();
}

// Workspace of knn_points_run: the grid of n centres, then the cell sort of m queries.
size_t knn_points_workspace(int32_t n, int32_t m) {
    const KnnLayout L = knn_layout(n);
    return L.bytes + knn_query_layout(L.cap_cells, m).bytes;
}

// The 16 nearest centres of m points (pts[i].w = 0: none, list -1) into knn [m][16]
// (16-byte aligned); workspace: knn_points_workspace(n, m) bytes, 256-byte aligned.
cudaError_t knn_points_run(int32_t n, const float4 *pos, int32_t m, const float4 *pts, void *workspace,
                           int32_t *knn, cudaStream_t s) {
    const KnnLayout L = knn_layout(n);
    cudaError_t e = knn_build(n, pos, workspace, L, s);
    if (e != cudaSuccess || m <= 0) return e;
    const KnnQueryLayout Q = knn_query_layout(L.cap_cells, m);
    void *qws = static_cast<char *>(workspace) + L.bytes;
    uint32_t *keys[2] = {at<uint32_t>(qws, Q.keys0), at<uint32_t>(qws, Q.keys1)};
    uint32_t *vals[2] = {at<uint32_t>(qws, Q.vals0), at<uint32_t>(qws, Q.vals1)};
    k_knn_point_keys<<<ceil_div_u64(m, 256), 256, 0, s>>>(pts, m, at<KnnGrid>(workspace, L.grid),
                                                          (uint32_t)((1ull << Q.bits) - 1), keys[0]);
    e = radix_sort(keys, vals, (uint32_t)m, Q.bits, at<uint32_t>(qws, Q.hist),
                   at<uint32_t>(qws, Q.partials), s);
    if (e != cudaSuccess) return e;
    const int res = ((Q.bits + 7) / 8) & 1;
    k_knn_points<<<ceil_div_u64(m, kQueryThreads), kQueryThreads, 0, s>>>(at<float4>(workspace, L.spos), at<uint32_t>(workspace, L.starts),
                                                     at<uint32_t>(workspace, L.bcount), at<KnnGrid>(workspace, L.grid),
                                                     pts, vals[res], m, knn);
    return cudaGetLastError();
}

}  // namespace ges

extern "C" ges_status ges_knn(int32_t n, const float *pos_op, void *workspace, size_t workspace_bytes, int32_t *knn,
                              void *stream) {
    GES_RANGE();
    if (n < GES_KNN_K || (uint64_t)n > (1ull << 26) || !pos_op || !workspace || !knn) return GES_ERR_INVALID_ARG;
    if (((uintptr_t)pos_op & 15u) || ((uintptr_t)workspace & 255u) || ((uintptr_t)knn & 3u))
        return GES_ERR_INVALID_ARG;
    const KnnLayout L = knn_layout(n);
    if (workspace_bytes < L.bytes) return GES_ERR_INVALID_ARG;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    const float4 *pos = reinterpret_cast<const float4 *>(pos_op);
    if (knn_build(n, pos, workspace, L, s) != cudaSuccess) return GES_ERR_CUDA;
    k_knn_query<<<ceil_div_u64(n, kQueryThreads), kQueryThreads, 0, s>>>(at<float4>(workspace, L.spos), at<uint32_t>(workspace, L.starts),
                                                    at<KnnGrid>(workspace, L.grid), n, knn);
    return cudaGetLastError() == cudaSuccess ? GES_OK : GES_ERR_CUDA;
}

extern "C" size_t ges_knn_points_workspace_bytes(int32_t n, int32_t m) {
    if (n < GES_KNN_K || (uint64_t)n > (1ull << 26) || m < 1 || (uint64_t)m > (1ull << 28)) return 0;
    return knn_points_workspace(n, m);
}

extern "C" ges_status ges_knn_points(int32_t n, const float *pos_op, int32_t m, const float *points,
                                     void *workspace, size_t workspace_bytes, int32_t *knn, void *stream) {
    GES_RANGE();
    if (n < GES_KNN_K || (uint64_t)n > (1ull << 26) || m < 1 || (uint64_t)m > (1ull << 28)) return GES_ERR_INVALID_ARG;
    if (!pos_op || !points || !workspace || !knn) return GES_ERR_INVALID_ARG;
    if (((uintptr_t)pos_op & 15u) || ((uintptr_t)points & 15u) || ((uintptr_t)workspace & 255u) ||
        ((uintptr_t)knn & 15u))
        return GES_ERR_INVALID_ARG;
    if (workspace_bytes < knn_points_workspace(n, m)) return GES_ERR_INVALID_ARG;
    return knn_points_run(n, reinterpret_cast<const float4 *>(pos_op), m, reinterpret_cast<const float4 *>(points),
                          workspace, knn, static_cast<cudaStream_t>(stream)) == cudaSuccess
               ? GES_OK
               : GES_ERR_CUDA;
}
