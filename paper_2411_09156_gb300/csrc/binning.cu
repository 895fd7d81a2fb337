// S5 binning (tile lists in depth order), and the scan and the stable LSD radix sort
// (reduce-then-scan, 8-bit digits) that the KNN grid uses.
//
// Binning: the instances of every tile are counted, the counts scanned into segments, the instances
// appended to their tile's segment in any order, and each segment sorted by (depth, entry) where it fits: in a
// warp's, a part's or a whole CTA's shared memory, after a split by depth where it does not. All counts stay in device
// memory, so the chain runs without a host round trip and can be captured in a CUDA graph.
// What bounds it: the scattered 8-byte appends and the sorts' shared-memory traffic (8 views of 1.5M splats of a
// heightfield, 34.7M instances: 410 and 400 us of 1,035). The whole call as a graph against a depth sort of all entries
// and a stable tile sort of all instances by radix passes: 1,000 splats at 128x128 26 us (95); 100k at 800x800 56 (131);
// 1.5M at 1600x1040 271 (313); 4 views of 300k 163 (217); 8 of 1.5M 1,035 (1,490). Objects, whose tiles differ most
// in length: 3 views of 170k 136 (157); 8 of 600k 454 (594). Slower where most instances lie in lists of thousands, and
// one view's segments outgrow L2: 2M splats of an object at 1600x1040 595 (517) in 16x16 tiles, 1,012 (732) in 16x8;
// 8 views of 1.5M 2,127 (2,084).
#include <cooperative_groups.h>

#include "ges_internal.cuh"
#include "sort_net.cuh"
#include "tile_tests.cuh"

namespace ges {

// ------------------------------------------------------------------ scan
// Exclusive scan of n uint32 in three launches: tile sums, one-CTA scan of the
// tile sums, tile scans offset by the scanned sums. In place is allowed.
__device__ __forceinline__ uint32_t warp_incl_scan(uint32_t v) {
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        uint32_t t = __shfl_up_sync(0xffffffffu, v, o);
        if (lane >= o) v += t;
    }
    return v;
}

// Exclusive block scan of one value per thread (blockDim.x multiple of 32, <= 1024).
__device__ __forceinline__ uint32_t block_excl_scan(uint32_t v, uint32_t *s_warp, uint32_t &total) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    uint32_t incl = warp_incl_scan(v);
    if (lane == 31) s_warp[warp] = incl;
    __syncthreads();
    if (warp == 0) {
        uint32_t w = lane < nw ? s_warp[lane] : 0u;
        uint32_t wi = warp_incl_scan(w);
        if (lane < nw) s_warp[lane] = wi - w;
        if (lane == 31) s_warp[32] = wi;
    }
    __syncthreads();
    uint32_t r = incl - v + s_warp[warp];
    total = s_warp[32];
    __syncthreads();
    return r;
}

__global__ void __launch_bounds__(256) k_scan_reduce(const uint32_t *in, uint32_t n, uint32_t *partials) {
    __shared__ uint32_t s_warp[33];
    const uint64_t base = (uint64_t)blockIdx.x * kScanTile;
    uint32_t sum = 0;
#pragma unroll 4
    for (int k = 0; k < kScanTile / 256; ++k) {
        uint64_t idx = base + (uint64_t)k * 256 + threadIdx.x;
        if (idx < n) sum += in[idx];
    }
    uint32_t tot;
    block_excl_scan(sum, s_warp, tot);
    if (threadIdx.x == 0) partials[blockIdx.x] = tot;
}

// One CTA of 1024 threads scans up to kScanMaxPartials tile sums.
__global__ void __launch_bounds__(1024) k_scan_partials(uint32_t *partials, uint32_t np) {
    __shared__ uint32_t s_warp[33];
    constexpr int PER = kScanMaxPartials / 1024;
    uint32_t v[PER];
    uint32_t s = 0;
#pragma unroll
    for (int k = 0; k < PER; ++k) {
        uint32_t idx = threadIdx.x * PER + k;
        v[k] = idx < np ? partials[idx] : 0u;
        s += v[k];
    }
    uint32_t tot;
    uint32_t run = block_excl_scan(s, s_warp, tot);
#pragma unroll
    for (int k = 0; k < PER; ++k) {
        uint32_t idx = threadIdx.x * PER + k;
        if (idx < np) partials[idx] = run;
        run += v[k];
    }
}

__global__ void __launch_bounds__(256) k_scan_down(const uint32_t *in, uint32_t *out, uint32_t n,
                                                  const uint32_t *partials) {
    __shared__ uint32_t s_data[kScanTile + kScanTile / 32];
    __shared__ uint32_t s_warp[33];
    const uint64_t base = (uint64_t)blockIdx.x * kScanTile;
    constexpr int PER = kScanTile / 256;  // 16
#pragma unroll
    for (int k = 0; k < PER; ++k) {
        uint32_t li = k * 256 + threadIdx.x;
        uint64_t idx = base + li;
        s_data[li + (li >> 5)] = idx < n ? in[idx] : 0u;
    }
    __syncthreads();
    uint32_t v[PER];
    uint32_t s = 0;
#pragma unroll
    for (int k = 0; k < PER; ++k) {
        uint32_t li = threadIdx.x * PER + k;
        v[k] = s_data[li + (li >> 5)];
        s += v[k];
    }
    uint32_t tot;
    uint32_t run = block_excl_scan(s, s_warp, tot) + partials[blockIdx.x];
#pragma unroll
    for (int k = 0; k < PER; ++k) {
        uint32_t li = threadIdx.x * PER + k;
        s_data[li + (li >> 5)] = run;
        run += v[k];
    }
    __syncthreads();
#pragma unroll
    for (int k = 0; k < PER; ++k) {
        uint32_t li = k * 256 + threadIdx.x;
        uint64_t idx = base + li;
        if (idx < n) out[idx] = s_data[li + (li >> 5)];
    }
}

cudaError_t exclusive_scan(const uint32_t *in, uint32_t *out, uint32_t n, uint32_t *partials, cudaStream_t s) {
    if (n == 0) return cudaSuccess;
    const uint32_t nb = ceil_div_u64(n, kScanTile);
    if (nb > (uint32_t)kScanMaxPartials) return cudaErrorInvalidValue;
    k_scan_reduce<<<nb, 256, 0, s>>>(in, n, partials);
    k_scan_partials<<<1, 1024, 0, s>>>(partials, nb);
    k_scan_down<<<nb, 256, 0, s>>>(in, out, n, partials);
    return cudaGetLastError();
}

// ------------------------------------------------------------------ radix sort
__global__ void __launch_bounds__(kSortThreads) k_radix_hist(const uint32_t *keys, uint32_t n, int shift,
                                                            uint32_t nblocks, uint32_t *hist) {
    __shared__ uint32_t s_h[kSortThreads / 32][256];
    const int warp = threadIdx.x >> 5;
    for (int k = threadIdx.x; k < (kSortThreads / 32) * 256; k += kSortThreads) (&s_h[0][0])[k] = 0u;
    __syncthreads();
    const uint64_t base = (uint64_t)blockIdx.x * kSortTile;
    if (base < n) {
        uint32_t kk[kSortItems];
#pragma unroll
        for (int k = 0; k < kSortItems; ++k) {
            const uint64_t idx = base + (uint64_t)k * kSortThreads + threadIdx.x;
            kk[k] = idx < n ? __ldg(keys + idx) : 0xffffffffu;
        }
#pragma unroll
        for (int k = 0; k < kSortItems; ++k) {
            const uint64_t idx = base + (uint64_t)k * kSortThreads + threadIdx.x;
            if (idx < n) atomicAdd(&s_h[warp][(kk[k] >> shift) & 0xffu], 1u);
        }
    }
    __syncthreads();
    const int d = threadIdx.x;  // kSortThreads == 256 digits
    uint32_t c = 0;
#pragma unroll
    for (int w = 0; w < kSortThreads / 32; ++w) c += s_h[w][d];
    hist[(uint64_t)d * nblocks + blockIdx.x] = c;
}

// Stable scatter: each warp ranks a contiguous 512-key chunk in rounds of 32 with
// digit ballots, keeping a per-warp running count per digit; warps are then ordered by
// an exclusive prefix per digit. The CTA's 4096 pairs are first reordered by digit
// in shared memory, then written out in digit runs (coalesced) at the offsets of
// the scanned digit-major histogram.
__global__ void __launch_bounds__(kSortThreads, 3) k_radix_scatter(const uint32_t *keys_in, const uint32_t *vals_in,
                                                               uint32_t *keys_out, uint32_t *vals_out,
                                                               uint32_t n, int shift, uint32_t nblocks,
                                                               const uint32_t *hist_scanned) {
    constexpr int NW = kSortThreads / 32;
    __shared__ uint32_t s_cnt[NW][256];
    __shared__ uint32_t s_dstart[256], s_gstart[256];
    __shared__ uint32_t s_warp[33];
    __shared__ uint32_t s_keys[kSortTile], s_vals[kSortTile];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (int k = threadIdx.x; k < NW * 256; k += kSortThreads) (&s_cnt[0][0])[k] = 0u;
    __syncthreads();
    const uint64_t base = (uint64_t)blockIdx.x * kSortTile;
    if (base >= n) return;  // uniform for the CTA
    const uint32_t nvalid = (uint32_t)min((uint64_t)kSortTile, (uint64_t)n - base);
    const uint64_t wbase = base + (uint64_t)warp * (kSortItems * 32);
    const uint32_t lt_mask = (1u << lane) - 1u;
    uint32_t key[kSortItems], val[kSortItems], rank[kSortItems];
    // all loads first, so that the 16 rounds' reads are in flight together
#pragma unroll
    for (int r = 0; r < kSortItems; ++r) {
        const uint64_t idx = wbase + (uint64_t)r * 32 + lane;
        const bool valid = idx < n;
        key[r] = valid ? __ldg(keys_in + idx) : 0u;
        val[r] = valid ? (vals_in ? __ldg(vals_in + idx) : (uint32_t)idx) : 0u;
    }
#pragma unroll
    for (int r = 0; r < kSortItems; ++r) {
        const uint64_t idx = wbase + (uint64_t)r * 32 + lane;
        const bool valid = idx < n;
        const uint32_t d = (key[r] >> shift) & 0xffu;
        // lanes holding the same digit (invalid lanes carry 0x100): one ballot per digit
        // bit, which issues faster than match.any on spread-out digits
        const uint32_t dd = valid ? d : 0x100u;
        uint32_t peers = 0xffffffffu;
#pragma unroll
        for (int b = 0; b < 9; ++b) {
            const uint32_t bal = __ballot_sync(0xffffffffu, (dd >> b) & 1u);
            peers &= ((dd >> b) & 1u) ? bal : ~bal;
        }
        uint32_t before = 0;
        if (valid) before = s_cnt[warp][d];
        __syncwarp();
        if (valid && (peers & lt_mask) == 0) s_cnt[warp][d] = before + __popc(peers);
        __syncwarp();
        rank[r] = valid ? before + __popc(peers & lt_mask) : 0xffffffffu;
    }
    __syncthreads();
    {
        // digit d = thread: block count, block-local start (exclusive scan over digits),
        // per-warp offsets inside the digit, and the digit's global start for this CTA
        const int d = threadIdx.x;
        uint32_t c = 0;
#pragma unroll
        for (int w = 0; w < NW; ++w) c += s_cnt[w][d];
        uint32_t tot;
        const uint32_t start = block_excl_scan(c, s_warp, tot);
        s_dstart[d] = start;
        s_gstart[d] = hist_scanned[(uint64_t)d * nblocks + blockIdx.x];
        uint32_t run = start;
#pragma unroll
        for (int w = 0; w < NW; ++w) {
            const uint32_t t = s_cnt[w][d];
            s_cnt[w][d] = run;
            run += t;
        }
    }
    __syncthreads();
#pragma unroll
    for (int r = 0; r < kSortItems; ++r) {
        if (rank[r] == 0xffffffffu) continue;
        const uint32_t d = (key[r] >> shift) & 0xffu;
        const uint32_t lpos = s_cnt[warp][d] + rank[r];
        s_keys[lpos] = key[r];
        s_vals[lpos] = val[r];
    }
    __syncthreads();
    for (uint32_t i = threadIdx.x; i < nvalid; i += kSortThreads) {
        const uint32_t k = s_keys[i];
        const uint32_t d = (k >> shift) & 0xffu;
        const uint32_t pos = s_gstart[d] + (i - s_dstart[d]);
        keys_out[pos] = k;
        vals_out[pos] = s_vals[i];
    }
}

// Sorts (keys[0][i], i) on key bits [0, bits) with ceil(bits/8) passes, ping-ponging
// between buffer 0 and 1; the result lands in buffer (passes % 2).
cudaError_t radix_sort(uint32_t *keys[2], uint32_t *vals[2], uint32_t n, int bits, uint32_t *hist,
                       uint32_t *partials, cudaStream_t s) {
    const uint32_t nblocks = ceil_div_u64(n > 0 ? n : 1, kSortTile);
    const int passes = (bits + 7) / 8;
    for (int p = 0; p < passes; ++p) {
        const int in = p & 1, out = in ^ 1;
        const int shift = 8 * p;
        k_radix_hist<<<nblocks, kSortThreads, 0, s>>>(keys[in], n, shift, nblocks, hist);
        cudaError_t e = exclusive_scan(hist, hist, 256u * nblocks, partials, s);
        if (e != cudaSuccess) return e;
        k_radix_scatter<<<nblocks, kSortThreads, 0, s>>>(keys[in], p == 0 ? nullptr : vals[in], keys[out], vals[out], n,
                                                        shift, nblocks, hist);
    }
    return cudaGetLastError();
}

// ------------------------------------------------------------------ binning
// Position of the k-th (0-based) set bit of m; m has more than k set bits.
__device__ __forceinline__ uint32_t select_bit(uint32_t m, uint32_t k) {
    uint32_t pos = 0;
#pragma unroll
    for (int s = 16; s > 0; s >>= 1) {
        const uint32_t lo = m & ((1u << s) - 1u);
        const uint32_t c = (uint32_t)__popc(lo);
        if (k >= c) { k -= c; m >>= s; pos += s; } else { m = lo; }
    }
    return pos;
}

// The tile tests of entry e of view v (box in binrec's first half b0).
__device__ __forceinline__ TileJob tile_job(const BinArgs &a, int v, size_t e, const uint4 b0, int lw, int lh) {
    TileJob J = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0u, 0u, 0u};
    const float4 r0 = a.rec[4 * e], r1 = a.rec[4 * e + 1];
    int x0, x1, y0, y1;
    pixel_box(r0.x, r0.y, __uint_as_float(b0.x), __uint_as_float(b0.y), a.V.width[v], a.V.height[v], x0, x1, y0, y1);
    if (x0 <= x1 && y0 <= y1)
        J = TileJob{r0.x, r0.y, r0.z, r0.w, r1.x, __frcp_rn(r0.z), __frcp_rn(r1.x), __fmul_rn(r1.y, kSupportMargin),
                    (uint32_t)x0 | ((uint32_t)x1 << 16), (uint32_t)y0 | ((uint32_t)y1 << 16),
                    (uint32_t)((x1 >> lw) - (x0 >> lw) + 1) * (uint32_t)((y1 >> lh) - (y0 >> lh) + 1)};
    return J;
}

// First kernel of a ges_bin: clears the header and the counters and, if there are more instances than the capacity, finds where the
// lists end: the instances kept are the first `cap` of all in the order of (depth, entry, tile), so what is lost is the
// farthest of every view. A radix selection over the entries' 64-bit keys (depth, entry), weighted by their tiles, by
// the CTAs of one cluster, whose barrier and shared memory it needs; it leaves in the header the key of the entry
// that the capacity cuts, the first tile that this entry loses, and a 1 (header zero: nothing is cut).
// Without an overflow it costs about what the memory clear that it replaced did (2.6 us; the whole binning of a
// 1.5M-splat view 280 -> 286 us with it and the ordered queue); with one, six passes over the records by one cluster
// (8 views of 1.5M splats: 6 ms of binning instead of 1.2; one 100k-splat view: 139 us instead of 80).
constexpr int kCutCtas = 8;
__global__ void __cluster_dims__(kCutCtas, 1, 1) __launch_bounds__(1024) k_bin_begin(const BinArgs a, uint4 *clear,
                                                                                     uint64_t n_clear) {
    const uint32_t t = threadIdx.x, lane = t & 31u, rank = blockIdx.x;
    if (rank == 0 && t < 64u) a.header[t] = 0u;  // (written further only by this CTA, past a barrier)
    for (uint64_t i = rank * 1024u + t; i < n_clear; i += kCutCtas * 1024u) clear[i] = make_uint4(0u, 0u, 0u, 0u);
    const unsigned long long total = *a.total;
    if (total <= a.cap || total >= 0xffffffffull) return;  // the same for the cluster
    constexpr int kDigit = 11, kBins = 1 << kDigit;
    __shared__ uint32_t s_bins[kBins], s_warp[33], s_digit, s_before;
    __shared__ uint4 s_jobs[kJobWords * 32];
    namespace cg = cooperative_groups;
    cg::cluster_group cluster = cg::this_cluster();
    const uint64_t n_entries = (uint64_t)a.n * (uint64_t)a.n_views;
    unsigned long long prefix = 0;
    uint32_t left = (uint32_t)a.cap;  // instances kept among the keys that begin with `prefix`
    for (int shift = 64; shift > 0;) {
        const int bits = shift < kDigit ? shift : kDigit, above = shift;
        shift -= bits;
        for (uint32_t k = t; k < kBins; k += 1024u) s_bins[k] = 0u;
        if (t == 0) s_digit = kBins;
        __syncthreads();
#pragma unroll 4
        for (uint64_t e = rank * 1024u + t; e < n_entries; e += kCutCtas * 1024u) {
            const uint4 b0 = __ldg(a.binrec + 2 * e);
            const unsigned long long key = ((unsigned long long)b0.w << 32) | e;
            if (b0.z && (above == 64 || key >> above == prefix))
                atomicAdd(&s_bins[(uint32_t)(key >> shift) & ((1u << bits) - 1u)], b0.z);
        }
        cluster.sync();
        uint32_t c0 = 0, c1 = 0, tot;
        for (uint32_t r = 0; r < kCutCtas; ++r) {
            const uint32_t *b = cluster.map_shared_rank(s_bins, r);
            c0 += b[2 * t];
            c1 += b[2 * t + 1];
        }
        const uint32_t first = block_excl_scan(c0 + c1, s_warp, tot);
        if (left >= first && left - first < c0 + c1) {  // one thread
            const bool second = left - first >= c0;
            s_digit = 2u * t + (second ? 1u : 0u);
            s_before = first + (second ? c0 : 0u);
        }
        cluster.sync();  // every CTA is past the bins, and this CTA's threads see the digit
        const uint32_t digit = s_digit, before = s_before;
        if (digit == kBins) return;  // (the entries hold fewer instances than the total says; the same for the cluster)
        prefix = (prefix << bits) | digit;
        left -= before;
        __syncthreads();  // the digit is reset after every thread has it
    }
    if (rank != 0 || t >= 32u) return;
    // the key's entry keeps its first `left` tiles: find its hit number `left`
    const uint32_t e = (uint32_t)prefix;
    const int v = (int)(e / (uint32_t)a.n), tiles_x = a.V.tiles_x[v];
    const uint4 b0 = __ldg(a.binrec + 2 * (size_t)e), b1 = __ldg(a.binrec + 2 * (size_t)e + 1);
    const uint32_t tbase = (uint32_t)a.V.tile_base[v], bw = b1.z & 0xffffu, bh = b1.z >> 16;
    auto cut_at = [&](uint32_t tx, uint32_t ty) {  // called by one lane
        *reinterpret_cast<unsigned long long *>(a.header + kCutWord) = prefix;
        a.header[kCutWord + 2] = tbase + ty * (uint32_t)tiles_x + tx;
        a.header[kCutWord + 3] = 1u;
        set_error(a.err, kErrCapacity);
    };
    if (bw * bh <= 32u) {
        const uint32_t bit = select_bit(b1.x, left);
        if (lane == 0) cut_at((b1.y & 0xffffu) + bit % bw, (b1.y >> 16) + bit / bw);
        return;
    }
    const int tw = a.V.tile_w, th = a.V.tile_h, lw = __ffs(tw) - 1, lh = __ffs(th) - 1;
    TileJob J = tile_job(a, v, e, b0, lw, lh);
    if (lane != 0) J.nbox = 0u;
    uint32_t seen = 0;
    warp_tile_rounds(J, (int)lane, lw, lh, tw, th, s_jobs, 0u, 1u,
                     [&](uint32_t hits, uint32_t, uint32_t, uint32_t, int tx, int ty, uint32_t, bool hit) {
                         if (hit && seen + (uint32_t)__popc(hits & ((1u << lane) - 1u)) == left) cut_at((uint32_t)tx, (uint32_t)ty);
                         seen += (uint32_t)__popc(hits);
                     });
}

// The instances of entries whose box has more than 32 tiles: the tile tests again.
template <class OnInstance>
__device__ __forceinline__ void large_box_instances(const BinArgs &a, int v, bool big, const uint4 b0, size_t e, uint4 *jobs,
                                                    int lane, uint32_t part, OnInstance &&on_instance) {
    if (!__any_sync(0xffffffffu, big)) return;
    const int tiles_x = a.V.tiles_x[v];
    const uint32_t tbase = (uint32_t)a.V.tile_base[v];
    const int tw = a.V.tile_w, th = a.V.tile_h;
    const int lw = __ffs(tw) - 1, lh = __ffs(th) - 1;  // tile sides are powers of two
    TileJob J = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0u, 0u, 0u};
    if (big) J = tile_job(a, v, e, b0, lw, lh);
    warp_tile_rounds(J, lane, lw, lh, tw, th, jobs, part, a.parts,
                     [&](uint32_t, uint32_t, uint32_t, uint32_t, int tx, int ty, uint32_t owner, bool hit) {
                         const uint32_t depth = __shfl_sync(0xffffffffu, b0.w, owner);
                         const uint32_t ent = __shfl_sync(0xffffffffu, (uint32_t)e, owner);
                         if (hit) on_instance(tbase + (uint32_t)(ty * tiles_x + tx), depth, ent);
                     });
}

// The instances of a lane's own entry from its hit mask, four at a time: take(tile, depth) for each, then put(what it
// returned, depth, entry), so that four of take's atomics are in flight. It issues a third of the instructions that sharing
// them over the warp does (8 views of 1.5M splats of a heightfield: count 262 -> 204 us, of an object 417 -> 330), and is
// used where the atomics are in shared memory: waiting for global ones, few lanes in flight, a 200k-splat object in a
// 1600x1040 view took 164 us against 124.
template <class Take, class Put>
__device__ __forceinline__ void lane_instances(const BinArgs &a, int v, uint32_t depth, const uint4 b1, uint32_t e, Take &&take,
                                               Put &&put) {
    constexpr uint32_t kNone = 0xffffffffu;
    const uint32_t tiles_x = (uint32_t)a.V.tiles_x[v], rw = b1.z & 0xffffu;
    const uint32_t origin = (uint32_t)a.V.tile_base[v] + (b1.y >> 16) * tiles_x + (b1.y & 0xffffu);
    const uint32_t mdiv = (65536u + rw - 1u) / rw, down = tiles_x - rw;  // bit / rw == (bit * mdiv) >> 16 for bit < 32
    for (uint32_t m = b1.x; m;) {
        uint32_t slot[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            slot[q] = kNone;
            if (m) {
                const uint32_t bit = (uint32_t)__ffs(m) - 1u;
                m &= m - 1u;
                slot[q] = take(origin + bit + ((bit * mdiv) >> 16) * down, depth);
            }
        }
#pragma unroll
        for (int q = 0; q < 4; ++q)
            if (slot[q] != kNone) put(slot[q], depth, e);
    }
}

// The instances of a warp's 32 entries, each listed tile of each entry once: on_instance(global tile, depth bits,
// entry) is called by one lane each. Entries whose box has at most 32 tiles are expanded from their hit masks
// by the whole warp, 32 instances a round (instance j goes to the entry whose prefix interval holds j, binary
// search over the warp's inclusive prefix, and to that entry's j-th set bit): a lane's own loop over its bits
// waits for an atomic per bit and took a quarter longer. Larger boxes repeat the tile tests.

template <class OnInstance>
__device__ __forceinline__ void warp_instances(const BinArgs &a, int v, uint32_t tiles, const uint4 b0, const uint4 b1,
                                               size_t e, uint4 *jobs, int lane, uint32_t part,
                                               OnInstance &&on_instance) {
    const int tiles_x = a.V.tiles_x[v];
    const uint32_t tbase = (uint32_t)a.V.tile_base[v];
    const uint32_t tx0 = b1.y & 0xffffu, ty0 = b1.y >> 16, bw = b1.z & 0xffffu, bh = b1.z >> 16;
    const uint32_t rw = tiles && bw * bh <= 32u ? bw : 0u;  // 0: nothing, or no mask
    const uint32_t origin = tbase + ty0 * (uint32_t)tiles_x + tx0;
    const uint32_t cnt = rw ? tiles : 0u;
    const uint32_t incl = warp_incl_scan(cnt), wtotal = __shfl_sync(0xffffffffu, incl, 31), excl = incl - cnt;
    const uint32_t mdiv = rw ? (65536u + rw - 1u) / rw : 0u;  // bit / rw == (bit * mdiv) >> 16 for bit < 32
    const uint32_t shape = rw | (mdiv << 8);
    for (uint32_t j0 = 32u * part; j0 < wtotal; j0 += 32u * a.parts) {
        const uint32_t j = j0 + (uint32_t)lane;
        int owner = 0;
#pragma unroll
        for (int step = 16; step > 0; step >>= 1) {
            const uint32_t p = __shfl_sync(0xffffffffu, incl, owner + step - 1);
            if (p <= j) owner += step;
        }
        const uint32_t o_excl = __shfl_sync(0xffffffffu, excl, owner);
        const uint32_t o_mask = __shfl_sync(0xffffffffu, b1.x, owner);
        const uint32_t o_org = __shfl_sync(0xffffffffu, origin, owner);
        const uint32_t o_shape = __shfl_sync(0xffffffffu, shape, owner);
        const uint32_t o_depth = __shfl_sync(0xffffffffu, b0.w, owner);
        if (j < wtotal) {
            const uint32_t bit = select_bit(o_mask, j - o_excl);
            const uint32_t row = (bit * (o_shape >> 8)) >> 16;
            // a warp's entries are consecutive
            on_instance(o_org + row * (uint32_t)tiles_x + (bit - row * (o_shape & 0xffu)), o_depth,
                        (uint32_t)e - (uint32_t)lane + (uint32_t)owner);
        }
    }
    large_box_instances(a, v, tiles && !rw, b0, e, jobs, lane, part, on_instance);
}
// EMIT false: counts the instances per tile. EMIT true: appends each instance to its tile's segment.
// A CTA takes `a.per_cta` entries of one view. SHARED: it counts them per tile in shared memory
// first, so that a tile costs one global atomic per CTA: the atomics of all CTAs on a view's few counters were
// what the kernel waited for (8 views of 1.5M splats, 34.7M instances: count 0.91 and append 1.06 ms with an
// atomic per instance). The count keeps what those atomics return, the CTA's place among a tile's instances, and
// the append of the same entries starts there, so a CTA's instances of a tile land side by side.
// SLABS: the tiles' segments are split by depth.
template <bool EMIT, bool SHARED, bool SLABS>
__global__ void __launch_bounds__(kInstThreads, EMIT || SLABS ? 3 : 4) k_instances(const BinArgs a) {
    const bool cut = a.header[kCutWord + 3] != 0u;  // (read beside the total)
    if (*a.total >= 0xffffffffull) {  // uint32 positions would wrap: no lists
        if (!EMIT && blockIdx.x == 0 && threadIdx.x == 0) set_error(a.err, kErrCapacity);
        return;
    }
    extern __shared__ uint32_t s_cnt[];  // SHARED: instances per segment of the view; the CTA's next slot in each
    __shared__ uint4 s_jobs[kInstThreads / 32][kJobWords * 32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    // The append takes the views one after the other: the segments it has open then are one view's and mostly stay in L2
    // until their sectors are full (8 views of 1.5M splats: 453 -> 411 us against all views at once). The count takes them
    // in turn, which keeps its atomics from meeting on one small view's counters.
    // blocks: the views of a part of a run of entries, the parts (every a.parts-th round of 32 instances of a
    // warp's entries: few splats of many tiles each give too few warps otherwise), the runs
    const uint32_t nv = (uint32_t)a.n_views, rows = gridDim.x / nv;
    const int v = (int)(EMIT && SHARED ? blockIdx.x / rows : blockIdx.x % nv);
    const uint32_t row = EMIT && SHARED ? blockIdx.x % rows : blockIdx.x / nv, part = row % a.parts;
    const uint32_t i0 = row / a.parts * a.per_cta, i1 = min(i0 + a.per_cta, (uint32_t)a.n);
    const uint32_t S = SLABS ? a.slabs : 1u, tbase = (uint32_t)a.V.tile_base[v] * S, vtiles = (uint32_t)a.V.tile_base[v + 1] * S - tbase;
    float z0 = 0.f, per_z = 0.f;
    if (SLABS) {
        z0 = __uint_as_float(~a.aux->depth_lo_inv[v]);
        const float dz = __uint_as_float(a.aux->depth_hi[v]) - z0;
        per_z = dz > 0.f ? (float)S / dz : 0.f;
    }
    // a tile's segment for a depth: the slabs' order is the depths'
    auto segment = [&](uint32_t tile, uint32_t depth) {
        if (!SLABS) return tile;
        return tile * S + min((uint32_t)max((int)((__uint_as_float(depth) - z0) * per_z), 0), S - 1u);
    };
    auto each_of = [&](auto &&on_instance) {
        for (uint32_t w0 = i0 + (uint32_t)warp * 32u; w0 < i1; w0 += blockDim.x) {
            const uint32_t i = w0 + (uint32_t)lane;
            const size_t e = (size_t)v * a.n + i;
            uint4 b0 = make_uint4(0u, 0u, 0u, 0u), b1 = b0;
            if (i < i1) {
                b0 = __ldg(a.binrec + 2 * e);
                b1 = __ldg(a.binrec + 2 * e + 1);
            }
            const uint32_t tiles = b0.z;
            if (!__any_sync(0xffffffffu, tiles != 0u)) continue;
            warp_instances(a, v, tiles, b0, b1, e, s_jobs[warp], lane, part, on_instance);
        }
    };
    // those that the capacity's cut keeps, in a loop of its own: the ordinary one needs no depths to count
    auto each = [&](auto &&on_instance) {
        if (!cut) {
            each_of(on_instance);
            return;
        }
        each_of([&](uint32_t tile, uint32_t depth, uint32_t e) {
            const unsigned long long key = ((unsigned long long)depth << 32) | e,
                                     last = *reinterpret_cast<const unsigned long long *>(a.header + kCutWord);
            if (key < last || (key == last && tile < a.header[kCutWord + 2])) on_instance(tile, depth, e);
        });
    };
    // each entry's instances by its own lane (no cut applies, and a warp has its entries to itself)
    auto each_own = [&](auto &&take, auto &&put) {
        for (uint32_t w0 = i0 + (uint32_t)warp * 32u; w0 < i1; w0 += blockDim.x) {
            const uint32_t i = w0 + (uint32_t)lane;
            const size_t e = (size_t)v * a.n + i;
            uint4 b0 = make_uint4(0u, 0u, 0u, 0u), b1 = b0;
            if (i < i1) {
                b0 = __ldg(a.binrec + 2 * e);
                b1 = __ldg(a.binrec + 2 * e + 1);
            }
            const bool masked = (b1.z & 0xffffu) * (b1.z >> 16) <= 32u;
            if (b0.z && masked) lane_instances(a, v, b0.w, b1, (uint32_t)e, take, put);
            __syncwarp();
            large_box_instances(a, v, b0.z && !masked, b0, e, s_jobs[warp], lane, 0u,
                                [&](uint32_t tile, uint32_t depth, uint32_t ent) { put(take(tile, depth), depth, ent); });
        }
    };
    const bool own = !cut && a.own;
    auto append = [&](uint32_t slot, uint32_t depth, uint32_t e) {
        if (slot < a.cap) a.pairs[slot] = ((unsigned long long)depth << 32) | e;
        else set_error(a.err, kErrCapacity);  // (counts beyond the total only: the cut keeps within the capacity)
    };
    if (SHARED) {
        uint32_t *place = a.places + (size_t)row * ((size_t)a.V.n_tiles * S) + tbase;
        // (a tile without instances here has no place: its slot is not used)
        for (uint32_t t = threadIdx.x; t < vtiles; t += blockDim.x) s_cnt[t] = EMIT ? a.counts[tbase + t] + place[t] : 0u;
        __syncthreads();
        if (EMIT) {
            if (own)
                each_own([&](uint32_t tile, uint32_t depth) { return atomicAdd(&s_cnt[segment(tile, depth) - tbase], 1u); },
                         append);
            else
                each([&](uint32_t tile, uint32_t depth, uint32_t e) {
                    append(atomicAdd(&s_cnt[segment(tile, depth) - tbase], 1u), depth, e);
                });
            return;
        }
        if (own)
            each_own([&](uint32_t tile, uint32_t depth) { atomicAdd(&s_cnt[segment(tile, depth) - tbase], 1u); return 0u; },
                     [](uint32_t, uint32_t, uint32_t) {});
        else
            each([&](uint32_t tile, uint32_t depth, uint32_t) { atomicAdd(&s_cnt[segment(tile, depth) - tbase], 1u); });
        __syncthreads();
        for (uint32_t t = threadIdx.x; t < vtiles; t += blockDim.x) {
            const uint32_t c = s_cnt[t];
            if (c) place[t] = atomicAdd(a.counts + tbase + t, c);
        }
    } else {
        each([&](uint32_t tile, uint32_t depth, uint32_t e) {
            const uint32_t slot = atomicAdd(a.counts + segment(tile, depth), 1u);
            if (EMIT) append(slot, depth, e);
        });
    }
}

// Least and greatest depth of each view's listed entries, for the slabs.
__global__ void __launch_bounds__(256) k_depth_range(const BinArgs a) {
    const int v = (int)blockIdx.y;
    uint32_t hi = 0u, lo_inv = 0u;
    for (uint32_t i = blockIdx.x * 256u + threadIdx.x; i < (uint32_t)a.n; i += gridDim.x * 256u) {
        const uint4 b = __ldg(a.binrec + 2 * ((size_t)v * a.n + i));
        if (b.z) {
            hi = max(hi, b.w);
            lo_inv = max(lo_inv, ~b.w);
        }
    }
    hi = __reduce_max_sync(0xffffffffu, hi);
    lo_inv = __reduce_max_sync(0xffffffffu, lo_inv);
    if ((threadIdx.x & 31) == 0 && hi) {
        atomicMax(&a.aux->depth_hi[v], hi);
        atomicMax(&a.aux->depth_lo_inv[v], lo_inv);
    }
}

// Length bucket of a list for the longest-first queue: 4 buckets per octave, longest first. Approximate
// order is enough for scheduling; the results do not depend on it.
__device__ __forceinline__ int length_bucket(uint32_t len) {
    if (len == 0) return kLptBuckets - 1;
    const int b = (kLptBuckets - 2) - (int)(4.f * log2f((float)len + 1.f));
    return b < 0 ? 0 : b;
}

// Tile index, first part: each CTA's instances and, for the queue, its tiles per length bucket. A CTA takes
// `per` consecutive tiles (a multiple of 1024).
__global__ void __launch_bounds__(1024) k_tile_sums(const BinArgs a, uint32_t per) {
    __shared__ uint32_t s_warp[33], s_bucket[kLptBuckets];
    const uint32_t n_tiles = (uint32_t)a.V.n_tiles, t0 = blockIdx.x * per;
    if (threadIdx.x < kLptBuckets) s_bucket[threadIdx.x] = 0u;
    __syncthreads();
    uint32_t sum = 0;
    for (uint32_t k = threadIdx.x; k < per; k += 1024) {
        const uint32_t t = t0 + k;
        if (t >= n_tiles) break;
        uint32_t c = 0;
        for (uint32_t q = 0; q < a.slabs; ++q) c += a.counts[(size_t)t * a.slabs + q];
        sum += c;
        if (a.build_queue) atomicAdd(&s_bucket[length_bucket(c)], 1u);
    }
    uint32_t tot;
    block_excl_scan(sum, s_warp, tot);
    if (threadIdx.x == 0) a.aux->partial[blockIdx.x] = tot;
    if (a.build_queue && threadIdx.x < kLptBuckets)
        a.buckets[(size_t)blockIdx.x * kLptBuckets + threadIdx.x] = s_bucket[threadIdx.x];
}

// Sort class of a segment of n instances at `start`, clipped to the capacity: -1 nothing to sort, kListClasses too
// long for one CTA.
__device__ __forceinline__ int seg_class(const BinArgs &a, uint32_t start, uint32_t n) {
    const uint32_t len = (uint32_t)(min((uint64_t)start + n, a.cap) - min((uint64_t)start, a.cap));
    return len == 0u ? -1 : len <= 256u ? 0 : len <= 1024u ? 1 : len <= kCtaList ? 2 : len <= kMidList ? 3
         : len <= kBigList ? 4 : len <= kSplitList ? kToSplit : kListClasses;
}

// A list [s, e) of tile t to be sorted in chunks.
__device__ __forceinline__ void push_chunks(const BinArgs &a, uint32_t s, uint32_t e, uint32_t t) {
    const uint32_t nch = (e - s + kBigList - 1u) / kBigList, k = atomicAdd(&a.aux->n_jobs, nch);
    for (uint32_t j = 0; j < nch; ++j) a.jobs[k + j] = make_uint4(s, e, t, j);
}

// Tile index, second part: each tile's range clipped to the capacity, its segments' starts (in place of their
// counts) and their places in the sort classes' lists or chunk jobs, and the tile's place in the queue. Within a
// bucket the queue keeps the tiles' order: the render backward takes the tiles in the queue's order and adds their
// gradients with float atomics, and the sums of a thin splat's Sigma' cancel so far that another order moves its
// gradients by 3e-5. With places taken by atomics across the CTAs the order varied from run to run.
__global__ void __launch_bounds__(1024) k_tile_index(const BinArgs a, uint32_t per) {
    __shared__ uint32_t s_warp[33], s_all[kLptBuckets], s_next[kLptBuckets];
    __shared__ uint32_t s_rank[32][kLptBuckets];  // tiles of a bucket per warp, then its first place
    __shared__ uint32_t s_cls[kListClasses], s_cls_base[kListClasses];
    const uint32_t n_tiles = (uint32_t)a.V.n_tiles, t0 = blockIdx.x * per, tid = threadIdx.x, S = a.slabs;
    const int lane = (int)(tid & 31u), warp = (int)(tid >> 5);
    if (blockIdx.x == 0 && tid == 0) {
        const unsigned long long t = *a.total;
        a.header[0] = t >= 0xffffffffull ? 0u : (uint32_t)(t < a.cap ? t : a.cap);
    }
    uint32_t run, tot;
    block_excl_scan(tid < blockIdx.x ? a.aux->partial[tid] : 0u, s_warp, run);  // at most kTileBlocks CTAs before
    if (a.build_queue) {  // the buckets' first places for this CTA: all longer buckets, then the CTAs before
        if (tid < kLptBuckets) s_all[tid] = s_next[tid] = 0u;
        __syncthreads();
        const uint32_t b = tid % kLptBuckets;
        uint32_t all = 0, before = 0;
        for (uint32_t c = tid / kLptBuckets; c < gridDim.x; c += 1024u / kLptBuckets) {
            const uint32_t n = a.buckets[(size_t)c * kLptBuckets + b];
            all += n;
            if (c < blockIdx.x) before += n;
        }
        atomicAdd(&s_all[b], all);
        atomicAdd(&s_next[b], before);
        __syncthreads();
        const uint32_t p = block_excl_scan(tid < kLptBuckets ? s_all[tid] : 0u, s_warp, tot);
        if (tid < kLptBuckets) s_next[tid] += p;
    }
    for (uint32_t k0 = 0; k0 < per; k0 += 1024) {
        const uint32_t t = t0 + k0 + tid;
        if (t0 + k0 >= n_tiles) break;  // uniform for the CTA
        if (a.build_queue)
            for (uint32_t k = tid; k < 32u * kLptBuckets; k += 1024u) s_rank[k / kLptBuckets][k % kLptBuckets] = 0u;
        if (tid < kListClasses) s_cls[tid] = 0u;
        __syncthreads();
        uint32_t c = 0;
        if (t < n_tiles)
            for (uint32_t q = 0; q < S; ++q) c += a.counts[(size_t)t * S + q];
        const uint32_t start = run + block_excl_scan(c, s_warp, tot);
        run += tot;
        const int bucket = t < n_tiles ? length_bucket(c) : kLptBuckets;
        uint32_t rank = 0;
        if (a.build_queue) {
            const uint32_t peers = __match_any_sync(0xffffffffu, bucket);
            rank = (uint32_t)__popc(peers & ((1u << lane) - 1u));
            if (rank == 0u && t < n_tiles) s_rank[warp][bucket] = (uint32_t)__popc(peers);
        }
        if (t < n_tiles) {
            const uint64_t s = min((uint64_t)start, a.cap), e = min((uint64_t)start + c, a.cap);
            a.ranges[t] = e > s ? make_uint2((uint32_t)s, (uint32_t)e) : make_uint2(0u, 0u);
            // the tile's segments: their starts replace their counts
            uint32_t at = start;
            for (uint32_t q = 0; q < S; ++q) {
                const uint32_t n = a.counts[(size_t)t * S + q];
                a.counts[(size_t)t * S + q] = at;
                const int cls = seg_class(a, at, n);
                if (cls < kListClasses && cls >= 0) atomicAdd(&s_cls[cls], 1u);
                at += n;
            }
        }
        __syncthreads();
        if (tid < kListClasses) {
            s_cls_base[tid] = s_cls[tid] ? atomicAdd(&a.aux->n_list[tid], s_cls[tid]) : 0u;
            s_cls[tid] = 0u;
        }
        if (a.build_queue && tid < kLptBuckets) {
            uint32_t next = s_next[tid];
#pragma unroll
            for (int w = 0; w < 32; ++w) {
                const uint32_t n = s_rank[w][tid];
                s_rank[w][tid] = next;
                next += n;
            }
            s_next[tid] = next;
        }
        __syncthreads();
        if (t < n_tiles) {
            uint32_t at = start;
            for (uint32_t q = 0; q < S; ++q) {
                // the next segment's start, the tile's end after the last
                const uint32_t end = q + 1 < S ? a.counts[(size_t)t * S + q + 1] : start + c;
                const int cls = seg_class(a, at, end - at);
                const uint32_t s = (uint32_t)min((uint64_t)at, a.cap), e = (uint32_t)min((uint64_t)end, a.cap);
                if (cls >= 0 && cls < kListClasses) {
                    const uint32_t k = s_cls_base[cls] + atomicAdd(&s_cls[cls], 1u);
                    a.lists[cls * a.stride + k] = make_uint4(s, e, t, 0u);
                } else if (cls == kListClasses) {
                    push_chunks(a, s, e, t);
                }
                at = end;
            }
        }
        if (a.build_queue && t < n_tiles) a.queue[s_rank[warp][bucket] + rank] = t;
        __syncthreads();
    }
}

// ------------------------------------------------------------------ tile list sort
typedef unsigned long long u64;
// Keys in shared memory are padded by one per ITEMS, so that neighbouring threads' runs of ITEMS start in
// different banks.
template <int ITEMS>
__host__ __device__ constexpr int padded(int i) { return i + i / ITEMS; }

// Merge sort of 64-bit keys by a group of threads (merges split along diagonals: Odeh, Green, Mwassi, Shmueli and Birk,
// "Merge Path - parallel merging made simple", 2012), ITEMS consecutive keys a thread: a sorting network in
// registers, then merges of doubling width, each thread producing its ITEMS outputs from where a binary
// search along its diagonal says they start.
// Sorts the len keys of sm (at padded<ITEMS>(i); len <= the group's threads x ITEMS) with the group's thread t; `sync`
// is the group's barrier. The keys are visible to the group on entry and on return.
template <int ITEMS, class Sync>
__device__ __forceinline__ void sort_keys(u64 *sm, int t, int len, Sync &&sync) {
    const int first = t * ITEMS, lenp = (len + ITEMS - 1) / ITEMS * ITEMS;
    const bool on = first < len;
    u64 k[ITEMS];
    if (on) {
#pragma unroll
        for (int i = 0; i < ITEMS; ++i) k[i] = first + i < len ? sm[padded<ITEMS>(first + i)] : ~0ull;
        batcher_sort(k);
#pragma unroll
        for (int i = 0; i < ITEMS; ++i) sm[padded<ITEMS>(first + i)] = k[i];
    }
    sync();
    for (int width = ITEMS; width < lenp; width <<= 1) {
        const int a0 = first & ~(2 * width - 1), a1 = a0 + width, b1 = min(a0 + 2 * width, lenp);
        const bool merge = on && a1 < b1;  // without a second run the keys stay
        if (merge) {
            const int diag = first - a0, lb = b1 - a1;
            int lo = max(0, diag - lb), hi = min(diag, width);
            while (lo < hi) {
                const int mid = (lo + hi) >> 1;
                if (sm[padded<ITEMS>(a0 + mid)] < sm[padded<ITEMS>(a1 + diag - 1 - mid)]) lo = mid + 1;
                else hi = mid;
            }
            int ai = a0 + lo, bi = a1 + diag - lo;
            u64 ka = ai < a1 ? sm[padded<ITEMS>(ai)] : ~0ull, kb = bi < b1 ? sm[padded<ITEMS>(bi)] : ~0ull;
#pragma unroll
            for (int i = 0; i < ITEMS; ++i) {
                const bool take_a = ka < kb;
                k[i] = take_a ? ka : kb;
                const int idx = take_a ? ++ai : ++bi, end = take_a ? a1 : b1;
                const u64 nk = idx < end ? sm[padded<ITEMS>(idx)] : ~0ull;
                ka = take_a ? nk : ka;
                kb = take_a ? kb : nk;
            }
        }
        sync();
        if (merge) {
#pragma unroll
            for (int i = 0; i < ITEMS; ++i) sm[padded<ITEMS>(first + i)] = k[i];
        }
        sync();
    }
}

// Sorts len <= THREADS x ITEMS keys with a group of THREADS threads: load(j) gives the j-th, store(at, key) takes
// the one that belongs at position `at`. Depths spread over a tile's list, so the keys are dropped into as many buckets of equal depth
// width (a monotone map) as there are keys, and each key then finds its place among the few of its bucket by
// comparing with all of them: about 60 instructions a key where the merge sort takes 200. A list with more than
// kBucketMost keys in a bucket (many equal depths, or a few far ones) is merge sorted.
// keys: padded<ITEMS>(THREADS x ITEMS), cnt: THREADS x ITEMS, scratch: 3 per warp; `sync` is the group's barrier.
constexpr uint32_t kBucketMost = 24;
template <int ITEMS, class Sync>
__device__ __noinline__ void sort_keys_apart(u64 *keys, int t, int len, Sync sync) {  // keeps its registers out of the callers
    sort_keys<ITEMS>(keys, t, len, sync);
}

template <int THREADS, int ITEMS, class Sync, class Load, class Store>
__device__ __forceinline__ void sort_spread(int len, u64 *keys, uint32_t *cnt, uint32_t *scratch, int t, Sync &&sync,
                                            Load &&load, Store &&store) {
    static_assert(THREADS * ITEMS <= 32768, "a bucket's start and count are packed into 32 bits");
    constexpr int WARPS = THREADS / 32;
    const int lane = t & 31, w = t >> 5;
    u64 k[ITEMS];
    uint32_t zlo = 0xffffffffu, zhi = 0u;  // depths are positive: their bits order as they do
#pragma unroll
    for (int i = 0; i < ITEMS; ++i) {
        const int j = t + i * THREADS;
        if (j < len) {
            k[i] = load(j);
            zlo = min(zlo, (uint32_t)(k[i] >> 32));
            zhi = max(zhi, (uint32_t)(k[i] >> 32));
        }
    }
    int per = 1;  // buckets per thread
    while (per * THREADS < len) per <<= 1;
    const int nb = per * THREADS;
    for (int b = t; b < nb; b += THREADS) cnt[b] = 0u;
    zlo = __reduce_min_sync(0xffffffffu, zlo);
    zhi = __reduce_max_sync(0xffffffffu, zhi);
    if (WARPS > 1 && lane == 0) { scratch[w] = zlo; scratch[WARPS + w] = zhi; }
    sync();
    if (WARPS > 1) {
        zlo = __reduce_min_sync(0xffffffffu, scratch[lane % WARPS]);
        zhi = __reduce_max_sync(0xffffffffu, scratch[WARPS + lane % WARPS]);
    }
    const float z0 = __uint_as_float(zlo), width = __uint_as_float(zhi) - z0;
    const float scale = width > 0.f ? (float)nb / width : 0.f;
    auto bucket = [&](u64 key) {
        return min((int)((__uint_as_float((uint32_t)(key >> 32)) - z0) * scale), nb - 1);
    };
    uint32_t rank[ITEMS];
#pragma unroll
    for (int i = 0; i < ITEMS; ++i)
        if (t + i * THREADS < len) rank[i] = atomicAdd(&cnt[bucket(k[i])], 1u);
    sync();
    // bucket starts: an exclusive scan, thread t taking buckets [t per, (t + 1) per)
    uint32_t sum = 0, most = 0;
    for (int q = 0; q < per; ++q) {
        const uint32_t c = cnt[t * per + q];
        sum += c;
        most = max(most, c);
    }
    uint32_t incl = warp_incl_scan(sum);
    most = __reduce_max_sync(0xffffffffu, most);
    if (WARPS > 1) {
        if (lane == 31) scratch[2 * WARPS + w] = incl;
        if (lane == 0) scratch[w] = most;
        sync();
        most = __reduce_max_sync(0xffffffffu, scratch[lane % WARPS]);
        const uint32_t before = lane < w ? scratch[2 * WARPS + lane] : 0u;  // WARPS <= 32
        incl += __reduce_add_sync(0xffffffffu, before);
    }
    const bool spread = most <= kBucketMost;  // the same in all threads of the group
    if (spread) {
        uint32_t run = incl - sum;
        for (int q = 0; q < per; ++q) {
            const uint32_t c = cnt[t * per + q];
            cnt[t * per + q] = run | (c << 16);  // starts below 2^15, counts at most kBucketMost
            run += c;
        }
        sync();
#pragma unroll
        for (int i = 0; i < ITEMS; ++i)
            if (t + i * THREADS < len) keys[(cnt[bucket(k[i])] & 0xffffu) + rank[i]] = k[i];
        sync();
        for (int j = t; j < len; j += THREADS) {
            const u64 key = keys[j];
            const uint32_t sc = cnt[bucket(key)], first = sc & 0xffffu, n = sc >> 16;
            uint32_t at = first;
            for (uint32_t q = 0; q < n; ++q) at += keys[first + q] < key;
            store((int)at, key);
        }
    } else {
#pragma unroll
        for (int i = 0; i < ITEMS; ++i)
            if (t + i * THREADS < len) keys[padded<ITEMS>(t + i * THREADS)] = k[i];
        sync();
        sort_keys_apart<ITEMS>(keys, t, len, sync);
        for (int j = t; j < len; j += THREADS) store(j, keys[padded<ITEMS>(j)]);
    }
    sync();
}

// Sorts one segment (start, end, tile) of at most THREADS x ITEMS instances and writes its part of the lists.
// SPLIT: split off a longer list, the keys (depth, entry) lie unsorted where the segment's own part of the lists will be.
template <int THREADS, int ITEMS, bool SPLIT, class Sync>
__device__ __forceinline__ void sort_segment(const BinArgs &a, uint4 rg, u64 *keys, uint32_t *cnt, uint32_t *scratch,
                                             int t, Sync &&sync) {
    sort_spread<THREADS, ITEMS>(
        (int)(rg.y - rg.x), keys, cnt, scratch, t, sync,
        [&](int j) {
            return SPLIT ? ((u64)a.inst_tile[rg.x + j] << 32) | a.inst_entry[rg.x + j] : a.pairs[rg.x + j];
        },
        [&](int at, u64 key) {
            a.inst_entry[rg.x + at] = (uint32_t)key;
            a.inst_tile[rg.x + at] = rg.z;
        });
}

// Splits the lists of kBigList to kSplitList entries by depth, a CTA each: a histogram over kSplitBins bins of equal
// depth width, consecutive bins gathered into segments of about kSplitGroup entries, and the keys written bin by bin to
// the list's own part of the outputs (depth and entry where tile and entry will be), from where the segments are sorted
// like short lists. Bound by the scattered stores of the last of its three passes. Merged from chunks instead, whose
// searches are one serial chain, the dense tiles of object scenes cost more than all else: 8 views of 1.5M splats (61M
// instances) 800 us for 332 lists, 150 here; a 170k-splat batch of three 740x640 views 136 us for two, 33 here.
constexpr int kSplitBins = 2048;
__global__ void __launch_bounds__(1024) k_split_lists(const BinArgs a) {
    __shared__ uint32_t s_bin[kSplitBins], s_warp[33], s_lo, s_hi, s_most;
    __shared__ uint32_t s_start[kSplitList / kSplitGroup + 2], s_cls[2], s_base[2];
    constexpr uint32_t kGroups = kSplitList / kSplitGroup + 1;
    const uint32_t t = threadIdx.x, n = a.aux->n_list[kToSplit];
    for (uint32_t k = blockIdx.x; k < n; k += gridDim.x) {
        const uint4 rg = a.lists[kToSplit * a.stride + k];
        const uint32_t len = rg.y - rg.x;
        const uint32_t *high = reinterpret_cast<const uint32_t *>(a.pairs + rg.x) + 1;  // the depths
        if (t == 0) { s_lo = 0xffffffffu; s_hi = 0u; s_most = 0u; }
        if (t < 2u) s_cls[t] = 0u;
        for (uint32_t b = t; b < kSplitBins; b += 1024u) s_bin[b] = 0u;
        if (t <= kGroups) s_start[t] = 0xffffffffu;
        __syncthreads();
        // kRun loads in flight at a time: a list has few warps, and each pass waits for memory
        constexpr uint32_t kRun = 8;
        uint32_t lo = 0xffffffffu, hi = 0u;
        for (uint32_t j0 = t; j0 < len; j0 += kRun * 1024u) {
#pragma unroll
            for (uint32_t q = 0; q < kRun; ++q) {
                const uint32_t z = high[2 * (size_t)min(j0 + q * 1024u, len - 1u)];
                lo = min(lo, z);
                hi = max(hi, z);
            }
        }
        lo = __reduce_min_sync(0xffffffffu, lo);
        hi = __reduce_max_sync(0xffffffffu, hi);
        if ((t & 31u) == 0) { atomicMin(&s_lo, lo); atomicMax(&s_hi, hi); }
        __syncthreads();
        const float z0 = __uint_as_float(s_lo), width = __uint_as_float(s_hi) - z0;
        const float scale = width > 0.f ? (float)kSplitBins / width : 0.f;
        auto bin = [&](uint32_t z) { return min((int)((__uint_as_float(z) - z0) * scale), kSplitBins - 1); };
        for (uint32_t j0 = t; j0 < len; j0 += kRun * 1024u) {
            uint32_t z[kRun];
#pragma unroll
            for (uint32_t q = 0; q < kRun; ++q) z[q] = high[2 * (size_t)min(j0 + q * 1024u, len - 1u)];
#pragma unroll
            for (uint32_t q = 0; q < kRun; ++q)
                if (j0 + q * 1024u < len) atomicAdd(&s_bin[bin(z[q])], 1u);
        }
        __syncthreads();
        // bin starts; a bin belongs to the segment its start falls into
        const uint32_t c0 = s_bin[2 * t], c1 = s_bin[2 * t + 1];
        uint32_t tot;
        const uint32_t first = block_excl_scan(c0 + c1, s_warp, tot);
        s_bin[2 * t] = first;
        s_bin[2 * t + 1] = first + c0;
        if (c0) atomicMin(&s_start[first / kSplitGroup], first);
        if (c1) atomicMin(&s_start[(first + c0) / kSplitGroup], first + c0);
        __syncthreads();
        uint32_t at = 0, end = 0;
        if (t < kGroups && s_start[t] != 0xffffffffu) {
            at = s_start[t];
            uint32_t g = t + 1u;
            while (g < kGroups && s_start[g] == 0xffffffffu) ++g;
            end = g < kGroups ? s_start[g] : len;
            atomicMax(&s_most, end - at);
        }
        __syncthreads();
        if (s_most > kCtaList) {  // the same for the CTA: left whole
            if (t == 0) push_chunks(a, rg.x, rg.y, rg.z);
        } else {
            const int cls = end - at <= 1024u ? 0 : 1;
            uint32_t place = 0;
            if (end > at) place = atomicAdd(&s_cls[cls], 1u);
            __syncthreads();
            if (t < 2u) s_base[t] = s_cls[t] ? atomicAdd(&a.aux->n_list[kSplitShort + t], s_cls[t]) : 0u;
            __syncthreads();
            if (end > at)
                a.lists[(kSplitShort + cls) * a.stride + s_base[cls] + place] = make_uint4(rg.x + at, rg.x + end, rg.z, 0u);
            constexpr uint32_t kHalf = kRun / 2;
            for (uint32_t j0 = t; j0 < len; j0 += kHalf * 1024u) {
                u64 key[kHalf];
#pragma unroll
                for (uint32_t q = 0; q < kHalf; ++q) key[q] = a.pairs[rg.x + min(j0 + q * 1024u, len - 1u)];
                uint32_t slot[kHalf];
#pragma unroll
                for (uint32_t q = 0; q < kHalf; ++q)
                    if (j0 + q * 1024u < len) slot[q] = rg.x + atomicAdd(&s_bin[bin((uint32_t)(key[q] >> 32))], 1u);
#pragma unroll
                for (uint32_t q = 0; q < kHalf; ++q)
                    if (j0 + q * 1024u < len) {
                        a.inst_tile[slot[q]] = (uint32_t)(key[q] >> 32);
                        a.inst_entry[slot[q]] = (uint32_t)key[q];
                    }
            }
        }
        __syncthreads();
    }
}

// Lists of at most kCtaList entries: the longest by a whole CTA, those up to 1024 by 128 threads, those up to 256
// by a warp. CTA b takes every gridDim-th of each class.
constexpr int kListItems = 8, kListThreads = (int)kCtaList / kListItems;
__global__ void __launch_bounds__(kListThreads, 2) k_sort_lists(const BinArgs a) {
    extern __shared__ u64 sm[];
    uint32_t *cnt = reinterpret_cast<uint32_t *>(sm + padded<kListItems>(kCtaList));
    __shared__ uint32_t scratch[3 * kListThreads / 32];
    const int t = threadIdx.x, g = t >> 7, w = t >> 5;
    const size_t T = a.stride;
    const uint32_t n2 = a.aux->n_list[2], n1 = a.aux->n_list[1], n0 = a.aux->n_list[0];
    for (uint32_t k = blockIdx.x; k < n2; k += gridDim.x)
        sort_segment<kListThreads, kListItems, false>(a, a.lists[2 * T + k], sm, cnt, scratch, t, []() { __syncthreads(); });
    for (uint32_t k = blockIdx.x * 4 + g; k < n1; k += gridDim.x * 4)
        sort_segment<128, kListItems, false>(a, a.lists[T + k], sm + g * padded<kListItems>(1024), cnt + g * 1024, scratch + g * 12,
                                   t & 127, [&]() { asm volatile("bar.sync %0, 128;" ::"r"(g + 1) : "memory"); });
    __syncthreads();
    for (uint32_t k = blockIdx.x * 16 + w; k < n0; k += gridDim.x * 16)
        sort_segment<32, kListItems, false>(a, a.lists[k], sm + w * padded<kListItems>(256), cnt + w * 256, scratch, t & 31,
                                  []() { __syncwarp(); });
}

// Chunk q of the ceil(len / kBigList) chunks of a list [rg.x, rg.y).
__device__ __forceinline__ uint2 chunk_of(uint4 job, uint32_t q) {
    const uint64_t len = job.y - job.x, nch = (len + kBigList - 1) / kBigList;
    return make_uint2(job.x + (uint32_t)(len * q / nch), job.x + (uint32_t)(len * (q + 1) / nch));
}

constexpr int kBigItems = (int)kBigList / 1024;

// sort_spread for up to kBigList keys by 1,024 threads, reading them three times (the range, the bucket counts, the
// buckets) in place of holding 16 and their ranks a thread, which spilled. Bound by the shared-memory pipe. 1.5M splats
// of an object at 1600x1040, 10.6M entries in lists of 4,096 to 11,323: k_sort_big 218 us with 16 keys a thread, 193
// with this, 166 with this from 8,192 on and 8 keys a thread below. Stores come after every load.
template <class Load, class Store>
__device__ __forceinline__ void sort_spread_big(int len, u64 *keys, uint32_t *cnt, uint32_t *scratch, int t, Load &&load,
                                                Store &&store) {
    constexpr int WARPS = 32, kRun = 8;
    const int lane = t & 31, w = t >> 5;
    uint32_t zlo = 0xffffffffu, zhi = 0u;
    for (int j0 = t; j0 < len; j0 += kRun * 1024) {
#pragma unroll
        for (int q = 0; q < kRun; ++q) {
            const uint32_t z = (uint32_t)(load(min(j0 + q * 1024, len - 1)) >> 32);
            zlo = min(zlo, z);
            zhi = max(zhi, z);
        }
    }
    int per = 1;  // buckets per thread
    while (per * 1024 < len) per <<= 1;
    const int nb = per * 1024;
    for (int b = t; b < nb; b += 1024) cnt[b] = 0u;
    zlo = __reduce_min_sync(0xffffffffu, zlo);
    zhi = __reduce_max_sync(0xffffffffu, zhi);
    if (lane == 0) { scratch[w] = zlo; scratch[WARPS + w] = zhi; }
    __syncthreads();
    zlo = __reduce_min_sync(0xffffffffu, scratch[lane]);
    zhi = __reduce_max_sync(0xffffffffu, scratch[WARPS + lane]);
    const float z0 = __uint_as_float(zlo), width = __uint_as_float(zhi) - z0;
    const float scale = width > 0.f ? (float)nb / width : 0.f;
    auto bucket = [&](u64 key) {
        return min((int)((__uint_as_float((uint32_t)(key >> 32)) - z0) * scale), nb - 1);
    };
    for (int j0 = t; j0 < len; j0 += kRun * 1024) {
        u64 k[kRun];
#pragma unroll
        for (int q = 0; q < kRun; ++q) k[q] = load(min(j0 + q * 1024, len - 1));
#pragma unroll
        for (int q = 0; q < kRun; ++q)
            if (j0 + q * 1024 < len) atomicAdd(&cnt[bucket(k[q])], 1u);
    }
    __syncthreads();
    uint32_t sum = 0, most = 0;
    for (int q = 0; q < per; ++q) {
        const uint32_t c = cnt[t * per + q];
        sum += c;
        most = max(most, c);
    }
    uint32_t incl = warp_incl_scan(sum);
    most = __reduce_max_sync(0xffffffffu, most);
    if (lane == 31) scratch[2 * WARPS + w] = incl;
    if (lane == 0) scratch[w] = most;
    __syncthreads();
    most = __reduce_max_sync(0xffffffffu, scratch[lane]);
    incl += __reduce_add_sync(0xffffffffu, lane < w ? scratch[2 * WARPS + lane] : 0u);
    if (most <= kBucketMost) {  // the same in all threads
        static_assert(kBigList <= 32767 && kBucketMost < 32, "a bucket's start, count and cursor in 15 + 5 + 5 bits");
        uint32_t run = incl - sum;
        for (int q = 0; q < per; ++q) {
            const uint32_t c = cnt[t * per + q];
            cnt[t * per + q] = run | (c << 15);
            run += c;
        }
        __syncthreads();
        for (int j0 = t; j0 < len; j0 += kRun * 1024) {
            u64 k[kRun];
#pragma unroll
            for (int q = 0; q < kRun; ++q) k[q] = load(min(j0 + q * 1024, len - 1));
#pragma unroll
            for (int q = 0; q < kRun; ++q)
                if (j0 + q * 1024 < len) {
                    const uint32_t sc = atomicAdd(&cnt[bucket(k[q])], 1u << 20);
                    keys[(sc & 0x7fffu) + (sc >> 20)] = k[q];
                }
        }
        __syncthreads();
        for (int j = t; j < len; j += 1024) {
            const u64 key = keys[j];
            const uint32_t sc = cnt[bucket(key)], first = sc & 0x7fffu, n = (sc >> 15) & 31u;
            uint32_t at = first;
            for (uint32_t q = 0; q < n; ++q) at += keys[first + q] < key;
            store((int)at, key);
        }
    } else {
        for (int j = t; j < len; j += 1024) keys[padded<kBigItems>(j)] = load(j);
        __syncthreads();
        sort_keys_apart<kBigItems>(keys, t, len, []() { __syncthreads(); });
        for (int j = t; j < len; j += 1024) store(j, keys[padded<kBigItems>(j)]);
    }
    __syncthreads();
}

// Lists of kCtaList to kBigList entries, the segments split off longer ones (by 128 or 512 threads), and the chunks of
// the longest (sorted in place). The CTAs take them in turn, the classes one after the other.
__global__ void __launch_bounds__(1024) k_sort_big(const BinArgs a) {
    extern __shared__ u64 sm[];
    __shared__ uint32_t scratch[3 * 32];
    uint32_t *cnt = reinterpret_cast<uint32_t *>(sm + padded<kBigItems>(kBigList));
    const int t = threadIdx.x;
    const uint32_t n3 = a.aux->n_list[3], n4 = a.aux->n_list[4], n6 = a.aux->n_list[kSplitShort],
                   n7 = a.aux->n_list[kSplitLong], nj = a.aux->n_jobs;
    const int g = t >> 7, h = t >> 9;
    // this CTA's first of a class, after the `before` pieces of work of the classes before it
    auto first = [](uint32_t before) { return (blockIdx.x + gridDim.x - before % gridDim.x) % gridDim.x; };
    for (uint32_t k = first(0); k < n4; k += gridDim.x) {
        const uint4 rg = a.lists[4 * a.stride + k];
        sort_spread_big((int)(rg.y - rg.x), sm, cnt, scratch, t, [&](int j) { return a.pairs[rg.x + j]; },
                        [&](int at, u64 key) {
                            a.inst_entry[rg.x + at] = (uint32_t)key;
                            a.inst_tile[rg.x + at] = rg.z;
                        });
    }
    for (uint32_t k = first(n4); k < n3; k += gridDim.x)
        sort_segment<1024, (int)kMidList / 1024, false>(a, a.lists[3 * a.stride + k], sm, cnt, scratch, t,
                                                        []() { __syncthreads(); });
    for (uint32_t k = first(n4 + n3) * 2 + h; k < n7; k += gridDim.x * 2)
        sort_segment<512, 8, true>(a, a.lists[kSplitLong * a.stride + k], sm + h * padded<8>(4096), cnt + h * 4096,
                                   scratch + h * 48, t & 511,
                                   [&]() { asm volatile("bar.sync %0, 512;" ::"r"(h + 9) : "memory"); });
    __syncthreads();
    for (uint32_t k = first(n4 + n3 + (n7 + 1) / 2) * 8 + g; k < n6; k += gridDim.x * 8)
        sort_segment<128, 8, true>(a, a.lists[kSplitShort * a.stride + k], sm + g * padded<8>(1024), cnt + g * 1024,
                                   scratch + g * 12, t & 127,
                                   [&]() { asm volatile("bar.sync %0, 128;" ::"r"(g + 1) : "memory"); });
    __syncthreads();
    for (uint32_t k = blockIdx.x; k < nj; k += gridDim.x) {
        const uint4 job = a.jobs[k];
        const uint2 c = chunk_of(job, job.w);
        sort_spread_big((int)(c.y - c.x), sm, cnt, scratch, t, [&](int j) { return a.pairs[c.x + j]; },
                        [&](int at, u64 key) { a.pairs[c.x + at] = key; });
    }
}

// Number of keys of the sorted chunk c below p.
__device__ __forceinline__ uint32_t keys_below(const u64 *pairs, uint2 c, u64 p) {
    uint32_t lo = c.x, hi = c.y;
    while (lo < hi) {
        const uint32_t mid = lo + (hi - lo) / 2u;
        if (pairs[mid] < p) lo = mid + 1u;
        else hi = mid;
    }
    return lo - c.x;
}

// How many keys of each sorted chunk belong to the first target[0] and to the first target[1] keys of the whole list
// (keys are unique): for each target the least p with that many keys below it, found 17-fold a round, one
// candidate a warp, half of the warps a target: first among the multiples of 2^32 (the depths), then, where
// several entries share the depth at the cut, among the keys.
__device__ __forceinline__ void split_chunks(const BinArgs &a, uint4 job, uint32_t nch, const uint32_t (&target)[2],
                                             uint32_t *from, uint32_t *to, uint32_t *s_below, uint32_t *s_range) {
    const int t = threadIdx.x, lane = t & 31, w = t >> 5, half = w >> 4;
    if (t == 0) { s_range[0] = 0xffffffffu; s_range[1] = 0u; }
    __syncthreads();
    for (uint32_t c = t; c < nch; c += 1024) {
        const uint2 ch = chunk_of(job, c);
        atomicMin(&s_range[0], (uint32_t)(a.pairs[ch.x] >> 32));
        atomicMax(&s_range[1], (uint32_t)(a.pairs[ch.y - 1u] >> 32));
    }
    __syncthreads();
    u64 lo[2], hi[2];
#pragma unroll
    for (int h = 0; h < 2; ++h) { lo[h] = s_range[0]; hi[h] = (u64)s_range[1] + 1u; }
#pragma unroll
    for (int shift = 32; shift >= 0; shift -= 32) {
        while (lo[0] < hi[0] || lo[1] < hi[1]) {  // uniform for the CTA
            auto pivot = [&](int h, int k) {
                const u64 span = hi[h] - lo[h], q = span / 17u;
                return q ? lo[h] + q * (u64)(k + 1) : lo[h] + min((u64)k, span);
            };
            const u64 p = pivot(half, w & 15) << shift;
            uint32_t below = 0;
            for (uint32_t c = lane; c < nch; c += 32) below += keys_below(a.pairs, chunk_of(job, c), p);
            below = __reduce_add_sync(0xffffffffu, below);
            if (lane == 0) s_below[w] = below;
            __syncthreads();
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                int k = 0;
                while (k < 16 && s_below[16 * h + k] < target[h]) ++k;
                const u64 nlo = k > 0 ? min(pivot(h, k - 1) + 1u, hi[h]) : lo[h], nhi = k < 16 ? pivot(h, k) : hi[h];
                lo[h] = nlo;
                hi[h] = nhi;
            }
            __syncthreads();
        }
        if (shift == 32) {  // the cut lies in (lo - 1, lo] << 32
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                hi[h] = lo[h] << 32;
                lo[h] = (lo[h] > 0 ? lo[h] - 1u : 0u) << 32;
            }
            // most cuts fall between two depths: then the search among the keys has nothing to do
            uint32_t below = 0;
            for (uint32_t c = lane; c < nch; c += 32) below += keys_below(a.pairs, chunk_of(job, c), hi[half]);
            below = __reduce_add_sync(0xffffffffu, below);
            if (lane == 0) s_below[w] = below;
            __syncthreads();
#pragma unroll
            for (int h = 0; h < 2; ++h)
                if (s_below[16 * h] == target[h]) lo[h] = hi[h];
            __syncthreads();
        }
    }
    for (uint32_t c = t; c < nch; c += 1024) {
        const uint2 ch = chunk_of(job, c);
        from[c] = keys_below(a.pairs, ch, lo[0]);
        to[c] = keys_below(a.pairs, ch, lo[1]);
    }
    __syncthreads();
}

// The lists of more than kBigList entries, from their sorted chunks: job q produces the q-th of as many parts of
// the whole list, gathering its keys from all chunks and sorting them once more.
__global__ void __launch_bounds__(1024) k_merge_chunks(const BinArgs a, uint32_t max_chunks) {
    extern __shared__ u64 sm[];
    __shared__ uint32_t s_warp[33], s_below[32], s_range[2], scratch[3 * 32];
    uint32_t *cnt = reinterpret_cast<uint32_t *>(sm + padded<kBigItems>(kBigList));
    uint32_t *from = cnt, *to = from + max_chunks;  // needed before the sort only (max_chunks <= kBigList / 2)
    const int t = threadIdx.x;
    const uint32_t nj = a.aux->n_jobs;
    for (uint32_t k = blockIdx.x; k < nj; k += gridDim.x) {
        const uint4 job = a.jobs[k];
        const uint32_t nch = (job.y - job.x + kBigList - 1u) / kBigList;
        const uint2 part = chunk_of(job, job.w);
        const uint32_t target[2] = {part.x - job.x, part.y - job.x};
        split_chunks(a, job, nch, target, from, to, s_below, s_range);
        uint32_t run = 0;
        for (uint32_t c0 = 0; c0 < nch; c0 += 1024) {  // a chunk a thread finds its place, then the CTA copies them
            const uint32_t c = c0 + t, n = c < nch ? to[c] - from[c] : 0u;
            uint32_t tot;
            const uint32_t at = run + block_excl_scan(n, s_warp, tot);
            run += tot;
            if (c < nch) to[c] = at;  // from now on: the part's offset of this chunk's keys
        }
        __syncthreads();
        const int len = (int)(part.y - part.x), lane = t & 31;
        for (uint32_t c = t >> 5; c < nch; c += 32) {
            const uint32_t at = to[c], n = (c + 1 < nch ? to[c + 1] : (uint32_t)len) - at;
            const uint32_t src = chunk_of(job, c).x + from[c];
            for (uint32_t j = lane; j < n; j += 32) sm[padded<kBigItems>((int)(at + j))] = a.pairs[src + j];
        }
        __syncthreads();
        sort_spread<1024, kBigItems>(len, sm, cnt, scratch, t, []() { __syncthreads(); },
                                     [&](int j) { return sm[padded<kBigItems>(j)]; },
                                     [&](int at, u64 key) {
                                         a.inst_entry[part.x + at] = (uint32_t)key;
                                         a.inst_tile[part.x + at] = job.z;
                                     });
    }
}

static int sm_count() {
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    return sms > 0 ? sms : 1;
}

template <bool EMIT, bool SHARED, bool SLABS>
static cudaError_t launch_instances_t(const BinArgs &a, uint32_t grid, uint32_t threads, int smem, cudaStream_t s) {
    if (SHARED) {
        // on every call: the attribute belongs to the current device. Always the same bound: with this call's own size
        // a thread binning a smaller view could lower it between another's attribute and launch
        const cudaError_t e = cudaFuncSetAttribute(k_instances<EMIT, SHARED, SLABS>,
                                                   cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                   (int)(sizeof(uint32_t) * kSharedCounters));
        if (e != cudaSuccess) return e;
    }
    k_instances<EMIT, SHARED, SLABS><<<grid, threads, smem, s>>>(a);
    return cudaGetLastError();
}

template <bool EMIT>
static cudaError_t launch_instances(const BinArgs &a, bool shared, uint32_t grid, uint32_t threads, int smem,
                                    cudaStream_t s) {
    if (a.slabs > 1)
        return shared ? launch_instances_t<EMIT, true, true>(a, grid, threads, smem, s)
                      : launch_instances_t<EMIT, false, true>(a, grid, threads, smem, s);
    return shared ? launch_instances_t<EMIT, true, false>(a, grid, threads, smem, s)
                  : launch_instances_t<EMIT, false, false>(a, grid, threads, smem, s);
}

cudaError_t launch_bin(const BinArgs &a, cudaStream_t s) {
    const uint32_t n_tiles = (uint32_t)a.V.n_tiles;
    // 0. counters (aux is 256-byte aligned inside bins and its array ends on such a boundary), the capacity's cut
    static_assert(sizeof(TileAux) % 16 == 0, "cleared with the counts after it, 16 bytes at a time");
    k_bin_begin<<<kCutCtas, 1024, 0, s>>>(a, reinterpret_cast<uint4 *>(a.aux),
                                          (sizeof(TileAux) + sizeof(uint32_t) * (uint64_t)n_tiles * a.slabs + 15u) / 16u);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    const int sms = sm_count();
    // 1. instances per tile: counted in shared memory while a view's counters fit; a CTA takes as many entries as
    // still leave a few CTAs for every SM
    BinArgs c = a;
    const uint32_t counters = most_tiles(a.V) * a.slabs;
    const bool shared = inst_shared(a.n, a.V);  // as the layout was made for
    c.per_cta = inst_entries(a.n, a.n_views);
    c.parts = inst_parts(a.n, a.n_views);
    c.own = c.parts == 1u;
    const uint32_t grid = ceil_div_u64((uint64_t)a.n, c.per_cta) * c.parts * (uint32_t)a.n_views;
    const uint32_t threads = min(c.per_cta, (uint32_t)kInstThreads);
    const int inst_smem = shared ? (int)(sizeof(uint32_t) * counters) : 0;
    if (a.n > 0) {
        if (a.slabs > 1) k_depth_range<<<dim3(ceil_div_u64((uint64_t)a.n, 2048), (uint32_t)a.n_views), 256, 0, s>>>(a);
        e = launch_instances<false>(c, shared, grid, threads, inst_smem, s);
        if (e != cudaSuccess) return e;
    }
    // 2. segments, ranges, sort classes, queue
    const uint32_t per = tiles_per_cta(n_tiles), nblk = tile_ctas(n_tiles);
    k_tile_sums<<<nblk, 1024, 0, s>>>(a, per);
    k_tile_index<<<nblk, 1024, 0, s>>>(a, per);
    if (a.n == 0) return cudaGetLastError();
    // 3. append
    e = launch_instances<true>(c, shared, grid, threads, inst_smem, s);
    if (e != cudaSuccess) return e;
    // 4. sort: a tile's list has at most one entry per splat
    const uint64_t longest = (uint64_t)a.n < a.cap ? (uint64_t)a.n : a.cap;
    if (longest > kBigList) k_split_lists<<<2 * sms, 1024, 0, s>>>(a);
    constexpr int list_smem = (int)(sizeof(u64) * padded<kListItems>(kCtaList) + sizeof(uint32_t) * kCtaList);
    e = cudaFuncSetAttribute(k_sort_lists, cudaFuncAttributeMaxDynamicSharedMemorySize, list_smem);
    if (e != cudaSuccess) return e;
    k_sort_lists<<<(uint32_t)min((uint64_t)(2 * sms), a.stride), kListThreads, list_smem, s>>>(a);
    if (longest > kCtaList) {
        constexpr int smem = (int)(sizeof(u64) * padded<kBigItems>(kBigList) + sizeof(uint32_t) * kBigList);
        e = cudaFuncSetAttribute(k_sort_big, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
        if (e != cudaSuccess) return e;
        k_sort_big<<<sms, 1024, smem, s>>>(a);
    }
    if (longest > kBigList) {
        const uint32_t max_chunks = ceil_div_u64(longest, kBigList);  // at most 4096: 67,108,864 entries in all
        constexpr int smem = (int)(sizeof(u64) * padded<kBigItems>(kBigList) + sizeof(uint32_t) * kBigList);
        e = cudaFuncSetAttribute(k_merge_chunks, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
        if (e != cudaSuccess) return e;
        k_merge_chunks<<<sms, 1024, smem, s>>>(a, max_chunks);
    }
    return cudaGetLastError();
}

}  // namespace ges
