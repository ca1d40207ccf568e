// Adaptive Voronoi cell list (arXiv 1701.02059, "Spatial Searching
// Algorithm"): centroid M-step, Morton relabel of the centroids, exact
// nearest-centroid E-step on a centroid grid, stable counting sort of the
// particles with the state gather, cell radii and neighbouring-cell lists.
//
// Every discrete output (cell of each particle, storage permutation,
// centroids, neighbouring cells) equals the FP64 definition bit for bit:
// integer arithmetic where the definition is integer (M-step, sort), FP32
// prefilters with a proven rounding band and an FP64 re-decision inside the
// band where the definition compares FP64 distances.
#include "integrator.cuh"

#include <algorithm>

namespace orbc {

// ============================================================== M-step
// S_k = sum over the members (lipids; every particle of a protein cell set)
// of minimg(x_i - c_k) on the 2^-40 grid (int64, exact, order-independent),
// n_k = their count.  Warp-aggregated 64-bit atomics.
__global__ void k_mstep_accum(View v, const int* __restrict__ cell_of, long long* __restrict__ S,
                              int* __restrict__ cnt) {
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    bool act = i < v.N;
    int c = -1;
    long long d[3] = {0, 0, 0};
    if (act) {
        const int ci = cell_of[i];
        const Inst& I = v.inst[find_inst(v.inst_k0, v.B, ci)];
        if (centroid_member(I, v.type[i])) {
            c = ci;
            for (int a = 0; a < 3; a++)
                d[a] = minimg_q(v.xq[(size_t)a * v.N + i] - v.cq[(size_t)a * v.Ktot + c], I.boxq[a], I.periodic[a]);
        }
    }
    const unsigned full = 0xffffffffu;   // every lane of the warp reaches this point
    unsigned grp = __match_any_sync(full, c);
    int leader = __ffs(grp) - 1;
    int lane = threadIdx.x & 31;
    long long s0 = d[0], s1 = d[1], s2 = d[2];
    int n = (c >= 0) ? 1 : 0;
    // the group leader sums its members (exact integers, any order)
    long long a0 = 0, a1 = 0, a2 = 0;
    int an = 0;
    unsigned m = grp;
    while (m) {
        int src = __ffs(m) - 1;
        m &= m - 1;
        a0 += __shfl_sync(grp, s0, src);
        a1 += __shfl_sync(grp, s1, src);
        a2 += __shfl_sync(grp, s2, src);
        an += __shfl_sync(grp, n, src);
    }
    if (c >= 0 && lane == leader) {
        atomicAdd((unsigned long long*)&S[(size_t)0 * v.Ktot + c], (unsigned long long)a0);
        atomicAdd((unsigned long long*)&S[(size_t)1 * v.Ktot + c], (unsigned long long)a1);
        atomicAdd((unsigned long long*)&S[(size_t)2 * v.Ktot + c], (unsigned long long)a2);
        atomicAdd(&cnt[c], an);
    }
}

// c_k <- c_k + floor((2 S_k + n_k) / (2 n_k)); periodic axes wrap into [0, L).
// cmove: the move of each centroid; dmax: the largest one of an instance's, as
// FP32 bits rounded up (warp-reduced before the atomics).
__global__ void k_mstep_finish(View v, long long* __restrict__ S, int* __restrict__ cnt, int iter,
                               unsigned* __restrict__ dmax, float* __restrict__ cmove) {
    int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= v.Ktot) return;
    int b = find_inst(v.inst_k0, v.B, k);
    const Inst& I = v.inst[b];
    int n = iter < I.n_lloyd ? cnt[k] : 0;   // instances past their k-means rounds keep c
    float mv2 = 0.f;
    for (int a = 0; a < 3; a++) {
        long long c = v.cq[(size_t)a * v.Ktot + k];
        long long step = 0;
        if (n > 0) step = floor_div_ll(2 * S[(size_t)a * v.Ktot + k] + n, 2 * (long long)n);
        const float sf = ll_to_float(step) * (float)kGridInv;
        mv2 = fmaf(sf, sf, mv2);
        c += step;
        if (I.periodic[a]) c = floor_mod_ll(c, I.boxq[a]);
        v.cq[(size_t)a * v.Ktot + k] = c;
        S[(size_t)a * v.Ktot + k] = 0;
    }
    cnt[k] = 0;
    const float move = sqrtf(mv2) * 1.0001f + 1e-6f;
    cmove[k] = move;
    const unsigned grp = __match_any_sync(__activemask(), b);
    const unsigned mv = __reduce_max_sync(grp, __float_as_uint(move));
    if ((int)(threadIdx.x & 31) == __ffs(grp) - 1) atomicMax(&dmax[b], mv);
}

// Rebuild M-step on cell-sorted particles: one warp per cell sums its members'
// grid displacements (exact int64, shuffles), updates the centroid and
// folds it into the instance bounding box (block-level, then atomics).
__global__ void k_mstep_sorted(View v, long long* __restrict__ bb, unsigned* __restrict__ dmax) {
    __shared__ long long wmin[8][3], wmax[8][3];
    __shared__ int winst[8];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int k = blockIdx.x * 8 + warp;
    int b = -1;
    long long c[3] = {0, 0, 0};
    if (k < v.Ktot) {
        b = find_inst(v.inst_k0, v.B, k);
        const Inst& I = v.inst[b];
        const int s = v.cell_start[k], e = v.cell_start[k + 1];
        for (int a = 0; a < 3; a++) c[a] = v.cq[(size_t)a * v.Ktot + k];
        long long S0 = 0, S1 = 0, S2 = 0;
        int n = 0;
        const size_t N = v.N;
        for (int p = s + lane; p < e; p += 32) {
            if (!centroid_member(I, v.type[p])) continue;
            S0 += minimg_q(v.xq[p] - c[0], I.boxq[0], I.periodic[0]);
            S1 += minimg_q(v.xq[N + p] - c[1], I.boxq[1], I.periodic[1]);
            S2 += minimg_q(v.xq[2 * N + p] - c[2], I.boxq[2], I.periodic[2]);
            n++;
        }
        for (int off = 16; off; off >>= 1) {
            S0 += __shfl_xor_sync(0xffffffffu, S0, off);
            S1 += __shfl_xor_sync(0xffffffffu, S1, off);
            S2 += __shfl_xor_sync(0xffffffffu, S2, off);
            n += __shfl_xor_sync(0xffffffffu, n, off);
        }
        long long S[3] = {S0, S1, S2};
        float mv2 = 0.f;
        for (int a = 0; a < 3; a++) {
            long long step = 0;
            if (n > 0) step = floor_div_ll(2 * S[a] + n, 2 * (long long)n);
            const float sf = ll_to_float(step) * (float)kGridInv;
            mv2 = fmaf(sf, sf, mv2);
            c[a] += step;
            if (I.periodic[a]) c[a] = floor_mod_ll(c[a], I.boxq[a]);
        }
        if (lane == 0) {
            for (int a = 0; a < 3; a++) v.cq[(size_t)a * v.Ktot + k] = c[a];
            if (dmax) atomicMax(&dmax[b], __float_as_uint(sqrtf(mv2) * 1.0001f + 1e-6f));
        }
    }
    if (lane == 0) {
        winst[warp] = b;
        for (int a = 0; a < 3; a++) { wmin[warp][a] = c[a]; wmax[warp][a] = c[a]; }
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        int cur = -1;
        long long mn[3], mx[3];
        for (int w = 0; w <= 8; w++) {
            int bw = (w < 8) ? winst[w] : -2;
            if (bw != cur) {
                if (cur >= 0)
                    for (int a = 0; a < 3; a++) { atomicMin(&bb[cur * 6 + a], mn[a]); atomicMax(&bb[cur * 6 + 3 + a], mx[a]); }
                cur = bw;
                if (bw >= 0) for (int a = 0; a < 3; a++) { mn[a] = wmin[w][a]; mx[a] = wmax[w][a]; }
            } else if (bw >= 0) {
                for (int a = 0; a < 3; a++) { mn[a] = min(mn[a], wmin[w][a]); mx[a] = max(mx[a], wmax[w][a]); }
            }
        }
    }
}

__device__ inline long long warp_min_ll(long long x) {
    for (int off = 16; off; off >>= 1) x = min(x, __shfl_xor_sync(0xffffffffu, x, off));
    return x;
}

// M-step from the sums the B-A-O-A launch accumulated (same terms as
// k_mstep_sorted, so the same centroids): one thread per cell updates c_k,
// clears the sums for the next step and folds the centroid into the
// instance's bounding box and its largest move (reduced over the block before
// the atomics).  The blocks from rot_block on take the B-A-O-A's left-over
// rotations instead (rot_rest; one launch fewer than on their own).
__global__ void __launch_bounds__(256) k_mstep_apply(View v, long long* __restrict__ S, int* __restrict__ cnt,
                                                     long long* __restrict__ bb, unsigned* __restrict__ dmax,
                                                     int rot_block, const long long* __restrict__ steps, int fused,
                                                     const int* __restrict__ rot_list, const int* __restrict__ rot_n) {
    if ((int)blockIdx.x >= rot_block) {
        rot_rest(v, v, steps, fused, rot_list, rot_n, (blockIdx.x - rot_block) * blockDim.x + threadIdx.x,
                 (gridDim.x - rot_block) * blockDim.x);
        return;
    }
    __shared__ long long red[8][6];
    __shared__ unsigned redm[8];
    __shared__ int s_b;
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    const bool act = k < v.Ktot;
    const size_t K = v.Ktot;
    const int b = act ? find_inst(v.inst_k0, v.B, k) : -1;
    long long c[3] = {0, 0, 0};
    float mv2 = 0.f;
    if (act) {
        const Inst& I = v.inst[b];
        const int n = cnt[k];
        for (int a = 0; a < 3; a++) {
            c[a] = v.cq[a * K + k];
            long long step = 0;
            if (n > 0) step = floor_div_ll(2 * S[a * K + k] + n, 2 * (long long)n);
            const float sf = ll_to_float(step) * (float)kGridInv;
            mv2 = fmaf(sf, sf, mv2);
            c[a] += step;
            if (I.periodic[a]) c[a] = floor_mod_ll(c[a], I.boxq[a]);
            v.cq[a * K + k] = c[a];
            S[a * K + k] = 0;
        }
        cnt[k] = 0;
    }
    const unsigned mv = __float_as_uint(sqrtf(mv2) * 1.0001f + 1e-6f);
    if (threadIdx.x == 0) s_b = b;
    __syncthreads();
    if (!__syncthreads_and(b == s_b || !act)) {
        // a block with cells of several instances
        if (act) {
            atomicMax(&dmax[b], mv);
            for (int a = 0; a < 3; a++) { atomicMin(&bb[b * 6 + a], c[a]); atomicMax(&bb[b * 6 + 3 + a], c[a]); }
        }
        return;
    }
    // one set of atomics per block
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    for (int a = 0; a < 6; a++) {
        const long long m = warp_min_ll(act ? (a < 3 ? c[a] : -c[a - 3]) : 0x7fffffffffffffffll);
        if (lane == 0) red[w][a] = m;
    }
    const unsigned mw = __reduce_max_sync(0xffffffffu, act ? mv : 0u);
    if (lane == 0) redm[w] = mw;
    __syncthreads();
    if (threadIdx.x < 6) {
        long long m = red[0][threadIdx.x];
        for (int q = 1; q < 8; q++) m = min(m, red[q][threadIdx.x]);
        if (threadIdx.x < 3) atomicMin(&bb[s_b * 6 + threadIdx.x], m);
        else atomicMax(&bb[s_b * 6 + threadIdx.x], -m);
    } else if (threadIdx.x == 32) {
        unsigned m = redm[0];
        for (int q = 1; q < 8; q++) m = max(m, redm[q]);
        atomicMax(&dmax[s_b], m);
    }
}

// ============================================================== Morton relabel
__global__ void k_fill_bbox(long long* bb, int B) {
    for (int t = threadIdx.x; t < B * 6; t += blockDim.x) bb[t] = ((t % 6) < 3) ? 0x7fffffffffffffffll : (-0x7fffffffffffffffll - 1);
}

// Bounding box of each instance's centroids (exact int64 min/max), reduced
// per block before the atomics.
__global__ void k_bbox(View v, long long* __restrict__ bb /* [B][6] */) {
    __shared__ long long smin[256][3], smax[256][3];
    __shared__ int sb[256];
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    const int t = threadIdx.x;
    sb[t] = -1;
    if (k < v.Ktot) {
        sb[t] = find_inst(v.inst_k0, v.B, k);
        for (int a = 0; a < 3; a++) smin[t][a] = smax[t][a] = v.cq[(size_t)a * v.Ktot + k];
    }
    __syncthreads();
    if (t == 0) {
        int cur = -2;
        long long mn[3] = {0, 0, 0}, mx[3] = {0, 0, 0};
        for (int q = 0; q <= 256; q++) {
            int bq = (q < 256) ? sb[q] : -3;
            if (bq != cur) {
                if (cur >= 0)
                    for (int a = 0; a < 3; a++) { atomicMin(&bb[cur * 6 + a], mn[a]); atomicMax(&bb[cur * 6 + 3 + a], mx[a]); }
                cur = bq;
                if (bq >= 0) for (int a = 0; a < 3; a++) { mn[a] = smin[q][a]; mx[a] = smax[q][a]; }
            } else if (bq >= 0) {
                for (int a = 0; a < 3; a++) { mn[a] = min(mn[a], smin[q][a]); mx[a] = max(mx[a], smax[q][a]); }
            }
        }
    }
}

__device__ inline unsigned long long spread3(unsigned long long x) {
    x &= 0x1fffffull;
    x = (x | (x << 32)) & 0x1f00000000ffffull;
    x = (x | (x << 16)) & 0x1f0000ff0000ffull;
    x = (x | (x << 8)) & 0x100f00f00f00f00full;
    x = (x | (x << 4)) & 0x10c30c30c30c30c3ull;
    x = (x | (x << 2)) & 0x1249249249249249ull;
    return x;
}

// Key: 21 bits per axis, q = min(2^21 - 1, floor((c - lo) * 2^21 / (hi - lo)))
// in FP64 exactly as the definition (c - lo is exact on the grid).  Also
// copies the centroids for the permutation that follows.
__global__ void k_morton_keys(View v, const long long* __restrict__ bb, unsigned long long* __restrict__ key,
                              long long* __restrict__ cq_copy) {
    int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= v.Ktot) return;
    int b = find_inst(v.inst_k0, v.B, k);
    unsigned long long kk = 0;
    for (int a = 0; a < 3; a++) {
        const long long c = v.cq[(size_t)a * v.Ktot + k];
        cq_copy[(size_t)a * v.Ktot + k] = c;
        double lo = grid_to_double(bb[b * 6 + a]), hi = grid_to_double(bb[b * 6 + 3 + a]);
        double s = (hi > lo) ? __ddiv_rn(2097152.0, __dsub_rn(hi, lo)) : 0.0;
        double t = __dmul_rn(__dsub_rn(grid_to_double(c), lo), s);
        double f = floor(t);
        unsigned long long q = (f >= 2097151.0) ? 2097151ull : (unsigned long long)f;
        kk |= spread3(q) << a;
    }
    key[k] = kk;
}

// Sort of (instance, key, index): bitonic sort of 1024-element tiles in
// shared memory, then each element's rank inside its instance is its rank in
// its own tile plus, for every other tile of the instance, the number of
// smaller elements there (binary search).  Keys are unique with the index.
constexpr int kTile = 1024;

struct SortRec { unsigned long long key; int idx; int inst; };

__device__ inline bool rec_less(const SortRec& a, const SortRec& b) {
    if (a.inst != b.inst) return a.inst < b.inst;
    if (a.key != b.key) return a.key < b.key;
    return a.idx < b.idx;
}

// One tile of kTile records sorted by a block of kTile threads (bitonic):
// exchanges across warps go through shared memory, the strides below 32
// through shuffles.
__device__ inline SortRec shfl_rec(const SortRec& r, int m) {
    SortRec o;
    o.key = __shfl_xor_sync(0xffffffffu, r.key, m);
    o.idx = __shfl_xor_sync(0xffffffffu, r.idx, m);
    o.inst = __shfl_xor_sync(0xffffffffu, r.inst, m);
    return o;
}

__global__ void __launch_bounds__(kTile) k_tile_sort(View v, const unsigned long long* __restrict__ key,
                                                    SortRec* __restrict__ out) {
    __shared__ SortRec sh[kTile];
    const int t = threadIdx.x;
    const int k = blockIdx.x * kTile + t;
    SortRec r;
    if (k < v.Ktot) { r.key = key[k]; r.idx = k; r.inst = find_inst(v.inst_k0, v.B, k); }
    else { r.key = ~0ull; r.idx = 0x7fffffff; r.inst = 0x7fffffff; }
    // the padding records sort last, so the network stops at the tile's
    // record count rounded up
    const int m = min(kTile, v.Ktot - (int)blockIdx.x * kTile);
    for (int size = 2; size < 2 * m; size <<= 1) {
        for (int stride = size >> 1; stride > 0; stride >>= 1) {
            SortRec o;
            if (stride >= 32) {
                sh[t] = r;
                __syncthreads();
                o = sh[t ^ stride];
                __syncthreads();
            } else {
                o = shfl_rec(r, stride);
            }
            // the lower slot of an ascending pair keeps the smaller record
            const bool up = (t & size) == 0, lower = (t & stride) == 0;
            const bool take = (lower == up) ? rec_less(o, r) : rec_less(r, o);
            if (take) r = o;
        }
    }
    out[blockIdx.x * kTile + t] = r;
}

// ============================================================== centroid grid
// Fixed per-instance geometry (origin, edge, dims); edge cells extend to
// infinity, so the face-distance bound of the shell search stays valid for
// centroids and particles outside the box.
__device__ inline int grid_coord(long long xq, const Inst& I, int a, float& rel) {
    long long d = xq - I.gorg[a];
    if (I.periodic[a]) d = floor_mod_ll(d, I.boxq[a]);
    // >> 20: units of 2^-20 sigma, |.| < 2^31 for |d| < 2048 sigma
    long long s = d >> 20;
    if (s > 2147483647ll) s = 2147483647ll;
    if (s < -2147483647ll) s = -2147483647ll;
    rel = (float)(int)s * 9.5367431640625e-07f;
    int g = (int)floorf(rel * I.ginv[a]);
    if (g < 0) g = 0;
    if (g >= I.gdim[a]) g = I.gdim[a] - 1;
    return g;
}

// Centroid k's grid cell: counted (gcount), noted (gidx) and its FP32 position
// relative to the grid origin (cf).
__device__ inline int grid_count_one(const Inst& I, int k, long long x, long long y, long long z,
                                     int* __restrict__ gcount, int* __restrict__ gidx, float4* __restrict__ cf,
                                     float4* f = nullptr) {
    float r[3];
    const int gx = grid_coord(x, I, 0, r[0]), gy = grid_coord(y, I, 1, r[1]), gz = grid_coord(z, I, 2, r[2]);
    const long long g = I.g0 + ((long long)gz * I.gdim[1] + gy) * I.gdim[0] + gx;
    gidx[k] = (int)g;
    cf[k] = make_float4(r[0], r[1], r[2], 0.f);
    if (f) *f = make_float4(r[0], r[1], r[2], 0.f);
    atomicAdd(&gcount[g], 1);
    return (int)g;
}

__global__ void k_grid_count(View v, int* __restrict__ gcount, int* __restrict__ gidx, float4* __restrict__ cf) {
    int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= v.Ktot) return;
    const Inst& I = v.inst[find_inst(v.inst_k0, v.B, k)];
    grid_count_one(I, k, v.cq[k], v.cq[(size_t)v.Ktot + k], v.cq[(size_t)2 * v.Ktot + k], gcount, gidx, cf);
}

// Centroid k to its place in grid order.  The counts are taken down to zero,
// ready for the next count.
__device__ inline void grid_fill_one(const View& v, int k, const int* __restrict__ gidx, int* __restrict__ gcount,
                                     const float4* __restrict__ cf) {
    const int g = gidx[k];
    const int pos = v.gstart[g] + atomicSub(&gcount[g], 1) - 1;
    float4 c = cf[k];
    c.w = __int_as_float(k);
    v.gcf[pos] = c;
}

__global__ void k_grid_fill(View v, const int* __restrict__ gidx, int* __restrict__ gcount, const float4* __restrict__ cf) {
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k < v.Ktot) grid_fill_one(v, k, gidx, gcount, cf);
}

// rank -> new cell index; writes order[new] = old and the permuted centroids,
// and counts each into its grid cell.
// Tiles wholly below or above a record need no search (nearly sorted keys
// between rebuilds make this the common case).
constexpr int kBoundTiles = 1024;   // tiles whose bounds a block keeps in shared memory

__global__ void k_rank_scatter(View v, const SortRec* __restrict__ tiles, int ntiles, const long long* __restrict__ cq_old,
                               int* __restrict__ new_of_old, int* __restrict__ gcount, int* __restrict__ gidx,
                               float4* __restrict__ cf, long long* __restrict__ bb) {
    // first and last key of every tile and its instance (-1: several): most
    // tiles lie wholly below or above a record, which these settle without a
    // search
    __shared__ unsigned long long tmin[kBoundTiles], tmax[kBoundTiles];
    __shared__ int tinst[kBoundTiles];
    const bool cached = ntiles <= kBoundTiles;
    if (cached)
        for (int t = threadIdx.x; t < ntiles; t += blockDim.x) {
            // (the last tile ends in padding records)
            const int last = min(kTile, v.Ktot - t * kTile) - 1;
            const SortRec a = tiles[(size_t)t * kTile], b = tiles[(size_t)t * kTile + last];
            tmin[t] = a.key;
            tmax[t] = b.key;
            tinst[t] = a.inst == b.inst ? a.inst : -1;
        }
    __syncthreads();
    int pos = blockIdx.x * blockDim.x + threadIdx.x;   // position in the tiled array
    // the bounding boxes, read by the keys, empty for the next step
    // (ntiles * kTile >= K >= B)
    if (pos < v.B)
        for (int a = 0; a < 6; a++) bb[pos * 6 + a] = a < 3 ? 0x7fffffffffffffffll : (-0x7fffffffffffffffll - 1);
    if (pos >= ntiles * kTile) return;
    SortRec me = tiles[pos];
    if (me.idx >= v.Ktot) return;
    const Inst& I = v.inst[me.inst];
    // rank inside the instance: over every tile holding part of the instance,
    // (records smaller than me) - (records of smaller instances)
    SortRec first;
    first.inst = me.inst; first.key = 0; first.idx = -1;
    int rank = 0;
    int t0 = I.k0 / kTile, t1 = (I.k0 + I.K - 1) / kTile;
    for (int t = t0; t <= t1; t++) {
        if (cached && tinst[t] == me.inst) {
            // (equal keys go by index: searched)
            if (me.key > tmax[t]) { rank += min(kTile, v.Ktot - t * kTile); continue; }
            if (me.key < tmin[t]) continue;
        }
        const SortRec* T = tiles + (size_t)t * kTile;
        const SortRec tfirst = T[0], tlast = T[kTile - 1];
        int lo, lo2;
        if (rec_less(tlast, me)) lo = kTile;
        else if (!rec_less(tfirst, me)) lo = 0;
        else {
            int a = 0, c = kTile;
            while (a < c) { int mid = (a + c) >> 1; if (rec_less(T[mid], me)) a = mid + 1; else c = mid; }
            lo = a;
        }
        if (rec_less(tlast, first)) lo2 = kTile;
        else if (!rec_less(tfirst, first)) lo2 = 0;
        else {
            int a = 0, c = kTile;
            while (a < c) { int mid = (a + c) >> 1; if (rec_less(T[mid], first)) a = mid + 1; else c = mid; }
            lo2 = a;
        }
        rank += lo - lo2;
    }
    int nk = I.k0 + rank;
    new_of_old[me.idx] = nk;
    long long c[3];
    for (int a = 0; a < 3; a++) {
        c[a] = cq_old[(size_t)a * v.Ktot + me.idx];
        v.cq[(size_t)a * v.Ktot + nk] = c[a];
    }
    grid_count_one(I, nk, c[0], c[1], c[2], gcount, gidx, cf);
}

// ============================================================== small batches
// M-step, Morton relabel and centroid grid of one instance of up to kSmallK
// cells in one block: five launches (M-step, keys, tile sort, ranks, grid
// scan) of one to four blocks each otherwise, 32-45 us of the 98-136 us of a
// step on 2,304 to 62k particles.  The outputs are those launches' (the
// grid's order inside a cell aside, which nothing depends on).  The blocks
// after the first take the left-over rotations (see k_mstep_apply).
constexpr int kSmallK = 1024;
constexpr int kSmallG = 1 << 16;

__global__ void __launch_bounds__(kSmallK) k_relabel_small(
    View v, int mstep, long long* __restrict__ S, int* __restrict__ cnt, unsigned* __restrict__ dmax,
    long long* __restrict__ bb, int* __restrict__ new_of_old, int* gcount, int* __restrict__ gidx, float4* __restrict__ cf,
    int* gstart, const long long* __restrict__ steps, int fused, const int* __restrict__ rot_list,
    const int* __restrict__ rot_n) {
    if (blockIdx.x > 0) {
        rot_rest(v, v, steps, fused, rot_list, rot_n, (blockIdx.x - 1) * blockDim.x + threadIdx.x,
                 (gridDim.x - 1) * blockDim.x);
        return;
    }
    __shared__ long long sc[3][kSmallK];                  // centroids by old index
    __shared__ unsigned long long skey[kSmallK];
    __shared__ unsigned short sidx[kSmallK];
    __shared__ long long red[32][6];                      // per warp: min x, y, z, -max x, y, z
    __shared__ float redm[32];
    __shared__ long long s_lo[3], s_hi[3];
    __shared__ unsigned long long s_m[3];                 // s = 2^21 / (hi - lo) = s_m 2^(es - 63)
    __shared__ int s_sh[3], s_r[3];
    const int t = threadIdx.x, lane = t & 31, w = t >> 5;
    const int K = v.Ktot;
    const size_t Ks = K;
    const Inst& I = v.inst[0];
    // M-step (k_mstep_apply's update)
    long long c[3] = {0, 0, 0};
    float mv2 = 0.f;
    if (t < K) {
        const int n = mstep ? cnt[t] : 0;
        for (int a = 0; a < 3; a++) {
            c[a] = v.cq[a * Ks + t];
            if (mstep) {
                long long step = 0;
                if (n > 0) step = floor_div_ll(2 * S[a * Ks + t] + n, 2 * (long long)n);
                const float sf = ll_to_float(step) * (float)kGridInv;
                mv2 = fmaf(sf, sf, mv2);
                c[a] += step;
                if (I.periodic[a]) c[a] = floor_mod_ll(c[a], I.boxq[a]);
                S[a * Ks + t] = 0;
            }
            sc[a][t] = c[a];
        }
        if (mstep) cnt[t] = 0;
    }
    // bounding box and largest move
    for (int a = 0; a < 3; a++) {
        const long long mn = warp_min_ll(t < K ? c[a] : 0x7fffffffffffffffll);
        const long long mx = warp_min_ll(t < K ? -c[a] : 0x7fffffffffffffffll);
        if (lane == 0) { red[w][a] = mn; red[w][3 + a] = mx; }
    }
    {
        const float mv = __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(sqrtf(mv2) * 1.0001f + 1e-6f)));
        if (lane == 0) redm[w] = mv;
    }
    __syncthreads();
    if (w == 0) {
        for (int a = 0; a < 6; a++) {
            const long long m = warp_min_ll(red[lane][a]);
            if (lane == 0) { if (a < 3) s_lo[a] = m; else s_hi[a - 3] = -m; }
        }
        const unsigned mv = __reduce_max_sync(0xffffffffu, __float_as_uint(redm[lane]));
        if (lane == 0 && mstep) dmax[0] = mv;
        __syncwarp();
        if (lane < 3) {
            // the keys' scale as the definition computes it, split for the
            // integer evaluation below
            const long long D = s_hi[lane] - s_lo[lane];
            const double s = D > 0 ? __ddiv_rn(2097152.0, __dsub_rn(grid_to_double(s_hi[lane]), grid_to_double(s_lo[lane]))) : 0.0;
            const long long bits = __double_as_longlong(s);
            const int es = (int)(bits >> 52) - 1023;
            s_m[lane] = D > 0 ? ((unsigned long long)(bits & 0xfffffffffffffll) | (1ull << 52)) << 11 : 0ull;
            s_sh[lane] = D > 0 ? __clzll(D) - 1 : 0;
            s_r[lane] = D > 0 ? 7 + s_sh[lane] - es : 8;
        }
        if (lane < 6) bb[lane] = lane < 3 ? 0x7fffffffffffffffll : (-0x7fffffffffffffffll - 1);
    }
    __syncthreads();
    // Morton keys: q = floor(fl((c - lo) s)).  (c - lo) s to 2^-32 in integers
    // (FP64 here would wait for the FP64 pipe of one SM); only a fraction
    // within 2^-32 of one can round to the next integer, and takes FP64.
    unsigned long long key = ~0ull;
    int idx = 0x7fff;
    if (t < K) {
        key = 0;
        idx = t;
        for (int a = 0; a < 3; a++) {
            const unsigned long long d = (unsigned long long)(c[a] - s_lo[a]);
            const unsigned long long f = __umul64hi(d << s_sh[a], s_m[a]) >> s_r[a];
            unsigned long long q = f >> 32;
            if ((unsigned)f == 0xffffffffu) {
                const double lo = grid_to_double(s_lo[a]);
                const double s = __ddiv_rn(2097152.0, __dsub_rn(grid_to_double(s_hi[a]), lo));
                q = (unsigned long long)floor(__dmul_rn(__dsub_rn(grid_to_double(c[a]), lo), s));
            }
            key |= spread3(min(q, 2097151ull)) << a;
        }
    }
    // bitonic sort of (key, index) over the next power of two (whole warps)
    int P = 32;
    while (P < K) P <<= 1;
    for (int size = 2; size <= P; size <<= 1) {
        for (int stride = size >> 1; stride > 0; stride >>= 1) {
            unsigned long long ok = key;
            int oi = idx;
            if (stride >= 32) {
                if (t < P) { skey[t] = key; sidx[t] = (unsigned short)idx; }
                __syncthreads();
                if (t < P) { ok = skey[t ^ stride]; oi = sidx[t ^ stride]; }
                __syncthreads();
            } else if (t < P) {
                ok = __shfl_xor_sync(0xffffffffu, key, stride);
                oi = __shfl_xor_sync(0xffffffffu, idx, stride);
            }
            const bool lower = (t & stride) == 0, up = (t & size) == 0;
            const bool less = ok < key || (ok == key && oi < idx);
            if (t < P && (lower == up) == less && (ok != key || oi != idx)) { key = ok; idx = oi; }
        }
    }
    // the record of rank t: old cell idx becomes cell t
    int gc = 0;
    float4 f = make_float4(0.f, 0.f, 0.f, 0.f);
    if (t < K) {
        new_of_old[idx] = t;
        for (int a = 0; a < 3; a++) {
            c[a] = sc[a][idx];
            v.cq[a * Ks + t] = c[a];
        }
        gc = grid_count_one(I, t, c[0], c[1], c[2], gcount, gidx, cf, &f);
    }
    __threadfence();
    __syncthreads();
    // grid starts: exclusive scan of the counts (written by atomics above:
    // read past L1), a contiguous chunk per thread, the first eight counts
    // kept for the second pass
    const int G = (int)v.Gtot + 1, per = ((G + kSmallK - 1) / kSmallK + 3) & ~3, g0 = min(t * per, G), g1 = min(g0 + per, G);
    int4 k0 = make_int4(0, 0, 0, 0), k1 = k0;
    if (g0 + 8 <= g1) {
        k0 = __ldcg(reinterpret_cast<const int4*>(gcount + g0));
        k1 = __ldcg(reinterpret_cast<const int4*>(gcount + g0 + 4));
    } else {
        int q[8];
#pragma unroll
        for (int u = 0; u < 8; u++) q[u] = g0 + u < g1 ? __ldcg(gcount + g0 + u) : 0;
        k0 = make_int4(q[0], q[1], q[2], q[3]);
        k1 = make_int4(q[4], q[5], q[6], q[7]);
    }
    int sum = k0.x + k0.y + k0.z + k0.w + k1.x + k1.y + k1.z + k1.w;
    for (int g = g0 + 8; g < g1; g++) sum += __ldcg(gcount + g);
    int x = sum;
    for (int off = 1; off < 32; off <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, x, off);
        if (lane >= off) x += y;
    }
    int* wtot = reinterpret_cast<int*>(&red[0][0]);
    if (lane == 31) wtot[w] = x;
    __syncthreads();
    if (w == 0) {
        int s = wtot[lane];
        for (int off = 1; off < 32; off <<= 1) {
            const int y = __shfl_up_sync(0xffffffffu, s, off);
            if (lane >= off) s += y;
        }
        wtot[lane] = s;
    }
    __syncthreads();
    int run = x - sum + (w > 0 ? wtot[w - 1] : 0);
    {
        const int q[8] = {k0.x, k0.y, k0.z, k0.w, k1.x, k1.y, k1.z, k1.w};
#pragma unroll
        for (int u = 0; u < 8; u++) {
            if (g0 + u < g1) gstart[g0 + u] = run;
            run += q[u];
        }
    }
    for (int g = g0 + 8; g < g1; g++) {
        gstart[g] = run;
        run += __ldcg(gcount + g);
    }
    __threadfence();
    __syncthreads();
    if (t < K) {
        const int pos = __ldcg(gstart + gc) + atomicSub(&gcount[gc], 1) - 1;
        f.w = __int_as_float(t);
        v.gcf[pos] = f;
    }
}

// ============================================================== E-step
// Exact nearest centroid (ties to the lowest index) of every particle.
// FP32 distances relative to the grid origin have an absolute error below
// kBand (coordinates < 2048 sigma carry <= 1.3e-4 sigma each); the shell
// search stops once the unexplored region is farther than best + band, and
// every centroid within band of the FP32 best is re-scored in FP64 with the
// definition's operation order.  A single candidate in the band is the
// exact answer without FP64.
constexpr float kBandE = 2e-3f;
// margin of the FP32 certificates of the E-steps (coordinates up to ~2000 sigma)
constexpr float kCertMargin = 4e-3f;

__device__ inline float axis_dist(float p, float c, const Inst& I, int a) {
    float d = p - c;
    if (I.periodic[a]) d -= I.boxf[a] * rintf(d / I.boxf[a]);
    return d;
}

__device__ inline int wrap_idx(int x, int n) { x %= n; return x < 0 ? x + n : x; }

// Is grid index w (wrapped) inside the cube of Chebyshev radius r around g?
__device__ inline bool in_cube(const int w[3], const int g[3], int r, const Inst& I) {
    for (int a = 0; a < 3; a++) {
        if (I.periodic[a]) {
            if (2 * r + 1 >= I.gdim[a]) continue;
            int d = wrap_idx(w[a] - g[a], I.gdim[a]);
            if (min(d, I.gdim[a] - d) > r) return false;
        } else {
            if (w[a] < g[a] - r || w[a] > g[a] + r) return false;
        }
    }
    return true;
}

// Visit every grid cell of cube(r) \ cube(r - 1) exactly once (periodic axes
// wrap; once an axis is fully covered it is enumerated without repeats).
template <typename F>
__device__ inline void for_shell(const int g[3], int r, const Inst& I, F&& f) {
    int lo[3], hi[3];
    for (int a = 0; a < 3; a++) {
        if (I.periodic[a]) {
            if (2 * r + 1 >= I.gdim[a]) { lo[a] = 0; hi[a] = I.gdim[a] - 1; }
            else { lo[a] = g[a] - r; hi[a] = g[a] + r; }
        } else {
            lo[a] = max(0, g[a] - r);
            hi[a] = min(I.gdim[a] - 1, g[a] + r);
        }
    }
    for (int z = lo[2]; z <= hi[2]; z++)
        for (int y = lo[1]; y <= hi[1]; y++)
            for (int x = lo[0]; x <= hi[0]; x++) {
                int w[3] = { I.periodic[0] ? wrap_idx(x, I.gdim[0]) : x, I.periodic[1] ? wrap_idx(y, I.gdim[1]) : y,
                             I.periodic[2] ? wrap_idx(z, I.gdim[2]) : z };
                if (r > 0 && in_cube(w, g, r - 1, I)) continue;
                long long gg = I.g0 + ((long long)w[2] * I.gdim[1] + w[1]) * I.gdim[0] + w[0];
                f(gg);
            }
}

// lower bound of the distance from p to anything outside the searched cube
__device__ inline float shell_bound(const float p[3], const int g[3], int r, const Inst& I, bool& exhausted) {
    float lb = 3.0e38f;
    exhausted = true;
    for (int a = 0; a < 3; a++) {
        if (I.periodic[a]) {
            if (2 * r + 1 >= I.gdim[a]) continue;
            float h = I.gh[a];
            float lo = p[a] - (g[a] - r) * h, hi = (g[a] + r + 1) * h - p[a];
            lb = fminf(lb, fminf(lo, hi));
            exhausted = false;
        } else {
            if (g[a] - r > 0) { lb = fminf(lb, p[a] - (g[a] - r) * I.gh[a]); exhausted = false; }
            if (g[a] + r < I.gdim[a] - 1) { lb = fminf(lb, (g[a] + r + 1) * I.gh[a] - p[a]); exhausted = false; }
        }
    }
    return lb;
}

// lbound (nullable) receives a lower bound on the distance from the particle
// to every centroid but the one it is assigned: the second-best scanned
// distance or the bound on the unscanned shells, whichever is smaller (0
// when the winner was decided inside the tie band).
__device__ void estep_one(const View& v, int i, int* __restrict__ cell_out, float* __restrict__ lbound = nullptr) {
    int b = find_inst(v.inst_p0, v.B, i);
    const Inst& I = v.inst[b];
    long long xq[3] = { v.xq[i], v.xq[(size_t)v.N + i], v.xq[(size_t)2 * v.N + i] };
    float p[3];
    int g[3];
    for (int a = 0; a < 3; a++) g[a] = grid_coord(xq[a], I, a, p[a]);
    float best = 3.0e38f, second = 3.0e38f;     // FP32 distances squared
    float lbx = 3.0e38f;                         // bound on the unscanned shells
    int r = 0;
    const int rmax = max(I.gdim[0], max(I.gdim[1], I.gdim[2]));
    for (;; r++) {
        for_shell(g, r, I, [&](long long gg) {
            for (int q = v.gstart[gg]; q < v.gstart[gg + 1]; q++) {
                float4 c = v.gcf[q];
                float dx = axis_dist(p[0], c.x, I, 0), dy = axis_dist(p[1], c.y, I, 1), dz = axis_dist(p[2], c.z, I, 2);
                float d2 = fmaf(dx, dx, fmaf(dy, dy, dz * dz));
                second = fminf(second, fmaxf(best, d2));
                best = fminf(best, d2);
            }
        });
        bool ex;
        float lb = shell_bound(p, g, r, I, ex);
        if (ex || r >= rmax) break;
        if (best < 3.0e38f && lb > sqrtf(best) + kBandE) { lbx = lb; break; }
    }
    // second pass over the searched cube: candidates within the band
    float lim = sqrtf(best) + kBandE;
    float lim2 = lim * lim;
    int ncand = 0, k1 = -1, bestk = -1;
    double best64 = 0.0;
    for (int rr = 0; rr <= r; rr++) {
        for_shell(g, rr, I, [&](long long gg) {
            for (int q = v.gstart[gg]; q < v.gstart[gg + 1]; q++) {
                float4 c = v.gcf[q];
                float dx = axis_dist(p[0], c.x, I, 0), dy = axis_dist(p[1], c.y, I, 1), dz = axis_dist(p[2], c.z, I, 2);
                float d2 = fmaf(dx, dx, fmaf(dy, dy, dz * dz));
                if (d2 <= lim2) {
                    int k = __float_as_int(c.w);
                    ncand++;
                    if (ncand == 1) { k1 = k; continue; }
                    if (ncand == 2) {
                        best64 = dist2_grid_d(xq[0], xq[1], xq[2], v.cq[k1], v.cq[(size_t)v.Ktot + k1],
                                              v.cq[(size_t)2 * v.Ktot + k1], I);
                        bestk = k1;
                    }
                    double d64 = dist2_grid_d(xq[0], xq[1], xq[2], v.cq[k], v.cq[(size_t)v.Ktot + k],
                                              v.cq[(size_t)2 * v.Ktot + k], I);
                    if (d64 < best64 || (d64 == best64 && k < bestk)) { best64 = d64; bestk = k; }
                }
            }
        });
    }
    if (ncand == 0) {   // unreachable for finite input: the search covers every centroid
        flag_inst(v, I, kStatusGridRange);
        cell_out[i] = I.k0;
        if (lbound) lbound[i] = 0.f;
        return;
    }
    cell_out[i] = (ncand == 1) ? k1 : bestk;
    if (lbound) lbound[i] = (ncand == 1) ? fminf(sqrtf(second), lbx) : 0.f;
}

// ---- warp-cooperative search for instances without periodic axes: the
// 32 queries of a warp (consecutive storage slots, hence neighbours in space)
// share one grid region [lo - r, hi + r]; every lane scores every centroid
// of the region (broadcast loads), and the region grows by one ring until
// each lane's unexplored space is provably farther than its band.
// The centroids of the region's grid cells (ring: without those of the region
// at r - 1), f(centroid) with the whole warp.  A lane looks at a grid cell and
// loads its centroids, and the warp passes them round: on a membrane most of
// the 27 to 125 grid cells are empty, and one after the other each of them
// would cost the warp a chain of loads (160 against 112 us for the first
// round of 500,000 particles, 78 against 52 for the later ones).
template <typename F>
__device__ __forceinline__ void region_visit(const View& v, const Inst& I, const int lo[3], const int hi[3], int r,
                                             bool ring, F&& f) {
    const unsigned full = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    int a0[3], ext[3];
    for (int a = 0; a < 3; a++) {
        a0[a] = max(0, lo[a] - r);
        ext[a] = min(I.gdim[a] - 1, hi[a] + r) - a0[a] + 1;
    }
    const int n = ext[0] * ext[1] * ext[2];    // (the whole grid has up to 2^24 cells)
    for (int base = 0; base < n; base += 32) {
        const int t = base + lane;
        int s = 0, c = 0;
        if (t < n) {
            const int x = a0[0] + t % ext[0], y = a0[1] + t / ext[0] % ext[1], z = a0[2] + t / (ext[0] * ext[1]);
            const bool inner = ring && r > 0 && x >= lo[0] - r + 1 && x <= hi[0] + r - 1 && y >= lo[1] - r + 1 &&
                               y <= hi[1] + r - 1 && z >= lo[2] - r + 1 && z <= hi[2] + r - 1;
            if (!inner) {
                const long long gg = I.g0 + ((long long)z * I.gdim[1] + y) * I.gdim[0] + x;
                s = v.gstart[gg];
                c = v.gstart[gg + 1] - s;
            }
        }
        for (int u = 0;; u++) {
            unsigned m = __ballot_sync(full, c > u);
            if (!m) break;
            const float4 own = c > u ? v.gcf[s + u] : make_float4(0.f, 0.f, 0.f, 0.f);
            while (m) {
                const int src = __ffs(m) - 1;
                m &= m - 1;
                f(make_float4(__shfl_sync(full, own.x, src), __shfl_sync(full, own.y, src), __shfl_sync(full, own.z, src),
                              __shfl_sync(full, own.w, src)));
            }
        }
    }
}

__device__ inline float region_bound(const Inst& I, const float p[3], const int lo[3], const int hi[3], int r,
                                     bool& exhausted) {
    float lb = 3.0e38f;
    exhausted = true;
    for (int a = 0; a < 3; a++) {
        if (lo[a] - r > 0) { lb = fminf(lb, p[a] - (lo[a] - r) * I.gh[a]); exhausted = false; }
        if (hi[a] + r < I.gdim[a] - 1) { lb = fminf(lb, (hi[a] + r + 1) * I.gh[a] - p[a]); exhausted = false; }
    }
    return lb;
}

__device__ inline void warp_box(const int g[3], bool valid, int lo[3], int hi[3]) {
    for (int a = 0; a < 3; a++) {
        int l = valid ? g[a] : 0x7fffffff, h = valid ? g[a] : -1;
        for (int off = 16; off; off >>= 1) {
            l = min(l, __shfl_xor_sync(0xffffffffu, l, off));
            h = max(h, __shfl_xor_sync(0xffffffffu, h, off));
        }
        lo[a] = l;
        hi[a] = h;
    }
}

// The search of the lanes with `in` set (whose grid cells lie in lo..hi), by
// the whole warp.
__device__ __forceinline__ void estep_group(const View& v, const Inst& I, int i, bool in, const long long xq[3],
                                            const float p[3], const int lo[3], const int hi[3],
                                            int* __restrict__ cell_out, float* __restrict__ lbound) {
    float best = 3.0e38f, second = 3.0e38f;
    float lbr = 3.0e38f;    // bound on the unscanned region after the last ring
    int bk = -1;
    int r = 0;
    for (;; r++) {
        region_visit(v, I, lo, hi, r, true, [&](const float4 c) {
            const float dx = p[0] - c.x, dy = p[1] - c.y, dz = p[2] - c.z;
            const float d2 = fmaf(dx, dx, fmaf(dy, dy, dz * dz));
            if (d2 < best) { second = best; best = d2; bk = __float_as_int(c.w); }
            else if (d2 < second) second = d2;
        });
        bool ex;
        const float lb = region_bound(I, p, lo, hi, r, ex);
        lbr = ex ? 3.0e38f : lb;
        const bool done = !in || ex || (best < 3.0e38f && lb > sqrtf(best) + kBandE);
        if (__all_sync(0xffffffffu, done)) break;
    }
    // tie band: every centroid within the band of the FP32 best is re-scored in FP64
    const float lim = sqrtf(best) + kBandE;
    const bool amb = in && second <= lim * lim;
    if (__any_sync(0xffffffffu, amb)) {
        double best64 = 1e300;
        int bk64 = -1;
        region_visit(v, I, lo, hi, r, false, [&](const float4 c) {
            const float dx = p[0] - c.x, dy = p[1] - c.y, dz = p[2] - c.z;
            const float d2 = fmaf(dx, dx, fmaf(dy, dy, dz * dz));
            if (amb && d2 <= lim * lim) {
                const int k = __float_as_int(c.w);
                const double d64 = dist2_grid_d(xq[0], xq[1], xq[2], v.cq[k], v.cq[(size_t)v.Ktot + k],
                                                v.cq[(size_t)2 * v.Ktot + k], I);
                if (d64 < best64 || (d64 == best64 && k < bk64)) { best64 = d64; bk64 = k; }
            }
        });
        if (amb) bk = bk64;
    }
    if (in) {
        if (bk < 0) { flag_inst(v, I, kStatusGridRange); bk = I.k0; }
        cell_out[i] = bk;
        if (lbound) lbound[i] = amb ? 0.f : fminf(sqrtf(second), lbr);
    }
}

// list (nullable): search only the particles listed, *count of them (null:
// all of v.N), in list order, which keeps the lanes of a warp close in space.
// A warp whose particles lie in several places (its list runs on from one row
// of grid cells to another) takes up to eight of them one after the other
// (three: 112 us for the first round of 500,000 particles and 50 for the
// later ones, eight: 58 and 40, any number the same).
__global__ void k_estep_warp(View v, int* __restrict__ cell_out, float* __restrict__ lbound,
                             const int* __restrict__ list, const int* __restrict__ count) {
    const int q = blockIdx.x * blockDim.x + threadIdx.x;
    const bool valid = q < (count ? *count : v.N);
    const int i = valid ? (list ? list[q] : q) : 0;
    const int b = valid ? find_inst(v.inst_p0, v.B, i) : -1;
    int b0 = __shfl_sync(0xffffffffu, b, 0);
    const int bfirst = __reduce_max_sync(0xffffffffu, valid ? b : -1);
    if (b0 < 0) b0 = bfirst;
    const bool same = __all_sync(0xffffffffu, !valid || b == b0);
    if (b0 < 0) return;
    const Inst& I = v.inst[b0];
    const bool periodic = I.periodic[0] | I.periodic[1] | I.periodic[2];
    if (!same || periodic) {
        // mixed instances or periodic axes: per-thread shell search
        if (valid) estep_one(v, i, cell_out, lbound);
        return;
    }
    long long xq[3] = {0, 0, 0};
    float p[3] = {0, 0, 0};
    int g[3] = {0, 0, 0};
    if (valid) {
        xq[0] = v.xq[i]; xq[1] = v.xq[(size_t)v.N + i]; xq[2] = v.xq[(size_t)2 * v.N + i];
        for (int a = 0; a < 3; a++) g[a] = grid_coord(xq[a], I, a, p[a]);
    }
    int lo[3], hi[3];
    warp_box(g, valid, lo, hi);
    if (hi[0] - lo[0] <= 2 && hi[1] - lo[1] <= 2 && hi[2] - lo[2] <= 2) {
        estep_group(v, I, i, valid, xq, p, lo, hi, cell_out, lbound);
        return;
    }
    unsigned todo = __ballot_sync(0xffffffffu, valid);
    for (int part = 0; todo && part < 8; part++) {
        const int lead = __ffs(todo) - 1;
        bool in = (todo >> (threadIdx.x & 31)) & 1u;
        for (int a = 0; a < 3; a++) in = abs(g[a] - __shfl_sync(0xffffffffu, g[a], lead)) <= 1 && in;
        warp_box(g, in, lo, hi);
        estep_group(v, I, i, in, xq, p, lo, hi, cell_out, lbound);
        todo &= ~__ballot_sync(0xffffffffu, in);
    }
    // the others: per-thread search
    if ((todo >> (threadIdx.x & 31)) & 1u) estep_one(v, i, cell_out, lbound);
}

// The particles by grid cell, for the searches of the initialisation: the
// input's order need not be one in space, and a warp whose lanes lie apart
// searches thread by thread (500,000 particles, ten rounds and the search
// after them: 1,720 us, 500 in this order, 35 to make it).  Counts per grid cell (gcount, zero before and
// after), then each particle's place: its position and type in the second
// buffers, its slot in order.  The order within a grid cell changes nothing
// (each particle's search is its own, and the centroids' sums are integers).
__device__ inline long long grid_cell(const View& v, const Inst& I, int i) {
    int g[3];
    float p;
    for (int a = 0; a < 3; a++) g[a] = grid_coord(v.xq[(size_t)a * v.N + i], I, a, p);
    return I.g0 + ((long long)g[2] * I.gdim[1] + g[1]) * I.gdim[0] + g[0];
}

__global__ void k_grid_particles(View v, int* __restrict__ gcount) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < v.N) atomicAdd(&gcount[grid_cell(v, v.inst[find_inst(v.inst_p0, v.B, i)], i)], 1);
}

__global__ void k_grid_order(View v, View to, const int* __restrict__ gstart, int* __restrict__ gcount,
                             int* __restrict__ order) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= v.N) return;
    const long long g = grid_cell(v, v.inst[find_inst(v.inst_p0, v.B, i)], i);
    const int q = gstart[g] + atomicSub(&gcount[g], 1) - 1;
    for (int a = 0; a < 3; a++) to.xq[(size_t)a * v.N + q] = v.xq[(size_t)a * v.N + i];
    to.type[q] = v.type[i];
    order[q] = i;
}

// One particle's nearest centroid by a whole warp: the lanes share the grid
// cells of each shell (see estep_one for the bounds; the same answer: the
// FP32 best alone in its band, else the FP64 best, ties to the lowest index).
__device__ int estep_warp_one(const View& v, int i) {
    const int lane = threadIdx.x & 31;
    const unsigned full = 0xffffffffu;
    const Inst& I = v.inst[find_inst(v.inst_p0, v.B, i)];
    const long long xq[3] = { v.xq[i], v.xq[(size_t)v.N + i], v.xq[(size_t)2 * v.N + i] };
    float p[3];
    int g[3];
    for (int a = 0; a < 3; a++) g[a] = grid_coord(xq[a], I, a, p[a]);
    // visits the centroids of cube(r) (skipping cube(r - 1) when shell is set)
    auto scan = [&](int r, bool shell, auto&& f) {
        int lo[3], ext[3];
        for (int a = 0; a < 3; a++) {
            int l, h;
            if (I.periodic[a]) {
                if (2 * r + 1 >= I.gdim[a]) { l = 0; h = I.gdim[a] - 1; }
                else { l = g[a] - r; h = g[a] + r; }
            } else {
                l = max(0, g[a] - r);
                h = min(I.gdim[a] - 1, g[a] + r);
            }
            lo[a] = l;
            ext[a] = h - l + 1;
        }
        const long long n = (long long)ext[0] * ext[1] * ext[2];
        for (long long t = lane; t < n; t += 32) {
            const int x = lo[0] + (int)(t % ext[0]), y = lo[1] + (int)(t / ext[0] % ext[1]),
                      z = lo[2] + (int)(t / ((long long)ext[0] * ext[1]));
            const int w[3] = { I.periodic[0] ? wrap_idx(x, I.gdim[0]) : x, I.periodic[1] ? wrap_idx(y, I.gdim[1]) : y,
                               I.periodic[2] ? wrap_idx(z, I.gdim[2]) : z };
            if (shell && r > 0 && in_cube(w, g, r - 1, I)) continue;
            const long long gg = I.g0 + ((long long)w[2] * I.gdim[1] + w[1]) * I.gdim[0] + w[0];
            const int q1 = v.gstart[gg + 1];
            for (int q = v.gstart[gg]; q < q1; q++) {
                const float4 c = v.gcf[q];
                const float dx = axis_dist(p[0], c.x, I, 0), dy = axis_dist(p[1], c.y, I, 1), dz = axis_dist(p[2], c.z, I, 2);
                f(fmaf(dx, dx, fmaf(dy, dy, dz * dz)), __float_as_int(c.w));
            }
        }
    };
    float best = 3.0e38f;
    int r = 0;
    const int rmax = max(I.gdim[0], max(I.gdim[1], I.gdim[2]));
    for (;; r++) {
        scan(r, true, [&](float d2, int) { best = fminf(best, d2); });
        // non-negative floats order like their bits
        best = __uint_as_float(__reduce_min_sync(full, __float_as_uint(best)));
        bool ex;
        const float lb = shell_bound(p, g, r, I, ex);
        if (ex || r >= rmax || (best < 3.0e38f && lb > sqrtf(best) + kBandE)) break;
    }
    const float lim = sqrtf(best) + kBandE, lim2 = lim * lim;
    int ncand = 0, bk = 0x7fffffff;
    scan(r, false, [&](float d2, int k) { if (d2 <= lim2) { ncand++; bk = min(bk, k); } });
    ncand = (int)__reduce_add_sync(full, (unsigned)ncand);
    if (ncand == 0) {   // unreachable for finite input: the search covers every centroid
        if (lane == 0) flag_inst(v, I, kStatusGridRange);
        return I.k0;
    }
    if (ncand > 1) {
        // (squared distances are non-negative: their bits order like them)
        unsigned long long b64 = ~0ull;
        bk = 0x7fffffff;
        scan(r, false, [&](float d2, int k) {
            if (d2 > lim2) return;
            const unsigned long long d = (unsigned long long)__double_as_longlong(
                dist2_grid_d(xq[0], xq[1], xq[2], v.cq[k], v.cq[(size_t)v.Ktot + k], v.cq[(size_t)2 * v.Ktot + k], I));
            if (d < b64 || (d == b64 && k < bk)) { b64 = d; bk = k; }
        });
        unsigned long long m = b64;
        for (int off = 16; off; off >>= 1) m = min(m, (unsigned long long)__shfl_xor_sync(full, m, off));
        if (b64 != m) bk = 0x7fffffff;
    }
    return __reduce_min_sync(full, bk);
}

// Grid search for the particles the certified E-step could not decide, a
// warp each (one thread each took 70 us for the few of the 4M cell: a chain
// of dependent loads per shell); counts them into their cells.
__global__ void __launch_bounds__(128) k_estep_list(View v, const int* __restrict__ fb_list,
                                                    const int* __restrict__ fb_count, int* __restrict__ cell_out,
                                                    int* __restrict__ cnt) {
    const int n = *fb_count;
    for (int q = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; q < n; q += (gridDim.x * blockDim.x) >> 5) {
        const int i = fb_list[q];
        const int c = estep_warp_one(v, i);
        if ((threadIdx.x & 31) == 0) {
            cell_out[i] = c;
            atomicAdd(&cnt[c], 1);
        }
    }
}

// Largest move of the centroids now in each grid cell (FP32 bits:
// non-negative floats order like their bit patterns).
__global__ void k_grid_move(View v, const int* __restrict__ gidx, const float* __restrict__ cmove,
                            unsigned* __restrict__ gmove) {
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k < v.Ktot) atomicMax(&gmove[gidx[k]], __float_as_uint(cmove[k]));
}

// k-means E-step after the first round (Hamerly's bound): the particle's
// centroid of the previous round is still its nearest when the distance to
// it is below the previous lower bound on every other centroid, less the
// largest move of the M-step in between (FP32 with a margin); the bound is
// carried on, the others are listed for the grid search.  When the bound is
// below the grid edge, every centroid that could now be nearer lies in the
// 27 grid cells around the particle, and the largest move among those
// replaces the instance's largest move.
__global__ void __launch_bounds__(256) k_estep_bound(View v, const int* __restrict__ cell, float* __restrict__ lbound,
                                                     const float4* __restrict__ cf, const unsigned* __restrict__ dmax,
                                                     const unsigned* __restrict__ gmove, int* __restrict__ list,
                                                     int* __restrict__ count) {
    __shared__ int wcount[8], wbase[8], bbase;
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    bool need = false;
    if (i < v.N) {
        const int b = find_inst(v.inst_p0, v.B, i);
        const Inst& I = v.inst[b];
        float p[3];
        int g[3];
        for (int a = 0; a < 3; a++) g[a] = grid_coord(v.xq[(size_t)a * v.N + i], I, a, p[a]);
        const float4 c = cf[cell[i]];
        const float dx = axis_dist(p[0], c.x, I, 0), dy = axis_dist(p[1], c.y, I, 1), dz = axis_dist(p[2], c.z, I, 2);
        const float l0 = lbound[i];
        float dm = __uint_as_float(dmax[b]);
        if (gmove && l0 <= fminf(I.gh[0], fminf(I.gh[1], I.gh[2]))) {
            unsigned m = 0;
            for (int zz = -1; zz <= 1; zz++)
                for (int yy = -1; yy <= 1; yy++)
                    for (int xx = -1; xx <= 1; xx++) {
                        int w[3] = {g[0] + xx, g[1] + yy, g[2] + zz};
                        for (int a = 0; a < 3; a++)
                            w[a] = I.periodic[a] ? wrap_idx(w[a], I.gdim[a]) : min(max(w[a], 0), I.gdim[a] - 1);
                        m = max(m, gmove[I.g0 + ((long long)w[2] * I.gdim[1] + w[1]) * I.gdim[0] + w[0]]);
                    }
            dm = __uint_as_float(m);
        }
        const float l = l0 - dm;
        if (sqrtf(fmaf(dx, dx, fmaf(dy, dy, dz * dz))) + kCertMargin < l) lbound[i] = l;
        else need = true;
    }
    const unsigned m = __ballot_sync(0xffffffffu, need);
    if (lane == 0) wcount[warp] = __popc(m);
    __syncthreads();
    if (threadIdx.x == 0) {
        int tot = 0;
        for (int w = 0; w < 8; w++) { wbase[w] = tot; tot += wcount[w]; }
        bbase = tot ? atomicAdd(count, tot) : 0;
    }
    __syncthreads();
    if (need) list[bbase + wbase[warp] + __popc(m & ((1u << lane) - 1u))] = i;
}

// The previous rows with their cells renumbered and the renumbered cells'
// FP32 centroids (w = new index), so the E-step reads one record per
// candidate instead of three dependent loads; the first K threads also put
// the centroids in grid order (gcount not null).
constexpr int kRowLanes = 8;    // (a membrane's rows hold about 8 cells)
__global__ void k_cand_rows(View v, const int* __restrict__ cnt_old, const int* __restrict__ pad_old,
                            const int* __restrict__ new_of_old, const float4* __restrict__ cf,
                            float4* __restrict__ rows, const int* __restrict__ gidx, int* __restrict__ gcount) {
    const int q = blockIdx.x * blockDim.x + threadIdx.x;   // kRowLanes threads per row
    if (gcount && q < v.Ktot) grid_fill_one(v, q, gidx, gcount, cf);
    const int k = q / kRowLanes;
    if (k >= v.Ktot) return;
    const int n = min(cnt_old[k], kAdjRow);
    for (int r = q % kRowLanes; r < n; r += kRowLanes) {
        const int j = new_of_old[pad_old[(size_t)k * kAdjRow + r]];
        float4 c = cf[j];
        c.w = __int_as_float(j);
        rows[(size_t)k * kAdjRow + r] = c;
    }
}

// Rebuild E-step from the previous cell list (the paper's guess from the
// previous particle, made exact), one thread per particle: the candidates
// are the particle's previous cell and its previous neighbouring cells (one
// row; the lanes of a warp mostly share it), renumbered by the Morton
// relabel.  Every centroid outside the row was at least rho_k from the old
// centroid c_k when the list was built (rho_k: distance to the nearest
// non-neighbour), and every centroid has since moved at most dmax, so none
// of them is within best + band of the particle when
//   sqrt(best) + band < rho_k - 2 dmax - |x - c_k|   (FP32 with margins).
// Particles that fail the test take the grid search.  The others are counted
// into their cells (a histogram pass of its own cost 13 us at 4M).
__global__ void __launch_bounds__(128, 16) k_estep_rows(View v, const int* __restrict__ cell_old,
                                                    const int* __restrict__ cnt_old, const float4* __restrict__ rows,
                                                    const float* __restrict__ rho_old, const int* __restrict__ new_of_old,
                                                    const unsigned* __restrict__ dmax, int* __restrict__ cell_out,
                                                    int* __restrict__ fb_list, int* __restrict__ fb_count,
                                                    int* __restrict__ cnt) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    bool fail = false;
    int to = -1;
    if (i < v.N) {
        const int b = find_inst(v.inst_p0, v.B, i);
        const Inst& I = v.inst[b];
        long long xq[3];
        float p[3];
        for (int a = 0; a < 3; a++) {
            xq[a] = v.xq[(size_t)a * v.N + i];
            grid_coord(xq[a], I, a, p[a]);
        }
        const int ko = cell_old[i], kn = new_of_old[ko];
        const int a0 = ko * kAdjRow, a1 = a0 + min(cnt_old[ko], kAdjRow);
        float best = 3.0e38f, second = 3.0e38f, dself2 = 3.0e38f;
        int bk = -1;
        for (int r = a0; r < a1; r++) {
            const float4 c = rows[r];
            const int j = __float_as_int(c.w);
            if (j < I.k0 || j >= I.k0 + I.K) continue;    // a cell of the other set
            const float dx = axis_dist(p[0], c.x, I, 0), dy = axis_dist(p[1], c.y, I, 1), dz = axis_dist(p[2], c.z, I, 2);
            const float d2 = fmaf(dx, dx, fmaf(dy, dy, dz * dz));
            if (j == kn) dself2 = d2;
            if (d2 < best || (d2 == best && j < bk)) { second = best; best = d2; bk = j; }
            else if (d2 < second) second = d2;
        }
        const float lim = sqrtf(best) + kBandE;
        const float cert = rho_old[ko] - 2.0f * __uint_as_float(dmax[b]) - sqrtf(dself2) - kCertMargin;
        fail = bk < 0 || dself2 >= 3.0e38f || !(lim < cert);
        if (!fail) {
            to = bk;
            if (second <= lim * lim) {
                // tie band: FP64 among the row's candidates within it
                double best64 = 1e300;
                int bk64 = -1;
                for (int r = a0; r < a1; r++) {
                    const float4 c = rows[r];
                    const int j = __float_as_int(c.w);
                    if (j < I.k0 || j >= I.k0 + I.K) continue;
                    const float dx = axis_dist(p[0], c.x, I, 0), dy = axis_dist(p[1], c.y, I, 1),
                                dz = axis_dist(p[2], c.z, I, 2);
                    if (fmaf(dx, dx, fmaf(dy, dy, dz * dz)) <= lim * lim) {
                        const double d64 = dist2_grid_d(xq[0], xq[1], xq[2], v.cq[j], v.cq[(size_t)v.Ktot + j],
                                                        v.cq[(size_t)2 * v.Ktot + j], I);
                        if (d64 < best64 || (d64 == best64 && j < bk64)) { best64 = d64; bk64 = j; }
                    }
                }
                to = bk64;
            }
            cell_out[i] = to;
        }
    }
    // the counts of the sort that follows: one atomic per distinct cell of a warp
    const unsigned peers = __match_any_sync(0xffffffffu, to);
    if (to >= 0 && (int)(threadIdx.x & 31) == __ffs(peers) - 1) atomicAdd(&cnt[to], __popc(peers));
    // the rare failures to the grid search's list, one atomic per warp
    const unsigned m = __ballot_sync(0xffffffffu, fail);
    if (m) {
        const int lane = threadIdx.x & 31, first = __ffs(m) - 1;
        int base = 0;
        if (lane == first) base = atomicAdd(fb_count, __popc(m));
        base = __shfl_sync(0xffffffffu, base, first);
        if (fail) fb_list[base + __popc(m & ((1u << lane) - 1u))] = i;
    }
}

// ============================================================== stable counting sort
// Consecutive particles mostly share a cell: one atomic per distinct cell of
// a warp (lanes with the same cell found with a match).
__global__ void k_hist(int N, const int* __restrict__ cell, int* __restrict__ cnt) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    const int c = (i < N) ? cell[i] : -1;
    const unsigned peers = __match_any_sync(0xffffffffu, c);
    const int lane = threadIdx.x & 31;
    if (c >= 0 && lane == __ffs(peers) - 1) atomicAdd(&cnt[c], __popc(peers));
}

// Slot of each particle inside its cell's range (in any order across warps;
// the per-cell sort that follows restores the storage order).  The counts
// are taken down to zero, ready for the next histogram.  In a rebuild (B > 0,
// B <= N) it also does what the launches before it left to a later one: see
// ScratchReset.
__global__ void k_scatter(int N, const int* __restrict__ cell, const int* __restrict__ start, int* __restrict__ cnt,
                          int* __restrict__ tmp, int B, ScratchReset z) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < B) {
        z.dmax[i] = 0u;
        z.rmax[i] = 0u;
        if (z.advance) z.steps[i] += 1;
        if (i == 0) { *z.fb_count = 0; *z.rot_n = 0; *z.novf = 0; }
    }
    const int c = (i < N) ? cell[i] : -1;
    const unsigned peers = __match_any_sync(0xffffffffu, c);
    const int lane = threadIdx.x & 31;
    const int leader = __ffs(peers) - 1;
    int base = 0;
    if (c >= 0 && lane == leader) base = atomicSub(&cnt[c], __popc(peers)) - __popc(peers);
    base = __shfl_sync(peers, base, leader);
    if (c >= 0) tmp[start[c] + base + __popc(peers & ((1u << lane) - 1u))] = i;
}

// Sort each cell's slot list ascending (= old storage order), which makes the
// scatter stable.  One block per cell, bitonic in shared memory.
constexpr int kSegMax = 2048;
__global__ void k_segsort(int Ktot, const int* __restrict__ start, int* __restrict__ tmp, unsigned* status) {
    __shared__ int sh[kSegMax];
    for (int k = blockIdx.x; k < Ktot; k += gridDim.x) {
    int s = start[k], e = start[k + 1], n = e - s;
    if (n <= 128 || n > kSegMax) continue;   // warp kernel / k_segrank
    int m = 1;
    while (m < n) m <<= 1;
    for (int t = threadIdx.x; t < m; t += blockDim.x) sh[t] = (t < n) ? tmp[s + t] : 0x7fffffff;
    __syncthreads();
    for (int size = 2; size <= m; size <<= 1)
        for (int stride = size >> 1; stride > 0; stride >>= 1) {
            for (int t = threadIdx.x; t < m; t += blockDim.x) {
                int p = t ^ stride;
                if (p > t) {
                    bool up = (t & size) == 0;
                    int a = sh[t], c = sh[p];
                    if ((c < a) == up) { sh[t] = c; sh[p] = a; }
                }
            }
            __syncthreads();
        }
    for (int t = threadIdx.x; t < n; t += blockDim.x) tmp[s + t] = sh[t];
    __syncthreads();
    }
}

// Cells of up to 32 NE particles: one warp, bitonic network over NE values per
// lane (element e = lane + 32 q), shuffles for strides < 32.
template <int NE>
__device__ __forceinline__ void segsort_net(const int* __restrict__ tmp, int n, int (&val)[NE]) {
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int q = 0; q < NE; q++) val[q] = (lane + 32 * q < n) ? tmp[lane + 32 * q] : 0x7fffffff;
#pragma unroll
    for (int size = 2; size <= 32 * NE; size <<= 1) {
#pragma unroll
        for (int stride = size >> 1; stride > 0; stride >>= 1) {
            if (stride >= 32) {
                const int qs = stride >> 5;
#pragma unroll
                for (int q = 0; q < NE; q++) {
                    if (q & qs) continue;
                    const int e = lane + 32 * q;
                    const bool up = (e & size) == 0;
                    const int a = val[q], c = val[q + qs];
                    val[q] = up ? min(a, c) : max(a, c);
                    val[q + qs] = up ? max(a, c) : min(a, c);
                }
            } else {
#pragma unroll
                for (int q = 0; q < NE; q++) {
                    const int e = lane + 32 * q;
                    const int other = __shfl_xor_sync(0xffffffffu, val[q], stride);
                    const bool up = (e & size) == 0;
                    const bool lower = (e & stride) == 0;
                    val[q] = (lower == up) ? min(val[q], other) : max(val[q], other);
                }
            }
        }
    }
}
template <int NE>
__device__ inline void segsort_store(int s, int n, int* __restrict__ tmp) {
    const int lane = threadIdx.x & 31;
    int val[NE];
    segsort_net<NE>(tmp + s, n, val);
#pragma unroll
    for (int q = 0; q < NE; q++)
        if (lane + 32 * q < n) tmp[s + lane + 32 * q] = val[q];
}
__device__ inline void segsort_warp(int s, int n, int* __restrict__ tmp) {   // n <= 128
    if (n <= 64) segsort_store<2>(s, n, tmp);
    else segsort_store<4>(s, n, tmp);
}

__global__ void k_segsort_warp(int Ktot, const int* __restrict__ start, int* __restrict__ tmp) {
    const int k = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    if (k >= Ktot) return;
    const int s = start[k], n = start[k + 1] - s;
    if (n > 1 && n <= 128) segsort_warp(s, n, tmp);
}

// One cell by a block: bitonic in shared memory (sh, kSegMax ints) up to
// kSegMax slots.  Beyond it the parts of kSegMax are sorted so, and a slot's
// place is its rank in its own part and, by binary search, in each other one
// (slots are distinct), out being scratch.  (Counting the smaller slots of the
// whole cell instead, the rebuild of one cell of 6,200 particles took 1,497 us,
// 400 so.)
__device__ void segsort_block(int s, int n, int* tmp, int* out, int* sh) {
    for (int c = s; c < s + n; c += kSegMax) {
        const int nc = min(kSegMax, s + n - c);
        int m = 1;
        while (m < nc) m <<= 1;
        for (int t = threadIdx.x; t < m; t += blockDim.x) sh[t] = (t < nc) ? tmp[c + t] : 0x7fffffff;
        __syncthreads();
        for (int size = 2; size <= m; size <<= 1)
            for (int stride = size >> 1; stride > 0; stride >>= 1) {
                for (int t = threadIdx.x; t < m; t += blockDim.x) {
                    const int p = t ^ stride;
                    if (p > t) {
                        const bool up = (t & size) == 0;
                        const int a = sh[t], b = sh[p];
                        if ((b < a) == up) { sh[t] = b; sh[p] = a; }
                    }
                }
                __syncthreads();
            }
        for (int t = threadIdx.x; t < nc; t += blockDim.x) tmp[c + t] = sh[t];
        __syncthreads();
    }
    if (n <= kSegMax) return;
    for (int q = threadIdx.x; q < n; q += blockDim.x) {
        const int me = tmp[s + q], own = q - q % kSegMax;
        int r = q - own;
        for (int c = 0; c < n; c += kSegMax) {
            if (c == own) continue;
            int lo = s + c, hi = s + min(c + kSegMax, n);
            while (lo < hi) {
                const int mid = (lo + hi) >> 1;
                if (tmp[mid] < me) lo = mid + 1;
                else hi = mid;
            }
            r += lo - (s + c);
        }
        out[s + r] = me;
    }
    __syncthreads();
    for (int q = s + threadIdx.x; q < s + n; q += blockDim.x) tmp[q] = out[q];
    __syncthreads();
}

// The rebuild's form for large cells, a block per cell: the cells are few, and
// eight of them one after the other in a block made the rebuild of eight cells
// of 1,300 particles 473 us (144 so; one such cell alone 132).
__global__ void __launch_bounds__(256) k_segsort_cells(const int* __restrict__ start, int* __restrict__ tmp,
                                                       int* __restrict__ out) {
    __shared__ int sh[kSegMax];
    const int s = start[blockIdx.x], n = start[blockIdx.x + 1] - s;
    if (n > 128) segsort_block(s, n, tmp, out, sh);
    else if (n > 1 && threadIdx.x < 32) segsort_warp(s, n, tmp);
}

// Cells larger than kSegMax: each slot's rank among its cell's (distinct)
// old indices, O(n^2) per such cell; writes the ordered list to out.
__global__ void k_segrank(int N, const int* __restrict__ cell, const int* __restrict__ start, const int* __restrict__ tmp,
                          int* __restrict__ out) {
    int q = blockIdx.x * blockDim.x + threadIdx.x;   // slot in the scattered order
    if (q >= N) return;
    int c = cell[tmp[q]];
    int s = start[c], e = start[c + 1];
    if (e - s <= kSegMax) return;
    int me = tmp[q], r = 0;
    for (int t = s; t < e; t++) r += (tmp[t] < me);
    out[s + r] = me;
}

__global__ void k_segcopy(int N, const int* __restrict__ cell, const int* __restrict__ start, const int* __restrict__ src,
                          int* __restrict__ tmp) {
    int q = blockIdx.x * blockDim.x + threadIdx.x;
    if (q >= N) return;
    int c = cell[tmp[q]];
    if (start[c + 1] - start[c] > kSegMax) tmp[q] = src[q];
}

// ============================================================== gather + mirrors
// The mirrors hold x - c~ at 2^-26 sigma, where c~ is the centroid rounded to
// a multiple of 2^-26 sigma: then round(x - c~) = round(x) - c~ exactly, and
// a pair's integer displacement m_j + (c~_l - c~_k) - m_i depends on the two
// positions alone (and, on a periodic axis, on the image), not on which
// cells hold them, so FP32 pair forces do not change when the cell list is
// rebuilt.
__device__ inline long long mirror_ref(long long c) {
    return ((c + (1ll << (kMirrorShift - 1))) >> kMirrorShift) << kMirrorShift;
}
__device__ inline int mirror_coord(long long xq, long long cq, const Inst& I, int a, const View& v) {
    long long d = minimg_q(xq - mirror_ref(cq), I.boxq[a], I.periodic[a]);
    long long r = (d + (1ll << (kMirrorShift - 1))) >> kMirrorShift;
    if (r > 2147483647ll || r < -2147483647ll) { flag_inst(v, I, kStatusMirrorRange); r = 0; }
    return (int)r;
}

// Cell radius R_k = max_i |x_i - c_k| over the cell (all types), equal to
// the FP64 definition: FP32 from the exact mirror (error < 1e-6 sigma) finds
// the candidates within this band of the maximum, FP64 decides among them.
// A single candidate (nearly always) is only noted: an FP64 instruction holds
// the FP64 pipe for a whole warp's turn, and the few radii that a neighbour
// test inside its band or a getter wants in FP64 are computed there
// (cell_r2).
constexpr float kBandR = 1e-5f;

// Gather of the cell-sorted state: the particle of old slot so moves to slot p
// of cell k with its state, type and id and gets its exact mirror relative to
// that cell's centroid.  Every load and the mirror come before the first
// store: as far as the compiler knows the stores may alias the sources, and
// interleaved they would serialise the loads' latencies.
struct Moved {
    long long x[3], vq[3], nq[3], wq[3];
    unsigned id;
    int q0;          // p0 + id
    int4 m;
    float4 no;
};

__device__ __forceinline__ void move_load(const View& v, const View& o, const Inst& I, int k, int so, int p, Moved& g) {
    const size_t N = v.N;
    g.id = o.id[so];        // (first: the bond list's look-up waits for it)
    for (int a = 0; a < 3; a++) {
        g.x[a] = o.xq[a * N + so];
        g.vq[a] = o.vq[a * N + so];
        g.nq[a] = o.nq[a * N + so];
        g.wq[a] = o.wq[a * N + so];
    }
    const unsigned char t = o.type[so];
    g.m.x = mirror_coord(g.x[0], v.cq[k], I, 0, v);
    g.m.y = mirror_coord(g.x[1], v.cq[(size_t)v.Ktot + k], I, 1, v);
    g.m.z = mirror_coord(g.x[2], v.cq[(size_t)2 * v.Ktot + k], I, 2, v);
    g.q0 = I.p0 + (int)g.id;
    g.m.w = t | (v.bptr[g.q0] < v.bptr[g.q0 + 1] ? kMirrorBonded : 0);
    g.no.x = ll_to_float(g.nq[0]) * (float)kGridInv;
    g.no.y = ll_to_float(g.nq[1]) * (float)kGridInv;
    g.no.z = ll_to_float(g.nq[2]) * (float)kGridInv;
    g.no.w = __int_as_float(p);
}

__device__ __forceinline__ void move_store(const View& v, int k, int p, const Moved& g, long long* __restrict__ xref) {
    const size_t N = v.N;
    for (int a = 0; a < 3; a++) {
        v.xq[a * N + p] = g.x[a];
        v.vq[a * N + p] = g.vq[a];
        v.nq[a * N + p] = g.nq[a];
        v.wq[a * N + p] = g.wq[a];
        if (xref) xref[a * N + p] = g.x[a];
    }
    v.type[p] = (unsigned char)(g.m.w & 0xff);
    v.id[p] = g.id;
    v.cell[p] = k;
    v.slot_of_id[g.q0] = p;
}

// One thread per new slot (large cells; k_build_cells otherwise): the old slot
// is perm[p], the cell the E-step's result for it.
__global__ void __launch_bounds__(256) k_gather_particles(View v, View o, const int* __restrict__ perm,
                                                          const int* __restrict__ cell_new,
                                                          long long* __restrict__ xref) {
    const int p = blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= v.N) return;
    const int so = perm[p], k = cell_new[so];
    Moved g;
    move_load(v, o, v.inst[find_inst(v.inst_p0, v.B, p)], k, so, p, g);
    move_store(v, k, p, g, xref);
    v.mq[p] = g.m;
    v.mo[p] = g.no;
}

// Bitonic sort of 32 * NE records over a warp, slot lane + 32 u held in
// r[u] (records of r beyond NE untouched); slots at a distance >= 32 are
// exchanged inside a lane.
template <int NE>
__device__ inline void warp_bitonic_u32(unsigned (&r)[4], int lane) {
#pragma unroll
    for (int size = 2; size <= 32 * NE; size <<= 1) {
#pragma unroll
        for (int stride = size >> 1; stride > 0; stride >>= 1) {
            if (stride >= 32) {
                const int du = stride >> 5;
#pragma unroll
                for (int u = 0; u < NE; u++) {
                    if (u & du) continue;
                    const bool up = ((lane + 32 * u) & size) == 0;
                    const unsigned x = r[u], y = r[u + du];
                    r[u] = up ? min(x, y) : max(x, y);
                    r[u + du] = up ? max(x, y) : min(x, y);
                }
            } else {
#pragma unroll
                for (int u = 0; u < NE; u++) {
                    const int e = lane + 32 * u;
                    const unsigned o = __shfl_xor_sync(0xffffffffu, r[u], stride);
                    const bool up = (e & size) == 0;
                    const bool lower = (e & stride) == 0;
                    r[u] = (lower == up) ? min(r[u], o) : max(r[u], o);
                }
            }
        }
    }
}

// The squared radius of cell k by the FP64 definition, from the positions x
// that the cells were built from.
__device__ inline double cell_r2(const View& v, const long long* __restrict__ x, const Inst& I, int k) {
    const int p = v.rcand[k];
    if (p < 0) return v.R2[k];
    const size_t N = v.N, K = v.Ktot;
    return dist2_grid_d(x[p], x[N + p], x[2 * N + p], v.cq[k], v.cq[K + k], v.cq[2 * K + k], I);
}

__global__ void k_cell_r2(View v, const long long* __restrict__ x) {
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k < v.Ktot) v.R2[k] = cell_r2(v, x, v.inst[find_inst(v.inst_k0, v.B, k)], k);
}

// What the pair kernels and the neighbour search want of a cell, by one warp:
// the cell radius (in FP32, and the particle that sets it), the pair kernels'
// cell frame (its normal the mean bilayer director, +z without one) and, in
// each tile of 128 particles, every particle's rank along the tile's longer
// tangent extent.  rmax_bits: each instance's largest radius (FP32 bits).
struct CellSums {        // a lane's share, then the cell's
    float mx = 0.f, nx = 0.f, ny = 0.f, nz = 0.f;
    __device__ __forceinline__ static float dist(const int4& m) {
        const float dx = m.x * kMirrorUnit, dy = m.y * kMirrorUnit, dz = m.z * kMirrorUnit;
        return sqrtf(fmaf(dx, dx, fmaf(dy, dy, dz * dz)));
    }
    __device__ __forceinline__ void add(const int4& m, float x, float y, float z) {
        mx = fmaxf(mx, dist(m));
        if (bilayer(m.w & 0xff)) { nx += x; ny += y; nz += z; }
    }
    __device__ __forceinline__ void reduce() {
        for (int off = 16; off; off >>= 1) {
            mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, off));
            nx += __shfl_xor_sync(0xffffffffu, nx, off);
            ny += __shfl_xor_sync(0xffffffffu, ny, off);
            nz += __shfl_xor_sync(0xffffffffu, nz, off);
        }
    }
};

// The radius: of the particles within the band of the FP32 maximum (cand, the
// last of the nc in this lane) the only one is noted, or exact(), a lane's
// largest FP64 distance squared among its own, decides.
template <typename F>
__device__ __forceinline__ void cell_radius(const View& v, int k, int b, float mx, int cand, int nc, unsigned* rmax_bits,
                                            F&& exact) {
    const int lane = threadIdx.x & 31;
    nc = (int)__reduce_add_sync(0xffffffffu, (unsigned)nc);
    cand = __reduce_max_sync(0xffffffffu, cand);
    if (nc > 1) {
        // (the maximum over the lanes on the bit patterns: a non-negative
        // double's bits order like its value)
        unsigned long long bb = exact();
        for (int off = 16; off; off >>= 1) bb = max(bb, (unsigned long long)__shfl_xor_sync(0xffffffffu, bb, off));
        if (lane == 0) v.R2[k] = __longlong_as_double((long long)bb);
        cand = -1;
    } else if (nc == 0 && lane == 0) {
        v.R2[k] = 0.0;      // an empty cell
    }
    if (lane == 0) {
        v.rcand[k] = cand;
        v.Rf[k] = mx;
        // (a possibly stale value read through L1 saves nearly all atomics on
        // the one address)
        if (__float_as_uint(mx) > __ldca(rmax_bits + b)) atomicMax(&rmax_bits[b], __float_as_uint(mx));
    }
}

__device__ __forceinline__ unsigned long long exact_r2_bits(const View& v, const Inst& I, int k, int p) {
    const size_t N = v.N, K = v.Ktot;
    return (unsigned long long)__double_as_longlong(
        dist2_grid_d(v.xq[p], v.xq[N + p], v.xq[2 * N + p], v.cq[k], v.cq[K + k], v.cq[2 * K + k], I));
}

__device__ __forceinline__ Frame cell_frame(const View& v, int k, float nx, float ny, float nz) {
    const int lane = threadIdx.x & 31;
    const float nn = sqrtf(fmaf(nx, nx, fmaf(ny, ny, nz * nz)));
    if (nn > 1e-3f) { nx /= nn; ny /= nn; nz /= nn; }
    else { nx = 0.f; ny = 0.f; nz = 1.f; }
    const Frame F = tangent_frame(nx, ny, nz);
    if (lane < 3)
        v.cframe[3 * (size_t)k + lane] =
            lane == 0 ? make_float4(F.r[0], F.r[1], F.r[2], 0.f)
                      : (lane == 1 ? make_float4(F.r[3], F.r[4], F.r[5], 0.f) : make_float4(F.r[6], F.r[7], F.r[8], 0.f));
    return F;
}

// A tile of nt <= 32 NE particles (particle lane + 32 u at tangent coordinates
// ya[u], yb[u]) in the order of its longer tangent extent: rank lane + 32 u
// goes to the particle (r[u] & 127), none where r[u] is ~0.  32-bit records:
// the key quantised to 24 bits over the tile's extent (monotone), the tile
// index in the low 7 bits (equal keys go by index), sorted over the warp.
template <int NE>
__device__ __forceinline__ void tile_ranks(const float (&ya)[4], const float (&yb)[4], int nt, unsigned (&r)[4]) {
    const int lane = threadIdx.x & 31;
    float lo_a = 3.0e38f, hi_a = -3.0e38f, lo_b = 3.0e38f, hi_b = -3.0e38f;
#pragma unroll
    for (int u = 0; u < NE; u++)
        if (lane + 32 * u < nt) {
            lo_a = fminf(lo_a, ya[u]); hi_a = fmaxf(hi_a, ya[u]);
            lo_b = fminf(lo_b, yb[u]); hi_b = fmaxf(hi_b, yb[u]);
        }
    for (int off = 16; off; off >>= 1) {
        lo_a = fminf(lo_a, __shfl_xor_sync(0xffffffffu, lo_a, off));
        hi_a = fmaxf(hi_a, __shfl_xor_sync(0xffffffffu, hi_a, off));
        lo_b = fminf(lo_b, __shfl_xor_sync(0xffffffffu, lo_b, off));
        hi_b = fmaxf(hi_b, __shfl_xor_sync(0xffffffffu, hi_b, off));
    }
    const bool use_a = (hi_a - lo_a) >= (hi_b - lo_b);
    const float klo = use_a ? lo_a : lo_b, kext = use_a ? hi_a - lo_a : hi_b - lo_b;
    const float ksc = kext > 0.f ? 16777215.0f / kext : 0.f;
#pragma unroll
    for (int u = 0; u < NE; u++) {
        const int t = lane + 32 * u;
        const float y = use_a ? ya[u] : yb[u];
        r[u] = (t < nt) ? (min(16777215u, (unsigned)((y - klo) * ksc)) << 7) | (unsigned)t : 0xffffffffu;
    }
    warp_bitonic_u32<NE>(r, lane);
}

// Cell k from the gathered mirrors mq, mo (written by the same lanes, or by an
// earlier launch).
__device__ void cell_props(const View& v, int k, unsigned* rmax_bits) {
    const int lane = threadIdx.x & 31;
    const int b = find_inst(v.inst_k0, v.B, k);
    const Inst& I = v.inst[b];
    const int s = v.cell_start[k], e = v.cell_start[k + 1];
    CellSums c;
    for (int p = s + lane; p < e; p += 32) {
        const float4 no = v.mo[p];
        c.add(v.mq[p], no.x, no.y, no.z);
    }
    c.reduce();
    int cand = -1, nc = 0;
    for (int p = s + lane; p < e; p += 32)
        if (CellSums::dist(v.mq[p]) >= c.mx - kBandR) { cand = p; nc++; }
    cell_radius(v, k, b, c.mx, cand, nc, rmax_bits, [&] {
        unsigned long long bb = 0;
        for (int p = s + lane; p < e; p += 32)
            if (CellSums::dist(v.mq[p]) >= c.mx - kBandR) bb = max(bb, exact_r2_bits(v, I, k, p));
        return bb;
    });
    const Frame F = cell_frame(v, k, c.nx, c.ny, c.nz);
    for (int t0 = s; t0 < e; t0 += 128) {
        const int nt = min(128, e - t0);
        float ya[4], yb[4];
        for (int u = 0; u < 4; u++) {
            const int t = lane + 32 * u;
            ya[u] = 0.f; yb[u] = 0.f;
            if (t < nt) {
                const int4 m = v.mq[t0 + t];
                float h;
                F.apply(m.x * kMirrorUnit, m.y * kMirrorUnit, m.z * kMirrorUnit, ya[u], yb[u], h);
            }
        }
        unsigned r[4] = {~0u, ~0u, ~0u, ~0u};
        if (nt <= 64) tile_ranks<2>(ya, yb, nt, r);
        else tile_ranks<4>(ya, yb, nt, r);
        for (int u = 0; u < 4; u++) {
            if (r[u] == 0xffffffffu) continue;
            const int t = (int)(r[u] & 127u), q = lane + 32 * u;
            v.grank[t0 + t] = (unsigned char)q;
            v.mqr[t0 + q] = v.mq[t0 + t];
            v.mor[t0 + q] = v.mo[t0 + t];
        }
        __syncwarp();
    }
}

__global__ void __launch_bounds__(256, 6) k_cell_props(View v, unsigned* rmax_bits /* [B] */) {
    const int k = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    if (k < v.Ktot) cell_props(v, k, rmax_bits);
}

// A cell of more than 128 particles (its old slots sorted): the mirrors go
// through mq, mo.
__device__ __noinline__ void build_large(const View& v, const View& o, int k, int s, int n, const int* perm,
                                         long long* __restrict__ xref, unsigned* rmax_bits) {
    const Inst& I = v.inst[find_inst(v.inst_k0, v.B, k)];
    for (int p = s + (threadIdx.x & 31); p < s + n; p += 32) {
        Moved g;
        move_load(v, o, I, k, perm[p], p, g);
        move_store(v, k, p, g, xref);
        v.mq[p] = g.m;
        v.mo[p] = g.no;
    }
    __syncwarp();
    cell_props(v, k, rmax_bits);
}

// What a warp of k_build_cells keeps of its cell.
struct CellTile {
    int4 m[128];
    float nx[128], ny[128], nz[128];
    int so[128];
};

template <int NE>
__device__ __forceinline__ void tile_sort(const int* __restrict__ perm, int n, int* so) {
    const int lane = threadIdx.x & 31;
    int val[NE];
    segsort_net<NE>(perm, n, val);
#pragma unroll
    for (int u = 0; u < NE; u++) so[lane + 32 * u] = val[u];
}

template <int NE>
__device__ __forceinline__ void tile_write(const View& v, const CellTile& T, const Frame& F, int s, int n) {
    const int lane = threadIdx.x & 31;
    float ya[4], yb[4];
#pragma unroll
    for (int u = 0; u < NE; u++) {
        const int t = lane + 32 * u;
        ya[u] = yb[u] = 0.f;
        if (t < n) {
            float h;
            F.apply(T.m[t].x * kMirrorUnit, T.m[t].y * kMirrorUnit, T.m[t].z * kMirrorUnit, ya[u], yb[u], h);
        }
    }
    unsigned r[4];
    tile_ranks<NE>(ya, yb, n, r);
#pragma unroll
    for (int u = 0; u < NE; u++) {
        if (r[u] == 0xffffffffu) continue;
        const int t = (int)(r[u] & 127u), q = lane + 32 * u;
        v.grank[s + t] = (unsigned char)q;
        v.mqr[s + q] = T.m[t];
        v.mor[s + q] = make_float4(T.nx[t], T.ny[t], T.nz[t], __int_as_float(s + t));
    }
}

// The cell sort's last part, the gather and the cells' properties in one
// launch, a warp per cell, the mirrors in shared memory throughout.  Bound by
// the latency of the gather's loads (in 1,000,000 particles 42% of the DRAM
// bandwidth, warps waiting for loads half of the time): as launches of their
// own the three took 8, 51 and 27 us there, together 62, as the sorts and the
// sums of one warp run under the loads of others and the mirrors are not
// written and read back.  Registers decide: the mirrors in registers (80, 24
// warps an SM) 80 us, here 64 registers and 32 warps; 48 registers spill (75).
// Rebuild of the 4M cell 637 -> 555 us, of the 62k vesicle 94 -> 87.
constexpr int kBuildWarps = 4;
__global__ void __launch_bounds__(32 * kBuildWarps, 8)
    k_build_cells(View v, View o, int* __restrict__ perm, int* __restrict__ out, long long* __restrict__ xref,
                  unsigned* rmax_bits) {
    __shared__ CellTile tile[kBuildWarps];
    static_assert(sizeof(tile) >= kSegMax * sizeof(int), "the large cells' sort uses the tiles' memory");
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int k0 = blockIdx.x * kBuildWarps, k = k0 + w;
    const int s = k < v.Ktot ? v.cell_start[k] : 0, n = k < v.Ktot ? v.cell_start[k + 1] - s : 0;
    if (__syncthreads_or(n > 128))
        for (int c = k0; c < min(k0 + kBuildWarps, v.Ktot); c++) {
            const int sc = v.cell_start[c], nc = v.cell_start[c + 1] - sc;
            if (nc > 128) segsort_block(sc, nc, perm, out, reinterpret_cast<int*>(tile));
        }
    if (k >= v.Ktot) return;
    if (n > 128) {
        build_large(v, o, k, s, n, perm, xref, rmax_bits);
        return;
    }
    CellTile& T = tile[w];
    if (n <= 64) tile_sort<2>(perm + s, n, T.so);
    else tile_sort<4>(perm + s, n, T.so);
    __syncwarp();
    const int b = find_inst(v.inst_k0, v.B, k);
    const Inst& I = v.inst[b];
    CellSums c;
#pragma unroll 1
    for (int t = lane; t < n; t += 32) {
        Moved g;
        move_load(v, o, I, k, T.so[t], s + t, g);
        move_store(v, k, s + t, g, xref);
        T.m[t] = g.m;
        T.nx[t] = g.no.x; T.ny[t] = g.no.y; T.nz[t] = g.no.z;
        c.add(g.m, g.no.x, g.no.y, g.no.z);
    }
    __syncwarp();
    c.reduce();
    int cand = -1, nc = 0;
    for (int t = lane; t < n; t += 32)
        if (CellSums::dist(T.m[t]) >= c.mx - kBandR) { cand = s + t; nc++; }
    cell_radius(v, k, b, c.mx, cand, nc, rmax_bits, [&] {
        unsigned long long bb = 0;
        for (int t = lane; t < n; t += 32)
            if (CellSums::dist(T.m[t]) >= c.mx - kBandR) bb = max(bb, exact_r2_bits(v, I, k, s + t));
        return bb;
    });
    const Frame F = cell_frame(v, k, c.nx, c.ny, c.nz);
    if (n <= 64) tile_write<2>(v, T, F, s, n);
    else tile_write<4>(v, T, F, s, n);
}

// Mirrors of the current order (after integration without a rebuild),
// written where the pair kernel reads them: slot p of its cell's tile of 128
// goes to the tile's position grank[p].  flag (nullable): nothing to do if it
// holds the number of the skin test just taken.
__global__ void k_mirrors(View v, const int* __restrict__ flag, int test) {
    int p = blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= v.N || (flag && *flag == test)) return;
    size_t N = v.N;
    int c = v.cell[p];
    int b = find_inst(v.inst_p0, v.B, p);
    const Inst& I = v.inst[b];
    int4 m;
    m.x = mirror_coord(v.xq[p], v.cq[c], I, 0, v);
    m.y = mirror_coord(v.xq[N + p], v.cq[(size_t)v.Ktot + c], I, 1, v);
    m.z = mirror_coord(v.xq[2 * N + p], v.cq[(size_t)2 * v.Ktot + c], I, 2, v);
    const unsigned id = v.id[p];
    m.w = v.type[p] | (v.bptr[I.p0 + id] < v.bptr[I.p0 + id + 1] ? kMirrorBonded : 0);
    float4 no;
    no.x = ll_to_float(v.nq[p]) * (float)kGridInv;
    no.y = ll_to_float(v.nq[N + p]) * (float)kGridInv;
    no.z = ll_to_float(v.nq[2 * N + p]) * (float)kGridInv;
    no.w = __int_as_float(p);
    const int cs = v.cell_start[c];
    const int q = cs + ((p - cs) & ~127) + (int)v.grank[p];
    v.mqr[q] = m;
    v.mor[q] = no;
}

// ============================================================== neighbouring cells
// nbr(k) = { j : |c_k - c_j| < ((R_k + R_j) + r_s + 2 skin)(1 + 1e-12) },
// evaluated exactly as the FP64 definition for candidates within a band of
// the threshold, and by an FP32 test with margin elsewhere.
constexpr float kBandA = 2e-3f;

// The definition's FP64 test of (k, j), for the candidates that FP32 leaves
// undecided; d: the distance of the centroids.
__device__ inline bool adj_exact(const View& v, const Inst& I, int k, int j, double& d) {
    const size_t K = v.Ktot;
    d = __dsqrt_rn(dist2_grid_d(v.cq[k], v.cq[K + k], v.cq[2 * K + k], v.cq[j], v.cq[K + j], v.cq[2 * K + j], I));
    // same operation order as the definition: ((Rk + Rj) + rs) + (skin + skin)
    double tt = __dadd_rn(__dadd_rn(__dadd_rn(__dsqrt_rn(cell_r2(v, v.xq, I, k)), __dsqrt_rn(cell_r2(v, v.xq, I, j))), I.rs),
                          __dadd_rn(I.skin, I.skin));
    tt = __dmul_rn(tt, 1.0 + 1e-12);
    return d < tt;
}

constexpr int kAdjRaw = 2 * kAdjRow;        // room for neighbours and undecided candidates
constexpr int kAdjOpen = 1 << 30;           // mark of an undecided one (K < 2^30)

// The warp's share of the centroids of one set, searched through the set's
// grid G (own: the set of cell k, whose nearest non-neighbour bounds the
// E-step's certificate; the other set's cells join the row only): the lanes
// share the rows of grid cells of the cube that the reach R_k + R_max + r_s +
// 2 skin can touch.  Neighbours go to row, candidates within kBandA of the
// threshold with the mark kAdjOpen (EXACT: decided at once).
template <bool EXACT>
__device__ inline void adj_scan(const View& v, const Inst& I, const Inst& G, int k, float Rkf, float tailf, float reach,
                                bool own, long long cx, long long cy, long long cz, int* row, int* rown, float& rho) {
    const int lane = threadIdx.x & 31;
    float p[3];
    int g[3];
    g[0] = grid_coord(cx, G, 0, p[0]);
    g[1] = grid_coord(cy, G, 1, p[1]);
    g[2] = grid_coord(cz, G, 2, p[2]);
    // cube radius: the first shell beyond which nothing is within reach
    int R = 0;
    for (;; R++) {
        bool ex;
        const float lb = shell_bound(p, g, R, G, ex);
        if (ex || lb > reach) break;
    }
    int lo[3], ext[3];
    bool full[3];
    for (int a = 0; a < 3; a++) {
        int l, h;
        full[a] = false;
        if (G.periodic[a]) {
            if (2 * R + 1 >= G.gdim[a]) { l = 0; h = G.gdim[a] - 1; full[a] = true; }
            else { l = g[a] - R; h = g[a] + R; }
        } else {
            l = max(0, g[a] - R);
            h = min(G.gdim[a] - 1, g[a] + R);
        }
        lo[a] = l;
        ext[a] = h - l + 1;
    }
    const float reach2 = reach * reach;
    // one lane per (y, z) row of the cube: the row's grid cells are
    // contiguous along x, and so are their centroids in grid order (one
    // or two segments when a periodic x range wraps)
    auto axis_gap = [&](int a, int u) {
        if (full[a]) return 0.f;
        const float cl = (!G.periodic[a] && u == 0) ? -3.0e38f : u * G.gh[a];
        const float ch = (!G.periodic[a] && u == G.gdim[a] - 1) ? 3.0e38f : (u + 1) * G.gh[a];
        return fmaxf(fmaxf(cl - p[a], p[a] - ch), 0.f);
    };
    const int rows = ext[1] * ext[2];
    for (int t = lane; t < rows; t += 32) {
        const int y = lo[1] + t % ext[1], z = lo[2] + t / ext[1];
        const float gy = axis_gap(1, y), gz = axis_gap(2, z);
        if (fmaf(gy, gy, gz * gz) > reach2) continue;      // the whole row is beyond the reach
        const int w1 = G.periodic[1] ? wrap_idx(y, G.gdim[1]) : y;
        const int w2 = G.periodic[2] ? wrap_idx(z, G.gdim[2]) : z;
        const long long rowbase = G.g0 + ((long long)w2 * G.gdim[1] + w1) * G.gdim[0];
        int xa[2], xb[2], nseg = 1;
        xa[0] = lo[0];
        xb[0] = lo[0] + ext[0] - 1;
        if (G.periodic[0] && !full[0]) {
            const int a0 = wrap_idx(xa[0], G.gdim[0]), b0 = wrap_idx(xb[0], G.gdim[0]);
            if (a0 <= b0) { xa[0] = a0; xb[0] = b0; }
            else { xa[0] = a0; xb[0] = G.gdim[0] - 1; xa[1] = 0; xb[1] = b0; nseg = 2; }
        }
        for (int sg = 0; sg < nseg; sg++) {
            const int q1 = v.gstart[rowbase + xb[sg] + 1];
            for (int q = v.gstart[rowbase + xa[sg]]; q < q1; q++) {
                const float4 c = v.gcf[q];
                const int j = __float_as_int(c.w);
                const float dx = axis_dist(p[0], c.x, G, 0), dy = axis_dist(p[1], c.y, G, 1), dz = axis_dist(p[2], c.z, G, 2);
                const float df = sqrtf(fmaf(dx, dx, fmaf(dy, dy, dz * dz)));
                // FP32 prefilter: FP32 radii differ from the definition's
                // FP64 sum by far less than the band
                const float tf = (Rkf + v.Rf[j]) + tailf;
                bool in = df <= tf + kBandA, open = in && df >= tf - kBandA;
                if (EXACT && open) {
                    double d;
                    in = adj_exact(v, I, k, j, d);
                    open = false;
                }
                if (in) {
                    const int at = atomicAdd(rown, 1);
                    if (at < kAdjRaw) row[at] = open ? j | kAdjOpen : j;
                } else if (own) {
                    rho = fminf(rho, df);
                }
            }
        }
    }
}

// The same with every candidate decided in the scan (out of line: only when
// neighbours and undecided candidates together overflow the row's room).
static __device__ __noinline__ float adj_scan_exact(const View& v, const Inst& I, const Inst& G, int k, float reach, bool own,
                                                    int* row, int* rown, float rho) {
    const size_t K = v.Ktot;
    adj_scan<true>(v, I, G, k, v.Rf[k], I.rsf + 2.0f * I.skinf, reach, own, v.cq[k], v.cq[K + k], v.cq[2 * K + k], row, rown,
                   rho);
    return rho;
}

// Neighbouring cells, one warp per cell: candidates by adj_scan, the few
// undecided ones by the FP64 rule afterwards (FP64 code inside the scan cost
// it registers and spills), then the row sorted.  A membrane whose proteins
// have a cell set of their own searches that set's grid too, so that its rows
// hold the neighbouring cells of both sets.  Rows longer than kAdjRow are
// flagged (kStatusAdjOverflow) and truncated. Each entry gets the pair
// kernel's staging descriptor (particle range, exact centroid offset at 2^-26
// sigma) in the same fixed-stride row.
__global__ void __launch_bounds__(256, 6) k_adj_warp(View v, const unsigned* __restrict__ rmax_bits, int* __restrict__ count,
                           float* __restrict__ rho_out, int* __restrict__ pad /* [Ktot][kAdjRow] */) {
    __shared__ int row[8][kAdjRaw];
    __shared__ int rown[8];
    const int wb = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int k = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    if (k >= v.Ktot) return;
    const int b = find_inst(v.inst_k0, v.B, k);
    const Inst& I = v.inst[b];
    const float Rkf = v.Rf[k];
    const long long cx = v.cq[k], cy = v.cq[(size_t)v.Ktot + k], cz = v.cq[(size_t)2 * v.Ktot + k];
    // the cell's scalars in FP32: they only set the FP32 prefilter and the
    // search reach, whose band kBandA is far wider than their rounding
    const float tailf = I.rsf + 2.0f * I.skinf;
    if (lane == 0) rown[wb] = 0;
    __syncwarp();
    auto reach_of = [&](int s) { return ((Rkf + __uint_as_float(rmax_bits[s])) + tailf) + kBandA; };
    const float rho0 = reach_of(b) - kBandA;
    float rho = rho0;
    for (int s = b, own = 1; s >= 0; s = own ? I.partner : -1, own = 0)
        adj_scan<false>(v, I, v.inst[s], k, Rkf, tailf, reach_of(s), own != 0, cx, cy, cz, row[wb], &rown[wb], rho);
    __syncwarp();
    if (rown[wb] > kAdjRaw) {
        __syncwarp();
        if (lane == 0) rown[wb] = 0;
        __syncwarp();
        rho = adj_scan_exact(v, I, I, k, reach_of(b), true, row[wb], &rown[wb], rho0);
        if (I.partner >= 0) adj_scan_exact(v, I, v.inst[I.partner], k, reach_of(I.partner), false, row[wb], &rown[wb], 0.f);
        __syncwarp();
    }
    int n = min(rown[wb], kAdjRaw);
    {
        // the undecided ones, and the row without those that fail
        bool any = false;
        for (int u = lane; u < n; u += 32) any |= (row[wb][u] & kAdjOpen) != 0;
        if (__any_sync(0xffffffffu, any)) {
            int m = 0;
            for (int u0 = 0; u0 < n; u0 += 32) {
                int j = u0 + lane < n ? row[wb][u0 + lane] : -1;
                bool keep = j >= 0;
                if (keep && (j & kAdjOpen)) {
                    double d;
                    j &= ~kAdjOpen;
                    keep = adj_exact(v, I, k, j, d);
                    // (a cell of the own set)
                    if (!keep && j >= I.k0 && j < I.k0 + I.K) rho = fminf(rho, (float)d);
                }
                const unsigned bal = __ballot_sync(0xffffffffu, keep);
                if (keep) row[wb][m + __popc(bal & ((1u << lane) - 1u))] = j;
                m += __popc(bal);
                __syncwarp();
            }
            n = m;
        }
    }
    for (int off = 16; off; off >>= 1) rho = fminf(rho, __shfl_xor_sync(0xffffffffu, rho, off));
    __syncwarp();
    if (n > kAdjRow) {
        if (lane == 0) flag_inst(v, I, kStatusAdjOverflow);
        n = kAdjRow;
    }
    // ascending row: every entry goes to its rank (entries are distinct)
    int val[2], rk[2] = {0, 0};
    for (int u = 0; u < 2; u++) val[u] = (lane + 32 * u < n) ? row[wb][lane + 32 * u] : 0;
    for (int s2 = 0; s2 < n; s2++) {
        const int o = row[wb][s2];
        rk[0] += o < val[0];
        rk[1] += o < val[1];
    }
    for (int u = 0; u < 2; u++) {
        if (lane + 32 * u >= n) continue;
        const int j = val[u];
        pad[(size_t)k * kAdjRow + rk[u]] = j;
        // exact offset between the mirrors' reference points (multiples of
        // 2^-26 sigma; on a periodic axis less the image)
        const long long dx = minimg_q(mirror_ref(v.cq[j]) - mirror_ref(cx), I.boxq[0], I.periodic[0]);
        const long long dy = minimg_q(mirror_ref(v.cq[(size_t)v.Ktot + j]) - mirror_ref(cy), I.boxq[1], I.periodic[1]);
        const long long dz = minimg_q(mirror_ref(v.cq[(size_t)2 * v.Ktot + j]) - mirror_ref(cz), I.boxq[2], I.periodic[2]);
        AdjDesc d;
        d.start = v.cell_start[j];
        d.cnt = v.cell_start[j + 1] - d.start;
        const long long off[3] = {(dx + (1ll << (kMirrorShift - 1))) >> kMirrorShift,
                                  (dy + (1ll << (kMirrorShift - 1))) >> kMirrorShift,
                                  (dz + (1ll << (kMirrorShift - 1))) >> kMirrorShift};
        d.ox = (int)(unsigned)(unsigned long long)off[0];
        d.oy = (int)(unsigned)(unsigned long long)off[1];
        d.oz = (int)(unsigned)(unsigned long long)off[2];
        d.cell_turns = (unsigned)j;
        for (int a = 0; a < 3; a++) d.cell_turns |= turn_code(off[a]) << (kCellBits + 2 * a);
        v.adjd[(size_t)k * kAdjRow + rk[u]] = d;
    }
    if (lane == 0) {
        count[k] = n;
        rho_out[k] = rho;
    }
}

// CSR rows from the fixed-stride rows (for the getters).
__global__ void k_adj_csr(View v, const int* __restrict__ pad) {
    const int k = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int lane = threadIdx.x & 31;
    if (k >= v.Ktot) return;
    const int a0 = v.adj_ptr[k], n = v.adj_ptr[k + 1] - a0;
    for (int t = lane; t < n && a0 + t < v.adj_cap; t += 32) v.adj[a0 + t] = pad[(size_t)k * kAdjRow + t];
}

// ============================================================== host side
static inline int nblk(long long n, int t) { return (int)((n + t - 1) / t); }

void Ensemble::reset_scratch() {
    // every other scratch array starts at zero (alloc)
    k_fill_bbox<<<1, 64, 0, stream>>>(d_bbox, B);
    launches++;
    CK(cudaGetLastError());
    after_baoa_ = -1;
    ovf_clean_ = true;
}

void Ensemble::build_grid() {
    View v = view();
    k_grid_count<<<nblk(Ktot, 256), 256, 0, stream>>>(v, d_gcount, d_gidx, d_cf);
    launches++;
    CK(cudaGetLastError());
    scan_exclusive(d_gcount, d_gstart, Gtot + 1);
    k_grid_fill<<<nblk(Ktot, 256), 256, 0, stream>>>(v, d_gidx, d_gcount, d_cf);
    launches++;
    CK(cudaGetLastError());
}

void Ensemble::mstep_iter(const int* cell_of, int iter) {
    View v = view();
    k_mstep_accum<<<nblk(N, 256), 256, 0, stream>>>(v, cell_of, d_S, d_cnt);
    launches++;
    CK(cudaGetLastError());
    CK(cudaMemsetAsync(d_dmax, 0, sizeof(unsigned) * B, stream));
    k_mstep_finish<<<nblk(Ktot, 256), 256, 0, stream>>>(v, d_S, d_cnt, iter, d_dmax, d_cmove);
    launches++;
    CK(cudaGetLastError());
}

void Ensemble::mirrors(bool unless_exceeded) {
    k_mirrors<<<nblk(N, spread_block(N, 256)), spread_block(N, 256), 0, stream>>>(view(), unless_exceeded ? d_flag : nullptr,
                                                                                 skin_tests_);
    launches++;
    CK(cudaGetLastError());
}

// Skin trigger: has any particle moved more than the skin since the last
// rebuild?  FP32 estimate with a margin that errs towards rebuilding (a
// rebuild never changes the forces, only where they are found).  A yes is the
// test's number in flag, and in the host's copy (mapped memory).
__global__ void k_displacement(View v, const long long* __restrict__ xref, int test, volatile int* flag,
                               volatile int* host) {
    int p = blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= v.N) return;
    int b = find_inst(v.inst_p0, v.B, p);
    const Inst& I = v.inst[b];
    size_t N = v.N;
    float d2 = 0.f;
    for (int a = 0; a < 3; a++) {
        float d = ll_to_float(minimg_q(v.xq[a * N + p] - xref[a * N + p], I.boxq[a], I.periodic[a])) * (float)kGridInv;
        d2 = fmaf(d, d, d2);
    }
    float s = I.skinf * (1.0f - 1e-5f);
    if (d2 > s * s && *flag != test) {
        *flag = test;
        *host = test;
    }
}

// The test is launched as soon as the positions are there, and the host waits
// for it only after it has launched the rest of the update and the mirrors
// that a step without a rebuild needs: the answer's way to the host and the
// next launch's way back pass under them (1M cell with a skin of 0.3: 476 us a
// step when the host waited at once, 462 now).  After a yes the mirrors are
// left alone; the rebuild writes them anew.
void Ensemble::launch_skin_test() {
    skin_tests_ = skin_tests_ < 0x7fffffff ? skin_tests_ + 1 : 1;
    k_displacement<<<nblk(N, spread_block(N, 256)), spread_block(N, 256), 0, stream>>>(view(), d_xref, skin_tests_, d_flag,
                                                                                      skin_host_);
    launches++;
    CK(cudaGetLastError());
    CK(cudaEventRecord(skin_event_, stream));
}

bool Ensemble::skin_exceeded() {
    CK(cudaEventSynchronize(skin_event_));
    return *(volatile int*)skin_host_ == skin_tests_;
}

// The Lloyd rounds of the initialisation, on the particles by grid cell
// (their positions and types in the second state buffers, which the sort of
// finish_cells fills anew).  d_perm is left with the slots in that order.
void Ensemble::lloyd(int iters) {
    const View v = view(), by_cell = view_alt();
    k_grid_particles<<<nblk(N, 256), 256, 0, stream>>>(v, d_gcount);
    launches++;
    CK(cudaGetLastError());
    scan_exclusive(d_gcount, d_gstart, Gtot + 1);
    k_grid_order<<<nblk(N, 256), 256, 0, stream>>>(v, by_cell, d_gstart, d_gcount, d_perm);
    launches++;
    CK(cudaGetLastError());
    swap_state();
    for (int it = 0; it < iters; it++) {
        tic("grid");
        build_grid();
        toc();
        // the first round searches every particle and records a lower bound
        // on its second-nearest centroid; later rounds search only the
        // particles whose bound no longer certifies their centroid
        tic("estep");
        if (it == 0) estep(d_cell, d_lbound);
        else estep_bounded(d_cell);
        toc();
        tic("mstep");
        mstep_iter(d_cell, it);
        toc();
    }
    swap_state();
}

void Ensemble::estep(int* cell_out, float* lbound, const int* order) {
    k_estep_warp<<<nblk(N, 128), 128, 0, stream>>>(view(), cell_out, lbound, order, nullptr);
    launches++;
    CK(cudaGetLastError());
}

void Ensemble::estep_bounded(int* cell) {
    CK(cudaMemsetAsync(d_fbcount, 0, sizeof(int), stream));
    CK(cudaMemsetAsync(d_gmove, 0, sizeof(unsigned) * Gtot, stream));
    k_grid_move<<<nblk(Ktot, 256), 256, 0, stream>>>(view(), d_gidx, d_cmove, d_gmove);
    k_estep_bound<<<nblk(N, 256), 256, 0, stream>>>(view(), cell, d_lbound, d_cf, d_dmax, d_gmove, d_cell_tmp,
                                                    d_fbcount);
    k_estep_warp<<<nblk(N, 128), 128, 0, stream>>>(view(), cell, d_lbound, d_cell_tmp, d_fbcount);
    launches += 3;
    CK(cudaGetLastError());
}

void Ensemble::morton_relabel() {
    View v = view();
    if (!bbox_ready_) {
        k_bbox<<<nblk(Ktot, 256), 256, 0, stream>>>(v, d_bbox);
        launches++;
    }
    bbox_ready_ = false;
    k_morton_keys<<<nblk(Ktot, 256), 256, 0, stream>>>(v, d_bbox, d_keys, d_cq_tmp);
    launches++;
    int ntiles = nblk(Ktot, kTile);
    k_tile_sort<<<ntiles, kTile, 0, stream>>>(v, d_keys, (SortRec*)d_sortrec);
    launches++;
    k_rank_scatter<<<nblk((long long)ntiles * kTile, 256), 256, 0, stream>>>(v, (const SortRec*)d_sortrec, ntiles, d_cq_tmp,
                                                                            d_new_of_old, d_gcount, d_gidx, d_cf, d_bbox);
    launches++;
    CK(cudaGetLastError());
}

// (As many cells as a block has threads: 60,000 particles in 1,000 cells 120 us
// a step, 126 by the five launches, which cells beyond the limit take: 1,025
// cells 124, 1,100 126.)
bool Ensemble::small_cells() const { return B == 1 && Ktot <= kSmallK && Gtot < kSmallG; }

// Whether k_build_cells does the rebuild's last part, or the sort (a block per
// cell), the gather (a thread per particle) and the cells' properties a launch
// each.  The line lies where cells begin to exceed the 128 particles that a
// warp holds: steps of 60,000 particles at a mean of 61 a cell 118 us against
// 122, 95 118 / 122, 105 137 / 130, 128 159 / 130; of 605,000 417 / 432, 425 /
// 424, 435 / 431, 455 / 457; of 1,445,000 857 / 893, 862 / 886, 874 / 886,
// 950 / 949.
bool Ensemble::build_fused() const { return N <= 100ll * Ktot; }

// order: the slots in an order that keeps neighbours together (nullable).
void Ensemble::finish_cells(bool sums_ready, const int* order) {
    View v = view();
    const bool small = small_cells();
    if (small) {
        const int rot = after_baoa_ >= 0 ? 4 : 0;
        k_relabel_small<<<1 + rot, kSmallK, 0, stream>>>(v, sums_ready, d_msum, d_mcnt, d_dmax, d_bbox, d_new_of_old, d_gcount,
                                                         d_gidx, d_cf, d_gstart, d_step, after_baoa_, d_cell_tmp, d_rot_n);
        launches++;
        CK(cudaGetLastError());
        bbox_ready_ = false;
    } else {
        morton_relabel();
        scan_exclusive(d_gcount, d_gstart, Gtot + 1);
    }
    if (prev_adj_valid_) {
        k_cand_rows<<<nblk((long long)Ktot * kRowLanes, 256), 256, 0, stream>>>(v, d_adjcount, d_adjpad, d_new_of_old, d_cf,
                                                                          d_candrows, d_gidx, small ? nullptr : d_gcount);
        k_estep_rows<<<nblk(N, spread_block(N, 128)), spread_block(N, 128), 0, stream>>>(
            v, d_cell, d_adjcount, d_candrows, d_rho, d_new_of_old, d_dmax, d_cell_new, d_cell_tmp, d_fbcount, d_cnt);
        k_estep_list<<<152 * 4, 128, 0, stream>>>(v, d_cell_tmp, d_fbcount, d_cell_new, d_cnt);
        launches += 3;
        CK(cudaGetLastError());
    } else {
        if (!small) {
            k_grid_fill<<<nblk(Ktot, 256), 256, 0, stream>>>(v, d_gidx, d_gcount, d_cf);
            launches++;
        }
        estep(d_cell_new, nullptr, order);
        k_hist<<<nblk(N, 256), 256, 0, stream>>>(N, d_cell_new, d_cnt);
        launches++;
    }
    // stable counting sort
    scan_exclusive(d_cnt, d_cell_start, Ktot + 1);
    const ScratchReset z{d_dmax, d_rmax, d_step, after_baoa_ == 1, d_fbcount, d_rot_n, d_novf_n};
    after_baoa_ = -1;
    ovf_clean_ = true;
    k_scatter<<<nblk(N, 256), 256, 0, stream>>>(N, d_cell_new, d_cell_start, d_cnt, d_perm, B, z);
    launches++;
    CK(cudaGetLastError());
    // gather into the second buffer set, then swap
    swap_state();
    View nv = view();
    View ov = view_alt();
    if (build_fused()) {
        k_build_cells<<<nblk(Ktot, kBuildWarps), 32 * kBuildWarps, 0, stream>>>(nv, ov, d_perm, d_cell_tmp, d_xref, d_rmax);
        launches++;
    } else {
        const long long warps = (long long)Ktot * 32;
        k_segsort_cells<<<Ktot, 256, 0, stream>>>(d_cell_start, d_perm, d_cell_tmp);
        k_gather_particles<<<nblk(N, spread_block(N, 256)), spread_block(N, 256), 0, stream>>>(nv, ov, d_perm, d_cell_new, d_xref);
        k_cell_props<<<nblk(warps, spread_block(warps, 256)), spread_block(warps, 256), 0, stream>>>(nv, d_rmax);
        launches += 3;
    }
    CK(cudaGetLastError());
    // neighbouring cells
    k_adj_warp<<<nblk((long long)Ktot * 32, spread_block((long long)Ktot * 32, 256)), spread_block((long long)Ktot * 32, 256), 0, stream>>>(nv, d_rmax, d_adjcount, d_rho, d_adjpad);
    launches++;
    CK(cudaGetLastError());
    prev_adj_valid_ = true;
    csr_valid_ = false;
    cells_valid = true;
    forces_valid = false;
    list_valid = false;
    n_rebuilds++;
}

void Ensemble::cell_radii() {
    if (!cells_valid) return;
    // (with a skin the particles may have moved since the cells were built)
    k_cell_r2<<<nblk(Ktot, 256), 256, 0, stream>>>(view(), d_xref ? d_xref : d_state[cur_][0]);
    launches++;
    CK(cudaGetLastError());
}

void Ensemble::adjacency_csr() {
    if (csr_valid_ || !cells_valid) return;
    CK(cudaMemsetAsync(d_adjcount + Ktot, 0, sizeof(int), stream));
    scan_exclusive(d_adjcount, d_adj_ptr, Ktot + 1);
    k_adj_csr<<<nblk((long long)Ktot * 32, 256), 256, 0, stream>>>(view(), d_adjpad);
    launches++;
    CK(cudaGetLastError());
    csr_valid_ = true;
}

void Ensemble::rebuild(bool sums_ready) {
    // M-step on the cell-sorted particles, fused with the centroid bounding
    // box (and the B-A-O-A's left-over rotations)
    if (sums_ready && small_cells()) {
        // (part of the small batches' relabel)
        finish_cells(true);
        return;
    }
    if (sums_ready) {
        const int nb = nblk(Ktot, 256);
        k_mstep_apply<<<nb + (after_baoa_ >= 0 ? 152 : 0), 256, 0, stream>>>(
            view(), d_msum, d_mcnt, d_bbox, d_dmax, nb, d_step, after_baoa_, d_cell_tmp, d_rot_n);
    } else {
        k_mstep_sorted<<<nblk(Ktot, 8), 256, 0, stream>>>(view(), d_bbox, d_dmax);
    }
    launches++;
    CK(cudaGetLastError());
    bbox_ready_ = true;
    finish_cells(false);
}

}  // namespace orbc
