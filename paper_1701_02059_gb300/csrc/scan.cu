// Device-wide exclusive prefix sum of int32 counts (cell histograms, grid
// occupancy, bond counts) in one launch: every block scans 4,096 elements,
// publishes its total and obtains its prefix by looking back over the totals
// of the blocks before it (Merrill & Garland, "Single-pass parallel prefix
// scan with decoupled look-back", 2016).  The recursive form (block scans, a
// scan of the totals, a uniform add) took three to five launches and a second
// pass over the array.
#include "ensemble.cuh"

namespace orbc {

constexpr int kScanThreads = 512;
constexpr int kScanItems = 8;
constexpr int kScanBlock = kScanThreads * kScanItems;
constexpr unsigned kScanPolls = 1u << 22;   // bound of each wait for a predecessor

// st: one word per block, flag (1: total, 2: inclusive prefix) above the
// 32-bit value, all zero between launches; ctl: ticket and finished counters
// (zero between launches).  Blocks take their index from the ticket, so every
// block before a waiting one has started.
__global__ void __launch_bounds__(kScanThreads) k_scan(const int* __restrict__ in, int* __restrict__ out, long long n,
                                                       unsigned long long* __restrict__ st, unsigned* __restrict__ ctl,
                                                       unsigned* __restrict__ status) {
    __shared__ int wtot[kScanThreads / 32];
    __shared__ int s_prefix;
    __shared__ unsigned s_bid, s_last;
    const int t = threadIdx.x, lane = t & 31, w = t >> 5;
    const unsigned nb = gridDim.x;
    if (t == 0) s_bid = nb > 1 ? atomicAdd(&ctl[0], 1u) : 0u;
    __syncthreads();
    const unsigned bid = s_bid;
    const long long base = (long long)bid * kScanBlock + (long long)t * kScanItems;
    int v[kScanItems];
    if (base + kScanItems <= n) {
        // (allocations are 256-byte aligned and base is a multiple of 8)
        const int4 a = *reinterpret_cast<const int4*>(in + base), b = *reinterpret_cast<const int4*>(in + base + 4);
        v[0] = a.x; v[1] = a.y; v[2] = a.z; v[3] = a.w;
        v[4] = b.x; v[5] = b.y; v[6] = b.z; v[7] = b.w;
    } else {
#pragma unroll
        for (int q = 0; q < kScanItems; q++) v[q] = (base + q < n) ? in[base + q] : 0;
    }
    int sum = 0;
#pragma unroll
    for (int q = 0; q < kScanItems; q++) sum += v[q];
    int x = sum;
    for (int off = 1; off < 32; off <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, x, off);
        if (lane >= off) x += y;
    }
    if (lane == 31) wtot[w] = x;
    __syncthreads();
    if (w == 0) {
        int s = lane < kScanThreads / 32 ? wtot[lane] : 0;
        for (int off = 1; off < kScanThreads / 32; off <<= 1) {
            const int y = __shfl_up_sync(0xffffffffu, s, off);
            if (lane >= off) s += y;
        }
        const int total = __shfl_sync(0xffffffffu, s, kScanThreads / 32 - 1);
        if (lane < kScanThreads / 32) wtot[lane] = s;
        int prefix = 0;
        if (nb > 1) {
            if (lane == 0)
                atomicExch(&st[bid], ((bid == 0 ? 2ull : 1ull) << 32) | (unsigned)total);
            for (int end = (int)bid - 1; end >= 0; end -= 32) {
                // lane l waits for block end - l (a lane past the first block
                // counts as an inclusive prefix of 0)
                unsigned long long word = 2ull << 32;
                bool ok = true;
                if (end - lane >= 0) {
                    unsigned it = 0;
                    while (((word = *(volatile unsigned long long*)&st[end - lane]) >> 32) == 0ull && ++it < kScanPolls)
                        if (it > 64) __nanosleep(64);
                    ok = (word >> 32) != 0ull;
                }
                if (!__all_sync(0xffffffffu, ok)) {
                    if (lane == 0) atomicOr(status, kStatusTimeout);
                    break;
                }
                const unsigned incl = __ballot_sync(0xffffffffu, (word >> 32) == 2ull);
                const int first = incl ? __ffs(incl) - 1 : 31;
                prefix += __reduce_add_sync(0xffffffffu, lane <= first ? (unsigned)word : 0u);
                if (incl) break;
            }
            if (lane == 0 && bid > 0) atomicExch(&st[bid], (2ull << 32) | (unsigned)(prefix + total));
        }
        if (lane == 0) s_prefix = prefix;
    }
    __syncthreads();
    int excl = s_prefix + x - sum + (w > 0 ? wtot[w - 1] : 0);
    if (base + kScanItems <= n) {
        int o[kScanItems];
#pragma unroll
        for (int q = 0; q < kScanItems; q++) { o[q] = excl; excl += v[q]; }
        *reinterpret_cast<int4*>(out + base) = make_int4(o[0], o[1], o[2], o[3]);
        *reinterpret_cast<int4*>(out + base + 4) = make_int4(o[4], o[5], o[6], o[7]);
    } else {
#pragma unroll
        for (int q = 0; q < kScanItems; q++) {
            if (base + q < n) out[base + q] = excl;
            excl += v[q];
        }
    }
    if (nb == 1) return;
    // the last block to get here clears the words for the next launch: every
    // block has read its predecessors by then
    if (t == 0) s_last = atomicAdd(&ctl[1], 1u) == nb - 1 ? 1u : 0u;
    __syncthreads();
    if (!s_last) return;
    for (unsigned b = t; b < nb; b += kScanThreads) st[b] = 0ull;
    if (t < 2) ctl[t] = 0u;
}

void Ensemble::scan_exclusive(const int* in, int* out, long long n) {
    if (n <= 0) return;
    const long long nb = (n + kScanBlock - 1) / kScanBlock;
    if (scan_words_ < nb + 1) {
        // grown on demand (the set-up runs the largest scan of a step once)
        if (d_scan_) CK(cudaFreeAsync(d_scan_, stream));
        d_scan_ = nullptr;
        scan_words_ = 0;
        CK(cudaMallocAsync(&d_scan_, sizeof(unsigned long long) * (nb + 1), stream));
        CK(cudaMemsetAsync(d_scan_, 0, sizeof(unsigned long long) * (nb + 1), stream));
        scan_words_ = nb + 1;
    }
    k_scan<<<(int)nb, kScanThreads, 0, stream>>>(in, out, n, d_scan_ + 1, (unsigned*)d_scan_, d_status);
    launches++;
    CK(cudaGetLastError());
}

}  // namespace orbc
