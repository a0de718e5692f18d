// Index stage: uvw (metres) x frequency -> pixel, oversampled offset, w-plane.
//
// This is the pre-processing the thesis moves out of the gridder
// (Section 3.3.5): each record's uv coordinate becomes integer indices of
// the beta-oversampled grid (nearest neighbour, Section 2.3.6), and records
// whose footprint leaves the grid are dropped (Bounded Records Assumption,
// Section 2.3.1).  Every floating-point step is an explicitly rounded FP64
// intrinsic, so no multiply-add is ever fused and the result is bit-exact
// with any IEEE-754 implementation of the same sequence.
//
// FP64 division and square root are slow on this GPU, so the sequence has
// one division per channel (the factor f / c0, shared by u, v and w) and
// none per visibility; the w-plane (nearest in sqrt|w|, ties up) is a count
// of precomputed thresholds T_j = ((j - 1/2)/(P - 1))^2 w_max, found by
// binary search.  Each CTA builds both small tables in shared memory.
#include <algorithm>

#include "gw_internal.cuh"

namespace gw {

namespace {

constexpr int kChanCache = 1024;   // channel factors kept in shared memory
constexpr size_t kIndexSmemMax = 227 * 1024;
constexpr int64_t kIndexGlobalMax = 1 << 19;

// What the records are counted into (COUNT: 0 nothing, 1 the bins' counters, 2 a
// histogram of the CTA in shared memory, added to them at the end).
struct CountBins {
    BinGeom g;
    int P, smin, smax, ntiles;
    uint32_t* count;
    uint32_t* cursor;            // cleared for the scatter
    unsigned long long* work;    // valid records, sum of S^2
};

// With COUNT the atomics run beside the FP64 pipe, which bounds the kernel, and
// the binner reads the records once less.  Index and bin stages, us, counted
// apart / here: 8.3 M records over 8,192 bins, 4 polarisations' tables to 63: 522 /
// 479; over 16,384 centre bins 488 / 419; 1.03 M over 32,768 (global) 165 / 125.
template <int COUNT>
__global__ void __launch_bounds__(COUNT == 2 ? kBinSmThreads : 256)
    k_index(const double* __restrict__ uvw, const double* __restrict__ freq, int64_t nrow,
            const int64_t* __restrict__ d_nrow, int nchan, IndexParams p,
            gw_index_rec* __restrict__ out, unsigned long long* __restrict__ dropped,
            CountBins cb) {
    // [nc] channel factors f / c0, then [P - 1] plane thresholds as bit
    // patterns: non-negative finite doubles order like their int64 bits, so
    // the search compares integers (exactly the FP64 comparison)
    extern __shared__ __align__(16) double sh[];
    const int nc = min(nchan, kChanCache);
    const int nthr = p.P > 1 ? p.P - 1 : 0;
    double* sc = sh;
    long long* thr = reinterpret_cast<long long*>(sh + nc);
    for (int c = threadIdx.x; c < nc; c += blockDim.x) sc[c] = __ddiv_rn(__ldg(freq + c), kC0);
    for (int j = threadIdx.x; j < nthr; j += blockDim.x) thr[j] = wplane_threshold(j, p);
    // (the tables are padded to 16 bytes)
    uint32_t* hist = reinterpret_cast<uint32_t*>(sh + ((nc + nthr + 1) & ~1));
    if constexpr (COUNT == 2) clear_hist(hist, cb.ntiles);
    if constexpr (COUNT != 0) clear_cursors(cb.cursor, cb.ntiles);
    unsigned long long n_valid = 0, n_taps = 0;
    __syncthreads();
    if (d_nrow) nrow = min(nrow, *d_nrow);     // row count read on the device
    const int64_t nvis = nrow * (int64_t)nchan;
    unsigned int my_drops = 0;
    // (row, channel) of the grid-stride position, advanced without division
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    int64_t row = i / nchan;
    int chan = (int)(i - row * nchan);
    const int64_t srow = stride / nchan;
    const int schan = (int)(stride - srow * nchan);
    for (; i < nvis; i += stride) {
        const double f_c = chan < nc ? sc[chan] : __ddiv_rn(__ldg(freq + chan), kC0);
        gw_index_rec r;
        const bool valid = index_record(__ldg(uvw + 3 * row + 0), __ldg(uvw + 3 * row + 1),
                                        __ldg(uvw + 3 * row + 2), f_c, p, thr, r);
        if (!valid) ++my_drops;
        reinterpret_cast<int4*>(out)[i] = *reinterpret_cast<const int4*>(&r);
        if constexpr (COUNT != 0) {
            if (valid) {
                const int S = plane_support(r.plane, cb.P, cb.smin, cb.smax);
                ++n_valid;
                n_taps += (unsigned long long)(S * S);
                uint32_t* const to = COUNT == 2 ? hist : cb.count;
                each_bin(r, cb.g, cb.P, cb.smin, cb.smax, [&](int t) { atomicAdd(to + t, 1u); });
            }
        }
        row += srow;
        chan += schan;
        if (chan >= nchan) {
            chan -= nchan;
            ++row;
        }
    }
    // one atomic per warp
    for (int d = 16; d > 0; d >>= 1) my_drops += __shfl_down_sync(0xffffffffu, my_drops, d);
    if ((threadIdx.x & 31) == 0 && my_drops) atomicAdd(dropped, (unsigned long long)my_drops);
    if constexpr (COUNT != 0) {
        for (int d = 16; d > 0; d >>= 1) {
            n_valid += __shfl_down_sync(0xffffffffu, n_valid, d);
            n_taps += __shfl_down_sync(0xffffffffu, n_taps, d);
        }
        if ((threadIdx.x & 31) == 0 && n_valid) {
            atomicAdd(cb.work, n_valid);
            atomicAdd(cb.work + 1, n_taps);
        }
    }
    if constexpr (COUNT == 2) {
        __syncthreads();
        for (int t = threadIdx.x; t < cb.ntiles; t += kBinSmThreads)
            if (hist[t]) atomicAdd(cb.count + t, hist[t]);
    }
}

}  // namespace

bool launch_index(const double* uvw, const double* freq, int64_t nrow, int nchan,
                  const IndexParams& prm, gw_index_rec* out, unsigned long long* dropped,
                  cudaStream_t s, const int64_t* d_nrow, const IndexBins* bins) {
    const int64_t nvis = nrow * (int64_t)nchan;
    if (nvis <= 0) return false;
    int threads = 256;
    int64_t blocks = (nvis + threads - 1) / threads;
    if (blocks > current_sm_count() * 16) blocks = current_sm_count() * 16;
    const size_t tables = ((size_t)std::min(nchan, kChanCache) + (prm.P > 1 ? prm.P - 1 : 0) + 1) / 2 * 16;
    CountBins cb{};
    int mode = 0;
    size_t smem = tables;
    if (bins) {
        const int ntiles = bin_count(bins->g);
        cb = CountBins{bins->g, bins->P, bins->smin, bins->smax, ntiles, bins->sc->count,
                       bins->sc->cursor, bins->sc->work};
        mode = 1;
        if (bin_in_shared(nvis, bins->g)) {
            // the binner's CTAs; where those (more bins than kBinSmFewBins, or
            // few records a bin) leave SMs idle and a thread more than one
            // record, the FP64 work would wait for them: the counters
            // themselves for moderate numbers of centre bins, else counted
            // apart (footprint bins contend more)
            const size_t hsm = sizeof(uint32_t) * (size_t)((ntiles + 3) / 4 * 4);
            int per_sm = 0;
            if (tables + hsm <= kIndexSmemMax &&
                cudaFuncSetAttribute(k_index<2>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                     (int)kIndexSmemMax) == cudaSuccess)
                cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_index<2>, kBinSmThreads,
                                                              tables + hsm);
            const int64_t b = std::min((int64_t)per_sm * current_sm_count(), bin_sm_blocks(nvis, bins->g));
            mode = b >= current_sm_count() || (b > 0 && nvis <= b * kBinSmThreads) ? 2
                   : bins->g.mode == 1 && nvis <= kIndexGlobalMax                 ? 1
                                                                                  : 0;
            if (mode == 2) {
                blocks = b;
                threads = kBinSmThreads;
                smem = tables + hsm;
            }
        }
        if (mode) cudaMemsetAsync(cb.count, 0, sizeof(uint32_t) * ntiles, s);
    }
    auto go = [&](auto k) {
        k<<<(unsigned)blocks, threads, smem, s>>>(uvw, freq, nrow, d_nrow, nchan, prm, out, dropped, cb);
    };
    if (mode == 2) go(k_index<2>);
    else if (mode == 1) go(k_index<1>);
    else go(k_index<0>);
    note_launch();
    return mode != 0;
}

cudaError_t preload_index_kernels() {
    cudaFuncAttributes attr;
    cudaError_t e = cudaFuncGetAttributes(&attr, k_index<0>);
    if (e == cudaSuccess) e = cudaFuncGetAttributes(&attr, k_index<1>);
    if (e == cudaSuccess) e = cudaFuncGetAttributes(&attr, k_index<2>);
    return e;
}

}  // namespace gw
