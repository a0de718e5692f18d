// Device binner: groups visibility ids by grid tile.
//
// The thesis orders records by their position on the NN grid ("SS" mode,
// Section 3.3.5) because record order controls commit traffic.  Here the
// equivalent is a bin per grid tile (2^su x 2^sv pixels):
//   footprint mode: a record is listed in every tile its S_p x S_p footprint
//                   touches (the gridder owns a tile and needs all of them);
//   centre mode:    a record is listed once, in the tile of its pixel (the
//                   degridder reads a record's whole footprint).
// Steps: histogram (atomics; per-CTA shared histograms when the tile count
// allows) -> exclusive scan -> scatter (atomic cursors),
// and the scan cuts the bins into work items of at most item_max entries.
// Order within a bin is unspecified.
#include "gw_internal.cuh"

namespace gw {

namespace {

__device__ __forceinline__ gw_index_rec load_rec(const gw_index_rec* rec, int64_t i) {
    int4 v = __ldg(reinterpret_cast<const int4*>(rec) + i);
    return *reinterpret_cast<gw_index_rec*>(&v);
}

__global__ void k_count(const gw_index_rec* __restrict__ rec, int64_t nvis, DevCount dc, BinGeom g,
                        int P, int smin, int smax, uint32_t* __restrict__ count,
                        unsigned long long* __restrict__ work) {
    nvis = dc.clamp(nvis);
    unsigned long long n_valid = 0, n_taps = 0;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < nvis;
         i += (int64_t)gridDim.x * blockDim.x) {
        const gw_index_rec r = load_rec(rec, i);
        if (!(r.flags & GW_FLAG_VALID)) continue;
        const int S = plane_support(r.plane, P, smin, smax);
        ++n_valid;
        n_taps += (unsigned long long)(S * S);
        const TileRange t = tile_range(r, g, P, smin, smax);
        const int lbase = g.layer_tiles ? (r.plane / g.group_planes) * g.layer_tiles : 0;
        for (int tv = t.tv0; tv <= t.tv1; ++tv)
            for (int tu = t.tu0; tu <= t.tu1; ++tu)
                atomicAdd(count + lbase + tv * g.ntu + tu, 1u);
    }
    for (int d = 16; d > 0; d >>= 1) {
        n_valid += __shfl_down_sync(0xffffffffu, n_valid, d);
        n_taps += __shfl_down_sync(0xffffffffu, n_taps, d);
    }
    if ((threadIdx.x & 31) == 0 && n_valid) {
        atomicAdd(work, n_valid);
        atomicAdd(work + 1, n_taps);
    }
}

// Exclusive scans of count[] -> offsets[] and of the bins' work items ->
// item_off[], with zeroed cursors and the work items, in segments of kScanSeg
// bins, one CTA each.
// Up to kScanSingleMax bins one kernel does it: every CTA first sums the bins
// before its segment (at most 1 MB of counts, read from L2 by 1,024 threads),
// so no CTA waits for another.  A bin a thread: the scan of 8,192 bins of 9.9 M
// entries took 43 us with 8 bins and their items a thread.  Beyond, pass 0 writes each
// segment's totals, k_scan_top scans the totals in one CTA, and pass 1 finishes.
constexpr int kScanThreads = 1024;
constexpr int kScanSeg = kScanThreads;
constexpr int kScanSingleMax = 262144;

__device__ __forceinline__ void block_excl_scan2(uint32_t& a, uint32_t& b, uint32_t* sa,
                                                 uint32_t* sb) {
    // exclusive scan of (a, b) over the CTA (kScanThreads threads)
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    uint32_t ia = a, ib = b;
    for (int d = 1; d < 32; d <<= 1) {
        const uint32_t xa = __shfl_up_sync(0xffffffffu, ia, d);
        const uint32_t xb = __shfl_up_sync(0xffffffffu, ib, d);
        if (lane >= d) { ia += xa; ib += xb; }
    }
    if (lane == 31) { sa[warp] = ia; sb[warp] = ib; }
    __syncthreads();
    if (warp == 0) {
        uint32_t wa = sa[lane], wb = sb[lane];
        for (int d = 1; d < 32; d <<= 1) {
            const uint32_t xa = __shfl_up_sync(0xffffffffu, wa, d);
            const uint32_t xb = __shfl_up_sync(0xffffffffu, wb, d);
            if (lane >= d) { wa += xa; wb += xb; }
        }
        sa[lane] = wa;
        sb[lane] = wb;
    }
    __syncthreads();
    const uint32_t ba = warp ? sa[warp - 1] : 0u, bb = warp ? sb[warp - 1] : 0u;
    a = ba + ia - a;
    b = bb + ib - b;
}

// Work items of a warp's 32 bins (the lanes' sizes c, item counts ni, first
// entries ra and items rb).  The warp writes
// its bins one after another, so that a bin of thousands of items is not one
// thread's.
__device__ __forceinline__ void write_items(Item* __restrict__ items, int bin0, int lane, uint32_t c,
                                            uint32_t ni, uint32_t ra, uint32_t rb,
                                            const ItemRule& rule) {
    for (uint32_t left = __ballot_sync(0xffffffffu, ni != 0); left; left &= left - 1) {
        const int src = __ffs(left) - 1;
        const uint32_t nc = __shfl_sync(0xffffffffu, c, src), nn = __shfl_sync(0xffffffffu, ni, src);
        const uint32_t st = __shfl_sync(0xffffffffu, ra, src), o = __shfl_sync(0xffffffffu, rb, src);
        const uint32_t item_max = rule.size(nc);
        for (uint32_t k = lane; k < nn; k += 32) {
            Item it;
            it.tile = bin0 + src;
            it.start = (int32_t)(st + k * item_max);
            it.len = (int32_t)min(item_max, nc - k * item_max);
            it.pad = 0;
            items[o + k] = it;
        }
    }
}

// pass 0: segment totals; pass 1: the rest, from scanned totals; pass 2: all in
// one kernel.
__global__ void __launch_bounds__(kScanThreads) k_scan_seg(
    const uint32_t* __restrict__ count, int n, ItemRule rule, int pass,
    uint32_t* __restrict__ seg_tot, uint32_t* __restrict__ offsets,
    uint32_t* __restrict__ item_off, uint32_t* __restrict__ cursor, Item* __restrict__ items) {
    __shared__ uint32_t sa[32], sb[32];
    const int s0 = blockIdx.x * kScanSeg, i = s0 + (int)threadIdx.x, lane = threadIdx.x & 31;
    const uint32_t c = i < n ? count[i] : 0u, ni = rule.items(c);
    uint32_t ra = 0, rb = 0;
    if (pass == 2 && s0 > 0) {
        uint32_t pa = 0, pb = 0;                     // bins before this segment
        for (int k = threadIdx.x; k < s0 / 4; k += kScanThreads) {
            const uint4 q = __ldg(reinterpret_cast<const uint4*>(count) + k);
            pa += q.x + q.y + q.z + q.w;
            pb += rule.items(q.x) + rule.items(q.y) + rule.items(q.z) + rule.items(q.w);
        }
        pa = __reduce_add_sync(0xffffffffu, pa);
        pb = __reduce_add_sync(0xffffffffu, pb);
        if (lane == 0) {
            sa[threadIdx.x >> 5] = pa;
            sb[threadIdx.x >> 5] = pb;
        }
        __syncthreads();
        ra = __reduce_add_sync(0xffffffffu, sa[lane]);
        rb = __reduce_add_sync(0xffffffffu, sb[lane]);
        __syncthreads();
    }
    uint32_t ea = c, eb = ni;
    block_excl_scan2(ea, eb, sa, sb);
    if (pass == 0) {
        if (threadIdx.x == kScanThreads - 1) {
            seg_tot[2 * blockIdx.x] = ea + c;
            seg_tot[2 * blockIdx.x + 1] = eb + ni;
        }
        return;
    }
    if (pass == 1) {
        ra = seg_tot[2 * blockIdx.x];
        rb = seg_tot[2 * blockIdx.x + 1];
    }
    ra += ea;
    rb += eb;
    if (i < n) {
        offsets[i] = ra;
        item_off[i] = rb;
        cursor[i] = 0;
    }
    if (pass == 2 && i == n - 1) {
        offsets[n] = ra + c;
        item_off[n] = rb + ni;
    }
    if (!items) return;                              // (the allocation-free degrid path)
    write_items(items, i - lane, lane, c, ni, ra, rb, rule);
}

// Exclusive scan of the segment totals in place (one CTA, nseg <= 32 * 1024);
// writes the grand totals to offsets[n] and item_off[n].
__global__ void __launch_bounds__(kScanThreads) k_scan_top(uint32_t* __restrict__ seg_tot, int nseg,
                                                           int n, uint32_t* __restrict__ offsets,
                                                           uint32_t* __restrict__ item_off) {
    __shared__ uint32_t sa[32], sb[32];
    const int per = (nseg + kScanThreads - 1) / kScanThreads;
    const int lo = min(nseg, (int)threadIdx.x * per), hi = min(nseg, lo + per);
    uint32_t ta = 0, tb = 0;
    for (int i = lo; i < hi; ++i) {
        ta += seg_tot[2 * i];
        tb += seg_tot[2 * i + 1];
    }
    uint32_t ea = ta, eb = tb;
    block_excl_scan2(ea, eb, sa, sb);
    for (int i = lo; i < hi; ++i) {
        const uint32_t xa = seg_tot[2 * i], xb = seg_tot[2 * i + 1];
        seg_tot[2 * i] = ea;
        seg_tot[2 * i + 1] = eb;
        ea += xa;
        eb += xb;
    }
    if (threadIdx.x == kScanThreads - 1) {
        offsets[n] = ea;
        item_off[n] = eb;
    }
}

__global__ void k_scatter(const gw_index_rec* __restrict__ rec, int64_t nvis, DevCount dc,
                          BinGeom g, int P, int smin, int smax,
                          const uint32_t* __restrict__ offsets, uint32_t* __restrict__ cursor,
                          uint32_t* __restrict__ entries) {
    nvis = dc.clamp(nvis);
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < nvis;
         i += (int64_t)gridDim.x * blockDim.x) {
        const gw_index_rec r = load_rec(rec, i);
        if (!(r.flags & GW_FLAG_VALID)) continue;
        const TileRange t = tile_range(r, g, P, smin, smax);
        const int lbase = g.layer_tiles ? (r.plane / g.group_planes) * g.layer_tiles : 0;
        for (int tv = t.tv0; tv <= t.tv1; ++tv)
            for (int tu = t.tu0; tu <= t.tu1; ++tu) {
                const int tile = lbase + tv * g.ntu + tu;
                const uint32_t pos = atomicAdd(cursor + tile, 1u);
                entries[offsets[tile] + pos] = (uint32_t)i;
            }
    }
}

// Shared-memory variants (ntiles small enough for a per-CTA histogram): a
// CTA takes a contiguous chunk of records and counts its (record, tile)
// pairs with shared-memory atomics; only the non-zero bins reach global
// memory, one atomic each.  The scatter recounts its chunk, reserves one run
// per (CTA, tile) in the tile's bin with a single global atomic, and places
// the entries with shared-memory cursors that start at the run bases.

// Work on the records [c0, c1) of a CTA, kBinIlp loads of a thread in flight:
// one at a time with 512 threads, the loads' latency bounded these kernels (bin
// stage, us, before / now: 3.1 M records over 32,768 bins 275 / 199, 4.2 M over
// 2,048 and 16,384 258 / 229, 255 k over 4,096 39 / 32, 8.3 M over 8,192 261 /
// 259).  Lanes of one bin sharing an atomic (match_any) were slower: 437 / 337 on
// the first two.
constexpr int kBinIlp = 4;

template <class F>
__device__ __forceinline__ void each_record(const gw_index_rec* __restrict__ rec, int64_t c0,
                                            int64_t c1, F f) {
    for (int64_t i0 = c0 + threadIdx.x; i0 < c1; i0 += kBinIlp * kBinSmThreads) {
        gw_index_rec r[kBinIlp];
#pragma unroll
        for (int k = 0; k < kBinIlp; ++k) {
            const int64_t i = i0 + k * kBinSmThreads;
            if (i < c1) r[k] = load_rec(rec, i);
            else r[k].flags = 0;
        }
#pragma unroll
        for (int k = 0; k < kBinIlp; ++k)
            if (r[k].flags & GW_FLAG_VALID) f(r[k], (uint32_t)(i0 + k * kBinSmThreads));
    }
}

__global__ void __launch_bounds__(kBinSmThreads) k_count_sm(
    const gw_index_rec* __restrict__ rec, int64_t nvis, DevCount dc, BinGeom g, int P, int smin,
    int smax, int ntiles, uint32_t* __restrict__ count, uint32_t* __restrict__ cursor,
    unsigned long long* __restrict__ work) {
    extern __shared__ __align__(16) uint32_t hist[];
    nvis = dc.clamp(nvis);
    clear_hist(hist, ntiles);
    clear_cursors(cursor, ntiles);
    __syncthreads();
    const int64_t chunk = (nvis + gridDim.x - 1) / gridDim.x;
    const int64_t c0 = blockIdx.x * chunk, c1 = min(nvis, c0 + chunk);
    unsigned long long n_valid = 0, n_taps = 0;
    each_record(rec, c0, c1, [&](const gw_index_rec& r, uint32_t) {
        const int S = plane_support(r.plane, P, smin, smax);
        ++n_valid;
        n_taps += (unsigned long long)(S * S);
        each_bin(r, g, P, smin, smax, [&](int t) { atomicAdd(hist + t, 1u); });
    });
    __syncthreads();
    for (int t = threadIdx.x; t < ntiles; t += kBinSmThreads)
        if (hist[t]) atomicAdd(count + t, hist[t]);
    for (int d = 16; d > 0; d >>= 1) {
        n_valid += __shfl_down_sync(0xffffffffu, n_valid, d);
        n_taps += __shfl_down_sync(0xffffffffu, n_taps, d);
    }
    if ((threadIdx.x & 31) == 0 && n_valid) {
        atomicAdd(work, n_valid);
        atomicAdd(work + 1, n_taps);
    }
}

// SCAN: the scan of at most kScanFusedMax bins is part of the kernel: every CTA
// scans all the counts for itself, and each writes the offsets and work items of
// some segments of them.  One launch less: 30 k records over 512 bins 16.8 ->
// 13.1 us for the bin stage, 472 k over 1,128 23.4 -> 20.1; 8.3 M over 8,192
// 200 -> 197.
constexpr int kScanFusedMax = 8192;

template <bool SCAN>
__global__ void __launch_bounds__(kBinSmThreads) k_scatter_sm(
    const gw_index_rec* __restrict__ rec, int64_t nvis, DevCount dc, BinGeom g, int P, int smin,
    int smax, int ntiles, const uint32_t* __restrict__ count, uint32_t* __restrict__ offsets,
    uint32_t* __restrict__ item_off, uint32_t* __restrict__ cursor, Item* __restrict__ items,
    uint32_t* __restrict__ entries) {
    extern __shared__ __align__(16) uint32_t hist[];
    nvis = dc.clamp(nvis);
    constexpr int kSegs = kScanFusedMax / kScanSeg;
    uint32_t cnt[SCAN ? kSegs : 1];
    if constexpr (SCAN) {
#pragma unroll
        for (int k = 0; k < kSegs; ++k) {
            const int t = k * kScanSeg + (int)threadIdx.x;
            cnt[k] = t < ntiles ? __ldg(count + t) : 0u;
        }
    }
    clear_hist(hist, ntiles);
    __syncthreads();
    const int64_t chunk = (nvis + gridDim.x - 1) / gridDim.x;
    const int64_t c0 = blockIdx.x * chunk, c1 = min(nvis, c0 + chunk);
    each_record(rec, c0, c1, [&](const gw_index_rec& r, uint32_t) {
        each_bin(r, g, P, smin, smax, [&](int t) { atomicAdd(hist + t, 1u); });
    });
    __syncthreads();
    // this CTA's run in each bin: absolute position of its first entry
    if constexpr (SCAN) {
        __shared__ uint32_t sa[32], sb[32];
        const ItemRule rule(g);
        const int lane = threadIdx.x & 31;
        uint32_t ra = 0, rb = 0;                         // before the segment
#pragma unroll
        for (int k = 0; k < kSegs; ++k) {
            if (k * kScanSeg >= ntiles) break;
            const int t = k * kScanSeg + (int)threadIdx.x;
            const uint32_t c = cnt[k], ni = rule.items(c);
            uint32_t ea = c, eb = ni;
            block_excl_scan2(ea, eb, sa, sb);
            ea += ra;
            eb += rb;
            ra += sa[31];
            rb += sb[31];
            if (t < ntiles && hist[t]) hist[t] = ea + atomicAdd(cursor + t, hist[t]);
            if (k % gridDim.x == blockIdx.x) {
                if (t < ntiles) {
                    offsets[t] = ea;
                    item_off[t] = eb;
                }
                if (t == ntiles - 1) {
                    offsets[ntiles] = ra;
                    item_off[ntiles] = rb;
                }
                if (items) write_items(items, t - lane, lane, c, ni, ea, eb, rule);
            }
            __syncthreads();
        }
    } else {
        for (int t0 = threadIdx.x; t0 < ntiles; t0 += kBinIlp * kBinSmThreads) {
            uint32_t c[kBinIlp], o[kBinIlp];
#pragma unroll
            for (int k = 0; k < kBinIlp; ++k) {
                const int t = t0 + k * kBinSmThreads;
                c[k] = t < ntiles ? hist[t] : 0u;
                o[k] = c[k] ? __ldg(offsets + t) : 0u;
                c[k] = c[k] ? atomicAdd(cursor + t, c[k]) : 0u;
            }
#pragma unroll
            for (int k = 0; k < kBinIlp; ++k) {
                const int t = t0 + k * kBinSmThreads;
                if (t < ntiles) hist[t] = o[k] + c[k];
            }
        }
    }
    __syncthreads();
    each_record(rec, c0, c1, [&](const gw_index_rec& r, uint32_t id) {
        each_bin(r, g, P, smin, smax, [&](int t) { entries[atomicAdd(hist + t, 1u)] = id; });
    });
}

}  // namespace

void launch_bin(const gw_index_rec* rec, int64_t nvis, const BinGeom& g, int P, int smin, int smax,
                Scratch& sc, cudaStream_t s, DevCount dc, bool counted) {
    const int ntiles = bin_count(g);
    if (!counted) cudaMemsetAsync(sc.count, 0, sizeof(uint32_t) * ntiles, s);
    // per-CTA shared histograms where zeroing and flushing one stays a small
    // part of a CTA's work (bin_sm_blocks); sparser inputs keep the
    // global-atomic kernels, which spread over all SMs
    int sm_blocks = 0;
    const size_t hsm = sizeof(uint32_t) * (size_t)((ntiles + 3) / 4 * 4);
    if (bin_in_shared(nvis, g)) {
        int dev = 0, nsm = 0, c_sm = 0, s_sm = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
        // (the most that any call needs: another thread may be between its
        // setting and its launch)
        const int most = (int)sizeof(uint32_t) * kBinSmTilesMax;
        cudaFuncSetAttribute(k_count_sm, cudaFuncAttributeMaxDynamicSharedMemorySize, most);
        cudaFuncSetAttribute(k_scatter_sm<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, most);
        cudaFuncSetAttribute(k_scatter_sm<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, most);
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&c_sm, k_count_sm, kBinSmThreads, hsm);
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(
            &s_sm, ntiles <= kScanFusedMax ? k_scatter_sm<true> : k_scatter_sm<false>, kBinSmThreads, hsm);
        sm_blocks = (int)std::min<int64_t>((int64_t)std::min(c_sm, s_sm) * nsm,
                                           bin_sm_blocks(nvis, g));
    }
    const int threads = 256;
    int64_t blocks = (nvis + threads - 1) / threads;
    if (blocks > current_sm_count() * 8) blocks = current_sm_count() * 8;
    if (blocks < 1) blocks = 1;
    if (nvis > 0 && !counted) {
        if (sm_blocks > 0)
            k_count_sm<<<sm_blocks, kBinSmThreads, hsm, s>>>(rec, nvis, dc, g, P, smin, smax, ntiles,
                                                             sc.count, sc.cursor, sc.work);
        else
            k_count<<<(unsigned)blocks, threads, 0, s>>>(rec, nvis, dc, g, P, smin, smax, sc.count,
                                                         sc.work);
        note_launch();
    }
    const int nseg = (ntiles + kScanSeg - 1) / kScanSeg;
    if (sm_blocks > 0 && ntiles <= kScanFusedMax) {
        // (the cursors were cleared where the records were counted)
        k_scatter_sm<true><<<sm_blocks, kBinSmThreads, hsm, s>>>(
            rec, nvis, dc, g, P, smin, smax, ntiles, sc.count, sc.offsets, sc.item_off, sc.cursor,
            sc.items, sc.entries);
        note_launch();
        return;
    }
    if (ntiles <= kScanSingleMax || !sc.scan_tmp || ntiles > sc.scan_tmp_bins) {
        k_scan_seg<<<nseg, kScanThreads, 0, s>>>(sc.count, ntiles, ItemRule(g), 2, nullptr, sc.offsets,
                                                 sc.item_off, sc.cursor, sc.items);
        note_launch();
    } else {
        k_scan_seg<<<nseg, kScanThreads, 0, s>>>(sc.count, ntiles, ItemRule(g), 0, sc.scan_tmp,
                                                 sc.offsets, sc.item_off, sc.cursor, sc.items);
        k_scan_top<<<1, kScanThreads, 0, s>>>(sc.scan_tmp, nseg, ntiles, sc.offsets, sc.item_off);
        k_scan_seg<<<nseg, kScanThreads, 0, s>>>(sc.count, ntiles, ItemRule(g), 1, sc.scan_tmp,
                                                 sc.offsets, sc.item_off, sc.cursor, sc.items);
        note_launch(3);
    }
    if (nvis > 0) {
        if (sm_blocks > 0)
            k_scatter_sm<false><<<sm_blocks, kBinSmThreads, hsm, s>>>(
                rec, nvis, dc, g, P, smin, smax, ntiles, sc.count, sc.offsets, sc.item_off,
                sc.cursor, sc.items, sc.entries);
        else
            k_scatter<<<(unsigned)blocks, threads, 0, s>>>(rec, nvis, dc, g, P, smin, smax,
                                                           sc.offsets, sc.cursor, sc.entries);
        note_launch();
    }
}

cudaError_t preload_bin_kernels() {
    cudaFuncAttributes attr;
    cudaError_t e = cudaFuncGetAttributes(&attr, k_count);
    if (e == cudaSuccess) e = cudaFuncGetAttributes(&attr, k_count_sm);
    if (e == cudaSuccess) e = cudaFuncGetAttributes(&attr, k_scatter);
    if (e == cudaSuccess) e = cudaFuncGetAttributes(&attr, k_scatter_sm<false>);
    if (e == cudaSuccess) e = cudaFuncGetAttributes(&attr, k_scatter_sm<true>);
    if (e == cudaSuccess) e = cudaFuncGetAttributes(&attr, k_scan_seg);
    if (e == cudaSuccess) e = cudaFuncGetAttributes(&attr, k_scan_top);
    return e;
}

int64_t scan_tmp_words(int64_t ntiles) { return 2 * ((ntiles + kScanSeg - 1) / kScanSeg) + 2; }

}  // namespace gw
