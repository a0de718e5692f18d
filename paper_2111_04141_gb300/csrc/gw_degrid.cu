// Degridding kernel: the adjoint of gridding (operator G^T of Eq.
// (residualcalc), Section 1.6):
//     V[pol] = sum_{tv, tu} conj(K_i(tv, tu)) * G[pol][kv + tv][ku + tu],
// K_i the record's kernel (K_p[ov][ou], or its conjugate when w < 0).
// Tables of any storage kind are widened to FP32 on load, the sum is FP32,
// and the result is written in the plan's visibility kind.
//
// Three kernels:
// * k_degrid_staged (used by gw_degrid_vis): one CTA of 32 warps per SM
//   serves chunks of work items (at most 1,024 records centred in one tile of
//   16 x 16 points, or 32 x 32 to 128 x 128 for sparse inputs and wide
//   supports).  Warps 0-3 load the records' metadata (id, kernel slice, centre,
//   support) into one of two shared buffers, the next chunk's while all
//   warps compute the current one.  The CTA stages the tile's grid region
//   (the tile plus the chunk's largest half-support on every side) in
//   shared memory once, as polarisation pairs, at a row pitch padded to the
//   support residue (mod 8; 16 for one polarisation) that carries most of the
//   item's taps, and serves
//   all of the item's records from it, so the grid is read from L2/HBM
//   about once per tile instead of once per tap.  Warps claim records one at
//   a time, wide supports first.  One warp per record: lanes take
//   consecutive taps of the S x S footprint (flattened, so every lane is
//   busy), with kernel values loaded four steps ahead, packed FP32x2 FMAs
//   (plain ones for one polarisation) into K.re G and K.im G sums, and a
//   reduce-scatter over the lanes.  The tap column and the region offset
//   advance in one register.  4.2 M visibilities x 1, support 31 (31 steps of 32
//   taps): 3.00 ms with 714 instructions a record and the pitch padded mod 8,
//   2.40 with 550.
//   A region larger than the shared memory is served in bands of rows: every
//   record sums the tap rows in the band, and its sums wait in shared memory
//   for the next one.  (Read through L1/L2 instead, 32 B a tap, 1.04 M
//   visibilities x 4 polarisations with supports to 127 on an 8192^2 grid took
//   13.2 ms; in bands they take 3.0, the same items read in place where few
//   taps share a region 5.2.)  The L1 data pipe bounds it (90 % on the 4-pol
//   w-projection batch, 8.94 ms: 16-byte loads of staged points); before
//   its instructions were cut 32 warps of 64 registers beat 24 of 80 there,
//   9.34 against 9.52 ms, and 3.28 against 3.63 in bands, although some variants
//   spill (FP32 x 4: 88 bytes stored, 52 loaded).
// * k_degrid_direct (small calls): one launch, index records included; the same
//   per-record warp, reading the grid through L1/L2.
// * k_degrid (the allocation-free entry point, and degrid_kernel = 2): the same
//   over binned records, visited in 32 x 32 centre-tile order.
#include "gw_internal.cuh"

namespace gw {

namespace {

constexpr int kThreads = 256;

// A warp's sum of conj(K_i) G over one visibility's S x S footprint, read through
// L1/L2, in every lane: kernel slice K, centre (ku, kv), sg = -1 for the conjugate
// kernel.  Lanes take consecutive taps (t / S, t % S), the loads of four of a
// lane's steps in flight: latency bounds it.  A loop over the rows with lanes
// along them leaves lanes idle and the unrolling to the compiler, which took it
// one way or the other with the length of a slice: 258 k, support 7-127, 8192^2,
// x 4 4.6 or 9.7 ms, here 4.2; x 1 2.6, here 1.2.
template <int NPOL, int TK>
__device__ __forceinline__ void gather_sum(const DegridArgs& a, const typename TabElem<TK>::T* K,
                                           int S, int ku, int kv, float sg, int lane,
                                           float (&acc)[NPOL][2]) {
    using TE = TabElem<TK>;
    const int h = S >> 1, N = a.N;
    // K.re G and K.im G apart, as in the staged kernel: half the length of the
    // chains, and the sums of conj(K_i) at the end
    float2 a1[NPOL], a2[NPOL];
#pragma unroll
    for (int p = 0; p < NPOL; ++p) a1[p] = a2[p] = make_float2(0.f, 0.f);
    // tap (tv, tu), advanced without division
    const int dq = 32 / S, dr = 32 - dq * S;
    int tv = lane / S, tu = lane - tv * S;
#pragma unroll 4
    for (int t = lane; t < S * S; t += 32) {
        const float2 k = TE::load(K + t);
        const int64_t pix = (int64_t)(kv - h + tv) * N + (ku - h + tu);
#pragma unroll
        for (int p = 0; p < NPOL; ++p) {
            const float2 g = __ldg(a.grid + (int64_t)p * N * N + pix);
            a1[p].x = fmaf(k.x, g.x, a1[p].x);
            a1[p].y = fmaf(k.x, g.y, a1[p].y);
            a2[p].x = fmaf(k.y, g.x, a2[p].x);
            a2[p].y = fmaf(k.y, g.y, a2[p].y);
        }
        tu += dr;
        tv += dq;
        if (tu >= S) {
            tu -= S;
            ++tv;
        }
    }
    // (K.re - j s K.im) (G.re + j G.im)
#pragma unroll
    for (int p = 0; p < NPOL; ++p) {
        acc[p][0] = fmaf(sg, a2[p].y, a1[p].x);
        acc[p][1] = fmaf(-sg, a2[p].x, a1[p].y);
    }
#pragma unroll
    for (int p = 0; p < NPOL; ++p)
#pragma unroll
        for (int d = 16; d > 0; d >>= 1) {
            acc[p][0] += __shfl_xor_sync(0xffffffffu, acc[p][0], d);
            acc[p][1] += __shfl_xor_sync(0xffffffffu, acc[p][1], d);
        }
}

// Stores visibility i from every lane's copy of the sums.
template <int NPOL>
__device__ __forceinline__ void store_sums(const DegridArgs& a, int64_t i, int lane,
                                           const float (&acc)[NPOL][2]) {
    if (lane < NPOL) {
        float re = acc[0][0], im = acc[0][1];
#pragma unroll
        for (int p = 1; p < NPOL; ++p)
            if (lane == p) { re = acc[p][0]; im = acc[p][1]; }
        store_vis(a.vis_out, a.vis_kind, i * NPOL + lane, re * a.table_inv, im * a.table_inv);
    }
}

template <int NPOL, int TK>
__global__ void __launch_bounds__(kThreads) k_degrid(DegridArgs a) {
    using TT = typename TabElem<TK>::T;
    const int lane = threadIdx.x & 31;
    const int64_t warp0 = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
    const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
    if (a.row_count && *a.row_count >= a.few_rows) return;
    const uint32_t n = *a.n_entries;
    const int hb = a.beta / 2;
    for (int64_t e = warp0; e < n; e += nwarps) {
        const uint32_t id = __ldg(a.entries + e);
        int4 rv = __ldg(reinterpret_cast<const int4*>(a.rec) + id);
        const gw_index_rec r = *reinterpret_cast<gw_index_rec*>(&rv);
        const int S = __ldg(a.support + r.plane);
        const TT* K = reinterpret_cast<const TT*>(a.table) + __ldg(a.plane_off + r.plane) +
                      ((int64_t)(r.ov + hb) * a.beta + (r.ou + hb)) * slice_elems(S);
        // conj(K_i): K_i = K for w >= 0 (use conj K), K_i = conj K for w < 0 (use K)
        float acc[NPOL][2];
        gather_sum<NPOL, TK>(a, K, S, r.ku, r.kv, (r.flags & GW_FLAG_CONJ) ? -1.f : 1.f, lane, acc);
        store_sums<NPOL>(a, id, lane, acc);
    }
}

template <int NPOL, int TK>
void launch_t(const DegridArgs& a, int64_t nvis, int num_sms, cudaStream_t s) {
    int per_sm = 0;
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_degrid<NPOL, TK>, kThreads, 0);
    if (per_sm < 1) per_sm = 1;
    int64_t blocks = (nvis * 32 + kThreads - 1) / kThreads;
    blocks = std::min<int64_t>(blocks, (int64_t)num_sms * per_sm);
    if (blocks < 1) blocks = 1;
    k_degrid<NPOL, TK><<<(unsigned)blocks, kThreads, 0, s>>>(a);
    note_launch();
}

// Direct degridding for small inputs, the counterpart of the direct gridder:
// one launch and no bins.  A warp per visibility, whose lane 0 computes the
// index record (the same bit-exact FP64 sequence as the index stage) and
// broadcasts it; lanes over the flattened S x S taps read the grid through
// L1/L2.  Dropped visibilities are written as zeros, and the work counters
// accumulate as the binner's would.
constexpr int kDirectChanCache = 256;   // channel factors kept in shared memory

template <int NPOL, int TK>
__global__ void __launch_bounds__(kThreads) k_degrid_direct(DegridArgs a, DirectIndex di,
                                                            unsigned long long* __restrict__ work) {
    using TT = typename TabElem<TK>::T;
    extern __shared__ long long sh_idx[];
    __shared__ unsigned long long s_cnt[3];   // the block's valid, taps, dropped
    const int nthr = di.p.P > 1 ? di.p.P - 1 : 0;
    const int nc = min(di.nchan, kDirectChanCache);
    long long* thr = sh_idx;
    double* fc = reinterpret_cast<double*>(sh_idx + nthr);
    for (int j = threadIdx.x; j < nthr; j += blockDim.x) thr[j] = wplane_threshold(j, di.p);
    for (int c = threadIdx.x; c < nc; c += blockDim.x) fc[c] = __ddiv_rn(__ldg(di.freq + c), kC0);
    if (threadIdx.x < 3) s_cnt[threadIdx.x] = 0;
    __syncthreads();
    const int lane = threadIdx.x & 31;
    const int64_t warp0 = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
    const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
    const int hb = a.beta / 2;
    const int64_t nvis = di.nrow * (int64_t)di.nchan;
    unsigned long long n_valid = 0, n_taps = 0, n_drop = 0;
    for (int64_t i = warp0; i < nvis; i += nwarps) {
        int4 rv = make_int4(0, 0, 0, 0);
        if (lane == 0) {
            const int64_t row = i / di.nchan;
            const int chan = (int)(i - row * di.nchan);
            const double f_c = chan < nc ? fc[chan] : __ddiv_rn(__ldg(di.freq + chan), kC0);
            gw_index_rec r;
            index_record(__ldg(di.uvw + 3 * row + 0), __ldg(di.uvw + 3 * row + 1),
                         __ldg(di.uvw + 3 * row + 2), f_c, di.p, thr, r);
            rv = *reinterpret_cast<const int4*>(&r);
        }
        rv.x = __shfl_sync(0xffffffffu, rv.x, 0);
        rv.y = __shfl_sync(0xffffffffu, rv.y, 0);
        rv.z = __shfl_sync(0xffffffffu, rv.z, 0);
        rv.w = __shfl_sync(0xffffffffu, rv.w, 0);
        const gw_index_rec rc = *reinterpret_cast<const gw_index_rec*>(&rv);
        const bool valid = (rc.flags & GW_FLAG_VALID) != 0;
        const int S = valid ? __ldg(a.support + rc.plane) : 0;
        const int64_t kofs = valid ? __ldg(a.plane_off + rc.plane) +
                                         ((int64_t)(rc.ov + hb) * a.beta + (rc.ou + hb)) * slice_elems(S) : 0;
        if (lane == 0) {
            n_valid += valid;
            n_drop += !valid;
            n_taps += (unsigned long long)(S * S);
        }
#ifdef GW_DEBUG_BOUNDS
        // the slice, the footprint's pixels and the output row
        const int h = S >> 1, N = a.N;
        if (valid && !gw_in_bounds((a.table_elems == 0 || (kofs >= 0 && kofs + (int64_t)S * S <= a.table_elems)) &&
                                       rc.ku - h >= 0 && rc.ku + h < N && rc.kv - h >= 0 && rc.kv + h < N &&
                                       (a.vis_count == 0 || i < a.vis_count),
                                   a.queue ? a.queue + 1 : nullptr))
            continue;
#endif
        float acc[NPOL][2];
        if (valid) {
            gather_sum<NPOL, TK>(a, reinterpret_cast<const TT*>(a.table) + kofs, S, rc.ku, rc.kv,
                                 (rc.flags & GW_FLAG_CONJ) ? -1.f : 1.f, lane, acc);
        } else {
#pragma unroll
            for (int p = 0; p < NPOL; ++p) acc[p][0] = acc[p][1] = 0.f;
        }
        store_sums<NPOL>(a, i, lane, acc);
    }
    // counts are held by lane 0 of each warp: one global atomic per block
    if (lane == 0) {
        if (n_valid) {
            atomicAdd(&s_cnt[0], n_valid);
            atomicAdd(&s_cnt[1], n_taps);
        }
        if (n_drop) atomicAdd(&s_cnt[2], n_drop);
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        if (s_cnt[0]) {
            atomicAdd(work, s_cnt[0]);
            atomicAdd(work + 1, s_cnt[1]);
        }
        if (s_cnt[2]) atomicAdd(di.dropped, s_cnt[2]);
    }
}

template <int TK>
void launch_direct_k(const DegridArgs& a, const DirectIndex& di, unsigned long long* work,
                     cudaStream_t s) {
    const int64_t nvis = di.nrow * (int64_t)di.nchan;
    int64_t blocks = (nvis * 32 + kThreads - 1) / kThreads;
    if (blocks > current_sm_count() * 8) blocks = current_sm_count() * 8;
    const size_t smem = sizeof(long long) * (size_t)(di.p.P > 1 ? di.p.P - 1 : 0) +
                        sizeof(double) * (size_t)std::min(di.nchan, kDirectChanCache);
    const unsigned b = (unsigned)blocks;
    switch (a.npol) {
        case 1: k_degrid_direct<1, TK><<<b, kThreads, smem, s>>>(a, di, work); break;
        case 2: k_degrid_direct<2, TK><<<b, kThreads, smem, s>>>(a, di, work); break;
        case 3: k_degrid_direct<3, TK><<<b, kThreads, smem, s>>>(a, di, work); break;
        default: k_degrid_direct<4, TK><<<b, kThreads, smem, s>>>(a, di, work); break;
    }
    note_launch();
}

#ifndef GW_DEGRID_THREADS
#define GW_DEGRID_THREADS 1024
#endif
constexpr int kStagedThreads = GW_DEGRID_THREADS;
constexpr int kStagedMeta = 1024;   // records whose metadata a CTA stages at once
constexpr int kStagedPad = 4;       // zero elements after each staged plane
#ifndef GW_DEGRID_DEPTH
#define GW_DEGRID_DEPTH 4
#endif
constexpr int kStagedDepth = GW_DEGRID_DEPTH;   // steps of kernel values loaded ahead

// A chunk: at most kStagedMeta records of a work item (items longer than
// that are served in several chunks from one staged region), with its record
// metadata in one of two shared buffers.
struct StagedChunk {
    Item item;
    int c0, nc;     // first record of the chunk in the item, records in it
    int done;       // no work left
    int h;          // largest half-support of the chunk's records (the region's)
    int front, back, next;   // metadata placement, record claims
    int taps[16];   // taps of the chunk's records by S mod kRes
};

constexpr int kLoaderThreads = 128;                       // warps 0-3
constexpr int kMetaPerLoader = kStagedMeta / kLoaderThreads;
constexpr int kLoaderBatch = 4;                           // records whose loads a loader issues together

// Last word of a record's metadata: its support (bits 0-8), the conjugation
// (bit 9) and ceil(2^20 / S) (bits 10-30), with which a lane divides numbers up
// to 32 by S in one multiplication: their product is at most 32 above the
// multiple of 2^20 / S that it stands for, S <= 255.
constexpr uint32_t kMetaSupport = 0x1ffu, kMetaConj = 0x200u;
__device__ __forceinline__ uint32_t meta_support(int S) {
    return (uint32_t)S | (uint32_t)((1 << 20) + S - 1) / (uint32_t)S << 10;
}

__device__ __forceinline__ void loader_sync() {
    asm volatile("bar.sync 1, %0;" ::"n"(kLoaderThreads) : "memory");
}

// GEN: any tile size, regions in bands; otherwise 16 x 16 tiles whose largest
// region fits (a tap loop without the band's bounds: 3.11 against 3.31 ms on
// 4.2 M visibilities of one polarisation, support 31, before the pitch was
// padded for them).
template <int NPOL, int TK, bool GEN>
__global__ void __launch_bounds__(kStagedThreads) k_degrid_staged(DegridArgs a, int hmax, int cap) {
    using TE = TabElem<TK>;
    using TT = typename TE::T;
    constexpr int D = kStagedDepth;
    // grid region as polarisation pairs [NPOL / 2][RS][RS] of (G_p, G_p+1),
    // then [RS][RS] of the last polarisation if NPOL is odd (`cap` grid points
    // at most: larger regions are served in bands of rows); then two chunks'
    // record metadata, and the partial sums of records that span bands
    constexpr int NPR = NPOL / 2;
    extern __shared__ __align__(16) float4 reg[];
    __shared__ StagedChunk s_ch[2];
    if (a.row_count && *a.row_count < a.few_rows) return;
    uint4* meta0;
    {
        const int pm = cap + kStagedPad;
        meta0 = reinterpret_cast<uint4*>(reinterpret_cast<float2*>(reg + (size_t)NPR * pm) +
                                         (NPOL % 2 ? pm : 0));
    }
    float2* part = reinterpret_cast<float2*>(meta0 + 2 * kStagedMeta);   // [kStagedMeta][NPOL]
    const int T = GEN ? 1 << a.tile_shift : 16;
    const int lane = threadIdx.x & 31;
    const int N = a.N, hb = a.beta / 2;
    const uint32_t nitems = *a.item_count;
    const TT* __restrict__ tab = reinterpret_cast<const TT*>(a.table);
    constexpr int kElem = NPR ? 16 : 8;       // bytes of an element of the first plane
    // elements to a row of banks: 8 or 16 lanes of a load take one
    constexpr int kRes = 128 / kElem;
    constexpr uint32_t kPosOff = (1u << 20) - 1;
    const char* const regc = reinterpret_cast<const char*>(reg);
    // thread 0: the item being served and the next chunk's first record
    Item cur{};
    int next_c0 = 0;

    // The loader warps (0-3) pick the next chunk and load its records'
    // metadata (id, kernel slice offset, centre relative to the tile, the word
    // of kMetaSupport) into buffer `buf`, records wider than h_max / 2
    // first: warps claim records in this order, so the long ones start early
    // and the short ones even out the end of the chunk.  Each loader thread
    // issues the loads of its (up to 8) records kLoaderBatch at a time.
    auto load_chunk = [&](const int buf) {
        StagedChunk& c = s_ch[buf];
        if (threadIdx.x == 0) {
            c.done = 0;
            if (next_c0 == 0 || next_c0 >= cur.len) {
                const uint32_t it = atomicAdd(a.queue, 1u);
                c.done = it >= nitems;
                if (it < nitems) cur = a.items[it];
                next_c0 = 0;
            }
            const int nc = min(kStagedMeta, cur.len - next_c0);
            c.item = cur;
            c.c0 = next_c0;
            c.nc = nc;
            c.next = 0;
            c.front = 0;
            c.back = nc;
            // an item served in several chunks keeps one region for all of
            // them: the plan's largest half-support
            c.h = cur.len > kStagedMeta ? hmax : 0;
            for (int k = 0; k < 16; ++k) c.taps[k] = 0;
            next_c0 += nc;
        }
        loader_sync();
        if (c.done) return;
        const Item item = c.item;
        const int c0 = c.c0, nc = c.nc;
        const int tx0 = (item.tile % a.ntiles_u) * T;
        const int ty0 = (item.tile / a.ntiles_u) * T;
        uint4* meta = meta0 + buf * kStagedMeta;
        int hw = 0;
        for (int k0 = 0; k0 < kMetaPerLoader; k0 += kLoaderBatch) {
            uint32_t ids[kLoaderBatch];
            gw_index_rec rcs[kLoaderBatch];
#pragma unroll
            for (int k = 0; k < kLoaderBatch; ++k) {
                const int r = (k0 + k) * kLoaderThreads + threadIdx.x;
                ids[k] = r < nc ? __ldg(a.entries + item.start + c0 + r) : 0u;
            }
#pragma unroll
            for (int k = 0; k < kLoaderBatch; ++k) {
                const int r = (k0 + k) * kLoaderThreads + threadIdx.x;
                if (r < nc) {
                    int4 rv = __ldg(reinterpret_cast<const int4*>(a.rec) + ids[k]);
                    rcs[k] = *reinterpret_cast<gw_index_rec*>(&rv);
                }
            }
#pragma unroll
            for (int k = 0; k < kLoaderBatch; ++k) {
                const int r = (k0 + k) * kLoaderThreads + threadIdx.x;
                if (r < nc) {
                    const gw_index_rec rc = rcs[k];
                    const int S = __ldg(a.support + rc.plane), h = S >> 1;
                    const int64_t kofs = __ldg(a.plane_off + rc.plane) +
                                         ((int64_t)(rc.ov + hb) * a.beta + (rc.ou + hb)) * slice_elems(S);
                    uint32_t rel = (uint32_t)(rc.ku - tx0) | (uint32_t)(rc.kv - ty0) << 8;
                    uint32_t w = meta_support(S) | ((rc.flags & GW_FLAG_CONJ) ? kMetaConj : 0u);
#ifdef GW_DEBUG_BOUNDS
                    // the record's slice, centre tile, region and output row: a
                    // record that fails is replaced by a 1 x 1 one at the
                    // table's start, centred in the tile
                    const bool ok =
                        (a.table_elems == 0 || (kofs >= 0 && kofs + (int64_t)S * S <= a.table_elems)) &&
                        rc.ku - tx0 >= 0 && rc.ku - tx0 < T && rc.kv - ty0 >= 0 &&
                        rc.kv - ty0 < T && h <= hmax &&
                        (a.vis_count == 0 || ids[k] < (uint64_t)a.vis_count);
                    if (!gw_in_bounds(ok, a.queue + 1)) {
                        rel = 8u | 8u << 8;
                        w = meta_support(1);
                    }
#endif
                    const int pos =
                        h > hmax / 2 ? atomicAdd(&c.front, 1) : atomicSub(&c.back, 1) - 1;
#ifdef GW_DEBUG_BOUNDS
                    if (!gw_in_bounds(pos >= 0 && pos < nc, a.queue + 1)) continue;
                    if ((w & kMetaSupport) == 1u && S != 1) {
                        meta[pos] = make_uint4(0u, 0u, rel, w);
                        continue;
                    }
#endif
                    meta[pos] = make_uint4(ids[k], (uint32_t)kofs, rel, w);
                    hw = max(hw, h);
                    atomicAdd(&c.taps[S & (kRes - 1)], S * S);
                }
            }
            if ((k0 + kLoaderBatch) * kLoaderThreads >= nc) break;
        }
        hw = (int)__reduce_max_sync(0xffffffffu, (unsigned)hw);
        if (lane == 0 && hw > 0) atomicMax(&c.h, hw);
    };

    // sum of a record's polarisation over one band: stored, or added to the
    // bands before and kept for the bands after
    auto finish = [&](int r, int p, uint32_t id, int before, bool more, float re, float im) {
        if constexpr (GEN) {
            float2* w = part + r * NPOL + p;
            if (before > 0) {
                re += w->x;
                im += w->y;
            }
            if (more) {
                *w = make_float2(re, im);
                return;
            }
        }
        store_vis(a.vis_out, a.vis_kind, (int64_t)id * NPOL + p, re * a.table_inv,
                  im * a.table_inv);
    };

    if (threadIdx.x < kLoaderThreads) load_chunk(0);
    __syncthreads();
    for (int kc = 0;; ++kc) {
        const int buf = kc & 1;
        const StagedChunk& c = s_ch[buf];
        if (c.done) break;
        const Item item = c.item;
        const int c0 = c.c0, nc = c.nc;
        const int tx0 = (item.tile % a.ntiles_u) * T;
        const int ty0 = (item.tile / a.ntiles_u) * T;
        const uint4* meta = meta0 + buf * kStagedMeta;
        // the region: rows and columns [t0 - hi, t0 + T + hi) of the tile,
        // RS x RS values at row pitch RSP; each plane holds RS x RSP elements
        // and kStagedPad zeros (element RS * RSP is read by lanes without a
        // tap in a record's last step).  The kRes flattened taps of a load's
        // quarter (16 bytes) or half (8) that cross a footprint row end jump by
        // RSP - S elements: with RSP = S mod kRes the load stays free of bank
        // conflicts (8 bytes: 2 wavefronts, else 3), so the
        // pitch is padded to the residue of the supports that carry most of
        // the item's taps, where the shared memory allows (items served in
        // several chunks keep RSP = RS).  RS is even, so every part stays
        // 16-byte aligned.
        const int hi = c.h;
        const int RS = T + 2 * hi;
        int RSP = RS;
        if (item.len <= kStagedMeta) {
            int best = 0, bt = -1;
#pragma unroll
            for (int k = 1; k < kRes; k += 2)  // supports are odd
                if (c.taps[k] > bt) {
                    bt = c.taps[k];
                    best = k;
                }
            const int rsp = RS + ((best - RS) & (kRes - 1));
            if (RS * rsp <= cap || (GEN && RS * RS > cap)) RSP = rsp;
        }
        // bands of BR region rows, of equal height
        const int nb = !GEN || RS * RSP <= cap ? 1 : (RS + cap / RSP - 1) / (cap / RSP);
        const int BR = (RS + nb - 1) / nb;
        const int plane = BR * RSP + kStagedPad;
        const int zoff = BR * RSP;
        float2* single = reinterpret_cast<float2*>(reg + (size_t)NPR * plane);
        for (int band = 0; band < nb; ++band) {
            const int yb = GEN ? band * BR : 0, nrows = GEN ? min(BR, RS - yb) : RS;
            if (c0 == 0 || nb > 1) {
                const int rx0 = tx0 - hi, ry0 = ty0 - hi + yb;
                if (band > 0 && threadIdx.x == 0) s_ch[buf].next = 0;
                if (threadIdx.x < kStagedPad) {
#pragma unroll
                    for (int q = 0; q < NPR; ++q)
                        reg[(size_t)q * plane + zoff + threadIdx.x] = make_float4(0.f, 0.f, 0.f, 0.f);
                    if (NPOL % 2) single[zoff + threadIdx.x] = make_float2(0.f, 0.f);
                }
                // (one polarisation: one load a point, so four points a time;
                // 60 k x 1 on 8192^2 271 -> 206 us, with two no gain)
#pragma unroll(NPOL == 1 ? 4 : 1)
                for (int e0 = threadIdx.x; e0 < nrows * RS; e0 += kStagedThreads) {
                    const int y = e0 / RS, x = e0 - y * RS;
                    const int e = y * RSP + x;
                    const int gy = ry0 + y, gx = rx0 + x;
                    const bool in = gx >= 0 && gx < N && gy >= 0 && gy < N;
                    float2 g[NPOL];
#pragma unroll
                    for (int p = 0; p < NPOL; ++p)
                        g[p] = in ? __ldg(a.grid + ((int64_t)p * N + gy) * N + gx) : make_float2(0.f, 0.f);
#pragma unroll
                    for (int q = 0; q < NPR; ++q)
                        reg[(size_t)q * plane + e] = make_float4(g[2 * q].x, g[2 * q].y, g[2 * q + 1].x,
                                                                 g[2 * q + 1].y);
                    if (NPOL % 2) single[e] = g[NPOL - 1];
                }
                __syncthreads();
            }
            // the loaders prepare the next chunk, then join the record claims
            if (band == nb - 1 && threadIdx.x < kLoaderThreads) load_chunk(buf ^ 1);
            for (;;) {
                int r = 0;
                if (lane == 0) r = atomicAdd(&s_ch[buf].next, 1);
                r = __shfl_sync(0xffffffffu, r, 0);
                if (r >= nc) break;
                const uint4 m = meta[r];
                const uint32_t id = m.x;
                const int S = (int)(m.w & kMetaSupport);
                const uint32_t inv = m.w >> 10;
                const float sg = m.w & kMetaConj ? -1.f : 1.f;
                // region row and column of tap (0, 0): centre - h + hi; the tap rows
                // [tv0, tv1) lie in this band
                const int ry = (int)(m.z >> 8) - (S >> 1) + hi, rx = (int)(m.z & 0xffu) - (S >> 1) + hi;
                const int tv0 = GEN ? max(0, yb - ry) : 0;
                const int tv1 = GEN ? min(S, yb + nrows - ry) : S;
                if (GEN && tv1 <= tv0) continue;
                const TT* K = tab + m.y + tv0 * S;
                const int n = (tv1 - tv0) * S;
                // flattened taps t = lane + 32 i at pos = tap column << 20 | region
                // offset (bytes of a plane, below 2^20): 32 taps on, the column
                // is up by dr, or by dr - S and a row further where it wraps;
                // one comparison, select and addition for both parts
                const int dq = (int)(32u * inv >> 20), dr = 32 - dq * S;
                const int lq = (int)((uint32_t)lane * inv >> 20);
                const uint32_t wrap_at = (uint32_t)(S - dr) << 20;
                const uint32_t go_on = ((uint32_t)dr << 20) + (uint32_t)((dq * RSP + dr) * kElem);
                const uint32_t go_wrap = go_on - ((uint32_t)S << 20) + (uint32_t)((RSP - S) * kElem);
                const int tu = lane - lq * S;
                uint32_t pos = (uint32_t)tu << 20 |
                               (uint32_t)(((ry + tv0 - yb + lq) * RSP + rx + tu) * kElem);
                // a1 = sum K.re G, a2 = sum K.im G (packed FP32x2 FMAs); the
                // conjugation sign is applied once at the end
                float2 a1[NPOL], a2[NPOL];
#pragma unroll
                for (int p = 0; p < NPOL; ++p) a1[p] = a2[p] = make_float2(0.f, 0.f);
                auto tap = [&](const float2 k, const uint32_t o) {
                    if constexpr (NPOL == 1) {
                        // one use of each: packing K.re and K.im twice would cost
                        // more than the packed FMAs save
                        const float2 g = *reinterpret_cast<const float2*>(regc + o);
                        a1[0].x = fmaf(k.x, g.x, a1[0].x);
                        a1[0].y = fmaf(k.x, g.y, a1[0].y);
                        a2[0].x = fmaf(k.y, g.x, a2[0].x);
                        a2[0].y = fmaf(k.y, g.y, a2[0].y);
                    } else {
                        const float2 kxx = make_float2(k.x, k.x), kyy = make_float2(k.y, k.y);
#pragma unroll
                        for (int q = 0; q < NPR; ++q) {
                            const float4 g =
                                *reinterpret_cast<const float4*>(regc + q * plane * kElem + o);
                            const float2 g0 = make_float2(g.x, g.y), g1 = make_float2(g.z, g.w);
                            a1[2 * q] = __ffma2_rn(kxx, g0, a1[2 * q]);
                            a2[2 * q] = __ffma2_rn(kyy, g0, a2[2 * q]);
                            a1[2 * q + 1] = __ffma2_rn(kxx, g1, a1[2 * q + 1]);
                            a2[2 * q + 1] = __ffma2_rn(kyy, g1, a2[2 * q + 1]);
                        }
                        if (NPOL % 2) {
                            const float2 g = *reinterpret_cast<const float2*>(
                                regc + NPR * plane * kElem + o / 2);
                            a1[NPOL - 1] = __ffma2_rn(kxx, g, a1[NPOL - 1]);
                            a2[NPOL - 1] = __ffma2_rn(kyy, g, a2[NPOL - 1]);
                        }
                    }
                };
                auto advance = [&]() { pos += pos >= wrap_at ? go_wrap : go_on; };
                // steps 0 .. nfull - 1 have a tap on every lane, step nfull on
                // the lanes below n - 32 nfull.  Kernel values are loaded D steps
                // ahead, unconditionally: past the slice they read the next
                // slice or the table's zero slack, never used.
                const int nfull = (n - 1) >> 5;
                const TT* kp = K + lane;
                TT kq[D];
#pragma unroll
                for (int d = 0; d < D; ++d) kq[d] = __ldg(kp + 32 * d);
                kp += 32 * D;
                int i = 0;
                for (; i + D <= nfull; i += D) {
#pragma unroll
                    for (int d = 0; d < D; ++d) {
                        const float2 k = TE::cvt(kq[d]);
                        kq[d] = __ldg(kp + 32 * d);
                        tap(k, pos & kPosOff);
                        advance();
                    }
                    kp += 32 * D;
                }
                // the last (< D) full steps and the partial one
#pragma unroll
                for (int d = 0; d < D; ++d) {
                    if (i + d > nfull) break;
                    const bool live = i + d < nfull || lane + 32 * nfull < n;
                    tap(live ? TE::cvt(kq[d]) : make_float2(0.f, 0.f), live ? pos & kPosOff : (uint32_t)(zoff * kElem));
                    advance();
                }
                // conj(K_i) G with K_i = K (w >= 0) or conj K (w < 0):
                // re = sum K.re G.re + s K.im G.im, im = sum K.re G.im - s K.im G.re
                float acc[NPOL][2];
#pragma unroll
                for (int p = 0; p < NPOL; ++p) {
                    acc[p][0] = fmaf(sg, a2[p].y, a1[p].x);
                    acc[p][1] = fmaf(-sg, a2[p].x, a1[p].y);
                }
                // reduce-scatter over the lanes: of the 2 NPOL sums (8 for 3
                // polarisations, two of them zero) a lane keeps the half that
                // its top bit picks, and so on down to one, which the lanes
                // left sum; 6, 7 and 10 shuffles (1, 2 and 3-4 polarisations)
                // where whole sums took 10, 20 and 40
                constexpr int NV = NPOL == 3 ? 8 : 2 * NPOL;
                float v[NV];
#pragma unroll
                for (int k = 0; k < NV; ++k) v[k] = k < 2 * NPOL ? acc[k / 2][k % 2] : 0.f;
                int d = 16;
#pragma unroll
                for (int w = NV / 2; w > 0; w >>= 1, d >>= 1) {
                    const bool up = (lane & d) != 0;
#pragma unroll
                    for (int k = 0; k < w; ++k)
                        v[k] = (up ? v[k + w] : v[k]) +
                               __shfl_xor_sync(0xffffffffu, up ? v[k] : v[k + w], d);
                }
                constexpr int kLow = 32 / NV;     // lanes that hold parts of the same sum
#pragma unroll
                for (; d > 0; d >>= 1) v[0] += __shfl_xor_sync(0xffffffffu, v[0], d);
                // the lanes of the real part fetch the imaginary one
                const float im = __shfl_down_sync(0xffffffffu, v[0], kLow);
                if ((lane & (2 * kLow - 1)) == 0 && lane / (2 * kLow) < NPOL)
                    finish(r, lane / (2 * kLow), id, tv0, tv1 < S, v[0], im);
            }
            __syncthreads();   // band consumed; after the last, the next chunk's metadata is in place
        }
    }
}

template <int NPOL, int TK, bool GEN>
void launch_staged_g(const DegridArgs& a, int hmax, size_t cap, size_t part, int num_sms,
                     cudaStream_t s) {
    const size_t smem = (cap + kStagedPad) * NPOL * sizeof(float2) +
                        2 * kStagedMeta * sizeof(uint4) + part;
    // (the most that any call needs: another thread may be between its setting
    // and its launch)
    constexpr size_t most = kStagedSmemMax + kStagedPad * NPOL * sizeof(float2) +
                            2 * kStagedMeta * sizeof(uint4);
    cudaFuncSetAttribute(k_degrid_staged<NPOL, TK, GEN>,
                         cudaFuncAttributeMaxDynamicSharedMemorySize, (int)most);
    k_degrid_staged<NPOL, TK, GEN><<<num_sms, kStagedThreads, smem, s>>>(a, hmax, (int)cap);
    note_launch();
}

template <int NPOL, int TK>
void launch_staged_t(const DegridArgs& a, int hmax, int num_sms, cudaStream_t s) {
    // grid points of the largest region where it fits, else as many as fit
    // beside the partial sums of a chunk
    const int RS = (1 << a.tile_shift) + 2 * hmax;
    constexpr size_t point = NPOL * sizeof(float2);
    // with its padded pitch where that fits too
    size_t cap = (size_t)RS * (RS + (NPOL == 1 ? 16 : 8)), part = 0;
    if ((size_t)RS * RS * point > kStagedSmemMax) part = kStagedMeta * point;
    cap = std::min(cap, (kStagedSmemMax - part) / point / 4 * 4);
    if (part || a.tile_shift != 4)
        launch_staged_g<NPOL, TK, true>(a, hmax, cap, part, num_sms, s);
    else
        launch_staged_g<NPOL, TK, false>(a, hmax, cap, part, num_sms, s);
}

template <int TK>
void launch_staged_k(const DegridArgs& a, int hmax, int num_sms, cudaStream_t s) {
    switch (a.npol) {
        case 1: launch_staged_t<1, TK>(a, hmax, num_sms, s); break;
        case 2: launch_staged_t<2, TK>(a, hmax, num_sms, s); break;
        case 3: launch_staged_t<3, TK>(a, hmax, num_sms, s); break;
        default: launch_staged_t<4, TK>(a, hmax, num_sms, s); break;
    }
}

template <int TK>
void launch_k(const DegridArgs& a, int64_t nvis, int num_sms, cudaStream_t s) {
    switch (a.npol) {
        case 1: launch_t<1, TK>(a, nvis, num_sms, s); break;
        case 2: launch_t<2, TK>(a, nvis, num_sms, s); break;
        case 3: launch_t<3, TK>(a, nvis, num_sms, s); break;
        default: launch_t<4, TK>(a, nvis, num_sms, s); break;
    }
}

}  // namespace

cudaError_t preload_degrid_kernel(int npol, int table_kind) {
    cudaFuncAttributes attr;
    auto get = [&](auto f) { return cudaFuncGetAttributes(&attr, f); };
    const int tk = table_kind == GW_BF16X2 ? 1 : (table_kind == GW_F16X2 ? 2 : 0);
    switch (npol * 3 + tk) {
        case 3: return get(k_degrid<1, GW_C64>);
        case 4: return get(k_degrid<1, GW_BF16X2>);
        case 5: return get(k_degrid<1, GW_F16X2>);
        case 6: return get(k_degrid<2, GW_C64>);
        case 7: return get(k_degrid<2, GW_BF16X2>);
        case 8: return get(k_degrid<2, GW_F16X2>);
        case 9: return get(k_degrid<3, GW_C64>);
        case 10: return get(k_degrid<3, GW_BF16X2>);
        case 11: return get(k_degrid<3, GW_F16X2>);
        case 13: return get(k_degrid<4, GW_BF16X2>);
        case 14: return get(k_degrid<4, GW_F16X2>);
        default: return get(k_degrid<4, GW_C64>);
    }
}

void launch_degrid_staged(const DegridArgs& a, int hmax, int num_sms, cudaStream_t s) {
    cudaMemsetAsync(a.queue, 0, sizeof(uint32_t), s);
    switch (a.table_kind) {
        case GW_BF16X2: launch_staged_k<GW_BF16X2>(a, hmax, num_sms, s); break;
        case GW_F16X2: launch_staged_k<GW_F16X2>(a, hmax, num_sms, s); break;
        default: launch_staged_k<GW_C64>(a, hmax, num_sms, s); break;
    }
}

void launch_degrid_direct(const DegridArgs& a, const DirectIndex& di, unsigned long long* work,
                          cudaStream_t s) {
    if (di.nrow <= 0 || di.nchan <= 0) return;
    switch (a.table_kind) {
        case GW_BF16X2: launch_direct_k<GW_BF16X2>(a, di, work, s); break;
        case GW_F16X2: launch_direct_k<GW_F16X2>(a, di, work, s); break;
        default: launch_direct_k<GW_C64>(a, di, work, s); break;
    }
}

void launch_degrid(const DegridArgs& a, int64_t nvis, int num_sms, cudaStream_t s) {
    switch (a.table_kind) {
        case GW_BF16X2: launch_k<GW_BF16X2>(a, nvis, num_sms, s); break;
        case GW_F16X2: launch_k<GW_F16X2>(a, nvis, num_sms, s); break;
        default: launch_k<GW_C64>(a, nvis, num_sms, s); break;
    }
}

}  // namespace gw
