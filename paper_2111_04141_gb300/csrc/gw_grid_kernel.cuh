// Gridding kernel: w-projection convolutional gridding onto a complex grid.
// Included once per table kind by gw_grid_c64.cu, gw_grid_bf16.cu and
// gw_grid_f16.cu.
//
// Computes the Gridding Step of Algorithm convgriddingoversampling
// (Section 2.4.5) with the w-projection GCF (Section 1.7.1):
//     G[pol][kv + tv][ku + tu] += K_p[ov][ou](tv, tu) * V[pol]   (conj K if w < 0)
//
// Design (GB300):
// * A CTA (one per SM) owns one 64 (u) x 32 (v) tile of the grid for a work
//   item (a run of that tile's bin) and keeps the tile's accumulators in
//   registers, so each grid point is committed once per work item (vector
//   atomics, red.global).
// * Sixteen compute warps each own an 8 (u) x 16 (v) block; lane (lu, lv)
//   holds the points (lu, lv + 4 j), j = 0..3 ("slots" of 8 x 4 points), for
//   every polarisation.  Four slots per warp amortise each record's staged
//   visibility over up to 4 x 32 points.  (The lane layout is a compile-time
//   choice, kGridLanesU x kGridLanesV = 8 x 4 or 16 x 2; the text describes
//   the default.)
// * The work is bound by the gathers of kernel values from L2 (each a
//   4-row x 64-byte window of a table slice per slot) and by the FP32 pipe,
//   so the design keeps many gathers in flight and many warps issuing: 20
//   warps per SM (4 compute warps and one producer warp per scheduler, 96
//   registers per thread), each compute warp holding the kernel values of
//   the next R = 3 list entries in a ring of registers.
// * Four producer warps (one warpgroup) stage batches of 256 records into
//   shared memory: the record ids and index records are loaded for all rows
//   at once, the visibilities are copied straight into shared memory with
//   cp.async (or widened / weighted in registers for 16-bit or weighted
//   input), and every record is appended to the list of each compute warp
//   whose block its footprint meets, with the record's table offset for the
//   tile and the slots its rows meet (one 64-bit entry).  Compute warps
//   therefore only see records that touch them.
// * Hand-over through mbarriers: a compute warp waits only for the batch it
//   needs and releases it when done, so the sixteen compute warps run
//   independently; the producers wait until all of them have released a
//   buffer before refilling it.  Every wait is bounded: a wait that gives up
//   sets the plan's device status word and the kernel returns.
// * The producers pad every warp's list to a multiple of R and append R more
//   null entries (no loads, the all-zero visibility row), so the compute loop
//   has no tail tests: the kernel values of entry i + R are loaded into the
//   registers entry i has just used, and the last pass over a batch loads the
//   first entries of the next batch (the ring never drains between batches).
//   An entry loads the slots its record
//   meets and zeros for the others, and always updates all four slots (one
//   loop body, no per-entry jump: the code stays small at ring depth R).
// * Kernel values come from zero-padded slices (kGridPadC = 7 zero columns
//   and kGridPadR = 3 zero rows around each S x S slice, one compile-time
//   row stride per plan), so
//   lanes outside the footprint read zeros and slot addresses are immediate
//   offsets.
// * Per tap and polarisation the update is two packed FP32x2 FMAs (Blackwell
//   FFMA2) on the (re, im) accumulator pair:
//     acc += (K.re, K.re) (.) (V.re, V.im) + (K.im, K.im) (.) s (-V.im, V.re)
//   with s = -1 for the conjugate kernel (w < 0); the staged visibility is
//   the plain (weighted) value, the second operand is formed in registers.
// * Storage precision: the table element type is a template parameter
//   (complex FP32, or bfloat16 / float16 pairs widened to FP32 on load);
//   visibilities of any kind are widened to FP32 when staged; all
//   accumulation is FP32.  With an error grid the commit is compensated
//   (commit_compensated).
// * Where tables and visibilities are of one 16-bit kind, with two and more
//   polarisations and no weights, the compute warps are MmaWarp instead of
//   FmaWarp (kernels, us, of 1.41 M visibilities, support 7-83, 2348^2, 1 / 2 / 3 / 4
//   polarisations: 1,473 / 1,443 / 1,476 / 1,451 against 1,394 / 1,666 / 2,012 /
//   2,436; seven other shapes alike): the same
//   producers, tiles and hand-over, the products on the tensor cores.  An
//   FP32 warp issues 32 packed FMAs (two issue slots each) and about 40 other
//   instructions for an entry of 128 points and 4 polarisations; the tensor
//   cores take 8 entries with 8 products and some 120 others.  3.13 M
//   visibilities x 4 polarisations, 8192^2, 128 planes, support 7 -> 127,
//   bfloat16: 5.24 -> 3.16 ms (2.9e12 -> 4.8e12 point updates x pol / s).
//   FP32 operands split in two TF32 parts (three products a row) were slower
//   than the FMAs (4096^2 batch: 11.1 against 8.25 ms): the split and the
//   address arithmetic cost more than the FMAs they replace.
#pragma once

#include <type_traits>

#include "gw_internal.cuh"

// Kernel-value register sets in flight per FP32 compute warp (measured on the
// 4-pol w-projection batch: 16 compute warps with ring 3 beat 8 compute warps
// with rings of 2-10 entries at 168 registers).
#ifndef GW_GRID_RING
#define GW_GRID_RING 3
#endif

namespace gw {

namespace {

constexpr int kComputeWarps = 16;
#ifndef GW_GRID_PRODUCER_WARPS
#define GW_GRID_PRODUCER_WARPS 4
#endif
constexpr int kProducerWarps = GW_GRID_PRODUCER_WARPS;
constexpr int kProducerThreads = kProducerWarps * 32;
constexpr int kThreads = (kComputeWarps + kProducerWarps) * 32;
constexpr int kRows = 256;                             // staged rows of a buffer
constexpr int kPerLane = kRows / kProducerThreads;     // rows staged by each producer thread
constexpr int kProducerBar = 1;                        // named barrier of the producer warps

__device__ __forceinline__ gw_index_rec load_rec(const gw_index_rec* rec, uint32_t i) {
    int4 v = __ldg(reinterpret_cast<const int4*>(rec) + i);
    return *reinterpret_cast<gw_index_rec*>(&v);
}

// ---- mbarriers (shared memory, CTA scope) ----------------------------------
__device__ __forceinline__ uint32_t smem_u32(const void* p) {
    return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}
__device__ __forceinline__ void mbar_init(unsigned long long* bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count)
                 : "memory");
}
__device__ __forceinline__ void mbar_arrive(unsigned long long* bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(unsigned long long* bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(smem_u32(bar)), "r"(parity)
        : "memory");
    return ok != 0;
}
__device__ __forceinline__ uint64_t global_ns() {
    uint64_t t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}
// Waits for the completion of the barrier phase of the given parity; gives
// up after about two seconds (a batch hand-over takes microseconds).
__device__ __forceinline__ bool mbar_wait(unsigned long long* bar, uint32_t parity) {
    if (mbar_try_wait(bar, parity)) return true;
    const uint64_t t0 = global_ns();
    for (;;) {
        for (int k = 0; k < 64; ++k)
            if (mbar_try_wait(bar, parity)) return true;
        if (global_ns() - t0 > 2000000000ull) return false;
    }
}
__device__ __forceinline__ void producer_sync() {
    asm volatile("bar.sync %0, %1;" ::"n"(kProducerBar), "n"(kProducerThreads) : "memory");
}

// ---- asynchronous global -> shared copies ----------------------------------
__device__ __forceinline__ void cp_async16(void* dst, const void* src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_u32(dst)), "l"(src)
                 : "memory");
}
__device__ __forceinline__ void cp_async8(void* dst, const void* src) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(smem_u32(dst)), "l"(src)
                 : "memory");
}
__device__ __forceinline__ void cp_async4(void* dst, const void* src) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(smem_u32(dst)), "l"(src)
                 : "memory");
}
__device__ __forceinline__ void cp_async_wait_all() {
    asm volatile("cp.async.commit_group;\n\tcp.async.wait_all;" ::: "memory");
}

// Commit with the rounding error kept: the vector atomic returns the value
// it added to, so the exact error of the (round-to-nearest) sum it stored is
// recovered with Knuth's TwoSum and accumulated into a second grid.  The
// compensated value is grid + err (a Kahan-style sum of the commits).
__device__ __forceinline__ void commit_compensated(float2* g, float2* err, float2 val) {
    const float2 old = atomicAdd(g, val);
    float2 e;
    {
        const float s = __fadd_rn(old.x, val.x);
        const float bv = __fsub_rn(s, old.x);
        const float av = __fsub_rn(s, bv);
        e.x = __fadd_rn(__fsub_rn(old.x, av), __fsub_rn(val.x, bv));
    }
    {
        const float s = __fadd_rn(old.y, val.y);
        const float bv = __fsub_rn(s, old.y);
        const float av = __fsub_rn(s, bv);
        e.y = __fadd_rn(__fsub_rn(old.y, av), __fsub_rn(val.y, bv));
    }
    if (e.x != 0.f || e.y != 0.f) atomicAdd(err, e);
}

// ---- compute warps: FP32 FMAs --------------------------------------------------
// List entry: x = padded-table index of the tile origin relative to the record;
// y = record row in the batch (bits 0-8), conjugate kernel (bit 19), mask of
// the slots the record's rows meet (bits 20-23).
constexpr uint32_t kConjBit = 1u << 19;

// Packed FMAs of one entry into slots J0..J1 (compile-time range); A = V,
// Bv = s (-V.im, V.re) (unused for a real kernel).
template <int NPOL, int J0, int J1, class TE>
__device__ __forceinline__ void slot_fma(float2 (&acc)[4][NPOL], const typename TE::T (&Kr)[4],
                                         const float2 (&A)[NPOL], const float2 (&Bv)[NPOL]) {
#pragma unroll
    for (int j = J0; j <= J1; ++j) {
        const float2 kc = TE::cvt(Kr[j]);   // 16-bit pairs are widened here, at their use
        const float2 kxx = make_float2(kc.x, kc.x);
        const float2 kyy = make_float2(kc.y, kc.y);
#pragma unroll
        for (int p = 0; p < NPOL; ++p) acc[j][p] = __ffma2_rn(kxx, A[p], acc[j][p]);
        if constexpr (!TE::kReal) {
#pragma unroll
            for (int p = 0; p < NPOL; ++p) acc[j][p] = __ffma2_rn(kyy, Bv[p], acc[j][p]);
        }
    }
}

// Staged visibility of an entry and the second FMA operand s (-V.im, V.re)
// (not formed for a real kernel).
template <int NPOL, bool REAL>
__device__ __forceinline__ void load_v(float2 (&A)[NPOL], float2 (&Bv)[NPOL],
                                       const float2 (*vs)[NPOL], uint32_t ey) {
    const float2* row = vs[ey & 0x1ff];
    if (NPOL % 2 == 0) {
#pragma unroll
        for (int p = 0; p < NPOL; p += 2) {
            const float4 q = *reinterpret_cast<const float4*>(row + p);
            A[p] = make_float2(q.x, q.y);
            A[p + 1] = make_float2(q.z, q.w);
        }
    } else {
#pragma unroll
        for (int p = 0; p < NPOL; ++p) A[p] = row[p];
    }
    if constexpr (!REAL) {
        const float s = (ey & kConjBit) ? -1.f : 1.f;
#pragma unroll
        for (int p = 0; p < NPOL; ++p) Bv[p] = make_float2(-s * A[p].y, s * A[p].x);
    }
}

// Kernel values of one list entry, as stored: the slots in its mask, zero
// (all bits clear, +0 in every storage kind) for the others.
template <int SP, class TE>
__device__ __forceinline__ void load_masked(const typename TE::T* __restrict__ tab, const uint2 en,
                                            typename TE::T (&Kd)[4]) {
    using T = typename TE::T;
    const uint32_t m = en.y >> 20;
    const T* p_ = tab + (int)en.x;
    const T z{};
    Kd[0] = (m & 1u) ? __ldg(p_) : z;
    Kd[1] = (m & 2u) ? __ldg(p_ + kGridLanesV * SP) : z;
    Kd[2] = (m & 4u) ? __ldg(p_ + 2 * kGridLanesV * SP) : z;
    Kd[3] = (m & 8u) ? __ldg(p_ + 3 * kGridLanesV * SP) : z;
}

template <int NPOL, int SP, int TK>
struct FmaWarp {
    using TE = TabElem<TK>;
    using T = typename TE::T;
    using VT = float2;                         // staged visibility
    static constexpr int kPol = NPOL, R = GW_GRID_RING;
    static constexpr int kBlockU = kGridLanesU, kBlockV = 4 * kGridLanesV;
    static constexpr int kBatch = kRows;       // records staged at a time
    static constexpr uint32_t kZeroRow = kBatch;   // staged row that is always zero
    static constexpr int kVisRows = kBatch + 1;
    const T* __restrict__ tab;
    float2 acc[4][NPOL];                       // (re, im)
    // kernel-value ring, in the table's storage kind; finite values only
    // (zero, then table values), so the null entries' zero visibility row
    // contributes exact zeros
    T K[R][4];
    uint32_t ey[R];

    __device__ __forceinline__ FmaWarp(const GridArgs& a, int warp, int lane) {
        constexpr int blocks = kGridTileU / kBlockU;
        const int bu = (warp % blocks) * kBlockU, bv = (warp / blocks) * kBlockV;
        tab = reinterpret_cast<const T*>(a.ptable) + (bv + lane / kGridLanesU) * SP + bu +
              lane % kGridLanesU;
#pragma unroll
        for (int j = 0; j < 4; ++j)
#pragma unroll
            for (int p = 0; p < NPOL; ++p) acc[j][p] = make_float2(0.f, 0.f);
#pragma unroll
        for (int d = 0; d < R; ++d)
#pragma unroll
            for (int j = 0; j < 4; ++j) K[d][j] = T{};
    }
    // Fills the ring with the first R entries of a list.
    __device__ __forceinline__ void fill(const uint2* lst, const VT (*)[NPOL]) {
#pragma unroll
        for (int d = 0; d < R; ++d) {
            const uint2 en = lst[d];
            ey[d] = en.y;
            load_masked<SP, TE>(tab, en, K[d]);
        }
    }
    // One ring pass: the FMAs of the R entries in the ring, each followed by the
    // loads of the entry R positions later, taken from `next`.  Every entry
    // updates all four slots; the slots outside its mask add zeros (spare FMA
    // issue, but one short loop body per ring position and no per-entry jump).
    __device__ __forceinline__ void pass(const uint2* next, const VT (*vs)[NPOL], const VT (*)[NPOL]) {
#pragma unroll
        for (int d = 0; d < R; ++d) {
            float2 A[NPOL], Bv[NPOL];
            load_v<NPOL, TE::kReal>(A, Bv, vs, ey[d]);
            slot_fma<NPOL, 0, 3, TE>(acc, K[d], A, Bv);
            const uint2 en = next[d];
            ey[d] = en.y;
            load_masked<SP, TE>(tab, en, K[d]);
        }
    }
    // Commits the block's accumulators at (u0, v0) of `gbase` and clears them.
    __device__ __forceinline__ void commit(const GridArgs& a, float2* gbase, int u0, int v0, int lane) {
        const int N = a.N, u = u0 + lane % kGridLanesU;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const int v = v0 + lane / kGridLanesU + kGridLanesV * j;
#pragma unroll
            for (int p = 0; p < NPOL; ++p) {
                if (u < N && v < N && (acc[j][p].x != 0.f || acc[j][p].y != 0.f)) {
                    const float2 val = make_float2(acc[j][p].x * a.table_inv,
                                                   acc[j][p].y * a.table_inv);
                    const int64_t off = ((int64_t)p * N + v) * N + u;
                    if (a.grid_err) {
                        commit_compensated(gbase + off, a.grid_err + off, val);
                    } else {
                        atomicAdd(gbase + off, val);
                    }
                }
                acc[j][p] = make_float2(0.f, 0.f);
            }
        }
    }
    // Producer: visibility `id` (weighted) into a staged row.
    static __device__ __forceinline__ void stage(const GridArgs& a, bool copy, VT (&row)[NPOL],
                                                 uint32_t id) {
        if (copy) {
            const float2* src = reinterpret_cast<const float2*>(a.vis) + (int64_t)id * NPOL;
            if (NPOL % 2 == 0) {
#pragma unroll
                for (int p = 0; p < NPOL; p += 2) cp_async16(&row[p], src + p);
            } else {
#pragma unroll
                for (int p = 0; p < NPOL; ++p) cp_async8(&row[p], src + p);
            }
        } else {
#pragma unroll
            for (int p = 0; p < NPOL; ++p) {
                float2 v = load_vis(a.vis, a.vis_kind, (int64_t)id * NPOL + p);
                if (a.weight) {
                    const float w = __ldg(a.weight + (int64_t)id * NPOL + p);
                    v.x *= w;
                    v.y *= w;
                }
                row[p] = v;
            }
        }
    }
    // visibilities copied as they are: FP32 pairs without weights, with
    // the 16-byte alignment the 16-byte copies need (pairs of polarisations)
    static __device__ __forceinline__ bool copies(const GridArgs& a) {
        return a.vis_kind == GW_C64 && a.weight == nullptr &&
               (NPOL % 2 == 1 || reinterpret_cast<uintptr_t>(a.vis) % 16 == 0);
    }
    // Producer: list entries of a record (staged row r, footprint lower corner
    // (ulo, vlo) and upper corner relative to the tile).
    struct Entries {
        uint32_t base, ey;
        __device__ __forceinline__ Entries(const GridArgs& a, const gw_index_rec& rc, int plane, int S,
                                           int r, int ulo, int vlo) {
            const int64_t slice = __ldg(a.pplane_off + plane) +
                                  ((int64_t)(rc.ov + a.beta / 2) * a.beta + (rc.ou + a.beta / 2)) *
                                      (int64_t)(S + 2 * kGridPadR) * SP;
            // padded index of the tile origin relative to this record
            base = (uint32_t)((int)slice + (kGridPadR - vlo) * SP + kGridPadC - ulo);
            ey = (uint32_t)r | ((rc.flags & GW_FLAG_CONJ) ? kConjBit : 0u);
        }
        // entry of block (cu, cv), whose rows j0 .. j1 the footprint meets
        __device__ __forceinline__ uint2 operator()(int, int, int j0, int j1) const {
            const uint32_t mask = ((2u << (j1 / kGridLanesV)) - 1u) & ~((1u << (j0 / kGridLanesV)) - 1u);
            return make_uint2(base, ey | (mask << 20));
        }
        // first and last table element the entry's loads touch
        __device__ __forceinline__ void span(uint2, int cu, int cv, int j0, int j1, int64_t& lo,
                                             int64_t& hi) const {
            j0 = j0 / kGridLanesV * kGridLanesV;
            j1 = j1 / kGridLanesV * kGridLanesV + kGridLanesV - 1;
            lo = (int64_t)(int)base + (int64_t)(kBlockV * cv + j0) * SP + kBlockU * cu;
            hi = (int64_t)(int)base + (int64_t)(kBlockV * cv + j1) * SP + kBlockU * cu + kBlockU - 1;
        }
    };
};

// Commits the sums s0, s1 of points (u, v) and (u + 1, v), u even, of
// polarisation p: both in one 16-byte reduction where the grid's alignment
// allows (N is even).
__device__ __forceinline__ void commit_pair(const GridArgs& a, float2* gbase, int u, int v, int p,
                                            float2 s0, float2 s1) {
    const int N = a.N;
    const float4 q = make_float4(s0.x * a.table_inv, s0.y * a.table_inv, s1.x * a.table_inv,
                                 s1.y * a.table_inv);
    const bool n0 = q.x != 0.f || q.y != 0.f, n1 = q.z != 0.f || q.w != 0.f;
    if (u >= N || v >= N || !(n0 || n1)) return;
    const int64_t off = ((int64_t)p * N + v) * N + u;
    const float2 q0 = make_float2(q.x, q.y), q1 = make_float2(q.z, q.w);
    if (a.grid_err) {
        if (n0) commit_compensated(gbase + off, a.grid_err + off, q0);
        if (n1) commit_compensated(gbase + off + 1, a.grid_err + off + 1, q1);
    } else if ((reinterpret_cast<uintptr_t>(gbase) & 15u) == 0) {
        atomicAdd(reinterpret_cast<float4*>(gbase + off), q);
    } else {
        if (n0) atomicAdd(gbase + off, q0);
        if (n1) atomicAdd(gbase + off + 1, q1);
    }
}

// ---- compute warps over pair tables ---------------------------------------------
// Blocks of 16 (u) x 8 (v) points, kernel values in aligned pairs of horizontally
// adjacent points (layout at pair_table_pairs).  List entry: x = pair index of
// the block's column 0, row 0 (modulo 2^32; only columns and rows inside the
// footprint are loaded); y = record row in the batch (bits 0-7), pairs per
// table row less one (8-14), conjugate kernel (15), rows (16-23) and column
// pairs (24-31) that the footprint meets.
constexpr uint32_t kPairConj = 1u << 15;
constexpr int kPairRows = 16, kPairCols = 24;

// Producer: list entries of a record over the pair tables.
struct PairEntries {
    static constexpr int kBlockU = 16, kBlockV = 8;
    uint32_t base, ey;
    int Q, pc0;
    __device__ __forceinline__ PairEntries(const GridArgs& a, const gw_index_rec& rc, int plane, int S,
                                       int r, int ulo, int vlo) {
        Q = (S + 1) / 2;                       // pairs per table row
        // the copy of the slice whose pairs line up with the tile's even
        // columns, and the pair column of the tile's column 0
        const int odd = ulo & 1;
        pc0 = (odd - ulo) / 2;
        const int64_t slice =
            __ldg(a.pair_off + plane) +
            (2 * ((int64_t)(rc.ov + a.beta / 2) * a.beta + (rc.ou + a.beta / 2)) + odd) *
                (int64_t)(S * Q);
        base = (uint32_t)slice + (uint32_t)(pc0 - vlo * Q);
        ey = (uint32_t)r | (uint32_t)(Q - 1) << 8 | ((rc.flags & GW_FLAG_CONJ) ? kPairConj : 0u);
    }
    __device__ __forceinline__ uint2 operator()(int cu, int cv, int j0, int j1) const {
        const int pc = pc0 + kBlockU / 2 * cu;
        const int lo = max(0, -pc), hi = min(kBlockU / 2 - 1, Q - 1 - pc);
        const uint32_t rows = ((2u << j1) - 1u) & ~((1u << j0) - 1u);
        const uint32_t cols = (2u << hi) - (1u << lo);
        return make_uint2(base + (uint32_t)(kBlockV * cv * Q + kBlockU / 2 * cu),
                          ey | rows << kPairRows | cols << kPairCols);
    }
    // first and last pair the entry's loads touch
    __device__ __forceinline__ void span(uint2 e, int cu, int, int j0, int j1, int64_t& lo,
                                         int64_t& hi) const {
        const int pc = pc0 + kBlockU / 2 * cu;
        lo = (int64_t)(uint32_t)(e.x + (uint32_t)(j0 * Q + max(0, -pc)));
        hi = (int64_t)(uint32_t)(e.x + (uint32_t)(j1 * Q + min(kBlockU / 2 - 1, Q - 1 - pc)));
    }
};

// A pair of the FP32 table, zero where `on` is false: one predicated load.  (A
// conditional one became a branch: 4.2 M visibilities x 1, support 31, 2.94 ms, so
// 2.82.  With two polarisations, and in FmaWarp, the conditional loads schedule
// better: the same x 2 3.887 against 3.957 ms (eight runs each, all within 0.005 of
// that) and the 4096^2 batch 8.23 against 8.79.)
__device__ __forceinline__ float4 load_pair(const float4* __restrict__ p, bool on) {
    float4 v;
    asm("{.reg .pred q; setp.ne.u32 q, %5, 0;\n"
        " mov.f32 %0, 0f00000000; mov.f32 %1, 0f00000000;\n"
        " mov.f32 %2, 0f00000000; mov.f32 %3, 0f00000000;\n"
        " @q ld.global.nc.v4.f32 {%0, %1, %2, %3}, [%4];}"
        : "=&f"(v.x), "=&f"(v.y), "=&f"(v.z), "=&f"(v.w)
        : "l"(p), "r"((uint32_t)on));
    return v;
}

// FP32 tables with one or two polarisations.  With so few FMAs an entry the
// gathers bound the kernel (each a quarter-warp's cache lines), and a 16-byte
// load of a pair takes 8 lanes through one 128-byte row: about 7.5 lines for
// 64 points against 11.5 for two 8-byte loads of 8 x 4 points.  4.2 M
// visibilities, 1 polarisation, support 31, 2048^2: 3.65 ms with FmaWarp; here
// 3.30 / 3.23 / 2.98 / 2.90 with 3 / 4 / 5 / 6 entries in flight (2.82 with
// predicated loads).  With more
// polarisations the FMAs share the bound and the 8 x 16 blocks of FmaWarp
// stay ahead (4: 8.2 against 9.2 ms on the 4096^2 batch).
// Lane (g, r) = (lane % 8, lane / 8): points 2 g, 2 g + 1 of rows r and r + 4.
template <int NPOL>
struct PairWarp {
    using VT = float2;                         // staged visibility
    static constexpr int kPol = NPOL, R = NPOL == 1 ? 6 : 5;   // entries in flight
    static constexpr int kBlockU = 16, kBlockV = 8;
    static constexpr int kBatch = kRows - 1;   // rows 0 .. 254, and the zero row 255
    static constexpr uint32_t kZeroRow = kBatch;
    static constexpr int kVisRows = kRows;
    float2 acc[4][NPOL];                       // (row slot, point of the pair), (re, im)
    float4 K[R][2];
    uint32_t ey[R];
    const float4* __restrict__ tab;
    uint32_t g, r;

    __device__ __forceinline__ PairWarp(const GridArgs& a, int, int lane) {
        tab = reinterpret_cast<const float4*>(a.pair_table);
        g = lane & 7;
        r = lane >> 3;
#pragma unroll
        for (int j = 0; j < 4; ++j)
#pragma unroll
            for (int p = 0; p < NPOL; ++p) acc[j][p] = make_float2(0.f, 0.f);
    }
    // kernel values of an entry, zero outside its footprint
    __device__ __forceinline__ void load(int d, const uint2 en) {
        const uint32_t q = ((en.y >> 8) & 0x7fu) + 1u, off = en.x + g + r * q;
        const uint32_t c = 1u << (kPairCols + g);
        const uint32_t m0 = c | 1u << (kPairRows + r), m1 = c | 1u << (kPairRows + 4 + r);
        ey[d] = en.y;
        if constexpr (NPOL == 1) {
            K[d][0] = load_pair(tab + off, (~en.y & m0) == 0);
            K[d][1] = load_pair(tab + (off + 4 * q), (~en.y & m1) == 0);
        } else {
            const float4 z = make_float4(0.f, 0.f, 0.f, 0.f);
            K[d][0] = (en.y & m0) == m0 ? __ldg(tab + off) : z;
            K[d][1] = (en.y & m1) == m1 ? __ldg(tab + (off + 4 * q)) : z;
        }
    }
    __device__ __forceinline__ void fill(const uint2* lst, const VT (*)[NPOL]) {
#pragma unroll
        for (int d = 0; d < R; ++d) load(d, lst[d]);
    }
    // one ring pass: the FMAs of the R entries in the ring, each followed by
    // the loads of the entry R positions later
    __device__ __forceinline__ void pass(const uint2* next, const VT (*vs)[NPOL], const VT (*)[NPOL]) {
#pragma unroll
        for (int d = 0; d < R; ++d) {
            const float2* row = vs[ey[d] & 0xffu];
            const float s = (ey[d] & kPairConj) ? -1.f : 1.f;
            float2 A[NPOL], Bv[NPOL];
#pragma unroll
            for (int p = 0; p < NPOL; ++p) {
                A[p] = row[p];
                Bv[p] = make_float2(-s * A[p].y, s * A[p].x);
            }
#pragma unroll
            for (int j = 0; j < 2; ++j)
#pragma unroll
                for (int i = 0; i < 2; ++i) {
                    const float kr = i ? K[d][j].z : K[d][j].x, ki = i ? K[d][j].w : K[d][j].y;
#pragma unroll
                    for (int p = 0; p < NPOL; ++p) {
                        float2& c = acc[2 * j + i][p];
                        c = __ffma2_rn(make_float2(kr, kr), A[p], c);
                        c = __ffma2_rn(make_float2(ki, ki), Bv[p], c);
                    }
                }
            load(d, next[d]);
        }
    }
    __device__ __forceinline__ void commit(const GridArgs& a, float2* gbase, int u0, int v0, int) {
#pragma unroll
        for (int j = 0; j < 2; ++j)
#pragma unroll
            for (int p = 0; p < NPOL; ++p) {
                commit_pair(a, gbase, u0 + 2 * (int)g, v0 + (int)r + 4 * j, p, acc[2 * j][p],
                            acc[2 * j + 1][p]);
                acc[2 * j][p] = acc[2 * j + 1][p] = make_float2(0.f, 0.f);
            }
    }
    static __device__ __forceinline__ bool copies(const GridArgs& a) {
        return FmaWarp<NPOL, 0, GW_C64>::copies(a);
    }
    static __device__ __forceinline__ void stage(const GridArgs& a, bool copy, VT (&row)[NPOL],
                                                 uint32_t id) {
        FmaWarp<NPOL, 0, GW_C64>::stage(a, copy, row, id);
    }
    using Entries = PairEntries;
};

// ---- compute warps: 16-bit tensor cores -----------------------------------------
// Tables and visibilities of one 16-bit kind: the products of 16-bit values
// are exact in FP32, so a group of 8 records is one m16n8k16 product per
// block row: rows of A the row's 16 points, K index the records' (re, im)
// kernel values as stored, columns of B the components (re, im) of the
// polarisations.  Its FP32 sums are added to the lane's accumulators with
// ordinary (rounded) additions.  The additions inside a product are not rounded
// to nearest one by one: they lose 3e-8 of the sum, always downwards, but replace
// sixteen roundings by one.  Errors against 64 bits on the stored values, here /
// FmaWarp, bfloat16, items of 1,024: 96 k x 4, 256^2, support 7-31 1.33 / 2.10 e-7,
// coherent 0.77 / 0.80 e-7; 29 k x 4, 1024^2, support 7-63 0.98 / 1.86 e-7, coherent 0.84 /
// 1.15 e-7; float16 alike.  Lane (g, t) = (lane / 4, lane % 4) loads
// column pair g of records t and t + 4 and holds polarisation t of points 2 g,
// 2 g + 1; pairs come from the pair tables (layout at pair_table_pairs).
template <int TK>
__device__ __forceinline__ void mma_16(float (&d)[4], const uint32_t (&a)[4],
                                       const uint32_t (&b)[2]) {
    if constexpr (TK == GW_BF16X2)
        asm("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, "
            "{%8,%9}, {%10,%10,%10,%10};"
            : "=f"(d[0]), "=f"(d[1]), "=f"(d[2]), "=f"(d[3])
            : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b[0]), "r"(b[1]), "f"(0.f));
    else
        asm("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, "
            "{%8,%9}, {%10,%10,%10,%10};"
            : "=f"(d[0]), "=f"(d[1]), "=f"(d[2]), "=f"(d[3])
            : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b[0]), "r"(b[1]), "f"(0.f));
}

template <int NPOL, int TK>
struct MmaWarp {
    using VT = uint32_t;                       // staged visibility, as stored
    static constexpr int kPol = NPOL, R = 8;   // records per group, one group in flight
    static constexpr int kBlockU = 16, kBlockV = 8;
    static constexpr int kBatch = kRows - 1;   // rows 0 .. 254, and the zero row 255
    static constexpr uint32_t kZeroRow = kBatch;
    static constexpr int kVisRows = kRows;
    float acc[8][4];                           // block row; point 2 g (re, im), point 2 g + 1
    uint2 K[8][2];
    uint32_t b[2];                             // operand B of the group in flight
    const uint2* __restrict__ tab;
    uint32_t g, t;

    __device__ __forceinline__ MmaWarp(const GridArgs& a, int, int lane) {
        tab = reinterpret_cast<const uint2*>(a.pair_table);
        g = lane >> 2;
        t = lane & 3;
#pragma unroll
        for (int j = 0; j < 8; ++j)
#pragma unroll
            for (int i = 0; i < 4; ++i) acc[j][i] = 0.f;
    }
    // position, row step and row mask of the lane's two records
    struct Cursor {
        uint32_t off[2], q[2], m[2];
    };
    __device__ __forceinline__ Cursor start(const uint2* lst, const VT (*vs)[NPOL]) {
        Cursor c;
#pragma unroll
        for (int k = 0; k < 2; ++k) {
            const uint2 en = lst[4 * k + t];
            c.off[k] = en.x + g;
            c.q[k] = ((en.y >> 8) & 0x7fu) + 1u;
            c.m[k] = (en.y >> (kPairCols + g)) & 1u ? en.y >> kPairRows : 0u;
            // column g of B: component (re, im) g & 1 of polarisation g / 2;
            // (K.re, K.im) multiply (V.re, -s V.im) or (V.im, s V.re), s = -1 for
            // the conjugate kernel
            uint32_t w = 0u;
            if (NPOL == 4 || (int)(g >> 1) < NPOL) {
                w = vs[en.y & 0xffu][g >> 1];
                w = __byte_perm(w, 0, (g & 1) ? 0x1032 : 0x3210) ^
                    ((~g << 31) ^ ((en.y & kPairConj) << 16));
            }
            b[k] = w;
        }
        return c;
    }
    // lanes outside the footprint read a zero pair (a select of the address:
    // 16 predicated loads with zeroed destinations do not fit the registers)
    __device__ __forceinline__ void load(int j, Cursor& c) {
#pragma unroll
        for (int k = 0; k < 2; ++k) {
            K[j][k] = __ldg(tab + (c.m[k] & (1u << j) ? c.off[k] : 0u));
            c.off[k] += c.q[k];
        }
    }
    __device__ __forceinline__ void fill(const uint2* lst, const VT (*vs)[NPOL]) {
        Cursor c = start(lst, vs);
#pragma unroll
        for (int j = 0; j < 8; ++j) load(j, c);
    }
    // one pass: the products of the group in flight, each row followed by its
    // loads for the next group
    __device__ __forceinline__ void pass(const uint2* next, const VT (*)[NPOL], const VT (*nvs)[NPOL]) {
        const uint32_t bc[2] = {b[0], b[1]};
        Cursor c = start(next, nvs);
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            const uint32_t a[4] = {K[j][0].x, K[j][0].y, K[j][1].x, K[j][1].y};
            float d[4];
            mma_16<TK>(d, a, bc);
#pragma unroll
            for (int i = 0; i < 4; i += 2) {
                const float2 q = __fadd2_rn(make_float2(acc[j][i], acc[j][i + 1]),
                                            make_float2(d[i], d[i + 1]));
                acc[j][i] = q.x;
                acc[j][i + 1] = q.y;
            }
            load(j, c);
        }
    }
    // Commits the block's accumulators (polarisations beyond NPOL hold zeros,
    // which are not committed).
    __device__ __forceinline__ void commit(const GridArgs& a, float2* gbase, int u0, int v0, int) {
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            commit_pair(a, gbase, u0 + 2 * (int)g, v0 + j, (int)t, make_float2(acc[j][0], acc[j][1]),
                        make_float2(acc[j][2], acc[j][3]));
#pragma unroll
            for (int i = 0; i < 4; ++i) acc[j][i] = 0.f;
        }
    }
    static __device__ __forceinline__ bool copies(const GridArgs& a) {
        return NPOL % 2 == 1 || reinterpret_cast<uintptr_t>(a.vis) % (4 * NPOL) == 0;
    }
    // Producer: visibility `id` into a staged row, with the widest copies its
    // alignment allows.
    static __device__ __forceinline__ void stage(const GridArgs& a, bool copy, VT (&row)[NPOL],
                                                 uint32_t id) {
        const uint32_t* src = reinterpret_cast<const uint32_t*>(a.vis) + (int64_t)id * NPOL;
        if (copy && NPOL == 4) {
            cp_async16(&row[0], src);
        } else if (copy && NPOL == 2) {
            cp_async8(&row[0], src);
        } else if (copy) {
#pragma unroll
            for (int p = 0; p < NPOL; ++p) cp_async4(&row[p], src + p);
        } else {
#pragma unroll
            for (int p = 0; p < NPOL; ++p) row[p] = __ldg(src + p);
        }
    }
    using Entries = PairEntries;
};

// PAIRS: the compute warps that read the pair tables.
template <int NPOL, int SP, int TK, bool PAIRS>
struct PickWarp { using W = FmaWarp<NPOL, SP, TK>; };
template <int NPOL, int SP, int TK>
struct PickWarp<NPOL, SP, TK, true> {
    using W = std::conditional_t<TK == GW_C64, PairWarp<NPOL>, MmaWarp<NPOL, TK>>;
};

template <class W, int B>
struct Smem {
    typename W::VT v[B][W::kVisRows][W::kPol];   // staged visibilities; row kZeroRow = 0
    // per warp: list entries, padded to a multiple of R, then R null entries
    uint2 list[B][kComputeWarps][kRows + 2 * W::R];
    int cnt[B][kComputeWarps];             // entries, padded to a multiple of R
    int tile[B];                           // tile of the batch; -1 = end of work
    int last[B];                           // batch ends its work item
    Item item;                             // producers: the current work item
    int done;                              // producers: no work item left
    unsigned long long full[B], empty[B];  // mbarriers
};

template <int NPOL, int SP, int TK, bool PAIRS, int B>
__global__ void __launch_bounds__(kThreads, 1) k_grid(GridArgs a) {
    using W = typename PickWarp<NPOL, SP, TK, PAIRS>::W;
    using VT = typename W::VT;
    constexpr int R = W::R, kBatch = W::kBatch, kBlockU = W::kBlockU, kBlockV = W::kBlockV;
    constexpr int kBlocksU = kGridTileU / kBlockU;
    constexpr uint32_t kZeroRow = W::kZeroRow;
    extern __shared__ __align__(128) unsigned char smem_raw[];
    Smem<W, B>& sm = *reinterpret_cast<Smem<W, B>*>(smem_raw);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int side = a.ntiles_u;

    // one-time set-up: barriers, the zero visibility row
    if (threadIdx.x == 0) {
        for (int b = 0; b < B; ++b) {
            mbar_init(&sm.full[b], kProducerThreads);
            mbar_init(&sm.empty[b], kComputeWarps * 32);
        }
    }
    for (int t = threadIdx.x; t < B * NPOL; t += kThreads)
        sm.v[t / NPOL][kZeroRow][t % NPOL] = VT{};
    __syncthreads();

    if (warp >= kComputeWarps) {
#ifdef GW_GRID_SETMAXNREG
        asm volatile("setmaxnreg.dec.sync.aligned.u32 40;" ::: "memory");
#endif
        // ----------------------------------------------------------- producers
        const int pt = threadIdx.x - kComputeWarps * 32;   // 0 .. kProducerThreads - 1
        const int pw = pt >> 5;
        // items [i0, *item_count): a band of tile rows, or all of them
        const uint32_t i0 = a.item_first ? *a.item_first : 0u;
        const uint32_t nitems = *a.item_count - i0;
        const bool copy_vis = W::copies(a);
        uint32_t nbatch = 0;
        for (;;) {
            int b = 0, nb_total = 1;
            bool done = false;
            Item item{};
            for (;;) {   // batches of the current work item
                const int buf = nbatch % B;
                if (nbatch >= (uint32_t)B &&
                    !mbar_wait(&sm.empty[buf], ((nbatch / B) - 1) & 1)) {
                    if (lane == 0) atomicOr(a.queue + 1, 1u);
                    return;
                }
                if (pw == 0) {
                    if (b == 0 && lane == 0) {
                        const uint32_t it = atomicAdd(a.queue, 1u);
                        sm.done = it >= nitems;
                        if (it < nitems) sm.item = a.items[i0 + it];
                    }
                    if (lane < kComputeWarps) sm.cnt[buf][lane] = 0;
                }
                producer_sync();
                if (b == 0) {
                    done = sm.done != 0;
                    if (!done) item = sm.item;
                    nb_total = done ? 1 : (item.len + kBatch - 1) / kBatch;
                }
                if (!done) {
                    // with w-layers (w-stacking) a tile id is layer * layer_tiles + tile
                    const int ltile = a.layer_tiles ? item.tile % a.layer_tiles : item.tile;
                    const int tu0 = (ltile % side) * kGridTileU;
                    const int tv0 = (ltile / side) * kGridTileV;
                    const int b0 = b * kBatch;
                    const int nb = min(kBatch, item.len - b0);
                    // all ids, then all index records of this thread's rows in flight
                    uint32_t ids[kPerLane];
                    gw_index_rec rcs[kPerLane];
#pragma unroll
                    for (int k = 0; k < kPerLane; ++k) {
                        const int r = k * kProducerThreads + pt;
                        ids[k] = r < nb ? __ldg(a.entries + item.start + b0 + r) : 0u;
                    }
#pragma unroll
                    for (int k = 0; k < kPerLane; ++k) {
                        const int r = k * kProducerThreads + pt;
                        if (r < nb) rcs[k] = load_rec(a.rec, ids[k]);
                    }
#pragma unroll
                    for (int k = 0; k < kPerLane; ++k) {
                        const int r = k * kProducerThreads + pt;
                        if (r >= nb) break;
                        const uint32_t id = ids[k];
                        const gw_index_rec rc = rcs[k];
                        W::stage(a, copy_vis, sm.v[buf][r], id);
                        // w-stacking records carry their layer in `plane`; the
                        // kernel is the plan's single (w = 0) plane
                        const int plane = (a.layer_tiles && !a.plane_groups) ? 0 : rc.plane;
                        const int S = __ldg(a.support + plane), h = S >> 1;
                        // footprint relative to the tile: [ulo, uhi] x [vlo, vhi]
                        const int ulo = rc.ku - h - tu0, uhi = rc.ku + h - tu0;
                        const int vlo = rc.kv - h - tv0, vhi = rc.kv + h - tv0;
                        const typename W::Entries entry(a, rc, plane, S, r, ulo, vlo);
                        const int cu0 = max(0, ulo) / kBlockU, cu1 = min(kGridTileU - 1, uhi) / kBlockU;
                        const int cv0 = max(0, vlo) / kBlockV, cv1 = min(kGridTileV - 1, vhi) / kBlockV;
                        for (int cv = cv0; cv <= cv1; ++cv) {
                            const int j0 = max(0, vlo - kBlockV * cv);
                            const int j1 = min(kBlockV - 1, vhi - kBlockV * cv);
                            for (int cu = cu0; cu <= cu1; ++cu) {
                                const int w = cv * kBlocksU + cu;
                                const uint2 e = entry(cu, cv, j0, j1);
#ifdef GW_DEBUG_BOUNDS
                                int64_t lo, hi;
                                entry.span(e, cu, cv, j0, j1, lo, hi);
                                const int64_t n = PAIRS ? a.pair_count : a.ptable_elems;
                                if (!gw_in_bounds(n == 0 || (lo >= 0 && lo <= hi && hi < n), a.queue + 1))
                                    continue;
#endif
                                const int pos = atomicAdd(&sm.cnt[buf][w], 1);
                                if (gw_in_bounds(pos < kBatch, a.queue + 1)) sm.list[buf][w][pos] = e;
                            }
                        }
                    }
                    if (copy_vis) cp_async_wait_all();
                }
                producer_sync();   // all rows staged, all list appends done
                if (pw == 0) {
                    // pad every warp's list to a multiple of R and put R null
                    // entries (no slots loaded, the zero visibility row) after it
                    if (lane < kComputeWarps) {
                        const int w = lane;
                        const int nf = sm.cnt[buf][w];
                        const int nfp = (nf + R - 1) / R * R;
                        const uint2 z = make_uint2(0u, kZeroRow);
                        for (int k = nf; k < nfp + R; ++k) sm.list[buf][w][k] = z;
                        sm.cnt[buf][w] = nfp;
                    }
                    if (lane == 0) {
                        sm.tile[buf] = done ? -1 : item.tile;
                        sm.last[buf] = done ? 1 : (b == nb_total - 1);
                    }
                    __syncwarp();
                }
                mbar_arrive(&sm.full[buf]);  // batch ready (every producer thread)
                ++nbatch;
                if (++b == nb_total) break;
            }
            if (done) break;
        }
        return;
    }

    // ---------------------------------------------------------------- consumers
#ifdef GW_GRID_SETMAXNREG
    asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(GW_GRID_SETMAXNREG) : "memory");
#endif
    const int bu = (warp % kBlocksU) * kBlockU, bv = (warp / kBlocksU) * kBlockV;
    W cw(a, warp, lane);

    // The ring runs across batches: the last pass over a batch's list loads
    // the first R entries of the next batch, so no batch starts with an empty
    // ring.  Lists are padded to a multiple of R and followed by R null
    // entries (the end-of-work batch has only those).
    if (!mbar_wait(&sm.full[0], 0)) {
        if (lane == 0) atomicOr(a.queue + 1, 1u);
        return;
    }
    cw.fill(sm.list[0][warp], sm.v[0]);
    uint32_t nbatch = 0;
    for (;;) {
        const int buf = nbatch % B;
        const int tile = sm.tile[buf];
        if (tile < 0) break;
        const int last = sm.last[buf];
        const int n = sm.cnt[buf][warp];
        const uint2* lst = sm.list[buf][warp];
        const int nbuf = (nbatch + 1) % B;
        const uint2* nlst = sm.list[nbuf][warp];
        for (int i = 0;; i += R) {
            const bool tail = i + R >= n;
            if (tail && !mbar_wait(&sm.full[nbuf], ((nbatch + 1) / B) & 1)) {
                if (lane == 0) atomicOr(a.queue + 1, 1u);
                return;
            }
            if (n == 0) {   // nothing of this batch for this warp
                cw.fill(nlst, sm.v[nbuf]);
                break;
            }
            cw.pass(tail ? nlst : lst + i + R, sm.v[buf], sm.v[tail ? nbuf : buf]);
            if (tail) break;
        }
        mbar_arrive(&sm.empty[buf]);  // buffer free (every lane, after its reads)
        ++nbatch;
        if (last) {
            // commit the tile's accumulators of this work item
            const int ltile = a.layer_tiles ? tile % a.layer_tiles : tile;
            float2* const gbase = a.grid + (a.layer_tiles ? (int64_t)(tile / a.layer_tiles) *
                                                                 a.layer_stride : 0);
            cw.commit(a, gbase, (ltile % a.ntiles_u) * kGridTileU + bu,
                      (ltile / a.ntiles_u) * kGridTileV + bv, lane);
        }
    }
}

// GW_GRID_BUFS staging buffers of 256 records.
#ifndef GW_GRID_BUFS
#define GW_GRID_BUFS 4
#endif
template <int NPOL, int SP, int TK, bool PAIRS>
void launch_sp(const GridArgs& a, int num_sms, cudaStream_t s) {
    constexpr int B = GW_GRID_BUFS;
    const size_t smem = sizeof(Smem<typename PickWarp<NPOL, SP, TK, PAIRS>::W, B>);
    cudaFuncSetAttribute(k_grid<NPOL, SP, TK, PAIRS, B>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                         (int)smem);
    int per_sm = 0;
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_grid<NPOL, SP, TK, PAIRS, B>, kThreads,
                                                  smem);
    if (per_sm < 1) per_sm = 1;
    k_grid<NPOL, SP, TK, PAIRS, B><<<num_sms * per_sm, kThreads, smem, s>>>(a);
    note_launch();
}

template <int NPOL, int TK>
void launch_t(const GridArgs& a, int num_sms, cudaStream_t s) {
    if constexpr (TK == GW_C64 && NPOL <= kPairPolMax) {
        launch_sp<NPOL, 0, TK, true>(a, num_sms, s);       // such plans have pair tables only
    } else {
        if constexpr ((TK == GW_BF16X2 || TK == GW_F16X2) && NPOL >= kMmaPolMin) {
            if (a.pair_table && a.vis_kind == TK && !a.weight) {
                launch_sp<NPOL, 0, TK, true>(a, num_sms, s);
                return;
            }
        }
        switch (a.pad_stride) {
#if GW_GRID_LANES_U == 16
            case 32: launch_sp<NPOL, 32, TK, false>(a, num_sms, s); break;
            case 48: launch_sp<NPOL, 48, TK, false>(a, num_sms, s); break;
            case 64: launch_sp<NPOL, 64, TK, false>(a, num_sms, s); break;
            case 96: launch_sp<NPOL, 96, TK, false>(a, num_sms, s); break;
            case 160: launch_sp<NPOL, 160, TK, false>(a, num_sms, s); break;
            default: launch_sp<NPOL, 288, TK, false>(a, num_sms, s); break;
#else
            case 24: launch_sp<NPOL, 24, TK, false>(a, num_sms, s); break;
            case 32: launch_sp<NPOL, 32, TK, false>(a, num_sms, s); break;
            case 48: launch_sp<NPOL, 48, TK, false>(a, num_sms, s); break;
            case 80: launch_sp<NPOL, 80, TK, false>(a, num_sms, s); break;
            case 144: launch_sp<NPOL, 144, TK, false>(a, num_sms, s); break;
            default: launch_sp<NPOL, 272, TK, false>(a, num_sms, s); break;
#endif
        }
    }
}

}  // namespace

// All gridder instantiations for one table kind.
template <int TK>
void launch_grid_kind(const GridArgs& a, int num_sms, cudaStream_t s) {
    switch (a.npol) {
        case 1: launch_t<1, TK>(a, num_sms, s); break;
        case 2: launch_t<2, TK>(a, num_sms, s); break;
        case 3: launch_t<3, TK>(a, num_sms, s); break;
        default: launch_t<4, TK>(a, num_sms, s); break;
    }
}


}  // namespace gw
