// rows_kernel.cuh -- the SpMM task kernel, Y = A X for one CSR orientation.
//
// Section 3.4 / Algorithm 1 of the paper: a nonzero a_ij scales the whole
// dense row X[j, :] into output row i, the row operation is vectorised (AVX
// in the paper, 16-byte lane loads here), and each output row has a single
// owner.
//
// Persistent warps walk the task list (plan.cpp), claiming their next tasks
// from an atomic counter (one task at a time for wide X rows, a few for narrow
// ones; FwdArgs::ctl), or, without a counter, with a stride of the grid's
// warp count.  Each warp stages a task's column indices, values and row
// pointers into shared memory with bulk asynchronous copies (cp.async.bulk,
// completion on an mbarrier) one task ahead, so the copy of task i+1 overlaps
// the gathers of task i -- the GPU form of the paper's asynchronous tile-row
// reads (Algorithm 1: read the tile rows asynchronously, multiply once they
// have arrived).  Every wait on a copy is bounded; on timeout the warp sets a
// status word, waits (bounded) for its other copy and exits.
//
// A warp is cut into G = 32 / LANES lane groups; LANES lanes cover one X row
// (each lane VEC consecutive elements, CH chunks of them).
//   short-row task: group g owns rows g, g+G, ... of the run and sums each
//                   row's nonzeros in order (with one lane per X row, k = 1
//                   takes the flat path and rows of up to 8 bytes the
//                   merge-based path; the MG instantiations cut the run
//                   into equal pieces per lane group instead: all three
//                   are described at their branches);
//   long row / hub segment: group g takes nonzeros g, g+G, g+2G, ...; the
//                   groups' partial sums are added by a fixed xor-shuffle
//                   tree; a segment writes its sum to a partial slot.
// All summation orders are fixed, so repeated calls give identical results.
#pragma once

#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include <mutex>
#include <type_traits>

#include "combine.cuh"
#include "internal.h"

namespace spmm {

// ------------------------------------------------------------ PTX helpers --
__device__ __forceinline__ uint32_t smem_u32(const void* p) {
    return (uint32_t)__cvta_generic_to_shared(p);
}
__device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}
__device__ __forceinline__ void fence_mbar_init() {
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}
__device__ __forceinline__ void fence_proxy_async() {
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}
__device__ __forceinline__ void mbar_arrive_expect_tx(uint64_t* bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes)
                 : "memory");
}
// 1-D bulk copy global -> shared; both addresses 16-byte aligned, bytes % 16
// == 0.  `policy` is an L2 cache policy (the streamed matrix is marked
// evict-first so it does not push the gathered X rows out of L2).
__device__ __forceinline__ void bulk_g2s(void* dst, const void* src, uint32_t bytes, uint64_t* bar,
                                         uint64_t policy) {
    asm volatile(
        "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint [%0], [%1], %2, [%3], "
        "%4;" ::"r"(smem_u32(dst)),
        "l"(src), "r"(bytes), "r"(smem_u32(bar)), "l"(policy)
        : "memory");
}
__device__ __forceinline__ uint64_t policy_evict_first() {
    uint64_t p;
    asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(p));
    return p;
}
__device__ __forceinline__ uint64_t policy_evict_last() {
    uint64_t p;
    asm volatile("createpolicy.fractional.L2::evict_last.b64 %0, 1.0;" : "=l"(p));
    return p;
}
__device__ __forceinline__ uint64_t policy_evict_normal() {
    uint64_t p;
    asm volatile("createpolicy.fractional.L2::evict_normal.b64 %0, 1.0;" : "=l"(p));
    return p;
}
// read-only global loads with an L2 cache policy
__device__ __forceinline__ float4 ldg_f4(const float* p, uint64_t pol) {
    float4 v;
    asm volatile("ld.global.nc.L2::cache_hint.v4.f32 {%0, %1, %2, %3}, [%4], %5;"
                 : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w)
                 : "l"(p), "l"(pol));
    return v;
}
__device__ __forceinline__ float2 ldg_f2(const float* p, uint64_t pol) {
    float2 v;
    asm volatile("ld.global.nc.L2::cache_hint.v2.f32 {%0, %1}, [%2], %3;" : "=f"(v.x), "=f"(v.y) : "l"(p), "l"(pol));
    return v;
}
__device__ __forceinline__ float ldg_f1(const float* p, uint64_t pol) {
    float v;
    asm volatile("ld.global.nc.L2::cache_hint.f32 %0, [%1], %2;" : "=f"(v) : "l"(p), "l"(pol));
    return v;
}
__device__ __forceinline__ uint4 ldg_u4(const void* p, uint64_t pol) {
    uint4 v;
    asm volatile("ld.global.nc.L2::cache_hint.v4.u32 {%0, %1, %2, %3}, [%4], %5;"
                 : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
                 : "l"(p), "l"(pol));
    return v;
}
__device__ __forceinline__ uint2 ldg_u2(const void* p, uint64_t pol) {
    uint2 v;
    asm volatile("ld.global.nc.L2::cache_hint.v2.u32 {%0, %1}, [%2], %3;" : "=r"(v.x), "=r"(v.y) : "l"(p), "l"(pol));
    return v;
}
__device__ __forceinline__ uint32_t ldg_u1(const void* p, uint64_t pol) {
    uint32_t v;
    asm volatile("ld.global.nc.L2::cache_hint.u32 %0, [%1], %2;" : "=r"(v) : "l"(p), "l"(pol));
    return v;
}
__device__ __forceinline__ uint32_t ldg_u16(const void* p, uint64_t pol) {
    unsigned short v;
    asm volatile("ld.global.nc.L2::cache_hint.u16 %0, [%1], %2;" : "=h"(v) : "l"(p), "l"(pol));
    return v;
}
__device__ __forceinline__ bool mbar_try_wait(uint64_t* bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}"
        : "=r"(ok)
        : "r"(smem_u32(bar)), "r"(parity)
        : "memory");
    return ok != 0;
}
__device__ __forceinline__ uint64_t global_timer_ns() {
    uint64_t t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}
// Wait for phase `parity` of `bar`; false if it did not complete within limit_ns.
__device__ __forceinline__ bool mbar_wait_bounded(uint64_t* bar, uint32_t parity, uint64_t limit_ns) {
    if (mbar_try_wait(bar, parity)) return true;
    const uint64_t t0 = global_timer_ns();
    for (;;) {
        for (int i = 0; i < 32; ++i)
            if (mbar_try_wait(bar, parity)) return true;
        if (global_timer_ns() - t0 > limit_ns) return false;
    }
}

// ------------------------------------------------------- element loading --
template <typename XT>
__device__ __forceinline__ float bits_to_f32(uint32_t b);
template <>
__device__ __forceinline__ float bits_to_f32<__nv_bfloat16>(uint32_t b) {
    return __uint_as_float(b << 16);
}
template <>
__device__ __forceinline__ float bits_to_f32<__half>(uint32_t b) {
    return __half2float(__ushort_as_half((unsigned short)b));
}

// VEC consecutive elements of X held as loaded (16-bit types stay packed two
// per 32-bit word until they are used, which halves the registers that hold
// loads in flight).  p is aligned to VEC * sizeof(XT).
template <typename XT, int VEC>
struct XVec {
    static_assert(sizeof(XT) == 2, "16-bit element path");
    static constexpr int kWords = (VEC + 1) / 2;
    uint32_t w[kWords];
    __device__ __forceinline__ void load(const XT* p, uint64_t pol) {
        if constexpr (VEC == 8) {
            uint4 v = ldg_u4(p, pol);
            w[0] = v.x; w[1] = v.y; w[2] = v.z; w[3] = v.w;
        } else if constexpr (VEC == 4) {
            uint2 v = ldg_u2(p, pol);
            w[0] = v.x; w[1] = v.y;
        } else if constexpr (VEC == 2) {
            w[0] = ldg_u1(p, pol);
        } else {
            w[0] = ldg_u16(p, pol);
        }
    }
    __device__ __forceinline__ float get(int i) const {
        return bits_to_f32<XT>((i & 1) ? (w[i >> 1] >> 16) : (w[i >> 1] & 0xffffu));
    }
    // the same elements from shared memory (VEC <= 2: rows of at most 4 bytes)
    __device__ __forceinline__ void load_sh(const XT* p) {
        static_assert(VEC <= 2, "shared-memory rows of at most 4 bytes");
        if constexpr (VEC == 2) w[0] = *reinterpret_cast<const uint32_t*>(p);
        else w[0] = *reinterpret_cast<const unsigned short*>(p);
    }
};

template <int VEC>
struct XVec<float, VEC> {
    float f[VEC];
    __device__ __forceinline__ void load(const float* p, uint64_t pol) {
        if constexpr (VEC == 4) {
            float4 v = ldg_f4(p, pol);
            f[0] = v.x; f[1] = v.y; f[2] = v.z; f[3] = v.w;
        } else if constexpr (VEC == 2) {
            float2 v = ldg_f2(p, pol);
            f[0] = v.x; f[1] = v.y;
        } else {
            f[0] = ldg_f1(p, pol);
        }
    }
    __device__ __forceinline__ float get(int i) const { return f[i]; }
    __device__ __forceinline__ void load_sh(const float* p) {
        static_assert(VEC == 1, "shared-memory rows of at most 4 bytes");
        f[0] = *p;
    }
};

// Store VEC floats to an address aligned to min(VEC, 4) * 4 bytes.
template <int VEC>
__device__ __forceinline__ void store_y(float* p, const float (&v)[VEC]) {
    if constexpr (VEC >= 4) {
#pragma unroll
        for (int i = 0; i < VEC; i += 4)
            __stcs(reinterpret_cast<float4*>(p + i), make_float4(v[i], v[i + 1], v[i + 2], v[i + 3]));
    } else if constexpr (VEC == 2) {
        __stcs(reinterpret_cast<float2*>(p), make_float2(v[0], v[1]));
    } else {
        __stcs(p, v[0]);
    }
}

// value of staged entry i (shared memory, raw bytes of the stored type)
template <int VMODE>
__device__ __forceinline__ float staged_val(const unsigned char* v, int i) {
    if constexpr (VMODE == 1) return reinterpret_cast<const float*>(v)[i];
    if constexpr (VMODE == 2) return __uint_as_float((uint32_t)reinterpret_cast<const unsigned short*>(v)[i] << 16);
    if constexpr (VMODE == 3) return __half2float(__ushort_as_half(reinterpret_cast<const unsigned short*>(v)[i]));
    return 1.0f;
}

template <int VMODE>
struct Layout {
    static constexpr int kValBytes = VMODE == 0 ? 0 : (VMODE == 1 ? 4 : 2);
    static constexpr int kColOff = 0;
    static constexpr int kValOff = kColBufInts * 4;
    static constexpr int kRpOff = kValOff + (VMODE ? kValBufBytes : 0);
    static constexpr int kBuf = kRpOff + kRpBufLongs * 8;       // bytes per staging buffer
    static constexpr int kWarp = 2 * kBuf + 16;                 // two buffers + two mbarriers
    static constexpr int kBlock = kWarpsPerBlock * kWarp;
    static_assert(kBuf % 16 == 0 && kWarp % 16 == 0, "16-byte aligned staging buffers");
};

struct Staged {
    const int32_t* col;         // col[i] = column of nonzero e0 + i
    const unsigned char* val;   // raw value bytes, entry i = nonzero e0 + i
    const int64_t* rpw;         // staged row_ptr[r0 ..] (short-row tasks)
    int e0;                     // low word of the task's first nonzero
    // start of row j among the task's nonzeros (the low words' difference)
    __device__ __forceinline__ int rp(int j) const {
        return entries_between(e0, (int)reinterpret_cast<const uint32_t*>(rpw)[2 * j]);
    }
};

__device__ __forceinline__ int64_t desc_e0(int z, int w) {
    return ((int64_t)(uint32_t)z) | ((int64_t)w << 32);
}

// Issue the bulk copies of one task into staging buffer `buf` (lane 0 only).
// Windows are widened to 16-byte boundaries; the arrays are padded on the
// device so the widened end stays inside the allocation.
template <int VMODE>
__device__ __forceinline__ void issue_task(const FwdArgs& a, const int4 d0, int64_t e1, unsigned char* buf,
                                           uint64_t* bar) {
    using Lay = Layout<VMODE>;
    const uint64_t pol = policy_evict_first();
    const int64_t e0 = desc_e0(d0.z, d0.w);
    const int64_t cs = e0 & ~(int64_t)3, ce = (e1 + 3) & ~(int64_t)3;
    const uint32_t cbytes = (uint32_t)((ce - cs) * 4);
    uint32_t vbytes = 0, rbytes = 0;
    int64_t vs = 0, rs = 0;
    if constexpr (VMODE != 0) {
        constexpr int epb = 16 / Lay::kValBytes;
        vs = e0 & ~(int64_t)(epb - 1);
        const int64_t ve = (e1 + epb - 1) & ~(int64_t)(epb - 1);
        vbytes = (uint32_t)((ve - vs) * Lay::kValBytes);
    }
    if (d0.y > 0) {
        rs = (int64_t)d0.x & ~(int64_t)1;
        const int64_t re = ((int64_t)d0.x + d0.y + 2) & ~(int64_t)1;
        rbytes = (uint32_t)((re - rs) * 8);
    }
    mbar_arrive_expect_tx(bar, cbytes + vbytes + rbytes);
    if (cbytes) bulk_g2s(buf + Lay::kColOff, a.col_idx + cs, cbytes, bar, pol);
    if constexpr (VMODE != 0)
        if (vbytes)
            bulk_g2s(buf + Lay::kValOff, reinterpret_cast<const unsigned char*>(a.val) + vs * Lay::kValBytes, vbytes,
                     bar, pol);
    if (rbytes) bulk_g2s(buf + Lay::kRpOff, a.row_ptr + rs, rbytes, bar, pol);
}

#ifndef SPMM_UNROLL_BYTES
#define SPMM_UNROLL_BYTES 64      // X bytes in flight per lane
#endif
#ifndef SPMM_K1_FLAT
#define SPMM_K1_FLAT 1            // k = 1 short-row runs: flat gather through shared memory
#endif
#ifndef SPMM_FLAT_UF
#define SPMM_FLAT_UF 8            // k = 1 flat path: nonzeros gathered per lane per round
#endif
#ifndef SPMM_MERGE
#define SPMM_MERGE 1              // one lane per X row: merge-based short-row runs
#endif

#ifndef SPMM_MIN_BLOCKS
#define SPMM_MIN_BLOCKS 3         // resident blocks per SM the register budget targets (80 registers)
#endif

// Resident blocks per SM that the register budget of an instantiation targets.
// Three blocks (80 registers a thread) measured faster than four (64) for
// every path but the pattern group merge over rows on 8 or more lanes
// (R-MAT scale 24, FP32: k = 1 1.10 -> 0.93 ms, k = 8 2.23 -> 1.92, 30
// PageRank iterations 35.9 -> 31.6 ms; k = 32 4.20 -> 4.34, k = 64
// 7.59 -> 7.91), which keeps four in its own variant (MG == 2).
// Two blocks, with twice the gathers in flight (up to 128 registers): where the
// staged values double the staging buffers, three blocks take 226 KB of
// shared memory and leave L1 next to nothing (weighted R-MAT, 4 M vertices,
// FP32, ms with three -> two: k = 1 0.395 -> 0.252, k = 2 0.424 -> 0.291, k = 8
// 0.684 -> 0.440; BF16 X, k = 16 0.771 -> 0.622; 2 M, k = 64 1.081 -> 0.834), and
// for rows on two chunks of single elements, whose walk keeps 16 rows' loads
// in flight (MG == 4; with three blocks it spills).  Pattern rows on one chunk lose (k = 8, 8 M vertices 0.90 ->
// 1.03 ms, k = 32, 4 M 1.03 -> 1.19).  The weighted group merge comes in both
// forms (MG == 1, MG == 3): lanes of 16 bytes run faster with three blocks while X
// fits L2 (k = 16, 37 MB of X: 0.152 against 0.162 ms) and with two beyond
// (134 MB: 0.836 against 0.569), narrower lanes always with two (k = 4, 67 MB
// 0.510 against 0.433).
template <int VMODE, int MG>
constexpr bool two_blocks() {
    return (VMODE != 0 && MG == 0) || MG == 3 || MG == 4;
}
template <int VMODE, int MG>
constexpr int min_blocks() {
    return (MG == 2 && VMODE == 0) ? 4 : two_blocks<VMODE, MG>() ? 2 : SPMM_MIN_BLOCKS;
}

// *p counted up, wrapping to zero after `last`; everything before it is visible
// to whoever sees the new count and then fences.
__device__ __forceinline__ unsigned int atom_inc_release(unsigned int* p, unsigned int last) {
    unsigned int old;
    asm volatile("atom.inc.release.gpu.global.u32 %0, [%1], %2;" : "=r"(old) : "l"(p), "r"(last) : "memory");
    return old;
}

// A segment of a split row has its partial in a.partials: returns the row's
// split if this was its last segment to arrive, -1 otherwise.  The arrival is a
// release, not a full fence, which would empty L1 as well.
__device__ __forceinline__ int segment_done(const FwdArgs& a, int slot, int lane) {
    if (!a.seg_done || (int64_t)slot >= a.n_slots) return -1;
    const int2 seg = a.slot_seg[slot];     // {split, segments of its row}
    __syncwarp();                          // the lanes' parts of the partial, before the arrival
    unsigned int before = 0;
    if (lane == 0) before = atom_inc_release(a.seg_done + seg.x, (unsigned int)seg.y - 1u);   // zero at the last
    return (int)__shfl_sync(0xffffffffu, before, 0) + 1 == seg.y ? seg.x : -1;
}

// ONE: one lane per X row (k == VEC, CH == 1); the lane geometry is then a
// compile-time constant and short-row runs take the flat (k = 1) or, for X
// rows of up to 8 bytes, the merge-based path.  MG != 0: several lanes per X
// row (CH == 1) and short-row runs merge-based over lane groups, with 3
// blocks per SM and 4 nonzeros in flight per group (MG == 1), 4 blocks and 2 in
// flight (MG == 2) or 2 blocks and 8 in flight (MG == 3).  MG == 4: a whole warp
// per X row of two chunks (odd k above 32), which takes a task's nonzeros as one
// stream, 8 + 8 rows in flight across the ends of the task's rows: the row walk
// has one row's loads in flight, and half of R-MAT's rows have fewer than four
// (FP16 k = 33, 700 K vertices 0.445 -> 0.378 ms, FP32 k = 33, 1 M 0.731 ->
// 0.551).  Rows on one chunk gain nothing (FP32 k = 31, 512 K 0.201 -> 0.210),
// nor does k = 64 on 32 lanes of two elements (2 M 0.795 -> 0.850).
// Warps per block: kWarpsPerBlock, or kHotWarps in one block per SM for the
// instantiations that keep the hot rows of X in shared memory (HOT).
template <bool HOT>
constexpr int warps_per_block() {
    return HOT ? kHotWarps : kWarpsPerBlock;
}

// HOT: one lane per X row of 4 bytes; a negative column index c names row ~c
// of the hot rows of X, which the block gathers into shared memory (after its
// warps' staging buffers) while its first tasks arrive, so those gathers leave
// the L1-to-L2 request path alone (hot.cu).
// Launches whose last warp resets the task counter: those of a few microseconds,
// where a memset before each would cost 3 us (k = 1, 512 K vertices 40.9 ->
// 37.4 us).  In the other instantiations the few instructions at the end
// change the compiled task loop for the worse (FP16 k = 33, 700 K vertices 443 ->
// 560 us), so their launches clear the counter first.
template <bool ONE, bool HOT, bool SEG>
constexpr bool self_reset() {
    return ONE || HOT || SEG;
}

// SEG: the warp that finishes a split row's last segment adds the row's partials
// (FwdArgs::seg_done); a variant of its own, since the other launches lose more
// to the registers this takes than the second launch costs them.
// MULTI: the tasks of several matrices (MultiArgs M, spmm_apply_batched),
// numbered one after the other; every task takes the matrix, X, Y, k and
// lane geometry of its own entry.  ga holds the launch-wide fields (task
// count, counter, status, wait bound).
template <typename XT, int VMODE, int VEC, int CH, bool COMP, bool ONE, int MG, bool HOT, bool MULTI, bool SEG>
__device__ __forceinline__ void rows_run(const FwdArgs& ga, const MultiArgs* M) {
    static_assert(!MULTI || (!ONE && MG == 0 && !HOT), "batched launches use the generic row walk");
    static_assert(!ONE || CH == 1, "one lane per row needs CH == 1");
    static_assert(MG == 0 || (!ONE && CH == (MG == 4 ? 2 : 1)), "merge over lane groups: several lanes, one chunk");
    static_assert(!HOT || (ONE && MG == 0 && VEC * sizeof(XT) <= 4), "hot rows in shared memory: <= 4-byte rows");
    constexpr int WPB = warps_per_block<HOT>();
    constexpr bool kFlat = ONE && VEC == 1 && SPMM_K1_FLAT;
    // merge-based runs pay off for X rows of up to 8 bytes; for 16-byte rows
    // (mostly gathered from DRAM) the row-per-lane walk measured faster
    constexpr bool kMerge = ONE && !kFlat && SPMM_MERGE && VEC * sizeof(XT) <= 8;
    // the same over lane groups, for rows that need several lanes (MG)
    constexpr bool kMergeG = MG != 0 && MG != 4;
    // a whole warp per X row: the run's nonzeros one after the other
    constexpr bool kWholeWarp = MG == 4;
    using Lay = Layout<VMODE>;
    // nonzeros in flight per lane group
    constexpr int kBytes = VEC * CH * (int)sizeof(XT);
    constexpr bool kWide = MULTI || (two_blocks<VMODE, MG>() && !HOT);
    constexpr int kU = SPMM_UNROLL_BYTES * (kWide ? 2 : 1) / kBytes;
    constexpr int U = kU < 2 ? 2 : (kU > 8 ? 8 : kU);
#ifndef SPMM_MERGE_UNROLL
#define SPMM_MERGE_UNROLL 2
#endif
    constexpr int UM = U < SPMM_MERGE_UNROLL ? U : SPMM_MERGE_UNROLL;   // merge path: nonzeros in flight per lane
#ifndef SPMM_MERGE_WIDE_UNROLL
#define SPMM_MERGE_WIDE_UNROLL 4
#endif
    // merge over lane groups: nonzeros in flight per group.  Values are read from
    // shared memory when they are used and the task state fits few registers, so
    // 4 in flight spill neither with values (2 before: k = 16 weighted, 37 MB of
    // X 0.168 -> 0.152 ms) nor without; 6 do (0.211).  The compensated form over
    // 16-byte lanes spills 60 bytes and is as fast as with 2 (k = 16, 1 M vertices
    // 256 us, 262).  Four blocks (MG == 2) spill 92 bytes with 2 in flight and 112 in
    // the form that adds split rows; min_blocks()'s figures have that in them.
    constexpr int kUW = MG == 4   ? 8
                        : MG == 3 ? 2 * SPMM_MERGE_WIDE_UNROLL
                        : MG == 1 ? SPMM_MERGE_WIDE_UNROLL
                                  : 2;
    constexpr int UW = MG == 4 ? kUW : U < kUW ? U : kUW;
    // Pieces whose length is no multiple of the batch diverge at their last batch
    // if the others carry no checks; the checks cost more where the lanes hold one
    // element or four blocks run (FP32 k = 7, 512 K vertices 0.102 -> 0.092 ms, k =
    // 32, 64 K 50 -> 41 us; but k = 16 weighted, 1 M 0.152 -> 0.188 ms).
    constexpr bool kWholeBatches = kMergeG && (VEC == 1 || MG == 2);
    extern __shared__ __align__(128) unsigned char smem[];
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    unsigned char* wb = smem + w * Lay::kWarp;
    uint64_t* bars = reinterpret_cast<uint64_t*>(wb + 2 * Lay::kBuf);
    const FwdArgs& a = ga;      // launch-wide fields (and, unless MULTI, the matrix's)
    const XT* hs = nullptr;     // hot rows of X in shared memory (HOT)
    const uint32_t n_tasks = (uint32_t)a.n_tasks;      // at most kMaxLaunchTasks
    const uint32_t W = gridDim.x * WPB;
    const uint32_t t = blockIdx.x * WPB + w;
    if (!HOT && t >= n_tasks) return;
    if (lane == 0) {
        mbar_init(&bars[0], 1);
        mbar_init(&bars[1], 1);
        fence_mbar_init();
    }
    __syncwarp();

    // a task's descriptor and where it ends (the next one's first nonzero)
    struct Desc {
        int4 a;
        int2 end;
    };
    auto load_desc = [&](const int4* p, Desc& x) {
        x.a = p[0];
        x.end = reinterpret_cast<const int2*>(p + 1)[1];
    };
    // returns the task's entry (MULTI: a binary search of the entries' first tasks)
    auto fetch = [&](uint32_t tt, Desc& x) -> int {
        if constexpr (MULTI) {
            int lo = 0, hi = M->n - 1;
            while (lo < hi) {
                const int mid = (lo + hi + 1) >> 1;
                if (M->off[mid] <= (int64_t)tt) lo = mid;
                else hi = mid - 1;
            }
            load_desc(M->ent[lo].tasks + ((int64_t)tt - M->off[lo]), x);
            return lo;
        } else {
            load_desc(a.tasks + tt, x);
            return 0;
        }
    };
    auto entry = [&](int e) -> const FwdArgs& {
        if constexpr (MULTI) return M->ent[e];
        else return a;
    };

    // lane geometry (of the current task's entry when MULTI)
    int lg = 0, LANES = 1, G = 32, g = 0, li = 0;
    bool act[CH];
    const XT* xb = nullptr;
    uint64_t xpol = 0;
    const FwdArgs* cur = &a;    // the entry of the task being computed
    auto set_geometry = [&](const FwdArgs& E) {
        lg = ONE ? 0 : kWholeWarp ? 5 : E.lanes_log2;
        LANES = 1 << lg;
        G = 32 >> lg;
        g = lane >> lg;
        li = lane & (LANES - 1);
#pragma unroll
        for (int c = 0; c < CH; ++c) act[c] = (li + c * LANES) < E.nvec;
        xb = reinterpret_cast<const XT*>(E.X) + (int64_t)li * VEC;
        xpol = E.x_evict_last ? policy_evict_last() : policy_evict_normal();
        cur = &E;
    };
    // load the X row of column index c (elements off.. of this lane's part)
    auto gather = [&](auto& xv, int64_t c, int off) {
        if constexpr (HOT) {
            if (c < 0) {
                xv.load_sh(hs + (int64_t)(~c) * VEC);
                return;
            }
        }
        xv.load(xb + (uint64_t)(uint32_t)c * (uint64_t)cur->ldx + off, xpol);
    };
    // copy the task in x (fetch) into buffer buf (lane 0 issues)
    auto stage = [&](int e, const Desc& x, int buf) {
        if (lane == 0)
            issue_task<VMODE>(entry(e), x.a, desc_e0(x.end.x, x.end.y), wb + buf * Lay::kBuf, &bars[buf]);
    };
    Desc nx;
    int ed = 0;
    if (!HOT || t < n_tasks) {
        ed = fetch(t, nx);
        set_geometry(entry(ed));
        stage(ed, nx, 0);
    }
    if constexpr (HOT) {
        // the hot rows of X (one 4-byte word each) while the first tasks arrive
        uint32_t* h4 = reinterpret_cast<uint32_t*>(smem + WPB * Lay::kWarp);
        const uint32_t* x4 = reinterpret_cast<const uint32_t*>(a.X);
        const uint64_t ld4 = (uint64_t)a.ldx / VEC;
#pragma unroll 4
        for (int i = threadIdx.x; i < (int)a.n_hot; i += WPB * 32) h4[i] = __ldg(x4 + (uint64_t)a.hot_cols[i] * ld4);
        hs = reinterpret_cast<const XT*>(h4);
        __syncthreads();
        if (t >= n_tasks) return;
    }
    // the current task: first row, kind, low word of its first nonzero, nonzeros
    int2 d0;
    int e0, n;
    auto take = [&](const Desc& x) {
        d0 = make_int2(x.a.x, x.a.y);
        e0 = x.a.z;
        n = entries_between(e0, x.end.x);
    };
    take(nx);
    // the next task: static stride, or the next of a chunk claimed from the
    // counter by lane 0
    uint32_t cnext = 0, cend = 0;
    auto next_task = [&](uint32_t cur) -> uint32_t {
        if (a.task_chunk == 0) return cur + W;
        if (cnext < cend) return cnext++;
        uint32_t v = 0;
        if (lane == 0) v = atomicAdd(self_reset<ONE, HOT, SEG>() ? &a.ctl->next : &a.ctl->cleared_next, 1u);
        cnext = W + __shfl_sync(0xffffffffu, v, 0) * (uint32_t)a.task_chunk;
        cend = cnext + a.task_chunk;
        return cnext++;
    };
    uint32_t tn = next_task(t);
    int en = 0;
    if (tn < n_tasks) en = fetch(tn, nx);
    uint32_t phase = 0;     // bit b = parity to wait for on buffer b
    int b = 0;

    for (;;) {
        // stage the next task into the other buffer (its readers are done)
        const bool more = tn < n_tasks;
        if (more) {
            __syncwarp();
            if (lane == 0) fence_proxy_async();
            stage(en, nx, b ^ 1);
        }
        // prefetch the descriptor after next
        const uint32_t tnn = more ? next_task(tn) : n_tasks;
        Desc mx{};
        int em = 0;
        if (tnn < n_tasks) em = fetch(tnn, mx);

        if (!mbar_wait_bounded(&bars[b], (phase >> b) & 1u, a.wait_ns)) {
            if (lane == 0) atomicOr(a.status, kStatusTimeout);
            if (more) mbar_wait_bounded(&bars[b ^ 1], (phase >> (b ^ 1)) & 1u, a.wait_ns);
            return;
        }
        phase ^= 1u << b;

        int ready = -1;         // split row that this task completes
        // ---- compute task (d0, e0, n) from buffer b
        if constexpr (MULTI) {
            if (cur != &entry(ed)) set_geometry(entry(ed));
        }
        {
            const FwdArgs& a = *cur;   // the task's entry (the launch's matrix unless MULTI)
            const unsigned char* buf = wb + b * Lay::kBuf;
            Staged st;
            st.e0 = e0;
            st.col = reinterpret_cast<const int32_t*>(buf + Lay::kColOff) + (e0 & 3);
            if constexpr (VMODE != 0) {
                constexpr int epb = 16 / Lay::kValBytes;
                st.val = buf + Lay::kValOff + (e0 & (epb - 1)) * Lay::kValBytes;
            } else {
                st.val = nullptr;
            }
            st.rpw = reinterpret_cast<const int64_t*>(buf + Lay::kRpOff) + (d0.x & 1);

            if (kFlat && d0.y > 0) {
                // k = 1, run of short rows: every lane gathers the task's
                // nonzeros as one flat array (lane, lane+32, ...) and writes each
                // product over its staged column index; then lane j adds the
                // products of rows j, j+32 in nonzero order from shared memory.
                const int nr = d0.y;
                int32_t* prod = const_cast<int32_t*>(st.col);
                constexpr int UF = SPMM_FLAT_UF;
                for (int base = 0; base < n; base += 32 * UF) {
                    float xv[UF], av[UF];
#pragma unroll
                    for (int u = 0; u < UF; ++u) {
                        const int idx = base + lane + 32 * u;
                        if (idx < n) {
                            const int64_t cidx = st.col[idx];
                            av[u] = staged_val<VMODE>(st.val, idx);
                            XVec<XT, 1> t1;
                            gather(t1, cidx, 0);
                            xv[u] = t1.get(0);
                        }
                    }
#pragma unroll
                    for (int u = 0; u < UF; ++u) {
                        const int idx = base + lane + 32 * u;
                        if (idx < n) prod[idx] = __float_as_int(av[u] * xv[u]);
                    }
                }
                __syncwarp();
                for (int j = lane; j < nr; j += 32) {
                    const int s = st.rp(j), e = st.rp(j + 1);
                    float acc = 0.f;
                    for (int i = s; i < e; i += 4) {          // four loads in flight, added in order
                        const float p0 = __int_as_float(prod[i]);
                        const float p1 = i + 1 < e ? __int_as_float(prod[i + 1]) : 0.f;
                        const float p2 = i + 2 < e ? __int_as_float(prod[i + 2]) : 0.f;
                        const float p3 = i + 3 < e ? __int_as_float(prod[i + 3]) : 0.f;
                        acc += p0;
                        if (i + 1 < e) acc += p1;
                        if (i + 2 < e) acc += p2;
                        if (i + 3 < e) acc += p3;
                    }
                    __stcs(a.Y + (int64_t)(d0.x + j) * a.ldy, acc);
                }
                fence_proxy_async();   // the products were written where the next copy lands
            } else if (kMerge && d0.y > 0) {
                // run of short rows, one lane per X row (merge-based): the task's
                // nonzeros are cut into 32 equal contiguous pieces, lane l taking
                // piece l, so every lane gathers about n/32 rows of X whatever
                // the row lengths.  A lane walks its piece in order and stores
                // the rows that lie wholly inside it.  A row that crosses piece
                // boundaries leaves a tail partial in each lane it continues out
                // of and a head partial in the lane where it ends; a segmented
                // scan (shfl_up) over the lanes' tails, keyed by row,
                // adds the tails, and the ending lane adds its head last.
                const int nr = d0.y;
                for (int j = lane; j < nr; j += 32)       // rows without nonzeros
                    if (st.rp(j) == st.rp(j + 1)) {
                        float z[VEC];
#pragma unroll
                        for (int v = 0; v < VEC; ++v) z[v] = 0.f;
                        store_y<VEC>(a.Y + (int64_t)(d0.x + j) * a.ldy, z);
                    }
                const int per = (n + 31) >> 5;
                const int cs = min(n, lane * per), ce = min(n, cs + per);
                float tail[VEC], head[VEC];
#pragma unroll
                for (int v = 0; v < VEC; ++v) tail[v] = 0.f, head[v] = 0.f;
                int key = -1 - lane;                      // tail row, or a key no other lane has
                int hrow = -1;                            // head row
                if (cs < ce) {
                    // r: the row holding nonzero cs (largest r with rp[r] <= e0 + cs)
                    int lo = 0, hi = nr - 1;
                    while (lo < hi) {
                        const int mid = (lo + hi + 1) >> 1;
                        if (st.rp(mid) <= cs) lo = mid;
                        else hi = mid - 1;
                    }
                    int r = lo;
                    int rs = st.rp(r), re = st.rp(r + 1);
                    float acc[VEC];
#pragma unroll
                    for (int v = 0; v < VEC; ++v) acc[v] = 0.f;
                    for (int i = cs; i < ce; i += UM) {
                        XVec<XT, VEC> xv[UM];
                        float av[UM];
#pragma unroll
                        for (int u = 0; u < UM; ++u)
                            if (i + u < ce) {
                                const int64_t cidx = st.col[i + u];
                                av[u] = staged_val<VMODE>(st.val, i + u);
                                gather(xv[u], cidx, 0);
                            }
#pragma unroll
                        for (int u = 0; u < UM; ++u)
                            if (i + u < ce) {
                                while (i + u >= re) {             // row r ended inside the piece
                                    if (rs < re) {
                                        if (rs >= cs) {
                                            store_y<VEC>(a.Y + (int64_t)(d0.x + r) * a.ldy, acc);
                                        } else {
                                            hrow = r;
#pragma unroll
                                            for (int v = 0; v < VEC; ++v) head[v] = acc[v];
                                        }
                                    }
#pragma unroll
                                    for (int v = 0; v < VEC; ++v) acc[v] = 0.f;
                                    ++r;
                                    rs = re;
                                    re = st.rp(r + 1);
                                }
#pragma unroll
                                for (int v = 0; v < VEC; ++v) acc[v] = fmaf(av[u], xv[u].get(v), acc[v]);
                            }
                    }
                    // the row holding nonzero ce - 1
                    if (re > ce) {
                        key = r;
#pragma unroll
                        for (int v = 0; v < VEC; ++v) tail[v] = acc[v];
                    } else if (rs >= cs) {
                        store_y<VEC>(a.Y + (int64_t)(d0.x + r) * a.ldy, acc);
                    } else {
                        hrow = r;
#pragma unroll
                        for (int v = 0; v < VEC; ++v) head[v] = acc[v];
                    }
                }
                // segmented inclusive scan of the tails (a row's tails sit in
                // consecutive lanes, so equal keys bound a segment)
#pragma unroll
                for (int off = 1; off < 32; off <<= 1) {
                    const int kup = __shfl_up_sync(0xffffffffu, key, off);
                    float up[VEC];
#pragma unroll
                    for (int v = 0; v < VEC; ++v) up[v] = __shfl_up_sync(0xffffffffu, tail[v], off);
                    if (lane >= off && kup == key)
#pragma unroll
                        for (int v = 0; v < VEC; ++v) tail[v] += up[v];
                }
#pragma unroll
                for (int v = 0; v < VEC; ++v) {
                    const float prev = __shfl_up_sync(0xffffffffu, tail[v], 1);
                    head[v] = prev + head[v];
                }
                if (hrow >= 0) store_y<VEC>(a.Y + (int64_t)(d0.x + hrow) * a.ldy, head);
            } else if (kMergeG && d0.y > 0) {
                // run of short rows, LANES lanes per X row (merge-based over lane
                // groups): the task's nonzeros are cut into G equal contiguous
                // pieces, group g taking piece g, so every group gathers about
                // n/G rows of X whatever the row lengths.  As in the one-lane
                // case, a row crossing pieces is finished by a segmented scan
                // over the groups' tails (shfl_up by multiples of LANES, so lane
                // li of a group meets lane li of the others) and its head.
                const int nr = d0.y;
                for (int j = g; j < nr; j += G)           // rows without nonzeros
                    if (st.rp(j) == st.rp(j + 1) && act[0]) {
                        float z[VEC];
#pragma unroll
                        for (int v = 0; v < VEC; ++v) z[v] = 0.f;
                        store_y<VEC>(a.Y + (int64_t)(d0.x + j) * a.ldy + li * VEC, z);
                    }
                const int per = (n + G - 1) / G;
                const int cs = min(n, g * per), ce = min(n, cs + per);
                float tail[VEC], head[VEC];
#pragma unroll
                for (int v = 0; v < VEC; ++v) tail[v] = 0.f, head[v] = 0.f;
                int key = -1 - g;                         // tail row, or a key no other group has
                int hrow = -1;                            // head row
                if (cs < ce) {
                    int lo = 0, hi = nr - 1;              // the row holding nonzero cs
                    while (lo < hi) {
                        const int mid = (lo + hi + 1) >> 1;
                        if (st.rp(mid) <= cs) lo = mid;
                        else hi = mid - 1;
                    }
                    int r = lo;
                    int rs = st.rp(r), re = st.rp(r + 1);
                    float acc[VEC];
#pragma unroll
                    for (int v = 0; v < VEC; ++v) acc[v] = 0.f;
                    auto end_row = [&]() {                // row r ends inside the piece
                        if (rs < re) {
                            if (rs >= cs) {
                                if (act[0]) store_y<VEC>(a.Y + (int64_t)(d0.x + r) * a.ldy + li * VEC, acc);
                            } else {
                                hrow = r;
#pragma unroll
                                for (int v = 0; v < VEC; ++v) head[v] = acc[v];
                            }
                        }
#pragma unroll
                        for (int v = 0; v < VEC; ++v) acc[v] = 0.f;
                        ++r;
                        rs = re;
                        re = st.rp(r + 1);
                    };
                    auto add = [&](XVec<XT, VEC>& x, int i) {
                        if (act[0]) {
                            const float av = staged_val<VMODE>(st.val, i);
#pragma unroll
                            for (int v = 0; v < VEC; ++v) acc[v] = fmaf(av, x.get(v), acc[v]);
                        }
                    };
                    int i = cs;
                    if constexpr (kWholeBatches) {        // without bounds checks, then the rest
                        for (; i + UW <= ce; i += UW) {
                            XVec<XT, VEC> xv[UW];
#pragma unroll
                            for (int u = 0; u < UW; ++u)
                                if (act[0]) gather(xv[u], st.col[i + u], 0);
#pragma unroll
                            for (int u = 0; u < UW; ++u) {
                                while (i + u >= re) end_row();
                                add(xv[u], i + u);
                            }
                        }
                        if (i < ce) {
                            XVec<XT, VEC> xv[UW];
#pragma unroll
                            for (int u = 0; u < UW - 1; ++u)
                                if (i + u < ce && act[0]) gather(xv[u], st.col[i + u], 0);
#pragma unroll
                            for (int u = 0; u < UW - 1; ++u)
                                if (i + u < ce) {
                                    while (i + u >= re) end_row();
                                    add(xv[u], i + u);
                                }
                        }
                    } else {
                        for (; i < ce; i += UW) {
                            XVec<XT, VEC> xv[UW];
#pragma unroll
                            for (int u = 0; u < UW; ++u)
                                if (i + u < ce && act[0]) gather(xv[u], st.col[i + u], 0);
#pragma unroll
                            for (int u = 0; u < UW; ++u)
                                if (i + u < ce) {
                                    while (i + u >= re) end_row();
                                    add(xv[u], i + u);
                                }
                        }
                    }
                    if (re > ce) {                        // the row holding nonzero ce - 1
                        key = r;
#pragma unroll
                        for (int v = 0; v < VEC; ++v) tail[v] = acc[v];
                    } else if (rs >= cs) {
                        if (act[0]) store_y<VEC>(a.Y + (int64_t)(d0.x + r) * a.ldy + li * VEC, acc);
                    } else {
                        hrow = r;
#pragma unroll
                        for (int v = 0; v < VEC; ++v) head[v] = acc[v];
                    }
                }
                for (int off = 1; off < G; off <<= 1) {
                    const int kup = __shfl_up_sync(0xffffffffu, key, off * LANES);
                    float up[VEC];
#pragma unroll
                    for (int v = 0; v < VEC; ++v) up[v] = __shfl_up_sync(0xffffffffu, tail[v], off * LANES);
                    if (g >= off && kup == key)
#pragma unroll
                        for (int v = 0; v < VEC; ++v) tail[v] += up[v];
                }
#pragma unroll
                for (int v = 0; v < VEC; ++v) head[v] += __shfl_up_sync(0xffffffffu, tail[v], LANES);
                if (hrow >= 0 && act[0]) store_y<VEC>(a.Y + (int64_t)(d0.x + hrow) * a.ldy + li * VEC, head);
            } else if (kWholeWarp && d0.y > 0) {
                // run of short rows, 32 lanes per X row: the warp takes the task's
                // nonzeros in order, UW rows of X requested while the UW before are
                // added, across the ends of rows; no bounds are checked inside a
                // whole batch, and every branch is the warp's.  Each row's sum is
                // that of the row walk, and no row beyond the run is written, whatever
                // a caller's task list says (spmm_apply_csr_static).
                const int nr = d0.y;
                int r = 0, re = st.rp(1);
                float acc[CH][VEC];
#pragma unroll
                for (int c = 0; c < CH; ++c)
#pragma unroll
                    for (int v = 0; v < VEC; ++v) acc[c][v] = 0.f;
                auto end_row = [&]() {
                    float* dst = a.Y + (int64_t)(d0.x + r) * a.ldy;
#pragma unroll
                    for (int c = 0; c < CH; ++c) {
                        if (act[c]) store_y<VEC>(dst + (li + c * 32) * VEC, acc[c]);
#pragma unroll
                        for (int v = 0; v < VEC; ++v) acc[c][v] = 0.f;
                    }
                    ++r;
                };
                auto add1 = [&](XVec<XT, VEC>(&x)[CH], int i) {
                    const float av = staged_val<VMODE>(st.val, i);
#pragma unroll
                    for (int c = 0; c < CH; ++c)
#pragma unroll
                        for (int v = 0; v < VEC; ++v) acc[c][v] = fmaf(av, x[c].get(v), acc[c][v]);
                };
                auto load1 = [&](XVec<XT, VEC>(&x)[CH], int i) {
                    const int64_t cidx = st.col[i];
#pragma unroll
                    for (int c = 0; c < CH; ++c)
                        if (act[c]) gather(x[c], cidx, c * 32 * VEC);
                };
                auto load = [&](XVec<XT, VEC>(&x)[UW][CH], int i) {
#pragma unroll
                    for (int u = 0; u < UW; ++u) load1(x[u], i + u);
                };
                auto add = [&](XVec<XT, VEC>(&x)[UW][CH], int i) {
                    if (i + UW <= re) {            // all in the current row
#pragma unroll
                        for (int u = 0; u < UW; ++u) add1(x[u], i + u);
                    } else {
#pragma unroll
                        for (int u = 0; u < UW; ++u) {
                            while (i + u >= re && r < nr) {
                                end_row();
                                re = st.rp(r + 1);
                            }
                            add1(x[u], i + u);
                        }
                    }
                };
                XVec<XT, VEC> xa[UW][CH], xb[UW][CH];
                const int full = n - n % UW;
                if (full > 0) load(xa, 0);
                int i = 0;
                for (; i < full; i += 2 * UW) {
                    if (i + UW < full) load(xb, i + UW);
                    add(xa, i);
                    if (i + UW < full) {
                        if (i + 2 * UW < full) load(xa, i + 2 * UW);
                        add(xb, i + UW);
                    }
                }
#pragma unroll
                for (int u = 0; u < UW - 1; ++u)
                    if (full + u < n) load1(xa[u], full + u);
#pragma unroll
                for (int u = 0; u < UW - 1; ++u)
                    if (full + u < n) {
                        while (full + u >= re && r < nr) {
                            end_row();
                            re = st.rp(r + 1);
                        }
                        add1(xa[u], full + u);
                    }
                while (r < nr) end_row();
            } else if (!kFlat && !kMerge && !kMergeG && !kWholeWarp && d0.y > 0) {
                // run of short rows: lane group g owns rows g, g+G, ...
                const int nr = d0.y;
                for (int j = g; j < nr; j += G) {
                    const int s = st.rp(j), e = st.rp(j + 1);
                    float acc[CH][VEC];
#pragma unroll
                    for (int c = 0; c < CH; ++c)
#pragma unroll
                        for (int v = 0; v < VEC; ++v) acc[c][v] = 0.f;
                    for (int i = s; i < e; i += U) {
                        XVec<XT, VEC> xv[U][CH];
#pragma unroll
                        for (int u = 0; u < U; ++u) {
                            if (i + u < e) {
                                const int64_t cidx = st.col[i + u];
#pragma unroll
                                for (int c = 0; c < CH; ++c)
                                    if (act[c]) gather(xv[u][c], cidx, c * LANES * VEC);
                            }
                        }
#pragma unroll
                        for (int u = 0; u < U; ++u)
                            if (i + u < e) {
                                const float av = staged_val<VMODE>(st.val, i + u);
#pragma unroll
                                for (int c = 0; c < CH; ++c)
#pragma unroll
                                    for (int v = 0; v < VEC; ++v) acc[c][v] = fmaf(av, xv[u][c].get(v), acc[c][v]);
                            }
                    }
                    float* dst = a.Y + (int64_t)(d0.x + j) * a.ldy;
#pragma unroll
                    for (int c = 0; c < CH; ++c)
                        if (act[c]) store_y<VEC>(dst + (li + c * LANES) * VEC, acc[c]);
                }
            } else if (COMP) {
                // one long row or hub segment, compensated: Neumaier summation of
                // the products, whose own rounding error fmaf recovers exactly
                float acc[CH][VEC], cmp[CH][VEC];
#pragma unroll
                for (int c = 0; c < CH; ++c)
#pragma unroll
                    for (int v = 0; v < VEC; ++v) acc[c][v] = 0.f, cmp[c][v] = 0.f;
                for (int i = g; i < n; i += G * U) {
                    XVec<XT, VEC> xv[U][CH];
                    float av[U];
#pragma unroll
                    for (int u = 0; u < U; ++u) {
                        const int idx = i + u * G;
                        if (idx < n) {
                            const int64_t cidx = st.col[idx];
                            av[u] = staged_val<VMODE>(st.val, idx);
#pragma unroll
                            for (int c = 0; c < CH; ++c)
                                if (act[c]) gather(xv[u][c], cidx, c * LANES * VEC);
                        }
                    }
#pragma unroll
                    for (int u = 0; u < U; ++u)
                        if (i + u * G < n) {
#pragma unroll
                            for (int c = 0; c < CH; ++c)
#pragma unroll
                                for (int v = 0; v < VEC; ++v) {
                                    const float x = xv[u][c].get(v);
                                    const float p = av[u] * x;
                                    const float pe = fmaf(av[u], x, -p);       // exact product error
                                    const float t = acc[c][v] + p;
                                    const float e = (fabsf(acc[c][v]) >= fabsf(p)) ? (acc[c][v] - t) + p
                                                                                   : (p - t) + acc[c][v];
                                    cmp[c][v] += e + pe;
                                    acc[c][v] = t;
                                }
                        }
                }
                for (int off = LANES; off < 32; off <<= 1)
#pragma unroll
                    for (int c = 0; c < CH; ++c)
#pragma unroll
                        for (int v = 0; v < VEC; ++v) {
                            const float s2 = __shfl_xor_sync(0xffffffffu, acc[c][v], off);
                            const float c2 = __shfl_xor_sync(0xffffffffu, cmp[c][v], off);
                            const float t = acc[c][v] + s2;
                            const float e = (fabsf(acc[c][v]) >= fabsf(s2)) ? (acc[c][v] - t) + s2
                                                                            : (s2 - t) + acc[c][v];
                            cmp[c][v] += c2 + e;
                            acc[c][v] = t;
                        }
                if (g == 0) {
                    if (d0.y == 0) {                   // whole row: one rounding of sum + compensation
#pragma unroll
                        for (int c = 0; c < CH; ++c)
#pragma unroll
                            for (int v = 0; v < VEC; ++v) acc[c][v] += cmp[c][v];
                        float* dst = a.Y + (int64_t)d0.x * a.ldy;
#pragma unroll
                        for (int c = 0; c < CH; ++c)
                            if (act[c]) store_y<VEC>(dst + (li + c * LANES) * VEC, acc[c]);
                    } else if ((int64_t)(-d0.y - 1) < a.n_slots) {   // segment: keep the pair for the combine pass
                        const int64_t slot = (int64_t)(-d0.y - 1) * a.k;
#pragma unroll
                        for (int c = 0; c < CH; ++c)
                            if (act[c]) {
                                store_y<VEC>(a.partials + slot + (li + c * LANES) * VEC, acc[c]);
                                store_y<VEC>(a.partials_comp + slot + (li + c * LANES) * VEC, cmp[c]);
                            }
                    } else if (lane == 0) {                // a slot beyond the scratch: write nothing
                        atomicOr(a.status, kStatusSlotRange);
                    }
                }
                if (SEG && d0.y < 0) ready = segment_done(a, -d0.y - 1, lane);
            } else {
                // one long row or one hub segment: nonzeros g, g+G, ... per group
                float acc[CH][VEC];
#pragma unroll
                for (int c = 0; c < CH; ++c)
#pragma unroll
                    for (int v = 0; v < VEC; ++v) acc[c][v] = 0.f;
                for (int i = g; i < n; i += G * U) {
                    XVec<XT, VEC> xv[U][CH];
#pragma unroll
                    for (int u = 0; u < U; ++u) {
                        const int idx = i + u * G;
                        if (idx < n) {
                            const int64_t cidx = st.col[idx];
#pragma unroll
                            for (int c = 0; c < CH; ++c)
                                if (act[c]) gather(xv[u][c], cidx, c * LANES * VEC);
                        }
                    }
#pragma unroll
                    for (int u = 0; u < U; ++u)
                        if (i + u * G < n) {
                            const float av = staged_val<VMODE>(st.val, i + u * G);
#pragma unroll
                            for (int c = 0; c < CH; ++c)
#pragma unroll
                                for (int v = 0; v < VEC; ++v) acc[c][v] = fmaf(av, xv[u][c].get(v), acc[c][v]);
                        }
                }
                for (int off = LANES; off < 32; off <<= 1)
#pragma unroll
                    for (int c = 0; c < CH; ++c)
#pragma unroll
                        for (int v = 0; v < VEC; ++v) acc[c][v] += __shfl_xor_sync(0xffffffffu, acc[c][v], off);
                if (d0.y < 0 && (int64_t)(-d0.y - 1) >= a.n_slots) {   // a slot beyond the scratch
                    if (lane == 0) atomicOr(a.status, kStatusSlotRange);
                } else if (g == 0) {
                    float* dst = (d0.y == 0) ? a.Y + (int64_t)d0.x * a.ldy
                                             : a.partials + (int64_t)(-d0.y - 1) * a.k;
#pragma unroll
                    for (int c = 0; c < CH; ++c)
                        if (act[c]) store_y<VEC>(dst + (li + c * LANES) * VEC, acc[c]);
                }
                if (SEG && d0.y < 0) ready = segment_done(a, -d0.y - 1, lane);
            }
        }
        if (SEG && ready >= 0) {   // add its segments' partials, in segment order, into Y
            // lane 0 saw the other warps' arrivals: its fence, then the warp's barrier, put every
            // lane's reads of their partials after them
            __threadfence();
            __syncwarp();
            const FwdArgs& a = *cur;
            combine_row(a.splits[ready], a.partials, a.Y, a.ldy, a.k, combine_lanes_log2(a.k), a.partials_comp, lane);
        }
        if (!more) break;
        take(nx);
        ed = en;
        nx = mx;
        en = em;
        tn = tnn;
        b ^= 1;
    }
}

// The end of a warp: the launch's last one leaves the task counter at zero for
// the next launch.  After a wait that ran out (in this launch or one not yet
// reported) some segments may be missing, so it clears the arrivals too.  Every
// warp's arrival here is a release and the last one's is followed by a fence, so
// the last warp sees each status bit, claim and segment arrival of the launch
// before it reads or clears them.
__device__ __forceinline__ void warp_done(const FwdArgs& ga, const MultiArgs* M) {
    if (!ga.ctl) return;
    __syncwarp();
    const int lane = threadIdx.x & 31;
    const unsigned int warps = gridDim.x * (blockDim.x >> 5);
    unsigned int old = 0;
    if (lane == 0) old = atom_inc_release(&ga.ctl->done, warps - 1);    // wraps to zero at the last
    if (__shfl_sync(0xffffffffu, old, 0) != warps - 1) return;
    __threadfence();
    __syncwarp();
    if (lane == 0) ga.ctl->next = 0;
    if (__ldcg(ga.status) == 0) return;
    for (int e = 0; e < (M ? M->n : 1); ++e) {
        const FwdArgs& a = M ? M->ent[e] : ga;
        if (a.seg_done)
            for (int64_t i = lane; i < a.n_splits; i += 32) a.seg_done[i] = 0;
    }
}

template <typename XT, int VMODE, int VEC, int CH, bool COMP, bool ONE, int MG = 0, bool HOT = false, bool SEG = false>
__global__ void __launch_bounds__(warps_per_block<HOT>() * 32, (HOT ? 1 : min_blocks<VMODE, MG>()))
    rows_kernel(const __grid_constant__ FwdArgs a) {
    rows_run<XT, VMODE, VEC, CH, COMP, ONE, MG, HOT, false, SEG>(a, nullptr);
    if constexpr (self_reset<ONE, HOT, SEG>()) warp_done(a, nullptr);
}

// the tasks of up to kMaxBatch matrices in one launch (spmm_apply_batched);
// two blocks per SM, so the per-task lane geometry fits in registers
template <typename XT, int VMODE, int VEC, int CH, bool COMP>
__global__ void __launch_bounds__(kWarpsPerBlock * 32, 2) rows_kernel_multi(const __grid_constant__ MultiArgs m) {
    rows_run<XT, VMODE, VEC, CH, COMP, false, 0, false, true, true>(m.g, &m);
    warp_done(m.g, &m);
}

template <typename XT, int VMODE, int VEC, int CH, bool COMP, bool ONE, int MG = 0, bool HOT = false, bool SEG = false>
cudaError_t launch_one(const FwdArgs& a, cudaStream_t s) {
    if constexpr (!SEG && !COMP && !HOT)
        if (a.seg_done) return launch_one<XT, VMODE, VEC, CH, COMP, ONE, MG, HOT, true>(a, s);
    using Lay = Layout<VMODE>;
    constexpr int WPB = warps_per_block<HOT>();
    constexpr int kStage = WPB * Lay::kWarp;      // staging buffers of the block's warps
    // per instantiation, computed once (thread-safe; a failure is reported to
    // every caller)
    static std::once_flag once;
    static int blocks_per_sm = 0, num_sms = 0, max_smem = 0;
    static cudaError_t setup = cudaSuccess;
    std::call_once(once, [] {
        cudaError_t e = cudaSuccess;
        int dev = 0, nb = 0, sms = 0, opt = 0;
        if (e == cudaSuccess) e = cudaGetDevice(&dev);
        if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
        if (e == cudaSuccess) e = cudaDeviceGetAttribute(&opt, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
        // the hot variant asks for the whole opt-in shared memory (its hot rows fill what the staging leaves)
        const int want = HOT ? opt : kStage;
        if (e == cudaSuccess && want > 48 * 1024)
            e = cudaFuncSetAttribute(rows_kernel<XT, VMODE, VEC, CH, COMP, ONE, MG, HOT, SEG>,
                                     cudaFuncAttributeMaxDynamicSharedMemorySize, want);
        if (e == cudaSuccess)
            e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, rows_kernel<XT, VMODE, VEC, CH, COMP, ONE, MG, HOT, SEG>,
                                                              WPB * 32, want);
        setup = e;
        num_sms = sms;
        max_smem = opt;
        // two blocks even where the registers of a compiler's choice would let a third in
        blocks_per_sm = nb < 1 ? 1 : (two_blocks<VMODE, MG>() && !HOT && nb > 2) ? 2 : nb;
    });
    if (setup != cudaSuccess) return setup;
    size_t smem = kStage;
    if constexpr (HOT) {
        smem += (size_t)a.n_hot * kHotRowBytes;
        if (smem > (size_t)max_smem || a.n_hot <= 0) return cudaErrorInvalidValue;
    }
    if (!self_reset<ONE, HOT, SEG>() && a.task_chunk > 0) {
        const cudaError_t e = cudaMemsetAsync(&a.ctl->cleared_next, 0, sizeof(unsigned int), s);
        if (e != cudaSuccess) return e;
    }
    const int64_t want = (a.n_tasks + WPB - 1) / WPB;
    const int64_t cap = (int64_t)blocks_per_sm * num_sms;
    const dim3 grid((unsigned)(want < cap ? want : cap));
    rows_kernel<XT, VMODE, VEC, CH, COMP, ONE, MG, HOT, SEG><<<grid, WPB * 32, smem, s>>>(a);
    return cudaGetLastError();
}

// One launch over the entries of M (generic row walk, two blocks per SM).
template <typename XT, int VMODE, int VEC, int CH, bool COMP>
cudaError_t launch_multi_one(const MultiArgs& m, cudaStream_t s) {
    using Lay = Layout<VMODE>;
    static std::once_flag once;
    static int blocks_per_sm = 0, num_sms = 0;
    static cudaError_t setup = cudaSuccess;
    std::call_once(once, [] {
        cudaError_t e = cudaSuccess;
        int dev = 0, nb = 0, sms = 0;
        if (Lay::kBlock > 48 * 1024)
            e = cudaFuncSetAttribute(rows_kernel_multi<XT, VMODE, VEC, CH, COMP>,
                                     cudaFuncAttributeMaxDynamicSharedMemorySize, Lay::kBlock);
        if (e == cudaSuccess) e = cudaGetDevice(&dev);
        if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
        if (e == cudaSuccess)
            e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, rows_kernel_multi<XT, VMODE, VEC, CH, COMP>,
                                                              kWarpsPerBlock * 32, Lay::kBlock);
        setup = e;
        num_sms = sms;
        blocks_per_sm = nb > 0 ? nb : 1;
    });
    if (setup != cudaSuccess) return setup;
    const int64_t want = (m.g.n_tasks + kWarpsPerBlock - 1) / kWarpsPerBlock;
    const int64_t cap = (int64_t)blocks_per_sm * num_sms;
    const dim3 grid((unsigned)(want < cap ? want : cap));
    rows_kernel_multi<XT, VMODE, VEC, CH, COMP><<<grid, kWarpsPerBlock * 32, Lay::kBlock, s>>>(m);
    return cudaGetLastError();
}

template <typename XT>
cudaError_t launch_rows_multi_t(const MultiArgs& m, int vmode, int vec, int ch, bool comp, cudaStream_t s) {
    if (m.g.n_tasks <= 0) return cudaSuccess;
#define SPMM_LAUNCH_MULTI(VM, V, C)                                                      \
    if (vmode == VM && vec == V && ch == C)                                              \
        return comp ? launch_multi_one<XT, VM, V, C, true>(m, s) : launch_multi_one<XT, VM, V, C, false>(m, s);
    if constexpr (sizeof(XT) == 4) {
        SPMM_LAUNCH_MULTI(0, 4, 1) SPMM_LAUNCH_MULTI(0, 2, 1) SPMM_LAUNCH_MULTI(0, 1, 1) SPMM_LAUNCH_MULTI(0, 1, 2)
        SPMM_LAUNCH_MULTI(1, 4, 1) SPMM_LAUNCH_MULTI(1, 2, 1) SPMM_LAUNCH_MULTI(1, 1, 1) SPMM_LAUNCH_MULTI(1, 1, 2)
    } else {
        constexpr int VM3 = std::is_same<XT, __half>::value ? 3 : 2;
        SPMM_LAUNCH_MULTI(0, 8, 1) SPMM_LAUNCH_MULTI(0, 4, 1) SPMM_LAUNCH_MULTI(0, 2, 1) SPMM_LAUNCH_MULTI(0, 1, 1)
        SPMM_LAUNCH_MULTI(0, 1, 2)
        SPMM_LAUNCH_MULTI(1, 8, 1) SPMM_LAUNCH_MULTI(1, 4, 1) SPMM_LAUNCH_MULTI(1, 2, 1) SPMM_LAUNCH_MULTI(1, 1, 1)
        SPMM_LAUNCH_MULTI(1, 1, 2)
        SPMM_LAUNCH_MULTI(VM3, 8, 1) SPMM_LAUNCH_MULTI(VM3, 4, 1) SPMM_LAUNCH_MULTI(VM3, 2, 1)
        SPMM_LAUNCH_MULTI(VM3, 1, 1) SPMM_LAUNCH_MULTI(VM3, 1, 2)
    }
#undef SPMM_LAUNCH_MULTI
    return cudaErrorInvalidValue;
}

// One lane per X row of at most 4 bytes, hot rows in shared memory.
template <typename XT>
cudaError_t launch_rows_hot_t(const FwdArgs& a, int vmode, int vec, cudaStream_t s) {
    if (a.n_tasks <= 0) return cudaSuccess;
#define SPMM_LAUNCH_HOT(VM, V)                                                           \
    if (vmode == VM && vec == V)                                                         \
        return a.compensated ? launch_one<XT, VM, V, 1, true, true, 0, true>(a, s)       \
                             : launch_one<XT, VM, V, 1, false, true, 0, true>(a, s);
    if constexpr (sizeof(XT) == 4) {
        SPMM_LAUNCH_HOT(0, 1) SPMM_LAUNCH_HOT(1, 1)
    } else {
        constexpr int VM3 = std::is_same<XT, __half>::value ? 3 : 2;
        SPMM_LAUNCH_HOT(0, 1) SPMM_LAUNCH_HOT(0, 2) SPMM_LAUNCH_HOT(1, 1) SPMM_LAUNCH_HOT(1, 2)
        SPMM_LAUNCH_HOT(VM3, 1) SPMM_LAUNCH_HOT(VM3, 2)
    }
#undef SPMM_LAUNCH_HOT
    return cudaErrorInvalidValue;
}

template <typename XT, bool ONE, int MG = 0>
cudaError_t launch_rows_t(const FwdArgs& a, int vmode, int vec, int ch, cudaStream_t s) {
    static_assert(!(ONE && MG), "one lane per row has no lane groups");
    if (a.n_tasks <= 0) return cudaSuccess;
#define SPMM_LAUNCH(VM, V, C)                                                            \
    if (vmode == VM && vec == V && ch == C)                                              \
        return a.compensated ? launch_one<XT, VM, V, C, true, ONE, MG>(a, s)             \
                             : launch_one<XT, VM, V, C, false, ONE, MG>(a, s);
    if constexpr (MG == 2) {     // float pattern rows of 4-element lanes only
        if constexpr (sizeof(XT) == 4) { SPMM_LAUNCH(0, 4, 1) }
    } else if constexpr (MG == 4) {   // a whole warp per X row, two chunks of single elements
        if constexpr (sizeof(XT) == 4) {
            SPMM_LAUNCH(0, 1, 2) SPMM_LAUNCH(1, 1, 2)
        } else {
            constexpr int VM3 = std::is_same<XT, __half>::value ? 3 : 2;
            SPMM_LAUNCH(0, 1, 2) SPMM_LAUNCH(1, 1, 2) SPMM_LAUNCH(VM3, 1, 2)
        }
    } else if constexpr (MG == 3) {   // staged values only
        if constexpr (sizeof(XT) == 4) {
            SPMM_LAUNCH(1, 4, 1) SPMM_LAUNCH(1, 2, 1) SPMM_LAUNCH(1, 1, 1)
        } else {
            constexpr int VM3 = std::is_same<XT, __half>::value ? 3 : 2;
            SPMM_LAUNCH(1, 4, 1) SPMM_LAUNCH(1, 2, 1) SPMM_LAUNCH(1, 1, 1)
            SPMM_LAUNCH(VM3, 4, 1) SPMM_LAUNCH(VM3, 2, 1) SPMM_LAUNCH(VM3, 1, 1)
        }
    } else if constexpr (MG == 1) {   // CH == 1, at most 4 elements per lane
        if constexpr (sizeof(XT) == 4) {
            SPMM_LAUNCH(0, 4, 1) SPMM_LAUNCH(0, 2, 1) SPMM_LAUNCH(0, 1, 1)
            SPMM_LAUNCH(1, 4, 1) SPMM_LAUNCH(1, 2, 1) SPMM_LAUNCH(1, 1, 1)
        } else {
            constexpr int VM3 = std::is_same<XT, __half>::value ? 3 : 2;
            SPMM_LAUNCH(0, 4, 1) SPMM_LAUNCH(0, 2, 1) SPMM_LAUNCH(0, 1, 1)
            SPMM_LAUNCH(1, 4, 1) SPMM_LAUNCH(1, 2, 1) SPMM_LAUNCH(1, 1, 1)
            SPMM_LAUNCH(VM3, 4, 1) SPMM_LAUNCH(VM3, 2, 1) SPMM_LAUNCH(VM3, 1, 1)
        }
    } else if constexpr (ONE) {  // CH == 1 only
        if constexpr (sizeof(XT) == 4) {
            SPMM_LAUNCH(0, 4, 1) SPMM_LAUNCH(0, 2, 1) SPMM_LAUNCH(0, 1, 1)
            SPMM_LAUNCH(1, 4, 1) SPMM_LAUNCH(1, 2, 1) SPMM_LAUNCH(1, 1, 1)
        } else {
            constexpr int VM3 = std::is_same<XT, __half>::value ? 3 : 2;  // own-type values
            SPMM_LAUNCH(0, 8, 1) SPMM_LAUNCH(0, 4, 1) SPMM_LAUNCH(0, 2, 1) SPMM_LAUNCH(0, 1, 1)
            SPMM_LAUNCH(1, 8, 1) SPMM_LAUNCH(1, 4, 1) SPMM_LAUNCH(1, 2, 1) SPMM_LAUNCH(1, 1, 1)
            SPMM_LAUNCH(VM3, 8, 1) SPMM_LAUNCH(VM3, 4, 1) SPMM_LAUNCH(VM3, 2, 1) SPMM_LAUNCH(VM3, 1, 1)
        }
    } else {
        if constexpr (sizeof(XT) == 4) {
            SPMM_LAUNCH(0, 4, 1) SPMM_LAUNCH(0, 2, 1) SPMM_LAUNCH(0, 1, 1)
            SPMM_LAUNCH(1, 4, 1) SPMM_LAUNCH(1, 2, 1) SPMM_LAUNCH(1, 1, 1)
        } else {
            constexpr int VM3 = std::is_same<XT, __half>::value ? 3 : 2;
            SPMM_LAUNCH(0, 8, 1) SPMM_LAUNCH(0, 4, 1) SPMM_LAUNCH(0, 2, 1) SPMM_LAUNCH(0, 1, 1)
            SPMM_LAUNCH(1, 8, 1) SPMM_LAUNCH(1, 4, 1) SPMM_LAUNCH(1, 2, 1) SPMM_LAUNCH(1, 1, 1)
            SPMM_LAUNCH(VM3, 8, 1) SPMM_LAUNCH(VM3, 4, 1) SPMM_LAUNCH(VM3, 2, 1) SPMM_LAUNCH(VM3, 1, 1)
        }
    }
#undef SPMM_LAUNCH
    return cudaErrorInvalidValue;
}

}  // namespace spmm
