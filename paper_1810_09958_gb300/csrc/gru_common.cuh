// gru_common.cuh -- device helpers shared by the GRU recurrence kernels.
#pragma once
#include <cstdint>

#include <cuda_bf16.h>

#include "ptx.cuh"

namespace isam {

constexpr uint32_t kSiteGruStep = 0x201;  // bounded wait for a round's vectors

// Branch-free gate nonlinearities (a data-dependent branch in the gate code
// would split warps for the rest of the step): __expf and the approximate
// __fdividef, exact in the limits (exp overflow gives 0 and +-1).
__device__ __forceinline__ float sigmoidf_fast(float v) { return __fdividef(1.0f, 1.0f + __expf(-v)); }
// tanh(v) = 1 - 2 / (1 + e^{2v})
__device__ __forceinline__ float tanhf_fast(float v) { return 1.0f - __fdividef(2.0f, 1.0f + __expf(2.0f * v)); }

// h' = (1 - z) n + z h and the candidate's argument x + r g, with the rounding
// written out: the one-layer and the two-layer kernels give the same bits.
__device__ __forceinline__ float gru_blend(float z, float n, float h) {
    return __fmaf_rn(z, h, __fmul_rn(__fsub_rn(1.0f, z), n));
}
__device__ __forceinline__ float gru_candidate(float x, float r, float g) { return tanhf_fast(__fmaf_rn(r, g, x)); }

__device__ __forceinline__ uint16_t f32_to_bf16_rne(float f) {
    return __bfloat16_as_ushort(__float2bfloat16_rn(f));
}

// Exchange ring of the recurrence.  A word holds kEmpty until its producer
// stores it: two bf16 values, never both 0xFFFF nor either of them, because
// the conversion to bf16 gives every NaN the pattern 0x7FFF.
constexpr int kSlots = 4;
constexpr uint32_t kEmpty = 0xFFFFFFFFu;

__device__ __forceinline__ uint4 ld_relaxed_gpu_v4(const void *p) {
    uint4 v;
    asm volatile("ld.relaxed.gpu.global.v4.u32 {%0, %1, %2, %3}, [%4];"
                 : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
                 : "l"(p)
                 : "memory");
    return v;
}

__device__ __forceinline__ uint32_t ld_relaxed_gpu(const uint32_t *p) {
    uint32_t v;
    asm volatile("ld.relaxed.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}

__device__ __forceinline__ void st_relaxed_gpu(uint32_t *p, uint32_t v) {
    asm volatile("st.relaxed.gpu.global.u32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}

__device__ __forceinline__ void fence_acq_rel_gpu() { asm volatile("fence.acq_rel.gpu;" ::: "memory"); }

// No half of the four words is 0xFFFF (a zero half of the complement: the
// borrow of the subtraction marks it, or a half above a marked one, so the
// answer over the whole word is exact).
__device__ __forceinline__ bool published(const uint4 &v) {
    const uint32_t m = ((~v.x - 0x00010001u) & v.x) | ((~v.y - 0x00010001u) & v.y) | ((~v.z - 0x00010001u) & v.z) |
                       ((~v.w - 0x00010001u) & v.w);
    return (m & 0x80008000u) == 0u;
}

// bounded_wait by every lane of a warp, with a warp-uniform result.
template <bool cluster_scope = false>
__device__ __forceinline__ bool all_wait(uint64_t *bar, uint32_t parity, const WaitCtx &w, uint32_t site) {
    return __all_sync(0xffffffffu, bounded_wait<cluster_scope>(bar, parity, w, site) ? 1 : 0) != 0;
}

// Waits ignoring the abort flag (lets work already issued complete).
__device__ inline void drain_bar(uint64_t *bar, uint32_t parity, unsigned long long timeout_ns) {
    const unsigned long long t0 = globaltimer();
    while (!mbar_try_wait(smem_u32(bar), parity))
        if (globaltimer() - t0 > timeout_ns) return;
}

// Gathers this warp's 16-byte pieces of a round's vectors: load l (piece
// l / LPA of the warp, batch rows 32 (l % LPA) + lane) is wanted where bit l of
// `mine` is set.  Every wanted piece is polled until its producer has stored
// it, and goes into the MMA's swizzled K-major tile; then the warp arrives on
// h_full.  False when the wait ran out or the CTA gave up.
template <int NL, int LPA>
__device__ __forceinline__ bool gather_tile(const uint16_t *src, uint8_t *dst, uint32_t mine, int src_stride,
                                            int dst_stride, uint64_t *h_full, int lane, const WaitCtx &w) {
    uint32_t pend = mine;
    unsigned long long t0 = 0;
    for (uint32_t it = 1;; ++it) {
        uint4 v[NL];
#pragma unroll
        for (int l = 0; l < NL; ++l)
            if (pend >> l & 1u) v[l] = ld_relaxed_gpu_v4(src + (l / LPA) * src_stride + (l % LPA) * 256);
#pragma unroll
        for (int l = 0; l < NL; ++l)
            if ((pend >> l & 1u) && published(v[l])) {
                *reinterpret_cast<uint4 *>(dst + (l / LPA) * dst_stride + (l % LPA) * 4096) = v[l];
                pend &= ~(1u << l);
            }
        if (__all_sync(0xffffffffu, pend == 0u)) break;
        if ((it & 15u) == 0u) {
            bool stop = *w.abort_flag != 0;
            if (t0 == 0) t0 = globaltimer();
            if (!stop && globaltimer() - t0 > w.timeout_ns) {
                report_timeout(w, kSiteGruStep);
                stop = true;
            }
            if (__any_sync(0xffffffffu, stop)) return false;
        }
    }
    fence_proxy_async_smem();
    __syncwarp();
    if (lane == 0) mbar_arrive(h_full);
    return true;
}

// Received partial rows: [source][row kind][half of the batch columns][unit][BP / 2],
// each half written by another warp.  16-byte piece c of a unit's half sits at
// c ^ recv_swizzle(unit), so that the gates' reads (8 or more units, few batch
// columns per warp) fall into different banks.
template <int BP>
__device__ __forceinline__ int recv_swizzle(int unit) {
    return BP == 32 ? (unit >> 1) & 3 : unit & 7;
}

// Floats from a row kind's first half to batch column b of a unit.
template <int BP, int UO>
__device__ __forceinline__ int recv_at(int unit, int b) {
    const int half = b / (BP / 2), c = b % (BP / 2);
    return (half * UO + unit) * (BP / 2) + (((c >> 2) ^ recv_swizzle<BP>(unit)) << 2) + (c & 3);
}

// Sends half `half` of the batch columns of this warp's 32 accumulator rows (at
// `acc`, TMEM lane = row) to their owners: dst is the half row in the owner's
// received rows, counted on the owner's barrier `bar`; only the npiece pieces of
// the whole row that hold the batch are sent.  Asynchronous remote stores: nothing
// here waits for them to land.
template <int BP>
__device__ __forceinline__ void push_rows(uint32_t acc, int half, int npiece, uint32_t dst, int unit, uint32_t bar) {
    constexpr int CH = BP / 2 < 32 ? BP / 2 : 32;  // columns per TMEM load
#pragma unroll
    for (int c0 = 0; c0 < BP / 2; c0 += CH) {
        const int col = half * (BP / 2) + c0;
        if (col / 4 >= npiece) break;
        uint32_t r[CH];
        if constexpr (CH == 16)
            tmem_ld16(acc + static_cast<uint32_t>(col), r);
        else
            tmem_ld32(acc + static_cast<uint32_t>(col), r);
        tmem_ld_wait(r);
#pragma unroll
        for (int c = 0; c < CH / 4; ++c)
            if (col / 4 + c < npiece)
                st_async_f4(dst + static_cast<uint32_t>(((c0 / 4 + c) ^ recv_swizzle<BP>(unit)) << 4),
                            make_float4(__uint_as_float(r[4 * c]), __uint_as_float(r[4 * c + 1]),
                                        __uint_as_float(r[4 * c + 2]), __uint_as_float(r[4 * c + 3])),
                            bar);
    }
    tc_fence_before();
}

// How partial rows cross the cluster: as bulk copies of whole half rows, or as
// 16-byte stores of the pieces that hold the batch.  The stores of a warp go to
// 32 different rows and take longer than the copies once a row is about three
// quarters full, at every hidden size: 40 steps (stores / copies) take 111.6 / 115.4
// us at hidden 1024 and batch 20, 115.7 / 116.0 at 24, 121.2 / 114.9 at 32, 170.6 /
// 172.1 at 48, 184.5 / 174.9 at 64; hidden 384, two splits: 101.8 / 102.4, 105.2 / 103.4,
// 112.8 / 107.5, 154.5 / 153.3, 179.1 / 168.0; hidden 256: 85.3 / 89.7, 89.5 / 90.3,
// 95.1 / 90.1, 133.8 / 136.4, 146.9 / 138.0.  At 128 padded rows (64 steps, hidden
// 1024) the two are equal at a full batch (527 / 529) and the stores ahead below it
// (441 / 482 at 96).
__host__ __device__ inline bool gru_push_bulk(int batch, int bp) { return bp < 128 && 4 * batch >= 3 * bp; }

// Staging buffers of push_rows_bulk, which rounds take in turn.
constexpr int kGruStages = 2;

// The same half rows through a staging copy: the warp writes those of other CTAs
// (`remote`) to `stage`, laid out as the owners hold them, then lane o sends owner
// o's `bytes` contiguous bytes as one bulk copy.  Whole half rows move (padding
// included); this CTA's own rows take the direct stores, npiece pieces each.  Warps
// w and w + 4, which share a lane quarter, each send what they wrote: one that has
// given up leaves the round, so no barrier may join them.
//
// A copy's end is seen on its owner's barrier only, so it is the exchange that lets
// a buffer be written again, in round k + 2 after round k.  A CTA that has gathered
// round k + 2's vectors has them from clusters that are through round k + 1; the CTAs
// of one such cluster have, between them, gathered round k + 1's vectors of every CTA;
// and an owner publishes those only after its rows of round k have landed.  One
// buffer would not do: for round k + 1's vectors the same argument gives the rows of
// round k - 1 only.  The second one takes 9 KB at 32 padded rows and four splits, 18
// KB at 64 and 21 KB in the two-layer kernel.
template <int BP>
__device__ __forceinline__ void push_rows_bulk(uint32_t acc, int half, int npiece, bool remote, uint8_t *stage_row,
                                               uint32_t dst, int unit, uint32_t bar, bool sends, uint32_t stage_part,
                                               uint32_t part_dst, uint32_t part_bar, uint32_t bytes) {
    constexpr int CH = BP / 2 < 32 ? BP / 2 : 32;
#pragma unroll
    for (int c0 = 0; c0 < BP / 2; c0 += CH) {
        const int col = half * (BP / 2) + c0;
        uint32_t r[CH];
        if constexpr (CH == 16)
            tmem_ld16(acc + static_cast<uint32_t>(col), r);
        else
            tmem_ld32(acc + static_cast<uint32_t>(col), r);
        tmem_ld_wait(r);
#pragma unroll
        for (int c = 0; c < CH / 4; ++c) {
            const uint32_t off = static_cast<uint32_t>(((c0 / 4 + c) ^ recv_swizzle<BP>(unit)) << 4);
            if (remote)
                *reinterpret_cast<uint4 *>(stage_row + off) = make_uint4(r[4 * c], r[4 * c + 1], r[4 * c + 2], r[4 * c + 3]);
            else if (col / 4 + c < npiece)
                st_async_f4(dst + off,
                            make_float4(__uint_as_float(r[4 * c]), __uint_as_float(r[4 * c + 1]),
                                        __uint_as_float(r[4 * c + 2]), __uint_as_float(r[4 * c + 3])),
                            bar);
        }
    }
    tc_fence_before();
    fence_proxy_async_smem();
    __syncwarp();
    if (sends) bulk_copy_cluster(part_dst, stage_part, bytes, part_bar);
    __syncwarp();
}

// Stores 16-byte pieces [c0, c1) (c1 - c0 a multiple of 4) of a weight row's K
// range from k0 on into this thread's TMEM lane, 4 columns a piece: zeros past
// K and where row is null.  The whole warp calls it.
__device__ __forceinline__ void tmem_load_row(uint32_t taddr, const uint16_t *row, int k0, int K, int c0, int c1) {
    for (int c = c0; c < c1; c += 4) {
        uint4 v[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const int k = k0 + (c + i) * 8;
            v[i] = row != nullptr && k < K ? __ldg(reinterpret_cast<const uint4 *>(row + k)) : make_uint4(0u, 0u, 0u, 0u);
        }
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const uint32_t q[4] = {v[i].x, v[i].y, v[i].z, v[i].w};
            tmem_st4(taddr + static_cast<uint32_t>((c + i) * 4), q);
        }
    }
}

}  // namespace isam
