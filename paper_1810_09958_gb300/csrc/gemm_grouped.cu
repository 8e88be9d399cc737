// gemm_grouped.cu -- many independent GEMMs in one persistent tcgen05 launch.
//
// The tiles of every problem form one list that the persistent CTAs walk
// round-robin (problems ordered by decreasing tile cost on the host), so the
// SMs stream the operands of several problems at once and the per-launch costs
// -- pipeline fill to the first data, the last tile's epilogue, the gap
// between kernels -- are paid once for the whole group instead of once per
// problem.  This is the paper's scheduler placing compute tiles across compute
// units (Sections 3.3-3.4) applied across a set of matrix multiplications.
//
// Per CTA: warp 0 TMA producer, warp 1 single-thread tcgen05.mma issuer into a
// double-buffered TMEM accumulator, warps 2 on epilogue storing C straight
// from TMEM (16-byte stores, or single floats when a row of C is not 16-byte
// aligned).  Layout (NN/TN/NT/TT) and tile width are per problem; a problem's
// tensor maps travel in the kernel parameters.
#include <algorithm>
#include <cstdlib>
#include <cstdio>
#include <cstring>
#include <memory>
#include <mutex>
#include <numeric>

#include "gemm_common.cuh"
#include "internal.h"
#include "ptx.cuh"

namespace isam {

namespace {

constexpr int kBM = 128;
constexpr int kBK = 64;
// Epilogue warps: one per TMEM lane quarter where the epilogue hides behind the
// next tile's main loop (two on alternate chunks cost the skinny sweep 0.6% and its
// E4M3 form 2%), two where a split tile's exchange is exposed
// (mixed groups in clusters: 31.2 -> 30.1 us, 25.5 -> 23.9, 33.8 -> 31.9).
__host__ __device__ constexpr int epi_warps(int log_split) { return log_split > 0 ? 8 : 4; }
constexpr int kThreads = (2 + epi_warps(1)) * 32;
constexpr int kMaxGroup = 64;
constexpr int kBNMax = 128;
constexpr int kAStage = kBM * kBK * 2;      // 16 KB
constexpr int kBStage = kBNMax * kBK * 2;   // 16 KB (either B layout at BN = 128)

enum : uint32_t {
    SITE_G_EMPTY = 0x401,
    SITE_G_TEMPTY = 0x402,
    SITE_G_FULL = 0x403,
    SITE_G_TFULL = 0x404,
    SITE_G_DONE = 0x406,
};

struct GroupProblem {
    int M, N, K;
    int m_tiles, n_tiles, kb_total;
    int a_mn, b_mn, bn;
    int panels;       // 128-row A panels per tile: 1, or 2 (256-row tiles for the heavy problems)
    int fp8;          // E4M3 operands (both K-major): 128-element K atoms
    int tile_start;   // first global tile index of this problem
    float alpha, beta;
    float *C;
};

constexpr int kMaxListed = 768;  // tiles of a group that travels with a tile list
constexpr int kMaxListCtas = 192;

struct GroupParams {
    int count, total_tiles, stages;
    int log_split;  // log2 of the CTAs (one cluster) that share each tile along K; then one tile per cluster
    int recv_bytes; // shared memory for the slices of a split tile
    int listed;  // 1: CTA i runs tiles list[first[i]] .. list[first[i + 1] - 1], else i, i + gridDim.x, ...
    unsigned long long timeout_ns;
    uint32_t *err;
    GroupProblem prob[kMaxGroup];
    CUtensorMap tmA[kMaxGroup];
    CUtensorMap tmB[kMaxGroup];
    uint16_t first[kMaxListCtas + 1];
    uint16_t list[kMaxListed];
};
static_assert(sizeof(GroupParams) <= 32764, "kernel parameters exceed 32764 bytes");

// The i-th tile of this CTA, -1 past the last.
__device__ __forceinline__ int cta_tile(const GroupParams &p, int i) {
    if (p.log_split > 0) return i == 0 ? static_cast<int>(blockIdx.x) >> p.log_split : -1;
    if (p.listed) {
        const int at = p.first[blockIdx.x] + i;
        return at < p.first[blockIdx.x + 1] ? p.list[at] : -1;
    }
    const int tile = static_cast<int>(blockIdx.x + i * gridDim.x);
    return tile < p.total_tiles ? tile : -1;
}

// 32 columns of a row of C that starts at any 4-byte boundary: `shift` single
// floats up to the next 16-byte boundary, then 16-byte pieces of the row moved
// down by as many.  (A float at a time, every store of a warp went to 32 rows:
// E4M3 group of 9, widths 10 to 255, 31.7 us against 20.9 at aligned widths.)
__device__ __forceinline__ void store_unaligned(float *dst, const uint32_t (&r)[32], int left, float alpha, float beta) {
    const int shift = static_cast<int>((16u - (static_cast<uint32_t>(reinterpret_cast<uintptr_t>(dst)) & 15u)) & 15u) >> 2;
    float v[36];
#pragma unroll
    for (int i = 0; i < 32; ++i) v[i] = alpha * __uint_as_float(r[i]);
    v[32] = v[33] = v[34] = v[35] = 0.0f;
#pragma unroll
    for (int i = 0; i < 3; ++i)
        if (i < shift && i < left) dst[i] = beta != 0.0f ? v[i] + beta * dst[i] : v[i];
    if (shift & 1)
#pragma unroll
        for (int i = 0; i < 35; ++i) v[i] = v[i + 1];
    if (shift & 2)
#pragma unroll
        for (int i = 0; i < 34; ++i) v[i] = v[i + 2];
    dst += shift;
    left = min(left, 32) - shift;
#pragma unroll
    for (int ch = 0; ch < 8; ++ch) {
        if (4 * ch + 4 <= left) {
            float4 *q = reinterpret_cast<float4 *>(dst + 4 * ch);
            float4 o = make_float4(v[4 * ch], v[4 * ch + 1], v[4 * ch + 2], v[4 * ch + 3]);
            if (beta != 0.0f) {
                const float4 cv = *q;
                o.x += beta * cv.x;
                o.y += beta * cv.y;
                o.z += beta * cv.z;
                o.w += beta * cv.w;
            }
            *q = o;
        } else {
#pragma unroll
            for (int e = 0; e < 4; ++e)
                if (4 * ch + e < left) dst[4 * ch + e] = beta != 0.0f ? v[4 * ch + e] + beta * dst[4 * ch + e] : v[4 * ch + e];
        }
    }
}

// The problem that owns `tile`, searched forward from `i` (a CTA visits its
// tiles in increasing order, listed or not, so each role keeps its index and the search
// advances by at most a few entries per tile instead of rescanning the table
// in parameter space).  Each role then copies the problem's fields into
// registers for the tile: through a reference the fields are read again from
// parameter space after every inline-asm statement with a memory clobber
// (each TMA, MMA and barrier operation), on the issue path of every k-block
// -- the copy made the sweep 3.5% faster.
__device__ __forceinline__ int find_problem(const GroupParams &p, int tile, int i) {
    while (i + 1 < p.count && p.prob[i + 1].tile_start <= tile) ++i;
    return i;
}

// Groups of few tiles, or with a few long ones, split every tile along K over the
// CTAs of a cluster, which run one tile and leave (see split_rule).
__global__ void __launch_bounds__(kThreads, 1) gemm_group_kernel(const __grid_constant__ GroupParams p) {
    const int ls = p.log_split;
    if (ls > 0 && !launch_shape_ok(p.err, 1u << ls, gridDim.x, 0x4F0u)) return;
    extern __shared__ uint8_t smem_raw[];
    uint8_t *smem = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) &
                                                ~static_cast<uintptr_t>(1023));
    const int ST = p.stages;
    uint8_t *sA = smem;
    uint8_t *sB = smem + static_cast<size_t>(ST) * kAStage;
    uint8_t *recv = sB + static_cast<size_t>(ST) * kBStage;
    uint64_t *bars = reinterpret_cast<uint64_t *>(recv + p.recv_bytes);
    uint64_t *full = bars;
    uint64_t *empty = bars + ST;
    uint64_t *tfull = empty + ST;
    uint64_t *tempty = tfull + 2;
    uint64_t *done = tempty + 2;
    uint64_t *red_full = done + 1;  // a split tile's slices have arrived
    uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(red_full + 1);
    volatile int *abort_flag = reinterpret_cast<volatile int *>(tmem_slot + 1);

    const int warp = threadIdx.x >> 5;
    const int lane = threadIdx.x & 31;
    constexpr uint32_t kTmemCols = 4 * kBNMax;  // two accumulators of two 128-row panels

    if (threadIdx.x == 0) {
        for (int i = 0; i < ST; ++i) {
            mbar_init(&full[i], 1);
            mbar_init(&empty[i], 1);
        }
        for (int i = 0; i < 2; ++i) {
            mbar_init(&tfull[i], 1);
            mbar_init(&tempty[i], epi_warps(ls));
        }
        mbar_init(done, epi_warps(ls));
        mbar_init(red_full, 1);
        *abort_flag = 0;
        fence_mbar_init();
    }
    __syncwarp();
    if (warp == 1) {
        tmem_alloc(tmem_slot, kTmemCols);
        tmem_relinquish();
    }
    tc_fence_before();
    __syncthreads();
    if (ls > 0) cluster_sync_all();
    tc_fence_after();
    const uint32_t tmem_base = *tmem_slot;
    const WaitCtx w{p.timeout_ns, p.err, abort_flag};
    // The previous kernel's results are complete from here on.
    griddep_launch_dependents();
    __syncwarp();
    griddep_wait();
    const uint32_t rank = ls > 0 ? cluster_ctarank() : 0u;
    bool arrived = false;  // at the cluster barrier before the exit
    // K atoms of a tile that this CTA multiplies.
    auto kb_from = [&](int kb_total) { return static_cast<int>((static_cast<long long>(rank) * kb_total) >> ls); };
    auto kb_to = [&](int kb_total) { return static_cast<int>((static_cast<long long>(rank + 1) * kb_total) >> ls); };

    if (warp == 0) {
        // ------------------------------------------------ TMA producer
        if (elect_one()) {
            int stage = 0, issued = 0, pi = 0;
            uint32_t phase = 0;
            bool ok = true;
            for (int n = 0, tile; ok && (tile = cta_tile(p, n)) >= 0; ++n) {
                pi = find_problem(p, tile, pi);
                const GroupProblem pr = p.prob[pi];  // a copy, see find_problem
                const int local = tile - pr.tile_start;
                const int mt = local % pr.m_tiles, nt = local / pr.m_tiles;
                const int panels = pr.panels;
                const uint32_t bbytes = pr.b_mn ? static_cast<uint32_t>((pr.bn + 63) / 64) * 8192u
                                                : static_cast<uint32_t>(pr.bn) * 128u;
                if (panels == 1) {
                    const int kb1 = kb_to(pr.kb_total);
                    for (int kb = kb_from(pr.kb_total); kb < kb1; ++kb) {
                        if (!bounded_wait(&empty[stage], phase ^ 1u, w, SITE_G_EMPTY)) {
                            ok = false;
                            break;
                        }
                        mbar_arrive_expect_tx(&full[stage], static_cast<uint32_t>(kAStage) + bbytes);
                        uint8_t *a = sA + static_cast<size_t>(stage) * kAStage;
                        uint8_t *b = sB + static_cast<size_t>(stage) * kBStage;
                        const int k0 = kb * (pr.fp8 ? 2 * kBK : kBK);  // in elements
                        if (pr.a_mn) {
                            tma_load_2d(&p.tmA[pi], &full[stage], a, mt * kBM, k0);
                            tma_load_2d(&p.tmA[pi], &full[stage], a + 8192, mt * kBM + 64, k0);
                        } else {
                            tma_load_2d(&p.tmA[pi], &full[stage], a, k0, mt * kBM);
                        }
                        if (pr.b_mn) {
                            for (int c = 0; c < (pr.bn + 63) / 64; ++c)
                                tma_load_2d(&p.tmB[pi], &full[stage], b + c * 8192, nt * pr.bn + c * 64, k0);
                        } else {
                            tma_load_2d(&p.tmB[pi], &full[stage], b, k0, nt * pr.bn);
                        }
                        ++issued;
                        if (++stage == ST) {
                            stage = 0;
                            phase ^= 1u;
                        }
                    }
                    continue;
                }
                // A k-block of a 256-row tile takes two consecutive stages:
                // panel 0 and the B block in the first, panel 1 in the second.
                const int r0 = mt * 2 * kBM, r1 = r0 + kBM;
                for (int kb = 0; kb < pr.kb_total; ++kb) {
                    const int k0 = kb * (pr.fp8 ? 2 * kBK : kBK);  // in elements
                    if (!bounded_wait(&empty[stage], phase ^ 1u, w, SITE_G_EMPTY)) {
                        ok = false;
                        break;
                    }
                    mbar_arrive_expect_tx(&full[stage], static_cast<uint32_t>(kAStage) + bbytes);
                    uint8_t *a = sA + static_cast<size_t>(stage) * kAStage;
                    uint8_t *b = sB + static_cast<size_t>(stage) * kBStage;
                    if (pr.a_mn) {
                        tma_load_2d(&p.tmA[pi], &full[stage], a, r0, k0);
                        tma_load_2d(&p.tmA[pi], &full[stage], a + 8192, r0 + 64, k0);
                    } else {
                        tma_load_2d(&p.tmA[pi], &full[stage], a, k0, r0);
                    }
                    if (pr.b_mn) {
                        for (int c = 0; c < (pr.bn + 63) / 64; ++c)
                            tma_load_2d(&p.tmB[pi], &full[stage], b + c * 8192, nt * pr.bn + c * 64, k0);
                    } else {
                        tma_load_2d(&p.tmB[pi], &full[stage], b, k0, nt * pr.bn);
                    }
                    ++issued;
                    if (++stage == ST) {
                        stage = 0;
                        phase ^= 1u;
                    }
                    if (!bounded_wait(&empty[stage], phase ^ 1u, w, SITE_G_EMPTY)) {
                        ok = false;
                        break;
                    }
                    mbar_arrive_expect_tx(&full[stage], static_cast<uint32_t>(kAStage));
                    a = sA + static_cast<size_t>(stage) * kAStage;
                    if (pr.a_mn) {
                        tma_load_2d(&p.tmA[pi], &full[stage], a, r1, k0);
                        tma_load_2d(&p.tmA[pi], &full[stage], a + 8192, r1 + 64, k0);
                    } else {
                        tma_load_2d(&p.tmA[pi], &full[stage], a, k0, r1);
                    }
                    ++issued;
                    if (++stage == ST) {
                        stage = 0;
                        phase ^= 1u;
                    }
                }
            }
            if (!ok) {
                const int pending = min(issued, ST);
                int s = stage;
                uint32_t ph = phase;
                for (int i = 0; i < pending; ++i) {
                    if (--s < 0) {
                        s = ST - 1;
                        ph ^= 1u;
                    }
                    drain_wait(&full[s], ph, p.timeout_ns);
                }
            }
        }
        __syncwarp();
    } else if (warp == 1) {
        // ------------------------------------------------ MMA issuer
        if (elect_one()) {
            int stage = 0, acc = 0, pi = 0;
            uint32_t phase = 0, acc_phase = 0;
            bool ok = true;
            for (int n = 0, tile; ok && (tile = cta_tile(p, n)) >= 0; ++n) {
                pi = find_problem(p, tile, pi);
                const GroupProblem pr = p.prob[pi];  // a copy, see find_problem
                const bool f8 = pr.fp8 != 0;
                const uint32_t idesc =
                    f8 ? idesc_e4m3_f32(kBM, pr.bn) : idesc_bf16_f32(kBM, pr.bn, pr.a_mn != 0, pr.b_mn != 0);
                if (!bounded_wait(&tempty[acc], acc_phase ^ 1u, w, SITE_G_TEMPTY)) break;
                tc_fence_after();
                const uint32_t d = tmem_base + static_cast<uint32_t>(acc * 2 * kBNMax);
                if (pr.panels == 1) {
                    const int kb0 = kb_from(pr.kb_total), kb1 = kb_to(pr.kb_total);
                    for (int kb = kb0; kb < kb1; ++kb) {
                        if (!bounded_wait(&full[stage], phase, w, SITE_G_FULL)) {
                            ok = false;
                            break;
                        }
                        tc_fence_after();
                        const uint32_t a0 = smem_u32(sA + static_cast<size_t>(stage) * kAStage);
                        const uint32_t b0 = smem_u32(sB + static_cast<size_t>(stage) * kBStage);
#pragma unroll
                        for (int k = 0; k < kBK / 16; ++k) {
                            const uint64_t ad = pr.a_mn ? sdesc_sw128(a0 + k * 2048, 8192, 1024)
                                                        : sdesc_sw128(a0 + k * 32, 16, 1024);
                            const uint64_t bd = pr.b_mn ? sdesc_sw128(b0 + k * 2048, 8192, 1024)
                                                        : sdesc_sw128(b0 + k * 32, 16, 1024);
                            if (f8)
                                umma_f8(d, ad, bd, idesc, (kb > kb0 || k > 0) ? 1u : 0u);
                            else
                                umma_bf16(d, ad, bd, idesc, (kb > kb0 || k > 0) ? 1u : 0u);
                        }
                        umma_commit(&empty[stage]);
                        if (++stage == ST) {
                            stage = 0;
                            phase ^= 1u;
                        }
                    }
                } else {
                    // 256-row tile: each k-block spans two stages, panel 0
                    // with the B block, then panel 1; both panels multiply
                    // the first stage's B, so both stages are freed after
                    // the k-block's last MMA.
                    for (int kb = 0; kb < pr.kb_total; ++kb) {
                        const int s0 = stage;
                        if (!bounded_wait(&full[s0], phase, w, SITE_G_FULL)) {
                            ok = false;
                            break;
                        }
                        if (++stage == ST) {
                            stage = 0;
                            phase ^= 1u;
                        }
                        tc_fence_after();
                        const uint32_t a0 = smem_u32(sA + static_cast<size_t>(s0) * kAStage);
                        const uint32_t b0 = smem_u32(sB + static_cast<size_t>(s0) * kBStage);
#pragma unroll
                        for (int k = 0; k < kBK / 16; ++k) {
                            const uint64_t ad = pr.a_mn ? sdesc_sw128(a0 + k * 2048, 8192, 1024)
                                                        : sdesc_sw128(a0 + k * 32, 16, 1024);
                            const uint64_t bd = pr.b_mn ? sdesc_sw128(b0 + k * 2048, 8192, 1024)
                                                        : sdesc_sw128(b0 + k * 32, 16, 1024);
                            if (f8)
                                umma_f8(d, ad, bd, idesc, (kb > 0 || k > 0) ? 1u : 0u);
                            else
                                umma_bf16(d, ad, bd, idesc, (kb > 0 || k > 0) ? 1u : 0u);
                        }
                        const int s1 = stage;
                        if (!bounded_wait(&full[s1], phase, w, SITE_G_FULL)) {
                            ok = false;
                            break;
                        }
                        if (++stage == ST) {
                            stage = 0;
                            phase ^= 1u;
                        }
                        tc_fence_after();
                        const uint32_t a1 = smem_u32(sA + static_cast<size_t>(s1) * kAStage);
#pragma unroll
                        for (int k = 0; k < kBK / 16; ++k) {
                            const uint64_t ad = pr.a_mn ? sdesc_sw128(a1 + k * 2048, 8192, 1024)
                                                        : sdesc_sw128(a1 + k * 32, 16, 1024);
                            const uint64_t bd = pr.b_mn ? sdesc_sw128(b0 + k * 2048, 8192, 1024)
                                                        : sdesc_sw128(b0 + k * 32, 16, 1024);
                            if (f8)
                                umma_f8(d + kBNMax, ad, bd, idesc, (kb > 0 || k > 0) ? 1u : 0u);
                            else
                                umma_bf16(d + kBNMax, ad, bd, idesc, (kb > 0 || k > 0) ? 1u : 0u);
                        }
                        umma_commit(&empty[s0]);
                        umma_commit(&empty[s1]);
                    }
                }
                if (!ok) break;
                umma_commit(&tfull[acc]);
                if (++acc == 2) {
                    acc = 0;
                    acc_phase ^= 1u;
                }
            }
        }
        __syncwarp();
    } else {
        // ------------------------------------------------ epilogue (warps 2-5, 2-9 in a cluster)
        const int ew = warp - 2;
        const int q = warp & 3;
        // Straight from TMEM to C: lane i holds row i of the warp's 32 rows,
        // 32 consecutive columns per TMEM load, stored as 16-byte pieces (or
        // single floats where C's rows are not 16-byte aligned).  No staging
        // buffer: the 32 KB it took is a seventh ring stage, and the
        // epilogue, which overlaps the next tile's main loop through the
        // second accumulator, has time for the scattered stores.
        int acc = 0, pi = 0;
        uint32_t acc_phase = 0;
        for (int n = 0, tile; (tile = cta_tile(p, n)) >= 0; ++n) {
            pi = find_problem(p, tile, pi);
            const GroupProblem pr = p.prob[pi];  // a copy, see find_problem
            const int local = tile - pr.tile_start;
            const int mt = local % pr.m_tiles, nt = local / pr.m_tiles;
            const int col0 = nt * pr.bn;
            const int nch = (pr.bn + 31) / 32;
            const bool vec = (pr.N & 3) == 0;
            if (!warp_wait(&tfull[acc], acc_phase, w, SITE_G_TFULL)) break;
            tc_fence_after();
            if (ls > 0) {
                // The ring's copies and products are done: it stages the tile.
                const int cw = chunk_cols(pr.bn), chunks = cw == 32 ? nch : 1;
                const bool none = kb_from(pr.kb_total) == kb_to(pr.kb_total);  // fewer K atoms than CTAs
                const uint32_t tb = tmem_base + (static_cast<uint32_t>(q * 32) << 16);
                if (ew == 0 && lane == 0) mbar_arrive_expect_tx(red_full, static_cast<uint32_t>(partial_bytes(pr.bn)));
                __syncwarp();
                split_push(smem, recv, red_full, q, lane, rank, ls, cw, chunks, [&](int col, uint32_t(&r)[32]) {
                    tmem_ld32(tb + col, r);
                    tmem_ld_wait(r);
                    if (none)
#pragma unroll
                        for (int i = 0; i < 32; ++i) r[i] = 0u;
                }, ew >> 2, 2);
                const bool got = warp_wait<true>(red_full, 0, w, SITE_G_TFULL);
                // No peer writes into this CTA any more; its own copies have been
                // read once every peer is here too.
                cluster_arrive_relaxed();
                arrived = true;
                if (got)
                    split_sum(recv, ew * 32 + lane, epi_warps(1) * 32, ls, cw, chunks, mt * kBM + (static_cast<int>(rank) << (7 - ls)), pr.M,
                              pr.N, col0, min(pr.N - col0, pr.bn), pr.alpha, pr.beta, nullptr, pr.C);
                __syncwarp();
                break;  // the cluster's only tile
            }
            for (int pn = 0; pn < pr.panels; ++pn) {
                const int grow = (mt * pr.panels + pn) * kBM + q * 32 + lane;
                const uint32_t tbase = tmem_base + (static_cast<uint32_t>(q * 32) << 16) +
                                       static_cast<uint32_t>(acc * 2 * kBNMax + pn * kBNMax);
                for (int j = 0; j < nch; ++j) {
                    uint32_t r[32];
                    tmem_ld32(tbase + j * 32, r);  // past bn: columns of the panel's own region
                    tmem_ld_wait(r);
                    if (grow < pr.M) {
                        float *crow = pr.C + static_cast<size_t>(grow) * pr.N;
                        const int cbase = col0 + j * 32;
                        const int left = min(pr.N, col0 + pr.bn) - cbase;  // columns of this chunk inside C
                        if (vec) {
#pragma unroll
                            for (int ch = 0; ch < 8; ++ch) {
                                if (4 * ch >= left) break;
                                float v[4];
#pragma unroll
                                for (int e = 0; e < 4; ++e) v[e] = pr.alpha * __uint_as_float(r[4 * ch + e]);
                                float4 *dst = reinterpret_cast<float4 *>(crow + cbase + 4 * ch);
                                if (pr.beta != 0.0f) {
                                    const float4 cv = *dst;
                                    v[0] += pr.beta * cv.x;
                                    v[1] += pr.beta * cv.y;
                                    v[2] += pr.beta * cv.z;
                                    v[3] += pr.beta * cv.w;
                                }
                                *dst = make_float4(v[0], v[1], v[2], v[3]);
                            }
                        } else {
                            store_unaligned(crow + cbase, r, left, pr.alpha, pr.beta);
                        }
                    }
                    __syncwarp();  // joined again before the next aligned tcgen05.ld
                }
            }
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(&tempty[acc]);
            __syncwarp();
            if (++acc == 2) {
                acc = 0;
                acc_phase ^= 1u;
            }
        }
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(done);
        __syncwarp();
    }

    if (ls > 0) {
        // Every CTA gets here, since every wait above is bounded.
        if (*abort_flag) {
            // After an abort, rows a peer sent may still be on their way.
            const unsigned long long t0 = globaltimer();
            while (globaltimer() - t0 < 50000ull) {
            }
        }
        __syncwarp();
        if (!arrived) cluster_arrive_relaxed();
        cluster_wait();
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 1) {
        bounded_wait(done, 0, w, SITE_G_DONE);
        __syncwarp();
        tc_fence_after();
        tmem_dealloc(tmem_base, kTmemCols);
    }
}

size_t group_smem_bytes(int stages, int recv_bytes) {
    return 1024 + static_cast<size_t>(stages) * (kAStage + kBStage) + static_cast<size_t>(recv_bytes) +
           (2 * stages + 6) * 8 + 16;
}

std::mutex g_group_mu;

// Operand microseconds of a K atom of a problem's tile on one SM.
float atom_us(const GroupProblem &pr) {
    const int b = pr.b_mn ? (pr.bn + 63) / 64 * 8192 : pr.bn * 128;
    return (pr.panels * kAStage + b) / 86350.0f;
}

// Gives each tile (costliest problems first) to the worker that is free first;
// returns when the last one ends.  cost: per problem; workers <= kMaxListCtas.
float share_out(const GroupParams &p, int workers, const float *cost, uint16_t *owner) {
    struct Slot {
        float end;
        int worker;
    };
    auto later = [](const Slot &a, const Slot &b) { return a.end > b.end; };
    Slot heap[kMaxListCtas];
    const int n = std::min(workers, p.total_tiles);
    for (int t = 0, i = 0; t < p.total_tiles; ++t) {
        while (i + 1 < p.count && p.prob[i + 1].tile_start <= t) ++i;
        if (t < n) {
            heap[t] = Slot{cost[i], t};
            if (owner) owner[t] = static_cast<uint16_t>(t);
            if (t + 1 == n) std::make_heap(heap, heap + n, later);
        } else {
            std::pop_heap(heap, heap + n, later);
            if (owner) owner[t] = static_cast<uint16_t>(heap[n - 1].worker);
            heap[n - 1].end += cost[i];
            std::push_heap(heap, heap + n, later);
        }
    }
    float longest = 0.0f;
    for (int i = 0; i < n; ++i) longest = std::max(longest, heap[i].end);
    return longest;
}

// Chooses how the tiles run: round-robin walk, tile list, or clusters that split
// each tile along K.
//
// The list gives each tile to the CTA that is free first, where that ends at
// least 3% before the walk.  A group of unlike problems otherwise hands the CTAs
// that hold the longest K as many further tiles as the others: 18 problems with K
// from 72 to 6424 62.2 -> 55.5 us, 16 with K from 112 to 5656 34.8 -> 27.4, the
// benchmark's bf16 sweep (K from 1760 to 4096) 126.8 -> 124.8; its E4M3 form takes
// 38.6 either way.
//
// A split (by 2, 4 or 8, where the device holds that many clusters) shortens the
// longest tile but costs each one an exchange and a new CTA, so it pays where
// tiles are few or a long K stands out: groups of 4 and 6 with K to 7758 30.4 -> 16.0
// and 32.5 -> 13.1 us, E4M3 group of 3 with K to 7520 21.2 -> 8.6.  (Over 24 drawn
// groups the geometric mean is 25.2 us without it, 23.0 with 0.5 to 1.5 us for a new
// CTA, 24.0 with 2.7.)  Above two tiles per SM it is not tried.
//
// ISAM_GROUP_ROUTE=walk, list, 2, 4 or 8 (CTAs that split a tile) forces one of them
// where the group allows it, for tests and measurements.
void split_rule(GroupParams &p, int grid, const DeviceState &ds) {
    p.listed = 0;
    p.log_split = 0;
    if (p.total_tiles > kMaxListed || grid > kMaxListCtas) return;
    const char *force = getenv("ISAM_GROUP_ROUTE");
    if (force && strcmp(force, "walk") == 0) return;
    float cost[kMaxGroup], walk[kMaxListCtas] = {};
    uint16_t owner[kMaxListed];
    bool tall = false;
    for (int i = 0; i < p.count; ++i) {
        cost[i] = p.prob[i].kb_total * atom_us(p.prob[i]) + 0.6f;
        tall = tall || p.prob[i].panels > 1;
    }
    for (int t = 0, i = 0; t < p.total_tiles; ++t) {
        while (i + 1 < p.count && p.prob[i + 1].tile_start <= t) ++i;
        walk[t % grid] += cost[i];
    }
    const float walked = *std::max_element(walk, walk + grid);
    float longest = share_out(p, grid, cost, owner);
    const bool list = force ? strcmp(force, "list") == 0 : longest <= 0.97f * walked;
    if (!list) longest = walked;
    if (force && !tall)
        for (int ls = 1; ls <= 3; ++ls)
            if (atoi(force) == 1 << ls && gemm_cluster_capacity(ds, 1 << ls) >= 1) p.log_split = ls;
    if (!force && !tall && p.total_tiles <= 2 * grid) {
        float best = 0.95f * (longest + 4.2f) - 4.2f;  // 4.2 us: launch, first data, last stores
        for (int ls = 1; ls <= 3; ++ls) {
            const int clusters = std::min(gemm_cluster_capacity(ds, 1 << ls), ds.num_sms >> ls);
            if (clusters < 1) continue;
            for (int i = 0; i < p.count; ++i) {
                const GroupProblem &pr = p.prob[i];
                cost[i] = ((pr.kb_total + (1 << ls) - 1) >> ls) * atom_us(pr) + 1.4f + 0.0176f * pr.bn +
                          0.054f * pr.bn / (1 << ls) + 1.0f;
            }
            const float us = share_out(p, clusters, cost, nullptr);
            if (us < best) {
                best = us;
                p.log_split = ls;
            }
        }
    }
    if (p.log_split > 0 || !list) return;
    p.listed = 1;
    uint16_t count[kMaxListCtas] = {}, at[kMaxListCtas];
    for (int t = 0; t < p.total_tiles; ++t) ++count[owner[t]];
    p.first[0] = 0;
    for (int c = 0; c < grid; ++c) p.first[c + 1] = static_cast<uint16_t>(p.first[c] + count[c]);
    std::copy(p.first, p.first + grid, at);
    for (int t = 0; t < p.total_tiles; ++t) p.list[at[owner[t]]++] = static_cast<uint16_t>(t);
}

// Fills p for a group of two or more but for its tensor maps; order[i]: the caller's
// index of problem i.  Host arithmetic only.
void group_plan(int count, const GemmDesc *g, const DeviceState &ds, GroupParams &p, int *order, int *grid_out) {
    auto atoms = [&](int i) { return (g[i].K + (g[i].fp8 ? 2 * kBK : kBK) - 1) / (g[i].fp8 ? 2 * kBK : kBK); };
    // Tile height: 256 rows (two 128-row panels sharing each B block) for
    // problems whose 128-row panel of A is 640 KB or more, which halves the
    // tile starts a CTA pays on them; kept at 128 rows when that would leave
    // fewer than two tiles per SM.
    int panels[kMaxGroup];
    {
        long long tall_tiles = 0;
        for (int i = 0; i < count; ++i) {
            const long long eb = g[i].fp8 ? 1 : 2;
            panels[i] = (g[i].M > kBM && static_cast<long long>(kBM) * g[i].K * eb >= 640 * 1024) ? 2 : 1;
            const int bn = std::min(kBNMax, (g[i].N + 15) / 16 * 16);
            tall_tiles += static_cast<long long>((g[i].M + kBM * panels[i] - 1) / (kBM * panels[i])) *
                          ((g[i].N + bn - 1) / bn);
        }
        if (tall_tiles < 2LL * ds.num_sms)
            for (int i = 0; i < count; ++i) panels[i] = 1;
        // ISAM_GROUP_PANELS=1 or 2 forces the tile height (2: every problem
        // taller than one panel), for tests and measurements.
        const char *fe = getenv("ISAM_GROUP_PANELS");
        const int forced = fe ? atoi(fe) : 0;
        if (forced == 1 || forced == 2)
            for (int i = 0; i < count; ++i) panels[i] = (forced == 2 && g[i].M > kBM) ? 2 : 1;
    }
    // Host-side order: problems with the costliest tiles first, so the
    // round-robin walk over tiles ends with the cheap ones.
    std::iota(order, order + count, 0);
    std::stable_sort(order, order + count,
                     [&](int a, int b) { return atoms(a) * panels[a] > atoms(b) * panels[b]; });

    memset(&p, 0, sizeof p);
    p.count = count;
    int tiles = 0;
    for (int s = 0; s < count; ++s) {
        const GemmDesc &d = g[order[s]];
        GroupProblem &pr = p.prob[s];
        pr.M = d.M;
        pr.N = d.N;
        pr.K = d.K;
        pr.fp8 = d.fp8;
        pr.a_mn = d.fp8 ? 0 : d.transA;
        pr.b_mn = (d.fp8 || d.transB == 1) ? 0 : 1;
        pr.bn = std::min(kBNMax, (d.N + 15) / 16 * 16);
        pr.panels = panels[order[s]];
        pr.m_tiles = (d.M + kBM * pr.panels - 1) / (kBM * pr.panels);
        pr.n_tiles = (d.N + pr.bn - 1) / pr.bn;
        pr.kb_total = atoms(order[s]);
        pr.tile_start = tiles;
        pr.alpha = d.alpha;
        pr.beta = d.beta;
        pr.C = d.C;
        tiles += pr.m_tiles * pr.n_tiles;
    }
    p.total_tiles = tiles;
    int grid = std::min(tiles, ds.num_sms);
    split_rule(p, grid, ds);
    if (p.log_split > 0) {
        grid = tiles << p.log_split;  // one tile per cluster: those that do not fit yet take turns
        for (int i = 0; i < count; ++i) p.recv_bytes = std::max(p.recv_bytes, partial_bytes(p.prob[i].bn));
    }
    int st = 8;
    while (st > 2 && group_smem_bytes(st, p.recv_bytes) > static_cast<size_t>(ds.max_smem_optin)) --st;
    p.stages = st;
    *grid_out = grid;
}

}  // namespace

int gemm_grouped_plan(int count, const GemmDesc *g, const DeviceState &ds, GroupedPlan *plan) {
    if (count == 1) {
        GemmPlan one;
        if (const int rc = gemm_plan(g[0], ds, &one)) return rc;
        *plan = GroupedPlan{one.split, 0, one.grid, one.stages};
        return ISAM_OK;
    }
    const auto p = std::make_unique<GroupParams>();
    int order[kMaxGroup], grid = 0;
    group_plan(count, g, ds, *p, order, &grid);
    *plan = GroupedPlan{1 << p->log_split, p->listed, grid, p->stages};
    return ISAM_OK;
}

int gemm_grouped_launch(int count, const GemmDesc *g, DeviceState &ds, cudaStream_t stream) {
    if (count < 1 || count > kMaxGroup)
        return set_error(ISAM_ERR_INVALID_ARG, "isam_gemm_grouped: count must be in [1, %d]", kMaxGroup);
    if (count == 1) {
        // Nothing to share the launch with: the planned tiles and split of a
        // single call.  Against this kernel, E4M3 / bf16: 384 x 128 x 4096 18.6 / 33.0
        // -> 5.9 / 7.1 us, 8192 x 256 x 8192 33.7 / 62.2 -> 25.5 / 47.1, 8192 x 8192 x
        // 1024 144 / 208 -> 75 / 98.
        GemmPlan plan;
        if (const int rc = gemm_plan(g[0], ds, &plan)) return rc;
        return gemm_launch(g[0], plan, ds, stream);
    }
    static GroupParams p;  // ~29 KB: built under the lock, copied into the launch
    std::lock_guard<std::mutex> lk(g_group_mu);
    int order[kMaxGroup], grid = 0;
    group_plan(count, g, ds, p, order, &grid);
    for (int s = 0; s < count; ++s) {
        const GemmDesc &d = g[order[s]];
        const GroupProblem &pr = p.prob[s];
        int rc;
        if (pr.fp8) {
            // 128-element (128-byte) K atoms of both K-major E4M3 operands.
            if ((rc = make_tmap_2d_u8(&p.tmA[s], d.A, d.K, d.M, static_cast<uint64_t>(d.K), 128, kBM))) return rc;
            if ((rc = make_tmap_2d_u8(&p.tmB[s], d.B, d.K, d.N, static_cast<uint64_t>(d.K), 128,
                                      static_cast<uint32_t>(pr.bn))))
                return rc;
        } else {
            if (pr.a_mn)
                rc = make_tmap_2d_bf16(&p.tmA[s], d.A, d.M, d.K, static_cast<uint64_t>(d.M) * 2, 64, 64);
            else
                rc = make_tmap_2d_bf16(&p.tmA[s], d.A, d.K, d.M, static_cast<uint64_t>(d.K) * 2, 64, kBM);
            if (rc) return rc;
            if (pr.b_mn)
                rc = make_tmap_2d_bf16(&p.tmB[s], d.B, d.N, d.K, static_cast<uint64_t>(d.N) * 2, 64, 64);
            else
                rc = make_tmap_2d_bf16(&p.tmB[s], d.B, d.K, d.N, static_cast<uint64_t>(d.K) * 2, 64,
                                       static_cast<uint32_t>(pr.bn));
            if (rc) return rc;
        }
    }
    p.timeout_ns = wait_timeout_ns();
    p.err = ds.err_word;
    const size_t smem = group_smem_bytes(p.stages, p.recv_bytes);
    if (const int rc = ensure_smem_optin(reinterpret_cast<const void *>(gemm_group_kernel), ds.max_smem_optin,
                                         ds.device, "cudaFuncSetAttribute(grouped gemm)"))
        return rc;
    cudaError_t e = launch_dependent(gemm_group_kernel, dim3(static_cast<unsigned>(grid)),
                                     (2 + epi_warps(p.log_split)) * 32, smem, stream, 1 << p.log_split, p);
    if (e != cudaSuccess) return cuda_error(e, "launch gemm_group_kernel");
    return ISAM_OK;
}

}  // namespace isam
