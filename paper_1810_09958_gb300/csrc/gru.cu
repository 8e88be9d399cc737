// gru.cu -- GRU forward over T steps on sm_103a.
//
// Recurrent scheduling after Section 3.6 of the paper: the loop body is
// scheduled once as a priming iteration (load the persistent weights and the
// initial state onto the compute units), a recursive iteration run T times
// that overwrites its own inputs, and a finish iteration (the last state is
// already in place in h_out).  The paper credits its GRU speed-up to fusion
// and to keeping reused data on chip (Section 5.1.2); here:
//
//   1. gx = x W^T + b_ih for all T steps is one GEMM (isam_gemm's kernel, bias
//      fused in its epilogue), written to a library workspace;
//   2. one persistent kernel runs the recurrence.  Hidden units are taken in
//      groups of 32; a group is a cluster of KS CTAs (KS = 4 at hidden 1024)
//      that split the reduction dimension of U h: CTA r keeps the 96 rows of U
//      for the group's r, z and n gates over its K quarter resident in tensor
//      memory for all T steps.  Per step each CTA gathers its quarter of
//      bf16(h_{t-1}) (all batch rows) from an exchange ring in global memory,
//      runs 16 tcgen05.mma (M = 128 with 96 rows used, N = 32 batch) into TMEM,
//      and pushes the partial rows of the units owned by each cluster peer
//      straight into that peer's shared memory; the owner sums the KS partials
//      in rank order, evaluates the gates in fp32 (h carried in fp32
//      registers) and publishes bf16(h_t) to the ring.  Every wait is bounded
//      in time.
#include <algorithm>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <mutex>
#include <utility>

#include <cuda_bf16.h>

#include "gru_common.cuh"
#include "internal.h"
#include "ptx.cuh"

namespace isam {

namespace {

constexpr int kGroup = 32;               // hidden units per group (one cluster)
constexpr int kRowsG = 3 * kGroup;       // 96 U rows per group (r, z, n)
constexpr int kBatchPad = 32;            // MMA N for batch <= 32 (the path with every feature)
constexpr int kBatchMax = 256;           // larger batches run in chunks of the padded width
constexpr int kGateWarps = 8;            // gather, push, gates
constexpr int kGateThreads = 32 * kGateWarps;
constexpr int kMmaWarp = 8;
constexpr int kHouseWarp = 9;            // ring and barrier upkeep; 9-11 drain a next layer's projection
constexpr int kThreads = 384;
constexpr int kAtomU = kRowsG * 128;     // one 64-wide K atom of the U slice (12 KB)
constexpr int kUPad = 32 * 128;          // the M = 128 MMA reads 32 rows past an atom
// The padded batch BP (32, 64 or 128) is the MMA's N: one K atom of h is BP
// rows of 128 bytes, and a received partial row holds BP batch values.
__host__ __device__ constexpr int atom_h_bytes(int bp) { return bp * 128; }
__host__ __device__ constexpr int recv_bytes(int bp) { return kRowsG * bp * 4; }

enum : uint32_t {
    SITE_GRU_H = 0x203,
    SITE_GRU_MMA = 0x204,
    SITE_GRU_RED = 0x205,
    SITE_GRU_W = 0x206,
};


struct GruParams {
    int T, H;
    int bstride;               // batch rows between two steps of gx / h_out (the full batch)
    int ks;                    // K splits per unit group = cluster size
    int ka;                    // 64-wide K atoms per CTA (all atoms of H, rounded up, / ks)
    int uo;                    // units whose gates one CTA evaluates (32 / ks)
    int n_cta;                 // (H / 32) * ks: CTAs of one chunk
    int chunks;                // batch chunks of this launch, bp rows each (the last may have fewer)
    int total;                 // batch rows of all of them
    const uint16_t *U;         // [3H][H] bf16 recurrent weights
    const float *gx;           // [T*bstride][3H], includes b_ih
    const float *b_hh;         // [3H]
    const float *h0;           // [total][H] or null
    float *h_out;              // [T][bstride][H]
    uint16_t *xb;              // the same states in bf16 (the next layer's GEMM input), or null
    uint16_t *hx;              // per chunk kSlots x [H/8 pieces][bp rows][8] bf16 exchange ring, kEmpty before launch
    int slot;                  // elements of one slot of the ring
    int reset_before;          // candidate's recurrent input U_n (r * h): two rounds per step
    int gx_parts;              // slabs summed into each projection value (1: gx = x W^T + b_ih)
    size_t gx_slab;            // floats between two slabs of gx
    const float *b_ih;         // [3H], added to the slab sum when gx_parts > 1 (else null)
    int has_next;              // also multiply the next layer's W by every loaded h
    float *gxp_out;            // [ks][T*batch][3H]: the next layer's projection, one slab per K rank
    int w_layer;               // the next layer's index in the tensor map of W
    // Layers that share a launch (POLL): `chunks` of them, each on its own n_cta
    // CTAs; the pointers above are the first one's (gxp_out: the last one's output).
    float *gxw;                // projections between them, [ks][T*batch][3H] each, kEmpty before launch
    size_t out_layer;          // floats between two layers of h_out
    int skip_publish_cta;      // debug: this CTA never publishes (-1: none)
    unsigned long long timeout_ns;
    uint32_t *err;
};

struct GruLayout {
    int off_w, off_h, off_recv, off_gx, off_stage, off_bars, total;
};

// Projection values a gate thread holds for one step: three gates of its
// (unit, batch) pairs, one per slab (as many slabs as K splits at bp = 32).
__host__ __device__ constexpr int gx_values(int ks, int bp) {
    return 3 * (kGroup / ks * bp / kGateThreads) * (bp == kBatchPad ? ks : 1);
}

// The partial rows of other CTAs' units that a CTA stages in a round.
__host__ __device__ constexpr int stage_bytes(int ks, int bp) { return bp < 128 ? recv_bytes(bp) / ks * (ks - 1) : 0; }

// [pad | next layer's W slice (has_next)] | h tile | 2 x partial rows |
// 2 x projection values of a step | kGruStages x staged partial rows |
// barriers.  The pad: W's product starts 32 rows
// before each atom.
__host__ __device__ inline GruLayout gru_layout(int ks, int ka, bool has_next, int bp = kBatchPad) {
    GruLayout L;
    L.off_w = kUPad;
    L.off_h = has_next ? kUPad + ka * kAtomU : 0;
    L.off_recv = L.off_h + ka * atom_h_bytes(bp);
    L.off_gx = L.off_recv + 2 * recv_bytes(bp);
    L.off_stage = L.off_gx + 2 * gx_values(ks, bp) * kGateThreads * 4;
    L.off_bars = L.off_stage + kGruStages * stage_bytes(ks, bp);
    L.total = L.off_bars + 192 + 1024;
    return L;
}

// Template arguments: KS, the K splits per unit group (cluster size, 4, 2 or
// 1), and BP, the padded batch (the MMA's N: 32, 64 or 128).  A CTA evaluates
// the gates of UO = 32 / KS units over BP batch rows, NP = UO * BP / 256
// (unit, batch) pairs per gate thread.  The next layer's product and the
// K-rank projection slabs exist for BP = 32 only.
//
// A round is one exchange of the recurrence: every CTA gathers its K range of
// the round's vectors (h_{t-1}, or r * h_{t-1} in the second round of a
// reset-before step), multiplies, reduces over the cluster, evaluates its
// gates and publishes its units' new vectors.  What bounds it is the chain of
// cross-SM latencies, so the exchange carries no flag: the ring's words hold
// kEmpty until their producer stores them, and the gather polls the data
// itself with plain 16-byte loads straight into registers and on into the
// MMA's swizzled shared-memory layout.  A published word is then visible one
// store plus one load later; a release, a counter, its poll and a TMA load
// (the exchange this replaced) were four such latencies one after another.
// Hidden 1024, batch 32: 609 -> 332 us for 128 steps, 2.5 us for one more; hidden
// 480, batch 5: 100 -> 51 us for 20 steps, 2.0 for one more.  Of the 2.5 us about
// 0.8 is the exchange, 0.3 the products, 0.5 push and reduction, 0.3 the gates; the
// rest has not been attributed.
//
// The ring is [piece of 8 units][batch row]: a CTA's words fill whole lines that
// no other CTA writes.  With the rows of 64 units interleaved (8 CTAs writing
// each line, 32 polling it) a step took 3.8 us.
//
//   warps 0-7   gather, push of the partial rows (6 of them), gates, publish;
//   warp 8      issues the MMAs once the tile has arrived;
//   warp 9      returns this CTA's words of an old slot to kEmpty and arms the
//               partial-row barrier; with a next layer, warps 9-11 drain its
//               projection from TMEM lanes 32-127.
//
// Ring reuse: round k reads slot k % 4, publishes to slot (k + 1) % 4 and
// empties slot (k + 3) % 4.  When a CTA has its round-k partial rows, its
// cluster has gathered round k's vectors from every CTA, so every CTA has
// finished gathering round k - 1's: that slot's words may be emptied.  The
// emptied words are performed (fence) before warp 9 arms round k + 1's
// barrier, on which this CTA's round k + 1 publication waits, and no CTA polls
// the slot again (round k + 3) before it has seen that publication.
//
// POLL: consecutive layers of a stack in one launch, each a step or two behind
// the one below: the words of a layer's projection slabs are kEmpty until the
// layer below stores them, and the gates poll those that their copy to shared
// memory found empty.  A stack then takes about T + 2 (layers - 1) steps instead
// of T times its layers: 39 reset-before steps of 3 layers at hidden 352, batch 4,
// 560 -> 217 us; 60 steps of 3 layers at hidden 96, batch 32, 506 -> 207; 20 steps of
// 2 layers at hidden 480, batch 5, 102 -> 66 (the next layer's projection alone was
// already overlapped before).
template <int KS, int BP, bool POLL = false>
__global__ void __launch_bounds__(kThreads, 1)
    gru_recurrent_kernel(const __grid_constant__ CUtensorMap tmWn, const GruParams p) {
    constexpr int UO = kGroup / KS;
    constexpr int NP = UO * BP / kGateThreads;
    constexpr int SL = BP == kBatchPad ? KS : 1;  // projection slabs a value can sum
    constexpr int AH = atom_h_bytes(BP);
    constexpr int BSTEP = kGateThreads / UO;
    constexpr int KAMAX = BP == 128 ? 4 : 7;      // most K atoms a CTA holds (gru_atoms)
    constexpr int LPA = BP / 32;                  // 16-byte loads per lane and atom
    constexpr int NL = KAMAX * LPA;
    if (!launch_shape_ok(p.err, static_cast<uint32_t>(KS), static_cast<uint32_t>(p.n_cta * p.chunks), 0x3F0u))
        return;
    // This CTA's chunk of the batch: independent sequences, which share nothing
    // with the other chunks of the launch but the weights.
    const int chunk = static_cast<int>(blockIdx.x) / p.n_cta;
    const int cta = static_cast<int>(blockIdx.x) - chunk * p.n_cta;
    const int layer = POLL ? chunk : 0;  // of this launch
    const int b0 = POLL ? 0 : chunk * BP;
    const int batch = min(BP, p.total - b0);
    const size_t set = static_cast<size_t>(KS) * p.gx_slab;  // one layer's slabs
    const float *const gx =
        POLL && layer > 0 ? p.gxw + (layer - 1) * set : p.gx + static_cast<size_t>(b0) * 3 * p.H;
    const int gx_parts = POLL && layer > 0 ? KS : p.gx_parts;
    const size_t h_base = POLL ? static_cast<size_t>(layer) * p.total * p.H : static_cast<size_t>(b0) * p.H;
    const float *const h0 = p.h0 != nullptr ? p.h0 + h_base : nullptr;
    float *const h_out = p.h_out + (POLL ? layer * p.out_layer : static_cast<size_t>(b0) * p.H);
    float *const gxp_out = POLL && layer + 1 < p.chunks ? p.gxw + layer * set : p.gxp_out;
    const float *const b_hh = p.b_hh + (POLL ? layer * 6 * p.H : 0);
    const float *const b_ih = POLL && layer > 0 ? b_hh - 3 * p.H : p.b_ih;
    const uint16_t *const U = p.U + (POLL ? static_cast<size_t>(layer) * 3 * p.H * p.H : 0);
    uint16_t *const xb = p.xb != nullptr ? p.xb + static_cast<size_t>(b0) * p.H : nullptr;
    uint16_t *const hx = p.hx + static_cast<size_t>(chunk) * kSlots * p.slot;
    const bool bulk = KS > 1 && gru_push_bulk(batch, BP);
    extern __shared__ uint8_t smem_raw[];
    uint8_t *smem = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) &
                                                ~static_cast<uintptr_t>(1023));
    const bool HN = POLL ? gxp_out != nullptr : p.has_next != 0;
    const GruLayout L = gru_layout(KS, p.ka, HN, BP);
    uint8_t *sW = smem + L.off_w;
    uint8_t *sH = smem + L.off_h;
    float *recv = reinterpret_cast<float *>(smem + L.off_recv);  // [2 round parity][ks src][3 gates][2 halves][uo][BP / 2]
    uint64_t *bars = reinterpret_cast<uint64_t *>(smem + L.off_bars);
    uint64_t *wbar = bars;                   // next layer's W slice landed
    uint64_t *h_full = bars + 1;             // the round's vectors are in shared memory
    uint64_t *mma_done = h_full + 1;         // MMAs of the round complete
    uint64_t *red_full = mma_done + 1;       // [2 round parity] all partial rows of my units arrived
    uint64_t *w_done = red_full + 2;         // [2 step parity] next layer's projection MMAs complete
    uint64_t *w_free = w_done + 2;           // [2 step parity] its accumulator drained
    uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(w_free + 2);
    volatile int *abort_flag = reinterpret_cast<volatile int *>(tmem_slot + 1);

    const int tid = threadIdx.x;
    const int warp = tid >> 5;
    const int lane = tid & 31;
    const int H = p.H;
    const int G = 3 * H;
    const int ka = p.ka;
    const int group = cta / KS;
    const uint32_t rank = KS > 1 ? cluster_ctarank() : 0u;
    const int unit0 = group * kGroup;
    const int atom0 = static_cast<int>(rank) * ka;
    const WaitCtx w{p.timeout_ns, p.err, abort_flag};

    if (tid == 0) {
        mbar_init(wbar, 1);
        mbar_init(h_full, kGateWarps);
        mbar_init(mma_done, 1);
        for (int i = 0; i < 2; ++i) {
            mbar_init(&red_full[i], 1);  // armed with the bytes of a round's partial rows
            mbar_init(&w_done[i], 1);
            mbar_init(&w_free[i], 3);
        }
        *abort_flag = 0;
        fence_mbar_init();
    }
    // The h tile starts as zeros: K columns past the matrix (and batch rows
    // past the batch) are never written.
    for (int i = tid; i < ka * AH / 16; i += kThreads) reinterpret_cast<uint4 *>(sH)[i] = make_uint4(0u, 0u, 0u, 0u);
    fence_proxy_async_smem();
    __syncwarp();
    // Columns 0 .. BP - 1: the recurrent product; 32-95 (BP = 32): the next
    // layer's projection, double-buffered by step parity; from kUCol on the
    // CTA's U slice, 32 columns per K atom.
    constexpr uint32_t kUCol = BP == kBatchPad ? 96 : BP;
    const uint32_t tmem_cols = kUCol + 32 * ka <= 256 ? 256u : 512u;
    if (warp == 0) {
        tmem_alloc(tmem_slot, tmem_cols);
        tmem_relinquish();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_d = *tmem_slot;
    // The projection (and what came before it) is complete from here on.
    griddep_launch_dependents();
    __syncwarp();
    griddep_wait();
    // ---- priming: the persistent weights.  U is the A operand of every round,
    // so it lives in tensor memory: an M = 128 MMA then reads only its 1 KB of
    // h from shared memory and sixteen of them take 376 cycles, against 760
    // with the 4 KB of A from shared memory (cycles from the first issue to the
    // commit's arrival).  Lane gate * 32 + u holds U row gate * H + unit0 + u,
    // two K elements per column; warps q and q + 4 load the two halves of lane
    // quarter q.
    if (warp < kGateWarps && (warp & 3) < 3) {
        const uint16_t *urow = U + (static_cast<size_t>(warp & 3) * H + unit0 + lane) * H;
        const int half = warp >> 2;  // of the row's K range
        tmem_load_row(tmem_d + (static_cast<uint32_t>((warp & 3) * 32) << 16) + kUCol, urow, atom0 * 64, H,
                      half * ka * 4, (half + 1) * ka * 4);
        tmem_st_wait();
    }
    tc_fence_before();
    __syncthreads();
    if (KS > 1) cluster_sync_all();  // peers' barriers exist before any remote store
    tc_fence_after();
    // A step is one round (all three gates' rows from h_{t-1}) or, with the
    // reset gate before the product, two: round 0 takes the r and z rows from
    // h_{t-1} and publishes r * h_{t-1}; round 1 takes the n rows from it.
    // Partial rows of a round for my units: KS sources x gates x UO rows, the
    // 16-byte pieces (4 batch columns) that hold the batch.
    const bool RB = p.reset_before != 0;
    const int nph = RB ? 2 : 1;
    const int rounds = p.T * nph;  // rounds with a recurrent product; the finish round of a next layer comes after
    const int npiece = (batch + 3) >> 2;
    auto round_bytes = [&](int ph) {
        const int rows = (RB ? (ph == 0 ? 2 : 1) : 3) * UO;  // from each source
        return static_cast<uint32_t>(rows * ((KS - 1) * (bulk ? BP * 4 : npiece * 16) + npiece * 16));
    };
    const uint32_t idesc = idesc_bf16_f32(128, BP, false, false);
    // A round in which the next layer's W multiplies the h_{t-1} just gathered.
    auto w_step = [&](int round) { return HN && round >= nph && round % nph == 0; };

    if (warp < kGateWarps) {
        // This CTA evaluates the gates of units unit0 + rank*UO + [0, UO); thread
        // tid takes unit ui = tid % UO and batch rows b = tid / UO + k * BSTEP.
        const int ui = tid % UO;
        const int j = unit0 + static_cast<int>(rank) * UO + ui;
        const bool publishes = static_cast<int>(blockIdx.x) != p.skip_publish_cta;
        const float bh_r = b_hh[j], bh_z = b_hh[H + j], bh_n = b_hh[2 * H + j];
        const float bi_r = b_ih ? b_ih[j] : 0.0f, bi_z = b_ih ? b_ih[H + j] : 0.0f,
                    bi_n = b_ih ? b_ih[2 * H + j] : 0.0f;
        // Unit pairs leave as one 32-bit word, stored by the even unit's lane.
        uint16_t *pub = hx + static_cast<size_t>(j >> 3) * (BP * 8) + (j & 7);
        auto publish = [&](int slot, int b, float v) {
            const uint32_t mine = f32_to_bf16_rne(v);
            const uint32_t next = __shfl_down_sync(0xffffffffu, mine, 1);
            if ((ui & 1) == 0 && b < batch && publishes)
                st_relaxed_gpu(reinterpret_cast<uint32_t *>(pub + static_cast<size_t>(slot) * p.slot + b * 8),
                               mine | (next << 16));
        };
        float hprev[NP];
#pragma unroll
        for (int k = 0; k < NP; ++k) {
            const int b = tid / UO + k * BSTEP;
            hprev[k] = (h0 != nullptr && b < batch) ? h0[static_cast<size_t>(b) * H + j] : 0.0f;
            publish(0, b, hprev[k]);
        }
        // Input projection of a step (independent of h): copied to shared memory
        // one step ahead, each thread its own values, so that nothing on the
        // recurrence's path waits for it (loads into registers made the gather
        // wait 1000 cycles a step for them).  gx is one slab holding x W^T +
        // b_ih (the GEMM's output), or KS slabs of K-rank partial products
        // computed by the layer below, summed after b_ih and in rank order
        // where the gates use them.
        float *sgx = reinterpret_cast<float *>(smem + L.off_gx) + tid;
        auto load_gx = [&](int tt) {
#pragma unroll
            for (int k = 0; k < NP; ++k) {
                const int b = tid / UO + k * BSTEP;
                const bool live = b < batch && tt < p.T;
                const float *g = gx + (live ? (static_cast<size_t>(tt) * p.bstride + b) * G + j : 0);
#pragma unroll
                for (int s = 0; s < SL; ++s) {
                    if (s > 0 && s >= gx_parts) break;
                    const float *gs = g + static_cast<size_t>(s) * p.gx_slab;
#pragma unroll
                    for (int q = 0; q < 3; ++q)
                        cp_async_f32(sgx + ((((tt & 1) * 3 + q) * NP + k) * SL + s) * kGateThreads, gs + q * H, live);
                }
            }
            cp_async_commit();
        };
        auto sum_gx = [&](int tt, int q, float bias, int k) {
            const float *v = sgx + (((tt & 1) * 3 + q) * NP + k) * SL * kGateThreads;
            float a = bias + v[0];
            if (SL > 1 && gx_parts > 1)
#pragma unroll
                for (int s = 1; s < SL; ++s) a += v[s * kGateThreads];
            return a;
        };
        // The words of step tt that the layer below had not stored when they were
        // copied: all of a thread's at once, until none is empty.
        auto poll_gx = [&](int tt) {
            constexpr int NV = 3 * NP * SL;
            float *at = sgx + (tt & 1) * NV * kGateThreads;
            const float *src[NP];
            uint32_t pend = 0;
#pragma unroll
            for (int k = 0; k < NP; ++k) {
                const int b = tid / UO + k * BSTEP;
                src[k] = gx + (static_cast<size_t>(tt) * p.bstride + b) * G + j;
#pragma unroll
                for (int q = 0; q < 3; ++q)
#pragma unroll
                    for (int sl = 0; sl < SL; ++sl) {
                        const int i = (q * NP + k) * SL + sl;
                        if (b < batch && __float_as_uint(at[i * kGateThreads]) == kEmpty) pend |= 1u << i;
                    }
            }
            unsigned long long t0 = 0;
#pragma unroll 1
            for (uint32_t it = 1; pend != 0u; ++it) {
                uint32_t v[NV];
#pragma unroll
                for (int i = 0; i < NV; ++i)
                    if (pend >> i & 1u)
                        v[i] = ld_relaxed_gpu(reinterpret_cast<const uint32_t *>(
                            src[i / SL % NP] + static_cast<size_t>(i % SL) * p.gx_slab + i / (NP * SL) * H));
#pragma unroll
                for (int i = 0; i < NV; ++i)
                    if ((pend >> i & 1u) && v[i] != kEmpty) {
                        at[i * kGateThreads] = __uint_as_float(v[i]);
                        pend &= ~(1u << i);
                    }
                if ((it & 15u) == 0u) {
                    if (*w.abort_flag) return false;
                    if (t0 == 0) t0 = globaltimer();
                    if (globaltimer() - t0 > w.timeout_ns) {
                        report_timeout(w, kSiteGruStep);
                        return false;
                    }
                }
            }
            return true;
        };
        load_gx(0);

        // Gather: warp q takes 16-byte pieces (8 units) q, q + 8, ... of the
        // CTA's K range, lane l the batch rows l, l + 32, ...: a piece's rows are
        // contiguous and come from one CTA, and the shared stores of 8 rows fall
        // into different banks.
        uint32_t mine = 0;  // bit a * LPA + i: this lane has that piece to fetch
#pragma unroll
        for (int a = 0; a < KAMAX; ++a)
#pragma unroll
            for (int i = 0; i < LPA; ++i)
                if (a < ka && lane + 32 * i < batch && (atom0 + a) * 64 + warp * 8 < H) mine |= 1u << (a * LPA + i);
        const uint16_t *src0 = hx + (static_cast<size_t>(atom0 * 8 + warp) * BP + lane) * 8;
        uint8_t *dst0 = sH + lane * 128 + ((warp ^ (lane & 7)) << 4);
        auto gather = [&](int round) {
            return gather_tile<NL, LPA>(src0 + static_cast<size_t>(round & (kSlots - 1)) * p.slot, dst0, mine, BP * 64,
                                        AH, h_full, lane, w);
        };

        // Push: row gate*32 + u of the partial product (TMEM lane = row) goes to
        // the cluster CTA that owns unit u, into its slot for this source rank.
        // Warps w and w + 4 share the TMEM lane quarter w % 4 = the gate, each
        // taking half of the batch columns.  Round 0 of a reset-before step sends
        // the r and z rows, round 1 the n rows.
        const int gate = warp & 3;
        const int half = warp >> 2;
        const uint32_t owner = static_cast<uint32_t>(lane / UO);
        const int oui = lane % UO;
        const int kind = ((static_cast<int>(rank) * 3 + (gate < 3 ? gate : 0)) * 2 + half) * UO;  // first half row at the owner
        const uint32_t push_dst = mapa_shared(smem_u32(recv + (kind + oui) * (BP / 2)), owner);
        const uint32_t push_bar = mapa_shared(smem_u32(red_full), owner);
        // Bulk form: staged as [round parity][gate][half][other owner][UO units][BP / 2].
        const int peer = static_cast<int>(owner) - (owner > rank ? 1 : 0);
        uint8_t *stage = smem + L.off_stage + ((gate < 3 ? gate : 0) * 2 + half) * (kGroup - UO) * (BP * 2);
        uint8_t *stage_row = stage + (peer * UO + oui) * (BP * 2);
        const uint32_t to = static_cast<uint32_t>(lane & (KS - 1));  // lanes 0 .. KS - 1 send to owner `lane`
        const bool sends = lane < KS && to != rank;
        const uint32_t stage_part = smem_u32(stage) + (to - (to > rank ? 1u : 0u)) * static_cast<uint32_t>(UO * BP * 2);
        const uint32_t part_dst = mapa_shared(smem_u32(recv + kind * (BP / 2)), to);
        const uint32_t part_bar = mapa_shared(smem_u32(red_full), to);
        auto push = [&](uint32_t par) {
            if (KS > 1 && BP < 128 && bulk)
                push_rows_bulk<BP>(tmem_d + (static_cast<uint32_t>(gate * 32) << 16), half, npiece, owner != rank,
                                   stage_row + par * stage_bytes(KS, BP), push_dst + par * recv_bytes(BP), oui,
                                   push_bar + par * 8u, sends, stage_part + par * stage_bytes(KS, BP),
                                   part_dst + par * recv_bytes(BP), part_bar + par * 8u,
                                   static_cast<uint32_t>(UO * BP * 2));
            else
                push_rows<BP>(tmem_d + (static_cast<uint32_t>(gate * 32) << 16), half, npiece,
                              push_dst + par * recv_bytes(BP), oui, push_bar + par * 8u);
        };

        auto write_out = [&](int tt) {
#pragma unroll
            for (int k = 0; k < NP; ++k) {
                const int b = tid / UO + k * BSTEP;
                if (b >= batch) continue;
                const size_t at = (static_cast<size_t>(tt) * p.bstride + b) * H + j;
                h_out[at] = hprev[k];
                if (xb != nullptr) xb[at] = f32_to_bf16_rne(hprev[k]);
            }
        };

        // ---- recursive iteration, T times (in nph rounds each), then, when the
        // next layer's projection is fused in, a finish round that only gathers
        // h_{T-1} for it.
        float zsave[NP];  // update gate between the two rounds of a step
        bool ok = true;
        const int gathers = rounds + (HN ? 1 : 0);
        int t = 0, ph = 0;
        for (int round = 0; round < gathers; ++round) {
            const uint32_t par = static_cast<uint32_t>(round & 1);
            // The next layer's product of the latest step still reads sH.
            if (HN && round > nph) {
                const int ws = (round - 1) / nph - 1;  // step parity index of that product
                if (!all_wait(&w_done[ws & 1], static_cast<uint32_t>(ws >> 1) & 1u, w, SITE_GRU_W)) {
                    ok = false;
                    break;
                }
            }
            if (!gather(round)) {
                ok = false;
                break;
            }
            if (ph == 0) {
                // While the MMAs run: the last step's state to h_out, the next
                // step's projection on its way to shared memory.  (Before the
                // gather, its fence and arrive waited for these accesses.)
                if (t > 0) write_out(t - 1);
                if (round == rounds) break;  // the finish round
                load_gx(t + 1);
            }
            if (gate < 3 && (bulk || half * (BP / 8) < npiece) && (!RB || (ph == 0 ? gate < 2 : gate == 2))) {
                if (!all_wait(mma_done, par, w, SITE_GRU_MMA)) {
                    ok = false;
                    break;
                }
                tc_fence_after();
                push(par);
            }
            // Projections of this step, before the partial rows arrive.
            float xr[NP], xz[NP], xn[NP];
            if (ph == 0) {
                cp_async_wait_all_but_last();
                if (POLL && layer > 0 && !__all_sync(0xffffffffu, poll_gx(t))) {
                    ok = false;
                    break;
                }
            }
#pragma unroll
            for (int k = 0; k < NP; ++k) {
                if (!RB || ph == 0) {
                    xr[k] = sum_gx(t, 0, bi_r, k);
                    xz[k] = sum_gx(t, 1, bi_z, k);
                }
                if (!RB || ph == 1) xn[k] = sum_gx(t, 2, bi_n, k);
            }
            if (!all_wait<true>(&red_full[par], static_cast<uint32_t>(round >> 1) & 1u, w, SITE_GRU_RED)) {
                ok = false;
                break;
            }
            const float *rv = recv + par * (recv_bytes(BP) / 4);
            const int next = (round + 1) & (kSlots - 1);
#pragma unroll
            for (int k = 0; k < NP; ++k) {
                const int b = tid / UO + k * BSTEP;
                float ghr = bh_r, ghz = bh_z, ghn = bh_n;
#pragma unroll
                for (int s = 0; s < KS; ++s) {  // partials summed in rank order
                    const float *rs = rv + s * 3 * UO * BP + recv_at<BP, UO>(ui, b);
                    if (!RB || ph == 0) {
                        ghr += rs[0];
                        ghz += rs[UO * BP];
                    }
                    if (!RB || ph == 1) ghn += rs[2 * UO * BP];
                }
                if (!RB) {
                    const float rg = sigmoidf_fast(xr[k] + ghr);
                    const float zg = sigmoidf_fast(xz[k] + ghz);
                    hprev[k] = gru_blend(zg, gru_candidate(xn[k], rg, ghn), hprev[k]);
                    publish(next, b, hprev[k]);
                } else if (ph == 0) {
                    const float rg = sigmoidf_fast(xr[k] + ghr);
                    zsave[k] = sigmoidf_fast(xz[k] + ghz);
                    publish(next, b, rg * hprev[k]);
                } else {
                    const float ng = tanhf_fast(xn[k] + ghn);
                    hprev[k] = gru_blend(zsave[k], ng, hprev[k]);
                    publish(next, b, hprev[k]);
                }
            }
            if (++ph == nph) {
                ph = 0;
                ++t;
            }
        }
        if (ok && !HN) write_out(p.T - 1);
    } else if (warp == kMmaWarp) {
        // The whole warp waits and one elected lane issues: under an elect.sync
        // branch the instruction's operands stay in uniform registers (16 to 23
        // cycles an MMA; 48 from a branch on the lane number).
        const bool lead = elect_one();
        if (lead) {
            mbar_arrive_expect_tx(&red_full[0], round_bytes(0));
            if (HN) {
                tma_prefetch_desc(&tmWn);
                mbar_arrive_expect_tx(wbar, static_cast<uint32_t>(ka * kAtomU));
                for (int a = 0; a < ka; ++a) tma_load_3d(&tmWn, wbar, sW + a * kAtomU, (atom0 + a) * 64, unit0, 3 * (p.w_layer + layer));
            }
        }
        __syncwarp();
        bool ok = true;
        if (HN) {
            ok = all_wait(wbar, 0, w, SITE_GRU_W);
            if (!ok) drain_bar(wbar, 0, p.timeout_ns);
        }
        const int last = rounds + (HN ? 1 : 0);
        int done_round = -1, w_issued = 0;  // for the drains after an abort
        for (int round = 0; ok && round < last; ++round) {
            const uint32_t par = static_cast<uint32_t>(round & 1);
            const bool finish = round == rounds;
            if (!all_wait(h_full, par, w, SITE_GRU_H)) {
                ok = false;
                break;
            }
            tc_fence_after();
            if (!finish) {
                if (lead) {
#pragma unroll
                    for (int a = 0; a < KAMAX; ++a) {
                        if (a >= ka) break;
                        const uint64_t hd = sdesc_sw128(smem_u32(sH + a * AH), 16, 1024);
                        const uint32_t ua = tmem_d + kUCol + static_cast<uint32_t>(a * 32);
#pragma unroll
                        for (int k = 0; k < 4; ++k)
                            umma_bf16_ts(tmem_d, ua + k * 8, hd + k * 2, idesc, (a > 0 || k > 0) ? 1u : 0u);
                    }
                    umma_commit(mma_done);
                }
                __syncwarp();
                done_round = round;
            }
            if (w_step(round)) {
                // The next layer's W times the h_{t-1} just used, after the
                // recurrent product in the tensor pipe.  Its A operand starts
                // 32 rows early (still inside shared memory: the pad precedes
                // W), so W's r, z and n rows land in TMEM lanes 32-127; two
                // accumulators by step parity.
                const int ws = round / nph - 1;
                if (ws >= 2 && !all_wait(&w_free[ws & 1], static_cast<uint32_t>((ws >> 1) - 1) & 1u, w, SITE_GRU_W)) {
                    ok = false;
                    break;
                }
                tc_fence_after();
                if (lead) {
                    const uint32_t col = 32u + 32u * static_cast<uint32_t>(ws & 1);
                    for (int a = 0; a < ka; ++a) {
                        const uint64_t wd = sdesc_sw128(smem_u32(sW + a * kAtomU) - 32u * 128u, 16, 1024);
                        const uint64_t hd = sdesc_sw128(smem_u32(sH + a * AH), 16, 1024);
#pragma unroll
                        for (int k = 0; k < 4; ++k)
                            umma_bf16(tmem_d + col, wd + k * 2, hd + k * 2, idesc, (a > 0 || k > 0) ? 1u : 0u);
                    }
                    umma_commit(&w_done[ws & 1]);
                }
                w_issued = ws + 1;
            }
            __syncwarp();
        }
        // Every product issued has completed before TMEM is released.
        if (done_round >= 0) drain_bar(mma_done, static_cast<uint32_t>(done_round & 1), p.timeout_ns);
        if (w_issued > 0)
            drain_bar(&w_done[(w_issued - 1) & 1], static_cast<uint32_t>((w_issued - 1) >> 1) & 1u, p.timeout_ns);
        __syncwarp();
    } else if (warp == kHouseWarp || HN) {
        const int last = rounds + (HN ? 1 : 0);
        // Units of this CTA: UO / 8 16-byte pieces per batch row.
        const int u0 = unit0 + static_cast<int>(rank) * UO;
        uint16_t *own = hx + static_cast<size_t>(u0 >> 3) * (BP * 8);
        for (int round = 0; round < last; ++round) {
            if (warp == kHouseWarp && round < rounds) {
                if (!all_wait<true>(&red_full[round & 1], static_cast<uint32_t>(round >> 1) & 1u, w, SITE_GRU_RED))
                    break;
                if (round >= 1) {
                    uint16_t *old = own + static_cast<size_t>((round + 3) & (kSlots - 1)) * p.slot;
                    for (int i = lane; i < UO / 8 * BP; i += 32)
                        if (i % BP < batch)
                            *reinterpret_cast<uint4 *>(old + i * 8) = make_uint4(kEmpty, kEmpty, kEmpty, kEmpty);
                    fence_acq_rel_gpu();
                }
                __syncwarp();
                if (lane == 0 && round + 1 < rounds)
                    mbar_arrive_expect_tx(&red_full[(round + 1) & 1], round_bytes((round + 1) % nph));
                __syncwarp();
            }
            if (w_step(round)) {
                // Next layer's projection of step ws over this CTA's K range:
                // TMEM lane 32 + gate*32 + u holds unit unit0 + u of that gate
                // for the 32 batch rows; row b goes to slab `rank`.
                const int ws = round / nph - 1;
                if (!all_wait(&w_done[ws & 1], static_cast<uint32_t>(ws >> 1) & 1u, w, SITE_GRU_W)) break;
                tc_fence_after();
                const int q = warp & 3;  // TMEM lane quarter 1, 2 or 3
                uint32_t r[32];
                tmem_ld32(tmem_d + (static_cast<uint32_t>(q * 32) << 16) + 32u + 32u * static_cast<uint32_t>(ws & 1), r);
                tmem_ld_wait(r);
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(&w_free[ws & 1]);
                float *dst = gxp_out + static_cast<size_t>(rank) * p.gx_slab +
                             static_cast<size_t>(ws) * p.bstride * G + (q - 1) * H + unit0 + lane;
#pragma unroll
                for (int c = 0; c < 32; ++c)
                    if (c < batch) {
                        if (POLL)  // any NaN but the empty word's pattern
                            st_relaxed_gpu(reinterpret_cast<uint32_t *>(dst + static_cast<size_t>(c) * G),
                                           r[c] == kEmpty ? 0x7FFFFFFFu : r[c]);
                        else
                            dst[static_cast<size_t>(c) * G] = __uint_as_float(r[c]);
                    }
            }
        }
    }

    // ---- teardown: release TMEM.
    __syncwarp();
    tc_fence_before();
    if (__syncthreads_or(*abort_flag) && tid == 0) {
        // After an abort, partial rows a peer sent may still be on their way.
        const unsigned long long t0 = globaltimer();
        while (globaltimer() - t0 < 50000ull) {
        }
    }
    __syncthreads();
    // No CTA leaves while a cluster peer may still write into its shared
    // memory (a peer that gave up on a wait can be behind by a round); every
    // wait above is bounded, so every CTA gets here.
    if (KS > 1) cluster_sync_all();
    if (warp == 0) {
        tc_fence_after();
        tmem_dealloc(tmem_d, tmem_cols);
    }
}

// K splits for a hidden size (the cluster size).  CTA k of a cluster takes
// the 64-wide K atoms k * ka .. k * ka + ka - 1 (ka = gru_atoms); the last
// range may end past the matrix, and a hidden of 64 j + 32 ends half an atom
// inside it: the tensor maps read zeros there on both sides of the product.
// 4 splits for multiples of 256, 2 for the other multiples of 128; otherwise
// one CTA per group up to 7 atoms (hidden <= 448), 2 up to 14 atoms and 4
// above, so that a CTA's slice of U, the next layer's slice of W (stacks) and
// its h tiles fit shared memory together at every multiple of 32.
int gru_splits(int H) {
    if (H % 256 == 0) return 4;
    if (H % 128 == 0) return 2;
    return H <= 448 ? 1 : H <= 896 ? 2 : 4;
}

// 64-wide K atoms per CTA: the hidden's atoms, rounded up, over the splits.
int gru_atoms(int H) {
    const int ks = gru_splits(H);
    return ((H + 63) / 64 + ks - 1) / ks;
}

size_t gru_smem_bytes(int H, bool has_next = false, int bp = kBatchPad) {
    return static_cast<size_t>(gru_layout(gru_splits(H), gru_atoms(H), has_next, bp).total);
}

int gru_cta_count(int H) { return H / kGroup * gru_splits(H); }

using GruKernel = void (*)(const CUtensorMap, const GruParams);

template <int BP>
GruKernel gru_kernel_for_bp(int ks) {
    return ks == 4 ? gru_recurrent_kernel<4, BP> : ks == 2 ? gru_recurrent_kernel<2, BP> : gru_recurrent_kernel<1, BP>;
}

// Padded batch widths a K-split count can run: 128 only with 4 splits (fewer
// splits leave 16 or 32 (unit, batch) pairs per thread, beyond the registers).
bool gru_bp_ok(int ks, int bp) { return bp == 32 || bp == 64 || (bp == 128 && ks == 4); }

// Several layers of a stack in one launch.
GruKernel gru_poll_kernel_for(int ks) {
    return ks == 4   ? gru_recurrent_kernel<4, kBatchPad, true>
           : ks == 2 ? gru_recurrent_kernel<2, kBatchPad, true>
                     : gru_recurrent_kernel<1, kBatchPad, true>;
}

GruKernel gru_kernel_for(int ks, int bp = kBatchPad) {
    if (bp == 128) return gru_recurrent_kernel<4, 128>;
    return bp == 64 ? gru_kernel_for_bp<64>(ks) : gru_kernel_for_bp<32>(ks);
}

// Opts every instantiation in to `bytes` of dynamic shared memory on the
// current device (ordinal `device`; the record is kept per device).
int gru_smem_attr(int bytes, int device) {
    const int ks[3] = {1, 2, 4}, bps[3] = {32, 64, 128};
    for (int k : ks)
        for (int bp : bps) {
            if (!gru_bp_ok(k, bp)) continue;
            const int rc = ensure_smem_optin(reinterpret_cast<const void *>(gru_kernel_for(k, bp)), bytes, device,
                                             "cudaFuncSetAttribute(gru)");
            if (rc) return rc;
        }
    for (int k : ks)
        if (const int rc = ensure_smem_optin(reinterpret_cast<const void *>(gru_poll_kernel_for(k)), bytes, device,
                                             "cudaFuncSetAttribute(gru)"))
            return rc;
    return ISAM_OK;
}

int ensure_ws(void **ptr, size_t *cap, size_t need, const char *what) {
    if (*cap >= need) return ISAM_OK;
    if (*ptr) cudaFree(*ptr);
    *ptr = nullptr;
    *cap = 0;
    cudaError_t e = cudaMalloc(ptr, need);
    if (e != cudaSuccess) return cuda_error(e, what);
    *cap = need;
    return ISAM_OK;
}

// Replaces a projection workspace that serves the call as it is by one of `need`
// bytes, or of twice its own, without freeing it: only layers that could share a
// launch ask for more, and a graph captured before may still use it.  What is kept
// adds up to less than the new one.  False (nothing changed) during a capture, which
// admits no allocation, and where no memory is found.
bool grow_projections(DeviceState &ds, size_t need, cudaStream_t stream) {
    cudaStreamCaptureStatus capture = cudaStreamCaptureStatusNone;
    if (ds.gru_gxp_olds == static_cast<int>(sizeof ds.gru_gxp_old / sizeof ds.gru_gxp_old[0]) ||
        cudaStreamIsCapturing(stream, &capture) != cudaSuccess || capture != cudaStreamCaptureStatusNone) {
        (void)cudaGetLastError();
        return false;
    }
    need = std::max(need, 2 * ds.gru_gxp_bytes);
    float *grown = nullptr;
    if (cudaMalloc(&grown, need) != cudaSuccess) {
        (void)cudaGetLastError();
        return false;
    }
    ds.gru_gxp_old[ds.gru_gxp_olds++] = ds.gru_gxp;
    ds.gru_gxp = grown;
    ds.gru_gxp_bytes = need;
    return true;
}

// Tensor map of the layers' W as [layer, 3 gates][H rows][H] (box: 96 rows of
// one group over one 64-wide K atom).
int weight_map(const uint16_t *Wt, int layers, int H, CUtensorMap *tm) {
    const uint64_t dims[3] = {static_cast<uint64_t>(H), static_cast<uint64_t>(H), 3 * static_cast<uint64_t>(layers)};
    const uint64_t strides[2] = {static_cast<uint64_t>(H) * 2, static_cast<uint64_t>(H) * H * 2};
    const uint32_t box[3] = {64, kGroup, 3};
    return make_tmap_3d_bf16(tm, Wt, dims, strides, box);
}

// Elements of one slot of the exchange ring: [H/8 pieces][bp rows][8].
int slot_elems(int H, int bp) { return H * bp; }

// Bytes of the rings of any call on a GB300.
constexpr size_t kRingsBytes = static_cast<size_t>(2) << 20;

// Bytes of a whole ring.
size_t ring_bytes(int H, int bp) { return static_cast<size_t>(kSlots) * slot_elems(H, bp) * sizeof(uint16_t); }

int gru_empty_rings(uint16_t *hx, size_t bytes, cudaStream_t stream) {
    const cudaError_t e = cudaMemsetAsync(hx, 0xFF, bytes, stream);  // kEmpty
    return e == cudaSuccess ? ISAM_OK : cuda_error(e, "emptying the GRU exchange rings");
}

// Chunks (or layers) of hidden H, gru_cta_count(H) CTAs each in clusters of its K
// splits, that kern keeps resident at once with `smem` bytes a CTA.
cudaError_t gru_resident(GruKernel kern, int H, size_t smem, int *chunks) {
    const int ks = gru_splits(H);
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = static_cast<unsigned>(ks);
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.gridDim = dim3(static_cast<unsigned>(gru_cta_count(H)), 1, 1);
    cfg.blockDim = dim3(kThreads, 1, 1);
    cfg.dynamicSmemBytes = smem;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    int clusters = 0;
    const cudaError_t e = cudaOccupancyMaxActiveClusters(&clusters, kern, &cfg);
    *chunks = clusters * ks / gru_cta_count(H);
    return e;
}

// Fills the shape fields of p and launches the
// recurrence: one cluster of KS CTAs per group of 32 units, as a plain cluster
// launch after checking that every cluster fits on the device at once (the
// exchange needs every CTA resident).  It is a dependent launch, whose set-up
// overlaps the projection: 1 to 3 us less a call at every length (off / on, 4, 24 and
// 128 steps: 17.0 / 15.7, 55.6 / 53.8 and 250.6 / 247.2 us at hidden 64, batch 5; 26.3 /
// 24.9, 74.8 / 73.5 and 331.5 / 330.6 at hidden 1024, batch 32).  No cooperative attribute: a launch that carries both it and the
// cluster shape can lose the cluster shape when a tool re-issues it, and the
// bounded waits already turn a CTA that never runs into ISAM_ERR_TIMEOUT.
//
// A batch of more rows than the padded width runs in chunks.  Chunks whose CTAs
// fit on the device together share a launch: a chunk's step is latency, so they
// cost little more than one (5 steps of 3 layers at hidden 160, batch 204: 354 ->
// 109 us; 70 steps at hidden 704, batch 102: 620 -> 353).
// `rings` exchange rings follow one another at p.hx, emptied by the caller
// (gru_empty_rings) ahead of the projection.
// With `layers` > 1 that many layers of a stack share the launch, p describing
// the first; their number must fit (gru_layers_together).
int launch_recurrent(GruParams &p, const CUtensorMap &tmWn, size_t smem, cudaStream_t stream, int rings = 1,
                     int bp = kBatchPad, int layers = 1) {
    const int H = p.H;
    p.ks = gru_splits(H);
    p.ka = gru_atoms(H);
    p.uo = kGroup / p.ks;
    p.n_cta = gru_cta_count(H);
    p.slot = slot_elems(H, bp);
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = static_cast<unsigned>(p.ks);
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.gridDim = dim3(static_cast<unsigned>(p.n_cta), 1, 1);
    cfg.blockDim = dim3(kThreads, 1, 1);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = stream;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    const GruKernel kern = layers > 1 ? gru_poll_kernel_for(p.ks) : gru_kernel_for(p.ks, bp);
    int resident = 0;
    cudaError_t e = gru_resident(kern, H, smem, &resident);
    if (e != cudaSuccess) return cuda_error(e, "cudaOccupancyMaxActiveClusters(gru)");
    // Chunks on the device at once; all layers have to be.
    const int fit = std::min(rings, resident);
    if (fit < layers || fit < 1)
        return set_error(ISAM_ERR_UNSUPPORTED,
                         "GRU recurrence: %d x %d CTAs in clusters of %d cannot be co-resident (%d x %d fit)",
                         layers, p.n_cta, p.ks, resident, p.n_cta);
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.numAttrs = 2;
    if (layers > 1) {
        p.chunks = layers;
        cfg.gridDim = dim3(static_cast<unsigned>(p.n_cta * layers), 1, 1);
        e = cudaLaunchKernelEx(&cfg, kern, tmWn, p);
        return e == cudaSuccess ? ISAM_OK : cuda_error(e, "launch gru_recurrent_kernel");
    }
    const int total = p.total;
    for (int b0 = 0; b0 < total; b0 += fit * bp) {
        GruParams c = p;
        c.total = std::min(fit * bp, total - b0);
        c.chunks = (c.total + bp - 1) / bp;
        c.gx += static_cast<size_t>(b0) * 3 * H;
        if (c.h0) c.h0 += static_cast<size_t>(b0) * H;
        c.h_out += static_cast<size_t>(b0) * H;
        if (c.xb) c.xb += static_cast<size_t>(b0) * H;
        c.hx += static_cast<size_t>(b0 / bp) * kSlots * p.slot;
        cfg.gridDim = dim3(static_cast<unsigned>(p.n_cta * c.chunks), 1, 1);
        e = cudaLaunchKernelEx(&cfg, kern, tmWn, c);
        if (e != cudaSuccess) return cuda_error(e, "launch gru_recurrent_kernel");
    }
    return ISAM_OK;
}

}  // namespace

namespace {

// bf16 copy of a layer's states (the next layer pair's GEMM input); n is a
// multiple of 4, both pointers 16-byte aligned.
__global__ void __launch_bounds__(256) states_to_bf16_kernel(const float4 *in, uint2 *out, size_t n4) {
    for (size_t i = blockIdx.x * static_cast<size_t>(blockDim.x) + threadIdx.x; i < n4;
         i += static_cast<size_t>(gridDim.x) * blockDim.x) {
        const float4 v = in[i];
        out[i] = make_uint2(static_cast<uint32_t>(f32_to_bf16_rne(v.x)) | (static_cast<uint32_t>(f32_to_bf16_rne(v.y)) << 16),
                            static_cast<uint32_t>(f32_to_bf16_rne(v.z)) | (static_cast<uint32_t>(f32_to_bf16_rne(v.w)) << 16));
    }
}

}  // namespace

int gru_plan(int layers, int batch, int hidden, int reset_before, int num_sms, int smem_optin, GruPlan *g) {
    const int H = hidden;
    if (layers < 1 || batch < 1 || batch > kBatchMax || H % 32 != 0 || H > 1024 || H < 32)
        return set_error(ISAM_ERR_UNSUPPORTED,
                         "isam_gru_forward: needs batch <= 256 and hidden a multiple of 32 in "
                         "[32, 1024] (batch=%d hidden=%d)",
                         batch, H);
    GruPlan q;
    q.ks = gru_splits(H);
    q.ka = gru_atoms(H);
    q.n_cta = gru_cta_count(H);
    if (q.n_cta > num_sms)
        return set_error(ISAM_ERR_UNSUPPORTED, "isam_gru_forward: %d CTAs cannot be co-resident", q.n_cta);
    // Padded batch of the recurrence (the MMA's N): 32 for batch <= 32, with
    // every feature; above that 64 or 128, the batch running in chunks of that
    // many rows (independent sequences).
    const bool chunked = batch > kBatchPad;
    q.bp = kBatchPad;
    if (chunked) {
        auto fits = [&](int cand) {
            return gru_bp_ok(q.ks, cand) && gru_smem_bytes(H, false, cand) <= static_cast<size_t>(smem_optin);
        };
        // Steps of a wider chunk take longer (in proportion 4.5 at 64 padded rows, 8.3
        // at 128), but chunks that do not fit on the device together run one after
        // another.  24 steps, hidden / batch in chunks of 64 and of 128: 256 / 128 87 and
        // 143 us, 512 / 128 98 and 160, 512 / 192 186 and 161, 768 / 96 184 and 149, 1024 /
        // 128 210 and 188, 1024 / 256 417 and 376; the choice is 1% behind at 192 rows of
        // hidden 768 and 1024 (292 and 289, 315 and 310).
        const int together = std::max(1, num_sms / q.n_cta);
        double best = 0.0;
        for (const auto &[cand, step_us] : {std::pair<int, double>{64, 4.5}, {128, 8.3}}) {
            if (!fits(cand)) continue;
            const int chunks = (batch + cand - 1) / cand;
            const double us = (chunks + together - 1) / together * step_us;
            if (q.bp == kBatchPad || us < best) {
                q.bp = cand;
                best = us;
            }
        }
    }
    const size_t smem_last = gru_smem_bytes(H, false, q.bp);
    const size_t smem_next = gru_smem_bytes(H, true);
    if (smem_last > static_cast<size_t>(smem_optin))
        return set_error(ISAM_ERR_UNSUPPORTED, "isam_gru_forward: hidden too large for shared memory");
    if (layers > 1 && !chunked && smem_next > static_cast<size_t>(smem_optin))
        return set_error(ISAM_ERR_UNSUPPORTED,
                         "isam_gru_forward_stack: hidden %d leaves no room for the next layer's "
                         "weights beside the recurrent ones (%zu bytes of shared memory)",
                         H, smem_next);
    q.chunks = (batch + q.bp - 1) / q.bp;
    q.smem = static_cast<int>(smem_last);
    if (layers == 1) {
        q.path = 0;
    } else if (chunked) {
        q.path = 3;
    } else {
        const char *nw = getenv("ISAM_NO_WAVE");
        if (!reset_before && !(nw && nw[0] == '1') && gru_wave_fits(H, batch, num_sms, smem_optin)) {
            q.path = 1;
            q.smem = static_cast<int>(gru_wave_smem_bytes(H));
        } else {
            q.path = 2;
            q.smem = static_cast<int>(smem_next);
        }
    }
    *g = q;
    return ISAM_OK;
}

// Layers of the per-layer chain whose CTAs fit on the device together, with at most
// 1 GB of projections between them.
static int gru_layers_together(int layers, int H, size_t gx_floats, const DeviceState &ds) {
    const int ks = gru_splits(H);
    int resident = 0;
    if (ensure_smem_optin(reinterpret_cast<const void *>(gru_poll_kernel_for(ks)), ds.max_smem_optin, ds.device,
                          "cudaFuncSetAttribute(gru)") != ISAM_OK ||
        gru_resident(gru_poll_kernel_for(ks), H, gru_smem_bytes(H, true), &resident) != cudaSuccess) {
        (void)cudaGetLastError();
        return 1;
    }
    const size_t set_bytes = static_cast<size_t>(ks) * gx_floats * sizeof(float);
    const long long by_size = 1 + static_cast<long long>((static_cast<size_t>(1) << 30) / set_bytes);
    return static_cast<int>(std::max<long long>(1, std::min<long long>({layers, resident, by_size})));
}

int gru_together(int layers, int T, int batch, int hidden, int reset_before, const DeviceState &ds, int *layers_together,
                 int *chunks_together) {
    GruPlan plan;
    int rc = gru_plan(layers, batch, hidden, reset_before, ds.num_sms, ds.max_smem_optin, &plan);
    if (rc) return rc;
    const size_t gx_floats = static_cast<size_t>(T) * batch * 3 * hidden;
    *layers_together = plan.path == 1 ? 2 : plan.path == 2 ? gru_layers_together(layers, hidden, gx_floats, ds) : 1;
    *chunks_together = 1;
    if (plan.chunks > 1) {
        if ((rc = gru_smem_attr(ds.max_smem_optin, ds.device))) return rc;
        int resident = 0;
        const cudaError_t e = gru_resident(gru_kernel_for(plan.ks, plan.bp), hidden, gru_smem_bytes(hidden, false, plan.bp),
                                           &resident);
        if (e != cudaSuccess) return cuda_error(e, "cudaOccupancyMaxActiveClusters(gru)");
        *chunks_together = std::max(1, std::min(plan.chunks, resident));
    }
    return ISAM_OK;
}

int gru_stack_launch(int layers, int T, int batch, int hidden, int reset_before, const uint16_t *x,
                     const uint16_t *W, const uint16_t *U, const float *b, const float *h0, float *h_out,
                     DeviceState &ds, cudaStream_t stream) {
    const int H = hidden;
    if ((reinterpret_cast<uintptr_t>(x) | reinterpret_cast<uintptr_t>(W) |
         reinterpret_cast<uintptr_t>(U) | reinterpret_cast<uintptr_t>(b) |
         reinterpret_cast<uintptr_t>(h0) | reinterpret_cast<uintptr_t>(h_out)) & 15u)
        return set_error(ISAM_ERR_UNSUPPORTED, "isam_gru_forward: pointers must be 16-byte aligned");
    GruPlan plan;
    int prc = gru_plan(layers, batch, H, reset_before, ds.num_sms, ds.max_smem_optin, &plan);
    if (prc != ISAM_OK) return prc;
    const bool chunked = batch > kBatchPad;  // path 3 when layers > 1
    const int bp = plan.bp;
    const size_t smem_last = gru_smem_bytes(H, false, bp);
    const size_t smem_next = gru_smem_bytes(H, true);

    int rc;
    const size_t seq_rows = static_cast<size_t>(T) * batch;
    const size_t gx_floats = seq_rows * 3 * H;
    if ((rc = ensure_ws(reinterpret_cast<void **>(&ds.gru_gx), &ds.gru_gx_bytes, gx_floats * sizeof(float),
                        "allocating the GRU projection workspace")))
        return rc;
    // Next layers' projections, sets of ks slabs, one per K rank: between the
    // layers of a launch, then two for those between launches (one read, one
    // written).
    const int ks = gru_splits(H);
    int together = plan.path == 2 ? gru_layers_together(layers, H, gx_floats, ds) : 1;
    const size_t set_floats = static_cast<size_t>(ks) * gx_floats;
    const size_t sets_held = ds.gru_gxp_bytes / (set_floats * sizeof(float));
    if (layers > 1 && !chunked && sets_held >= 2) {
        // Room for one layer after another; more only for layers that can share a launch.
        if (sets_held < static_cast<size_t>(together) + 1 &&
            !grow_projections(ds, static_cast<size_t>(together + 1) * set_floats * sizeof(float), stream))
            together = static_cast<int>(sets_held) - 1;
    } else if (layers > 1 && !chunked) {
        auto sets = [&] {
            return ensure_ws(reinterpret_cast<void **>(&ds.gru_gxp), &ds.gru_gxp_bytes,
                             static_cast<size_t>(together + 1) * set_floats * sizeof(float),
                             "allocating the stacked GRU projection workspace");
        };
        rc = sets();
        if (rc && together > 1) {  // no room for them all: one layer after another
            (void)cudaGetLastError();
            together = 1;
            rc = sets();
        }
        if (rc) return rc;
    }
    // Exchange rings: two for a layer pair, else one for each chunk of the batch or
    // layer of a launch, which empties what it uses.  All shapes fit the 2 MB taken
    // at first (four chunks of 64 rows, or two of 128, at hidden 1024; layers together
    // hold no more units than the device has SMs for), so the buffer does not move.
    const int rings = std::max(plan.chunks, together);
    if ((rc = ensure_ws(reinterpret_cast<void **>(&ds.gru_hx), &ds.gru_hx_bytes,
                        std::max(kRingsBytes, std::max(2, rings) * ring_bytes(H, bp)),
                        "allocating the GRU exchange buffer")))
        return rc;
    if ((rc = gru_smem_attr(ds.max_smem_optin, ds.device))) return rc;

    const size_t wsz = static_cast<size_t>(3) * H * H;
    // Input projection of layer l for all steps: gx = in W_l^T + b_ih_l
    // (M = T*batch, N = 3H, K = H).
    auto project = [&](const uint16_t *in, int l) {
        GemmDesc g{T * batch, 3 * H, H, 0, 1, 1.0f, 0.0f, in, W + l * wsz, ds.gru_gx, b + static_cast<size_t>(l) * 6 * H};
        GemmPlan plan;
        int r;
        if ((r = gemm_validate(g))) return r;
        if ((r = gemm_plan(g, ds, &plan))) return r;
        return gemm_launch(g, plan, ds, stream);
    };
    // One layer's recurrence.  Its projection is either ds.gru_gx (one slab,
    // b_ih included) or, for layer l > 0 of the per-layer chain, the slabs the
    // layer below computed; with has_next it computes layer l + 1's slabs.
    // The states in bf16 go to ds.gru_xb when a GEMM projects them for the next layer.
    // `n` > 1: that many layers from l on in one launch.
    auto recur = [&](int l, bool has_next, bool gx_from_below, bool to_gemm, int n = 1) {
        CUtensorMap tmWn;
        memset(&tmWn, 0, sizeof tmWn);
        int r;
        if ((has_next || n > 1) && (r = weight_map(W, layers, H, &tmWn))) return r;
        GruParams p{};
        p.T = T;
        p.U = U + l * wsz;
        p.total = batch;
        p.bstride = batch;
        p.H = H;
        if (!gx_from_below) {
            p.gx = ds.gru_gx;
            p.gx_parts = 1;
            p.b_ih = nullptr;
        } else {
            p.gx = ds.gru_gxp + (together - 1 + (l / together & 1)) * set_floats;
            p.gx_parts = ks;
            p.b_ih = b + static_cast<size_t>(l) * 6 * H;
        }
        p.gx_slab = gx_floats;
        p.has_next = has_next ? 1 : 0;
        p.gxp_out = has_next ? ds.gru_gxp + (together - 1 + ((l + n) / together & 1)) * set_floats : nullptr;
        p.w_layer = l + 1;
        p.gxw = ds.gru_gxp;
        p.out_layer = seq_rows * H;
        p.b_hh = b + static_cast<size_t>(l) * 6 * H + 3 * H;
        p.h0 = h0 ? h0 + static_cast<size_t>(l) * batch * H : nullptr;
        p.h_out = h_out + static_cast<size_t>(l) * seq_rows * H;
        p.xb = to_gemm ? ds.gru_xb : nullptr;
        p.hx = ds.gru_hx;
        p.reset_before = reset_before ? 1 : 0;
        p.skip_publish_cta = -1;
        if (const char *sk = getenv("ISAM_DEBUG_GRU_SKIP_CTA")) p.skip_publish_cta = atoi(sk);
        p.timeout_ns = wait_timeout_ns();
        p.err = ds.err_word;
        return launch_recurrent(p, tmWn, has_next || n > 1 ? smem_next : smem_last, stream, rings, bp, n);
    };
    // bf16 copy of layer l - 1's states as layer l's GEMM input.
    auto states_below = [&](int l) {
        const size_t n4 = seq_rows * H / 4;
        const int blocks = static_cast<int>(std::min<size_t>((n4 + 255) / 256, static_cast<size_t>(ds.num_sms) * 8));
        states_to_bf16_kernel<<<blocks, 256, 0, stream>>>(
            reinterpret_cast<const float4 *>(h_out + static_cast<size_t>(l - 1) * seq_rows * H),
            reinterpret_cast<uint2 *>(ds.gru_xb), n4);
        cudaError_t e = cudaGetLastError();
        return e == cudaSuccess ? ISAM_OK : cuda_error(e, "launch states_to_bf16_kernel");
    };

    // Batches wider than 32: every layer projects its input with the GEMM and
    // runs its recurrence in chunks.
    if (chunked) {
        if (layers > 1 && (rc = ensure_ws(reinterpret_cast<void **>(&ds.gru_xb), &ds.gru_xb_bytes,
                                          seq_rows * H * sizeof(uint16_t), "allocating the GRU layer-input buffer")))
            return rc;
        for (int l = 0; l < layers; ++l) {
            if ((rc = gru_empty_rings(ds.gru_hx, rings * ring_bytes(H, bp), stream))) return rc;
            if ((rc = project(l > 0 ? ds.gru_xb : x, l))) return rc;
            if ((rc = recur(l, false, false, l + 1 < layers))) return rc;
        }
        return ISAM_OK;
    }

    // Pairs of layers in one kernel (gru_wave.cu): layer l + 1 advances one
    // step behind layer l, its projection computed from the same h tiles.
    // Between pairs (and for an odd last layer) the layer below's states are
    // rounded to bf16 and projected by the GEMM.  (Storing them in bf16 from the
    // pair's kernel as well made its step 1.4% slower.)
    if (plan.path == 1) {
        if (layers > 2 && (rc = ensure_ws(reinterpret_cast<void **>(&ds.gru_xb), &ds.gru_xb_bytes,
                                          seq_rows * H * sizeof(uint16_t), "allocating the GRU layer-input buffer")))
            return rc;
        for (int l = 0; l < layers;) {
            if ((rc = gru_empty_rings(ds.gru_hx, gru_wave_ring_bytes(H), stream))) return rc;
            if (l > 0 && (rc = states_below(l))) return rc;
            if ((rc = project(l > 0 ? ds.gru_xb : x, l))) return rc;
            if (l + 1 < layers) {
                const size_t so = seq_rows * H;
                if ((rc = gru_wave_launch(T, batch, H, ds.gru_gx, U + l * wsz, W + (l + 1) * wsz, U + (l + 1) * wsz,
                                          b + static_cast<size_t>(l) * 6 * H, b + static_cast<size_t>(l + 1) * 6 * H,
                                          h0 ? h0 + static_cast<size_t>(l) * batch * H : nullptr,
                                          h0 ? h0 + static_cast<size_t>(l + 1) * batch * H : nullptr,
                                          h_out + static_cast<size_t>(l) * so, h_out + static_cast<size_t>(l + 1) * so,
                                          ds.gru_hx, ds, stream)))
                    return rc;
                l += 2;
            } else {
                if ((rc = recur(l, false, false, false))) return rc;
                l += 1;
            }
        }
        return ISAM_OK;
    }

    // Layer l's recurrence also computes layer l + 1's projection (its slabs),
    // which layer l + 1 sums as it goes: a step or two behind in the same launch,
    // or in the next one.
    for (int l = 0; l < layers; l += together) {
        const int n = std::min(together, layers - l);
        if ((rc = gru_empty_rings(ds.gru_hx, n * ring_bytes(H, bp), stream))) return rc;
        if (n > 1) {
            const cudaError_t e =
                cudaMemsetAsync(ds.gru_gxp, 0xFF, (n - 1) * set_floats * sizeof(float), stream);  // kEmpty
            if (e != cudaSuccess) return cuda_error(e, "emptying the stacked GRU projections");
        }
        if (l == 0 && (rc = project(x, 0))) return rc;
        if ((rc = recur(l, l + n < layers, l > 0, false, n))) return rc;
    }
    return ISAM_OK;
}

int gru_launch(int T, int batch, int hidden, const uint16_t *x, const uint16_t *W,
               const uint16_t *U, const float *b, const float *h0, float *h_out, DeviceState &ds,
               cudaStream_t stream, int reset_before) {
    return gru_stack_launch(1, T, batch, hidden, reset_before, x, W, U, b, h0, h_out, ds, stream);
}

}  // namespace isam

// ===========================================================================
// Allocation-free variant of the GRU forward.
//
// Some callers cannot let a library call cudaMalloc: a serving process whose
// device memory is all reserved up front by its framework's caching allocator
// (a raw cudaMalloc would fail or fragment that pool), or a latency-bound
// request path that forbids cudaMalloc/cudaFree because they can synchronise
// the whole device.  isam_gru_forward_noalloc serves them: its workspaces
// (device error word, hidden-state exchange ring, and the input projection of up to a chunk of time steps) live in the fixed array
// below, so the call allocates nothing.  It launches the same two kernels as
// isam_gru_forward, one time chunk after another, carrying h from one chunk to
// the next through h_out.
// ===========================================================================
namespace isam {
namespace {

constexpr size_t kNoAllocScratchBytes = static_cast<size_t>(8) << 20;  // 8 MiB
constexpr size_t kNaErrOff = 0;      // 16-byte device error word
constexpr size_t kNaHxOff = 256;     // the exchange ring

}  // namespace
}  // namespace isam

// Every GPU that loads this library holds these 8 MiB until the process exits.
static __device__ __align__(256) unsigned char g_gru_noalloc_scratch[isam::kNoAllocScratchBytes];

namespace isam {
namespace {

struct NoAllocDevice {
    bool ready = false;
    unsigned char *scratch = nullptr;  // device address of g_gru_noalloc_scratch
    int num_sms = 0;
    int smem_optin = 0;
};
NoAllocDevice g_noalloc[64];
std::mutex g_noalloc_mu;

// Once per device, with that device current: the array's device address and
// the device limits the launches need.  No allocation happens here.
int noalloc_setup(int dev, NoAllocDevice *nd) {
    int major = 0, minor = 0;
    cudaError_t e = cudaDeviceGetAttribute(&major, cudaDevAttrComputeCapabilityMajor, dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&minor, cudaDevAttrComputeCapabilityMinor, dev);
    if (e != cudaSuccess) return cuda_error(e, "isam_gru_forward_noalloc: device attributes");
    if (major != 10 || minor != 3)
        return set_error(ISAM_ERR_UNSUPPORTED,
                         "isam_gru_forward_noalloc: built for sm_103a (GB300); device %d is sm_%d%d",
                         dev, major, minor);
    void *ptr = nullptr;
    e = cudaGetSymbolAddress(&ptr, g_gru_noalloc_scratch);
    if (e != cudaSuccess || ptr == nullptr)
        return cuda_error(e, "isam_gru_forward_noalloc: cudaGetSymbolAddress(scratch)");
    if ((e = cudaDeviceGetAttribute(&nd->num_sms, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess ||
        (e = cudaDeviceGetAttribute(&nd->smem_optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev)) !=
            cudaSuccess)
        return cuda_error(e, "isam_gru_forward_noalloc: device attributes");
    nd->scratch = static_cast<unsigned char *>(ptr);
    nd->ready = true;
    return ISAM_OK;
}

}  // namespace
}  // namespace isam

extern "C" int isam_gru_forward_noalloc(int T, int batch, int hidden, const isam_bf16 *x,
                                        const isam_bf16 *W, const isam_bf16 *U, const float *b,
                                        const float *h0, float *h_out) {
    using namespace isam;
    const int H = hidden;
    if (T < 1 || batch < 1 || H < 1)
        return set_error(ISAM_ERR_INVALID_ARG, "isam_gru_forward_noalloc: sizes must be >= 1");
    if (!x || !W || !U || !b || !h_out)
        return set_error(ISAM_ERR_INVALID_ARG, "isam_gru_forward_noalloc: null pointer");
    if (batch > kBatchPad || H % 32 != 0 || H > 1024 || H < 32)
        return set_error(ISAM_ERR_UNSUPPORTED,
                         "isam_gru_forward_noalloc: needs batch <= 32 and hidden a multiple of 32 "
                         "in [32, 1024] (batch=%d hidden=%d)",
                         batch, H);
    if ((reinterpret_cast<uintptr_t>(x) | reinterpret_cast<uintptr_t>(W) |
         reinterpret_cast<uintptr_t>(U) | reinterpret_cast<uintptr_t>(b) |
         reinterpret_cast<uintptr_t>(h0) | reinterpret_cast<uintptr_t>(h_out)) & 15u)
        return set_error(ISAM_ERR_UNSUPPORTED,
                         "isam_gru_forward_noalloc: pointers must be 16-byte aligned");
    // Scratch layout: error word | exchange ring | projection chunk.
    const size_t gx_off = (kNaHxOff + ring_bytes(H, kBatchPad) + 255) / 256 * 256;
    const size_t step_bytes = static_cast<size_t>(batch) * 3 * H * sizeof(float);
    const long long chunk = static_cast<long long>((kNoAllocScratchBytes - gx_off) / step_bytes);
    if (chunk < 1)
        return set_error(ISAM_ERR_UNSUPPORTED,
                         "isam_gru_forward_noalloc: one step's projection (%zu bytes) exceeds the "
                         "%zu-byte scratch",
                         step_bytes, kNoAllocScratchBytes - gx_off);

    int dev = -1;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return cuda_error(e, "cudaGetDevice");
    if (dev < 0 || dev >= 64)
        return set_error(ISAM_ERR_UNSUPPORTED, "device ordinal %d out of range", dev);
    NoAllocDevice nd;
    {
        std::lock_guard<std::mutex> lk(g_noalloc_mu);
        if (!g_noalloc[dev].ready) {
            int rc = noalloc_setup(dev, &g_noalloc[dev]);
            if (rc) return rc;
        }
        nd = g_noalloc[dev];
        int rc0 = gru_smem_attr(nd.smem_optin, dev);
        if (rc0) return rc0;
    }
    const int n_cta = gru_cta_count(H);
    const size_t smem = gru_smem_bytes(H);
    if (n_cta > nd.num_sms || smem > static_cast<size_t>(nd.smem_optin))
        return set_error(ISAM_ERR_UNSUPPORTED, "isam_gru_forward_noalloc: hidden too large");

    uint32_t *err = reinterpret_cast<uint32_t *>(nd.scratch + kNaErrOff);
    uint16_t *hx = reinterpret_cast<uint16_t *>(nd.scratch + kNaHxOff);
    float *gx = reinterpret_cast<float *>(nd.scratch + gx_off);
    cudaStream_t stream = current_stream();

    // A device view for the shared GEMM launcher: limits plus the scratch error word.
    DeviceState view;
    view.device = dev;
    view.num_sms = nd.num_sms;
    view.max_smem_optin = nd.smem_optin;
    view.err_word = err;

    int rc;
    if ((e = cudaMemsetAsync(err, 0, 16, stream)) != cudaSuccess)
        return cuda_error(e, "clearing the scratch error word");
    CUtensorMap no_next;
    memset(&no_next, 0, sizeof no_next);
    const size_t step_elems = static_cast<size_t>(batch) * H;
    for (long long t0 = 0; t0 < T; t0 += chunk) {
        const int tc = static_cast<int>(T - t0 < chunk ? T - t0 : chunk);
        // Input projection of steps [t0, t0 + tc): gx = x W^T + b_ih.
        GemmDesc g{tc * batch, 3 * H, H, 0, 1, 1.0f, 0.0f, x + static_cast<size_t>(t0) * step_elems, W,
                   gx, b};
        if ((rc = gru_empty_rings(hx, ring_bytes(H, kBatchPad), stream))) return rc;
        GemmPlan plan;
        if ((rc = gemm_validate(g))) return rc;
        if ((rc = gemm_plan(g, view, &plan))) return rc;
        if ((rc = gemm_launch(g, plan, view, stream))) return rc;
        // Recurrence over the chunk, starting from h_{t0 - 1} (h0 for the first chunk).
        GruParams p{};
        p.T = tc;
        p.U = U;
        p.total = batch;
        p.bstride = batch;
        p.H = H;
        p.gx = gx;
        p.b_hh = b + 3 * H;
        p.h0 = t0 == 0 ? h0 : h_out + static_cast<size_t>(t0 - 1) * step_elems;
        p.h_out = h_out + static_cast<size_t>(t0) * step_elems;
        p.hx = hx;
        p.skip_publish_cta = -1;
        p.timeout_ns = wait_timeout_ns();
        p.err = err;
        p.reset_before = 0;  // the reset-after form only
        p.gx_parts = 1;
        p.gx_slab = 0;
        p.b_ih = nullptr;
        p.has_next = 0;
        p.gxp_out = nullptr;
        if ((rc = launch_recurrent(p, no_next, smem, stream))) return rc;
    }
    // Report device-side timeouts of this call before returning: the error
    // word is read back on the call's own stream (no wait on other streams),
    // then that stream alone is synchronised.
    uint32_t w[4] = {0, 0, 0, 0};
    if ((e = cudaMemcpyAsync(w, err, sizeof w, cudaMemcpyDeviceToHost, stream)) != cudaSuccess)
        return cuda_error(e, "isam_gru_forward_noalloc: reading the scratch error word");
    if ((e = cudaStreamSynchronize(stream)) != cudaSuccess)
        return cuda_error(e, "isam_gru_forward_noalloc: cudaStreamSynchronize");
    if (w[0] & DEV_ERR_LAUNCH_SHAPE)
        return set_error(ISAM_ERR_CUDA,
                         "isam_gru_forward_noalloc: the recurrent kernel found clusters of %u CTAs, "
                         "not the shape it was launched for; h_out is undefined",
                         w[3]);
    if (w[0] != 0)
        return set_error(ISAM_ERR_TIMEOUT,
                         "isam_gru_forward_noalloc: a bounded device wait ran out (site 0x%x, "
                         "block %u); h_out is undefined",
                         w[1], w[2]);
    return ISAM_OK;
}
