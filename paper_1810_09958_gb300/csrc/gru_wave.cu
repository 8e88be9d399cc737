// gru_wave.cu -- two stacked GRU layers in one persistent kernel.
//
// Layer b reads layer a's states, so step t of b can run as soon as step t of
// a is done: in round r the kernel advances layer a to step r and layer b to
// step r - 1, and two layers take T + 1 rounds instead of 2 T.  The grid is
// the single-layer recurrence's (hidden / 32 clusters of 4 CTAs, each CTA one
// K quarter of one group of 32 units).  Per round a CTA gathers its quarter of
// bf16(h_a at step r - 1) and of bf16(h_b at step r - 2) and multiplies
//
//   U_a h_a            -> layer a's recurrent term for step r
//   W_b h_a + U_b h_b  -> layer b's terms for step r - 1 (the same h_a tile:
//                         the input projection of the upper layer comes from
//                         data the lower layer already loaded, Section 5.1.2)
//
// All three weight slices are A operands in tensor memory (384 columns at
// hidden 1024).  Layer b's accumulator sums both products of its r and z rows
// (lanes 0-63) and keeps the candidate's input term W_n h_a (lanes 64-95) and
// recurrent term U_n h_b (lanes 96-127) apart, because r multiplies only the
// latter: W_n's lanes are zero over U_b's K range and U_n's over W_b's.  Four
// rows per unit then cross the cluster instead of six.
//
// The two layers are two groups of warps, each running the single-layer
// kernel's round (gather by polling the exchange ring, push, reduce, gates,
// publish; gru.cu says why and how the ring is reused) at its own pace; they
// meet only in the MMA warp, which needs layer a's tile for W_b.  A round is
// then one chain of cross-SM latencies for both layers: hidden 1024, batch 32,
// 128 steps take 382 us for two layers (2.8 us for one more round; one layer 332
// us), against 1089 us with a step counter, weights in shared memory and all six row
// kinds of layer b crossing the cluster.  (The common sum of the r and z rows changes
// their last bits, not the error: over 32 runs of two to four layers at hidden 256 to
// 1024 it is 1.0001 times what separate sums give against 64 bits.)  Layer a's projection
// x W_a^T + b_ih for all steps is a GEMM before the kernel.  Reset gate after
// the recurrent product, hidden a multiple of 256 (4 K splits), batch <= 32.
// Every wait is bounded.
#include <cstdio>
#include <cstdlib>
#include <mutex>

#include "gru_common.cuh"
#include "internal.h"
#include "ptx.cuh"

namespace isam {

namespace {

constexpr int kKS = 4;                   // K splits = cluster size
constexpr int kGroup = 32;               // hidden units per cluster
constexpr int kUO = kGroup / kKS;        // units whose gates a CTA evaluates (8)
constexpr int kBatchPad = 32;
constexpr int kGateWarps = 8;            // per layer: one (unit, batch) pair per thread
constexpr int kMmaWarp = 2 * kGateWarps;
constexpr int kHouseWarp = kMmaWarp + 1; // one per layer: ring and barrier upkeep
constexpr int kThreads = 32 * (kHouseWarp + 2);
constexpr int kMaxAtoms = 4;             // K atoms of a quarter (hidden <= 1024)
constexpr int kAtomH = kBatchPad * 128;  // one K atom of h (4 KB)
constexpr int kRowBytes = kBatchPad * 4; // a received partial row
// Rows per unit and source that a CTA receives: r, z, n of layer a; r, z, the
// candidate's input and recurrent terms of layer b.
__host__ __device__ constexpr int wave_rows(int layer) { return layer == 0 ? 3 : 4; }
// Rows of the other CTAs' units that a CTA stages in a round.
__host__ __device__ constexpr int wave_stage_bytes(int layer) { return wave_rows(layer) * (kGroup - kUO) * kRowBytes; }
__host__ __device__ constexpr int wave_recv_bytes(int layer) { return kKS * wave_rows(layer) * kUO * kRowBytes; }
// TMEM columns: layer a's accumulator, layer b's two (by round parity), then
// the weights, 32 columns per K atom: U_a, W_b, U_b.
constexpr uint32_t kColA = 0, kColB = 32, kColW = 96;
constexpr uint32_t kTmemCols = 512;

enum : uint32_t {
    SITE_WAVE_W = 0x221,
    SITE_WAVE_H = 0x222,
    SITE_WAVE_MMA = 0x223,
    SITE_WAVE_RED = 0x224,
};

struct WaveParams {
    int T, batch, H;
    int ka, n_cta, slot;
    const uint16_t *U_a, *W_b, *U_b;  // [3H][H]
    const float *gx_a;         // [T*batch][3H]: x W_a^T + b_ih_a
    const float *b_hh_a;       // [3H]
    const float *b_ih_b;       // [3H]
    const float *b_hh_b;       // [3H]
    const float *h0[2];        // [batch][H] or null, per layer
    float *out[2];             // [T][batch][H]
    uint16_t *hx[2];           // kSlots x [H/8 pieces][32 rows][8] bf16 exchange ring, kEmpty before launch
    int bulk;                  // partial rows cross the cluster as bulk copies (else as 16-byte stores)
    int skip_publish_cta;      // debug: this CTA never publishes (-1: none)
    unsigned long long timeout_ns;
    uint32_t *err;
};

struct WaveLayout {
    int off_h[2], off_recv[2], off_gx, off_stage[2], off_bars, total;
};

// h_a tile | h_b tile | partial rows of a, of b (2 round parities each) |
// layer a's projection of 2 steps | staged partial rows of a, of b (kGruStages
// buffers each) | barriers.
__host__ __device__ inline WaveLayout wave_layout(int ka) {
    WaveLayout L;
    L.off_h[0] = 0;
    L.off_h[1] = ka * kAtomH;
    L.off_recv[0] = 2 * ka * kAtomH;
    L.off_recv[1] = L.off_recv[0] + 2 * wave_recv_bytes(0);
    L.off_gx = L.off_recv[1] + 2 * wave_recv_bytes(1);
    L.off_stage[0] = L.off_gx + 2 * 3 * 32 * kGateWarps * 4;
    L.off_stage[1] = L.off_stage[0] + kGruStages * wave_stage_bytes(0);
    L.off_bars = L.off_stage[1] + kGruStages * wave_stage_bytes(1);
    L.total = L.off_bars + 256 + 1024;
    return L;
}

__global__ void __launch_bounds__(kThreads, 1) gru_wave_kernel(const WaveParams p) {
    if (!launch_shape_ok(p.err, static_cast<uint32_t>(kKS), static_cast<uint32_t>(p.n_cta), 0x3E0u)) return;
    extern __shared__ uint8_t smem_raw[];
    uint8_t *smem = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) &
                                                ~static_cast<uintptr_t>(1023));
    const WaveLayout L = wave_layout(p.ka);
    uint64_t *bars = reinterpret_cast<uint64_t *>(smem + L.off_bars);
    uint64_t *h_full = bars;              // [2 layers] the round's vectors are in shared memory
    uint64_t *mma_done = bars + 2;        // [2 layers] the round's products complete
    uint64_t *w_done = bars + 4;          // W_b h_a complete: h_a's tile may be overwritten
    uint64_t *red_full = bars + 5;        // [2 layers][2 round parities] all partial rows of my units arrived
    uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(red_full + 4);
    volatile int *abort_flag = reinterpret_cast<volatile int *>(tmem_slot + 1);

    const int tid = threadIdx.x;
    const int warp = tid >> 5;
    const int lane = tid & 31;
    const int H = p.H;
    const int G = 3 * H;
    const int T = p.T;
    const int ka = p.ka;
    const int group = blockIdx.x / kKS;
    const uint32_t rank = cluster_ctarank();
    const int unit0 = group * kGroup;
    const int atom0 = static_cast<int>(rank) * ka;
    const WaitCtx w{p.timeout_ns, p.err, abort_flag};

    if (tid == 0) {
        for (int i = 0; i < 2; ++i) {
            mbar_init(&h_full[i], kGateWarps);
            mbar_init(&mma_done[i], 1);
        }
        mbar_init(w_done, 1);
        for (int i = 0; i < 4; ++i) mbar_init(&red_full[i], 1);  // armed with the bytes of a round's partial rows
        *abort_flag = 0;
        fence_mbar_init();
    }
    // The h tiles start as zeros: batch rows past the batch are never written.
    for (int i = tid; i < 2 * ka * kAtomH / 16; i += kThreads) reinterpret_cast<uint4 *>(smem)[i] = make_uint4(0u, 0u, 0u, 0u);
    fence_proxy_async_smem();
    __syncwarp();
    if (warp == 0) {
        tmem_alloc(tmem_slot, kTmemCols);
        tmem_relinquish();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tmem_slot;
    // The projection (and what came before it) is complete from here on.
    griddep_launch_dependents();
    __syncwarp();
    griddep_wait();
    // ---- priming: the weights into tensor memory (warps q, q + 4, q + 8: the
    // three slices' rows of lane quarter q).
    if (warp < 12) {
        const int q = warp & 3, part = warp >> 2;
        const uint16_t *base = part == 0 ? p.U_a : part == 1 ? p.W_b : p.U_b;
        // Gate whose rows this quarter holds; layer b keeps W_n in quarter 2
        // and U_n in quarter 3.  Layer a's quarter 3 is never read.
        const int g = part == 0 ? (q < 3 ? q : -1) : part == 1 ? (q < 3 ? q : -1) : (q < 2 ? q : q == 3 ? 2 : -1);
        const uint16_t *row = g >= 0 ? base + (static_cast<size_t>(g) * H + unit0 + lane) * H : nullptr;
        tmem_load_row(tmem + (static_cast<uint32_t>(q * 32) << 16) + kColW + static_cast<uint32_t>(part * ka * 32), row,
                      atom0 * 64, H, 0, ka * 8);
        tmem_st_wait();
    }
    tc_fence_before();
    __syncthreads();
    cluster_sync_all();  // peers' barriers exist before any remote store
    tc_fence_after();
    const int npiece = (p.batch + 3) >> 2;  // 16-byte pieces of a partial row that hold the batch
    auto round_bytes = [&](int layer) {
        const int rows = wave_rows(layer) * kUO;  // from each source
        return static_cast<uint32_t>(rows * ((kKS - 1) * (p.bulk ? kRowBytes : npiece * 16) + npiece * 16));
    };

    if (warp < 2 * kGateWarps) {
        const int layer = warp / kGateWarps;
        const int lw = warp % kGateWarps;
        const int ltid = tid - layer * 32 * kGateWarps;
        uint8_t *sH = smem + L.off_h[layer];
        const int rows = wave_rows(layer);
        const int recv_buf = wave_recv_bytes(layer);
        float *recv = reinterpret_cast<float *>(smem + L.off_recv[layer]);  // [2][src][row kind][2 halves][unit][16]
        uint64_t *red = red_full + 2 * layer;
        // This CTA evaluates the gates of units unit0 + rank*8 + [0, 8); thread
        // ltid takes unit ltid % 8 and batch row ltid / 8.
        const int ui = ltid % kUO;
        const int b = ltid / kUO;
        const int j = unit0 + static_cast<int>(rank) * kUO + ui;
        const bool live = b < p.batch;
        const bool publishes = static_cast<int>(blockIdx.x) != p.skip_publish_cta;
        const float *bh = layer == 0 ? p.b_hh_a : p.b_hh_b;
        const float bh_r = bh[j], bh_z = bh[H + j], bh_n = bh[2 * H + j];
        const float bi_r = layer == 0 ? 0.0f : p.b_ih_b[j], bi_z = layer == 0 ? 0.0f : p.b_ih_b[H + j],
                    bi_n = layer == 0 ? 0.0f : p.b_ih_b[2 * H + j];
        uint16_t *hx = p.hx[layer];
        uint16_t *pub = hx + static_cast<size_t>(j >> 3) * (kBatchPad * 8) + b * 8 + (j & 7);
        auto publish = [&](int slot, float v) {
            const uint32_t mine = f32_to_bf16_rne(v);
            const uint32_t next = __shfl_down_sync(0xffffffffu, mine, 1);
            if ((ui & 1) == 0 && live && publishes)
                st_relaxed_gpu(reinterpret_cast<uint32_t *>(pub + static_cast<size_t>(slot) * p.slot), mine | (next << 16));
        };
        float h = (p.h0[layer] != nullptr && live) ? p.h0[layer][static_cast<size_t>(b) * H + j] : 0.0f;
        publish(0, h);
        float *sgx = reinterpret_cast<float *>(smem + L.off_gx) + ltid;
        auto load_gx = [&](int t) {
            const bool on = live && t < T;
            const float *g = p.gx_a + (on ? (static_cast<size_t>(t) * p.batch + b) * G + j : 0);
#pragma unroll
            for (int q = 0; q < 3; ++q) cp_async_f32(sgx + ((t & 1) * 3 + q) * 32 * kGateWarps, g + q * H, on);
            cp_async_commit();
        };
        if (layer == 0) load_gx(0);
        float *out = p.out[layer] + static_cast<size_t>(b) * H + j;
        const size_t out_step = static_cast<size_t>(p.batch) * H;

        uint32_t mine = 0;
#pragma unroll
        for (int a = 0; a < kMaxAtoms; ++a)
            if (a < ka && lane < p.batch) mine |= 1u << a;
        const uint16_t *src0 = hx + (static_cast<size_t>(atom0 * 8 + lw) * kBatchPad + lane) * 8;
        uint8_t *dst0 = sH + lane * 128 + ((lw ^ (lane & 7)) << 4);
        // Push: warp lw sends half lw / 4 of the batch columns of lane quarter lw % 4.
        const int q = lw & 3, half = lw >> 2;
        const bool pushes = q < rows && (p.bulk || half * (kBatchPad / 8) < npiece);
        const uint32_t owner = static_cast<uint32_t>(lane / kUO);
        const int oui = lane % kUO;
        const int qr = q < rows ? q : 0;
        const int kind = ((static_cast<int>(rank) * rows + qr) * 2 + half) * kUO;  // first half row at the owner
        const uint32_t push_dst = mapa_shared(smem_u32(recv) + static_cast<uint32_t>((kind + oui) * (kRowBytes / 2)), owner);
        const uint32_t push_bar = mapa_shared(smem_u32(red), owner);
        // Bulk form: staged as [round parity][row kind][half][other owner][8 units][16].
        const int peer = static_cast<int>(owner) - (owner > rank ? 1 : 0);
        uint8_t *stage = smem + L.off_stage[layer] + (qr * 2 + half) * (kGroup - kUO) * (kRowBytes / 2);
        uint8_t *stage_row = stage + (peer * kUO + oui) * (kRowBytes / 2);
        const uint32_t to = static_cast<uint32_t>(lane % kKS);  // lanes 0 .. 3 send to owner `lane`
        const bool sends = lane < kKS && to != rank;
        const uint32_t stage_part = smem_u32(stage) + (to - (to > rank ? 1u : 0u)) * static_cast<uint32_t>(kUO * kRowBytes / 2);
        const uint32_t part_dst = mapa_shared(smem_u32(recv) + static_cast<uint32_t>(kind * (kRowBytes / 2)), to);
        const uint32_t part_bar = mapa_shared(smem_u32(red), to);
        const uint32_t acc = tmem + (static_cast<uint32_t>(q * 32) << 16) + (layer == 0 ? kColA : kColB);

        // Step s of this layer; layer a gathers once more for layer b's last step.
        bool ok = true;
        const int gathers = layer == 0 ? T + 1 : T;
        for (int s = 0; s < gathers; ++s) {
            const uint32_t par = static_cast<uint32_t>(s & 1);
            // W_b h_a of the round before still reads the tile.
            if (layer == 0 && s >= 2 && !all_wait(w_done, par, w, SITE_WAVE_MMA)) {
                ok = false;
                break;
            }
            if (!gather_tile<kMaxAtoms, 1>(src0 + static_cast<size_t>(s & (kSlots - 1)) * p.slot, dst0, mine,
                                           kBatchPad * 64, kAtomH, &h_full[layer], lane, w)) {
                ok = false;
                break;
            }
            // While the MMAs run: the last step's state, the next step's projection.
            if (s > 0 && live) out[static_cast<size_t>(s - 1) * out_step] = h;
            if (s == T) break;
            if (layer == 0) load_gx(s + 1);
            if (pushes) {
                if (!all_wait(&mma_done[layer], par, w, SITE_WAVE_MMA)) {
                    ok = false;
                    break;
                }
                tc_fence_after();
                const uint32_t acc_now = acc + (layer == 0 ? 0u : 32u * par);
                const uint32_t buf = par * static_cast<uint32_t>(recv_buf);
                const uint32_t stage_buf = par * static_cast<uint32_t>(wave_stage_bytes(layer));
                if (p.bulk)
                    push_rows_bulk<kBatchPad>(acc_now, half, npiece, owner != rank, stage_row + stage_buf, push_dst + buf,
                                              oui, push_bar + par * 8u, sends, stage_part + stage_buf, part_dst + buf,
                                              part_bar + par * 8u, static_cast<uint32_t>(kUO * kRowBytes / 2));
                else
                    push_rows<kBatchPad>(acc_now, half, npiece, push_dst + buf, oui, push_bar + par * 8u);
            }
            float xr = bi_r, xz = bi_z, xn = bi_n;
            if (layer == 0) {
                cp_async_wait_all_but_last();
                const float *v = sgx + static_cast<int>(par) * 3 * 32 * kGateWarps;
                xr += v[0];
                xz += v[32 * kGateWarps];
                xn += v[2 * 32 * kGateWarps];
            }
            if (!all_wait<true>(&red[par], static_cast<uint32_t>(s >> 1) & 1u, w, SITE_WAVE_RED)) {
                ok = false;
                break;
            }
            // Partials summed over the 4 source ranks in rank order.
            const float *rv = recv + par * (recv_buf / 4) + recv_at<kBatchPad, kUO>(ui, b);
            auto part = [&](int src, int kind) { return rv[(src * rows + kind) * kUO * kBatchPad]; };
            float gr = bh_r, gz = bh_z, gn = bh_n;
#pragma unroll
            for (int src = 0; src < kKS; ++src) {
                gr += part(src, 0);
                gz += part(src, 1);
                if (layer == 0) {
                    gn += part(src, 2);
                } else {
                    xn += part(src, 2);
                    gn += part(src, 3);
                }
            }
            const float rg = sigmoidf_fast(xr + gr);
            const float zg = sigmoidf_fast(xz + gz);
            h = gru_blend(zg, gru_candidate(xn, rg, gn), h);
            publish((s + 1) & (kSlots - 1), h);
        }
        if (ok && layer == 1 && live) out[static_cast<size_t>(T - 1) * out_step] = h;
    } else if (warp == kMmaWarp) {
        const bool lead = elect_one();
        if (lead) {
            mbar_arrive_expect_tx(&red_full[0], round_bytes(0));
            mbar_arrive_expect_tx(&red_full[2], round_bytes(1));
        }
        __syncwarp();
        const uint32_t idesc = idesc_bf16_f32(128, kBatchPad, false, false);
        // Product of weight slice `part` with layer `layer`'s tile.
        auto issue = [&](int part, int layer, uint32_t d, bool fresh) {
#pragma unroll
            for (int a = 0; a < kMaxAtoms; ++a) {
                if (a >= ka) break;
                const uint64_t hd = sdesc_sw128(smem_u32(smem + L.off_h[layer] + a * kAtomH), 16, 1024);
                const uint32_t wa = tmem + kColW + static_cast<uint32_t>((part * ka + a) * 32);
#pragma unroll
                for (int k = 0; k < 4; ++k)
                    umma_bf16_ts(tmem + d, wa + k * 8, hd + k * 2, idesc, (!fresh || a > 0 || k > 0) ? 1u : 0u);
            }
        };
        int a_done = -1, b_done = -1;  // for the drains after an abort
        for (int r = 0; r <= T; ++r) {
            if (!all_wait(&h_full[0], static_cast<uint32_t>(r & 1), w, SITE_WAVE_H)) break;
            tc_fence_after();
            // Layer b's accumulator of this round, last read two rounds ago: its
            // warps gathered the previous round's tile after that.
            const uint32_t colb = kColB + 32u * static_cast<uint32_t>((r - 1) & 1);
            if (lead) {
                if (r < T) {
                    issue(0, 0, kColA, true);
                    umma_commit(&mma_done[0]);
                }
                if (r >= 1) {
                    issue(1, 0, colb, true);
                    umma_commit(w_done);
                }
            }
            __syncwarp();
            a_done = r;
            if (r >= 1) {
                if (!all_wait(&h_full[1], static_cast<uint32_t>((r - 1) & 1), w, SITE_WAVE_H)) break;
                tc_fence_after();
                if (lead) {
                    issue(2, 1, colb, false);
                    umma_commit(&mma_done[1]);
                }
                __syncwarp();
                b_done = r - 1;
            }
        }
        // Every product issued has completed before TMEM is released (the last
        // commit of this thread covers those before it).
        if (a_done >= 0 && a_done < T) drain_bar(&mma_done[0], static_cast<uint32_t>(a_done & 1), p.timeout_ns);
        if (a_done >= 1) drain_bar(w_done, static_cast<uint32_t>((a_done - 1) & 1), p.timeout_ns);
        if (b_done >= 0) drain_bar(&mma_done[1], static_cast<uint32_t>(b_done & 1), p.timeout_ns);
        __syncwarp();
    } else {
        // Ring and barrier upkeep of one layer (gru.cu).
        const int layer = warp - kHouseWarp;
        uint64_t *red = red_full + 2 * layer;
        uint16_t *own = p.hx[layer] + static_cast<size_t>((unit0 >> 3) + static_cast<int>(rank)) * (kBatchPad * 8);
        for (int s = 0; s < T; ++s) {
            if (!all_wait<true>(&red[s & 1], static_cast<uint32_t>(s >> 1) & 1u, w, SITE_WAVE_RED)) break;
            if (s >= 1) {
                if (lane < p.batch)
                    *reinterpret_cast<uint4 *>(own + static_cast<size_t>((s + 3) & (kSlots - 1)) * p.slot + lane * 8) =
                        make_uint4(kEmpty, kEmpty, kEmpty, kEmpty);
                fence_acq_rel_gpu();
            }
            __syncwarp();
            if (lane == 0 && s + 1 < T) mbar_arrive_expect_tx(&red[(s + 1) & 1], round_bytes(layer));
            __syncwarp();
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
    // memory; every wait above is bounded, so every CTA gets here.
    cluster_sync_all();
    if (warp == 0) {
        tc_fence_after();
        tmem_dealloc(tmem, kTmemCols);
    }
}

}  // namespace

size_t gru_wave_smem_bytes(int H) { return static_cast<size_t>(wave_layout(H / (kKS * 64)).total); }

size_t gru_wave_ring_bytes(int H) { return static_cast<size_t>(2) * kSlots * kBatchPad * H * sizeof(uint16_t); }

bool gru_wave_fits(int H, int batch, int num_sms, int smem_optin) {
    if (H % 256 != 0 || H < 256 || H > 1024 || batch < 1 || batch > kBatchPad) return false;
    if (H / kGroup * kKS > num_sms) return false;
    return gru_wave_smem_bytes(H) <= static_cast<size_t>(smem_optin);
}

bool gru_wave_supported(int H, int batch, const DeviceState &ds) {
    return gru_wave_fits(H, batch, ds.num_sms, ds.max_smem_optin);
}

int gru_wave_launch(int T, int batch, int H, const float *gx_a, const uint16_t *U_a, const uint16_t *W_b,
                    const uint16_t *U_b, const float *b_a, const float *b_b, const float *h0_a,
                    const float *h0_b, float *out_a, float *out_b, uint16_t *hx, DeviceState &ds,
                    cudaStream_t stream) {
    if (!gru_wave_supported(H, batch, ds))
        return set_error(ISAM_ERR_UNSUPPORTED, "two-layer GRU kernel: hidden %d, batch %d not supported", H, batch);
    WaveParams p{};
    p.T = T;
    p.batch = batch;
    p.H = H;
    p.ka = H / (kKS * 64);
    p.n_cta = H / kGroup * kKS;
    p.slot = kBatchPad * H;
    p.U_a = U_a;
    p.W_b = W_b;
    p.U_b = U_b;
    p.gx_a = gx_a;
    p.b_hh_a = b_a + 3 * H;
    p.b_ih_b = b_b;
    p.b_hh_b = b_b + 3 * H;
    p.h0[0] = h0_a;
    p.h0[1] = h0_b;
    p.out[0] = out_a;
    p.out[1] = out_b;
    p.hx[0] = hx;
    p.hx[1] = hx + static_cast<size_t>(kSlots) * p.slot;
    p.bulk = gru_push_bulk(batch, kBatchPad) ? 1 : 0;
    p.skip_publish_cta = -1;
    if (const char *s = getenv("ISAM_DEBUG_GRU_SKIP_CTA")) p.skip_publish_cta = atoi(s);
    p.timeout_ns = wait_timeout_ns();
    p.err = ds.err_word;

    int rc;
    if ((rc = ensure_smem_optin(reinterpret_cast<const void *>(gru_wave_kernel), ds.max_smem_optin, ds.device,
                                "cudaFuncSetAttribute(gru wave)")))
        return rc;
    const size_t smem = gru_wave_smem_bytes(H);
    cudaLaunchConfig_t cfg = {};
    // A plain cluster launch, once every cluster is known to fit at the same
    // time (the exchange needs every CTA resident); no cooperative
    // attribute, whose combination with the cluster shape a tool's re-issue
    // of the launch can drop.
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = kKS;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.gridDim = dim3(static_cast<unsigned>(p.n_cta), 1, 1);
    cfg.blockDim = dim3(kThreads, 1, 1);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = stream;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    int max_clusters = 0;
    cudaError_t e = cudaOccupancyMaxActiveClusters(&max_clusters, gru_wave_kernel, &cfg);
    if (e != cudaSuccess) return cuda_error(e, "cudaOccupancyMaxActiveClusters(gru wave)");
    if (max_clusters * kKS < p.n_cta)
        return set_error(ISAM_ERR_UNSUPPORTED, "two-layer GRU kernel: %d CTAs in clusters of 4 cannot be co-resident",
                         p.n_cta);
    // The caller has emptied the rings ahead of the projection.  A dependent launch
    // starts about 1.5 us earlier, but its clusters are placed around the projection's
    // last CTAs and a step takes 0.07 us longer: off / on 34.0 / 32.5 us for 4 steps at
    // hidden 1024, batch 32, 88.0 / 87.6 for 24, 112.0 / 112.1 for 32, 132.6 / 133.5 for
    // 40, 378 / 386 for 128.
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.numAttrs = T <= 32 ? 2 : 1;
    e = cudaLaunchKernelEx(&cfg, gru_wave_kernel, p);
    if (e != cudaSuccess) return cuda_error(e, "launch gru_wave_kernel");
    return ISAM_OK;
}

}  // namespace isam
