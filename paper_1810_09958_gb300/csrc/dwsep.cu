// dwsep.cu -- separable depthwise convolution (Listing 3 with s = 1, c = 1,
// zero border of one pixel) on sm_103a, in the factored form of Section 2.3:
// the 3x3 depthwise sum is formed first and the result is multiplied by the
// pointwise weights, a GEMM with M = N*H*W pixels, K = Cin, N = Cout.
//
// One persistent kernel, one CTA per SM, tiles of 128 pixels: a patch of one
// image.  Its input comes in 64-channel chunks by TMA, producer warps form the
// depthwise sums of a chunk in fp32, round them to bf16 and write the A tile
// straight into the tensor cores' 128-byte swizzled K-major layout, one warp
// multiplies it with the pointwise weights (resident for the whole kernel) into
// a double-buffered TMEM accumulator, and epilogue warps drain TMEM to C with
// bulk tensor stores (see dwsep_patch_kernel).
// The depthwise intermediate never leaves the chip.
#include <algorithm>
#include <cstdio>

#include "dw_common.cuh"
#include "internal.h"
#include "ptx.cuh"

namespace isam {

namespace {

constexpr int kBM = kPatchPixels;
enum : uint32_t {
    SITE_DW_AEMPTY = 0x301,
    SITE_DW_AFULL = 0x302,
    SITE_DW_TEMPTY = 0x303,
    SITE_DW_TFULL = 0x304,
    SITE_DW_W = 0x305,
    SITE_DW_RING = 0x306,
};

struct DwPatchParams {
    int H, W, Cin, Cout;
    int step;               // output channels of one grid row (a multiple of 32, or all of them)
    int ty, tx;             // patches per image: down, across
    int tiles;              // N * ty * tx
    int atoms;              // ceil(Cin / 64): 64-channel chunks of a patch, K atoms of its product
    int nchunks;            // ceil(step / 64) 64-wide column chunks of the weights
    int stages_p, stages_a; // patch chunks in flight, A ring depth
    const uint16_t *dw;
    unsigned long long timeout_ns;
    uint32_t *err;
};

constexpr int kPatchStagesMax = 4;
constexpr int kAStagesMax = 4;
constexpr int kPGroups = 2;
constexpr int kPProdWarps = kPGroups * kChunkWarps;
constexpr int kPLoadWarp = kPProdWarps;
constexpr int kPMmaWarp = kPProdWarps + 1;
constexpr int kPEpiWarp0 = kPMmaWarp + 1;  // warp w reads TMEM lane quarter w % 4
constexpr int kPEpiWarps = 8;
constexpr int kPThreads = (kPEpiWarp0 + kPEpiWarps) * 32;

struct DwPatchLayout {
    int off_w, off_a, off_stage, off_patch, off_dw, off_bars, total;
};

__host__ __device__ inline DwPatchLayout dw_patch_layout(int Cin, int Cout, int pw, int stages_p, int stages_a) {
    DwPatchLayout L;
    const int atoms = (Cin + 63) / 64;
    const int nchunks = (Cout + 63) / 64;
    L.off_w = 0;
    L.off_a = L.off_w + atoms * nchunks * 8192;
    L.off_stage = L.off_a + stages_a * kBM * 128;
    L.off_patch = L.off_stage + kPEpiWarps * 4096;
    L.off_dw = L.off_patch + stages_p * dw_patch_bytes(pw);
    L.off_bars = L.off_dw + 9 * atoms * 128;
    L.total = L.off_bars + 256 + 1024;
    return L;
}

// ---------------------------------------------------------------- patches
// Images of any width: a tile is a patch of 128 / PW rows x PW columns of one
// image, and its input (with a halo of one pixel) comes in chunks of 64 channels
// as 4-D TMA boxes.  Pixels outside the image are the tensor map's fill value,
// so the taps need no bounds test, and the output boxes are clipped the same
// way.
//
//   warps 0-15   depthwise producers in two groups of 8 that take alternate
//                chunks: thread = 4 channels of one column, walking down the
//                rows.  Each input row adds to the three outputs that see it,
//                so only 3 x 4 sums are live and an input is read from shared
//                memory once per column that needs it;
//   warp 16      loads the patches (two to four in flight);
//   warp 17      loads the pointwise weights once, issues the MMAs of a chunk
//                as soon as it is in the A ring;
//   warps 18-25  epilogue, two per TMEM lane quarter.
//
// What bounds it: with many patches the output writes (32 x 56 x 56, 128 -> 256
// at 24.3 us is 5.3 TB/s of unique bytes, a plain copy 6.8), with few the first
// patch's latency (5.6 us for any layer of up to one patch per SM).  Two kernels
// preceded it.  Whole image rows as tiles, the input rows in a shared-memory
// ring (widths to 128): its producers walked along the rows with a window of 12
// inputs in registers and a CTA barrier a tile, one A tile at a time, 30.4 us on
// the layer above; 16 x 112 x 112, 32 -> 64: 29.3 -> 17.1 us; 4 x 14 x 14,
// 32 -> 48: 9.6 -> 5.6 us.  Nine 16-byte taps an output from L1/L2 (other widths):
// 5 x 75 x 150, 48 -> 80: 26.0 -> 10.9 us; 2 x 130 x 180, 128 -> 128: 58 -> 13.6 us.
// Patches in flight on the first layer: 2 / 3 / 4 gave 29.6 / 25.8 / 25.1 us and a
// third A chunk at 3 patches 26.2, before TMA and MMA were issued under elect.sync.
template <int PW>
__global__ void __launch_bounds__(kPThreads, 1)
    dwsep_patch_kernel(const __grid_constant__ CUtensorMap tmX, const __grid_constant__ CUtensorMap tmW,
                       const __grid_constant__ CUtensorMap tmOut, const DwPatchParams p) {
    constexpr int PH = kBM / PW;                // patch rows
    constexpr int PBYTES = dw_patch_bytes(PW);
    extern __shared__ uint8_t smem_raw[];
    uint8_t *smem = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) &
                                                ~static_cast<uintptr_t>(1023));
    const DwPatchLayout L = dw_patch_layout(p.Cin, p.step, PW, p.stages_p, p.stages_a);
    uint8_t *sW = smem + L.off_w;
    uint8_t *sA = smem + L.off_a;
    uint8_t *sPatch = smem + L.off_patch;
    uint64_t *bars = reinterpret_cast<uint64_t *>(smem + L.off_bars);
    uint64_t *p_full = bars;                       // [stages_p] patch chunk landed
    uint64_t *p_empty = p_full + kPatchStagesMax;  // [stages_p] its producers have read it
    uint64_t *a_full = p_empty + kPatchStagesMax;  // [stages_a] A chunk written
    uint64_t *a_empty = a_full + kAStagesMax;      // [stages_a] its MMAs are done
    uint64_t *tfull = a_empty + kAStagesMax;       // [2]
    uint64_t *tempty = tfull + 2;                // [2]
    uint64_t *wbar = tempty + 2;
    uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(wbar + 1);
    volatile int *abort_flag = reinterpret_cast<volatile int *>(tmem_slot + 1);

    const int tid = threadIdx.x;
    const int warp = tid >> 5;
    const int lane = tid & 31;
    const int atoms = p.atoms, PS = p.stages_p, AS = p.stages_a;
    // This CTA's output channels: c0 .. c0 + cout - 1 (grid row blockIdx.y).
    const int c0 = static_cast<int>(blockIdx.y) * p.step;
    const int cout = min(p.step, p.Cout - c0);
    const int ncols = cout <= 64 ? 64 : (cout <= 128 ? 128 : 256);  // accumulator width (pow2)
    const uint32_t tmem_cols = 2u * static_cast<uint32_t>(ncols);
    const WaitCtx w{p.timeout_ns, p.err, abort_flag};

    if (tid == 0) {
        for (int s = 0; s < PS; ++s) {
            mbar_init(&p_full[s], 1);
            mbar_init(&p_empty[s], kChunkWarps);
        }
        for (int s = 0; s < AS; ++s) {
            mbar_init(&a_full[s], kChunkWarps);
            mbar_init(&a_empty[s], 1);
        }
        for (int i = 0; i < 2; ++i) {
            mbar_init(&tfull[i], 1);
            mbar_init(&tempty[i], kPEpiWarps);
        }
        mbar_init(wbar, 1);
        *abort_flag = 0;
        fence_mbar_init();
        tma_prefetch_desc(&tmX);
        tma_prefetch_desc(&tmW);
        tma_prefetch_desc(&tmOut);
    }
    __syncwarp();
    if (warp == kPMmaWarp) {
        tmem_alloc(tmem_slot, tmem_cols);
        tmem_relinquish();
    }
    // The previous kernel's results are complete from here on.
    griddep_launch_dependents();
    griddep_wait();
    // Taps as [9][atoms * 64], zero past Cin.
    uint32_t *sDw = reinterpret_cast<uint32_t *>(smem + L.off_dw);
    for (int i = tid; i < 9 * atoms * 32; i += kPThreads) {
        const int t = i / (atoms * 32), c2 = i - t * (atoms * 32);
        sDw[i] = 2 * c2 < p.Cin ? *reinterpret_cast<const uint32_t *>(p.dw + t * p.Cin + 2 * c2) : 0u;
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = *tmem_slot;
    const int per_img = p.ty * p.tx;

    if (warp < kPProdWarps) {
        // ------------------------------------------------ depthwise producers
        const int grp = warp / kChunkWarps;
        const int g = lane & 15;                                      // channels 4g .. 4g + 3 of the chunk
        const int walker = (warp % kChunkWarps) * 2 + (lane >> 4);   // column (and row segment) of this thread
        const int my_tiles = static_cast<int>(blockIdx.x) < p.tiles
                                 ? (p.tiles - 1 - static_cast<int>(blockIdx.x)) / static_cast<int>(gridDim.x) + 1
                                 : 0;
        const int items = my_tiles * atoms;
        int ps = grp % PS, as = grp % AS, chunk = grp % atoms, loaded = -1;
        uint32_t pph = static_cast<uint32_t>(grp / PS) & 1u, aph = static_cast<uint32_t>(grp / AS) & 1u;
        uint32_t wt[9][2];
        for (int it = grp; it < items; it += kPGroups) {
            if (chunk != loaded) {
#pragma unroll
                for (int t = 0; t < 9; ++t) {
                    const uint2 v = *reinterpret_cast<const uint2 *>(sDw + t * (atoms * 32) + chunk * 32 + g * 2);
                    wt[t][0] = v.x;
                    wt[t][1] = v.y;
                }
                loaded = chunk;
            }
            if (!__all_sync(0xffffffffu, bounded_wait(&p_full[ps], pph, w, SITE_DW_RING) &&
                                             bounded_wait(&a_empty[as], aph ^ 1u, w, SITE_DW_AEMPTY)))
                break;
            dw_chunk<PW>(sPatch + ps * PBYTES, sA + as * (kBM * 128), walker, g, wt);
            fence_proxy_async_smem();
            __syncwarp();
            if (lane == 0) {
                mbar_arrive(&p_empty[ps]);
                mbar_arrive(&a_full[as]);
            }
            for (int k = 0; k < kPGroups; ++k) {
                if (++ps == PS) {
                    ps = 0;
                    pph ^= 1u;
                }
                if (++as == AS) {
                    as = 0;
                    aph ^= 1u;
                }
                if (++chunk == atoms) chunk = 0;
            }
        }
        __syncwarp();
    } else if (warp == kPLoadWarp) {
        // ------------------------------------------------ patch loader
        if (elect_one()) {
            int st = 0, issued = 0;
            uint32_t ph = 0;
            bool ok = true;
            for (int tile = blockIdx.x; ok && tile < p.tiles; tile += gridDim.x) {
                const int n = tile / per_img, rem = tile - n * per_img;
                const int yt = rem / p.tx, xt = rem - yt * p.tx;
                for (int c = 0; c < atoms; ++c) {
                    if (!bounded_wait(&p_empty[st], ph ^ 1u, w, SITE_DW_RING)) {
                        ok = false;
                        break;
                    }
                    mbar_arrive_expect_tx(&p_full[st], static_cast<uint32_t>(PBYTES));
                    tma_load_4d(&tmX, &p_full[st], sPatch + st * PBYTES, c * 64, xt * PW - 1, yt * PH - 1, n);
                    ++issued;
                    if (++st == PS) {
                        st = 0;
                        ph ^= 1u;
                    }
                }
            }
            // Every copy already issued lands before the CTA can exit.
            for (int i = min(issued, PS); i > 0; --i) {
                if (--st < 0) {
                    st = PS - 1;
                    ph ^= 1u;
                }
                dw_drain(&p_full[st], ph, p.timeout_ns);
            }
        }
        __syncwarp();
    } else if (warp == kPMmaWarp) {
        // ------------------------------------------------ weights + MMA issuer
        const bool lead = elect_one();
        if (lead) {
            mbar_arrive_expect_tx(wbar, static_cast<uint32_t>(atoms * p.nchunks * 8192));
            for (int kb = 0; kb < atoms; ++kb)
                for (int c = 0; c < p.nchunks; ++c)
                    tma_load_2d(&tmW, wbar, sW + (kb * p.nchunks + c) * 8192, c0 + c * 64, kb * 64);
        }
        __syncwarp();
        bool ok = __all_sync(0xffffffffu, bounded_wait(wbar, 0, w, SITE_DW_W));
        if (!ok) dw_drain(wbar, 0, p.timeout_ns);
        const uint32_t idesc = idesc_bf16_f32(kBM, cout, false, true);
        int as = 0, acc = 0;
        uint32_t aph = 0, acc_phase = 0;
        for (int tile = blockIdx.x; ok && tile < p.tiles; tile += gridDim.x) {
            if (!__all_sync(0xffffffffu, bounded_wait(&tempty[acc], acc_phase ^ 1u, w, SITE_DW_TEMPTY))) break;
            const uint32_t d = tmem_base + static_cast<uint32_t>(acc * ncols);
            for (int c = 0; c < atoms; ++c) {
                if (!__all_sync(0xffffffffu, bounded_wait(&a_full[as], aph, w, SITE_DW_AFULL))) {
                    ok = false;
                    break;
                }
                tc_fence_after();
                if (lead) {
                    const uint32_t a0 = smem_u32(sA + as * (kBM * 128));
                    const uint32_t w0 = smem_u32(sW + c * (p.nchunks * 8192));
                    const int ks = min(4, (p.Cin - c * 64) / 16);
                    for (int k = 0; k < ks; ++k)
                        umma_bf16(d, sdesc_sw128(a0 + k * 32, 16, 1024), sdesc_sw128(w0 + k * 2048, 8192, 1024), idesc,
                                  (c > 0 || k > 0) ? 1u : 0u);
                    umma_commit(&a_empty[as]);
                    if (c + 1 == atoms) umma_commit(&tfull[acc]);
                }
                __syncwarp();
                if (++as == AS) {
                    as = 0;
                    aph ^= 1u;
                }
            }
            if (++acc == 2) {
                acc = 0;
                acc_phase ^= 1u;
            }
        }
        __syncwarp();
    } else if (warp >= kPEpiWarp0) {
        // ------------------------------------------------ epilogue
        // Two warps per TMEM lane quarter q, taking alternate 32-column chunks.
        // The quarter is 32 / PW whole patch rows: one box of the output map.
        const int q = warp & 3;
        const bool lead = elect_one();
        const int ew = warp - kPEpiWarp0;
        const int c_first = (ew >> 2) * 32;
        uint8_t *sb = smem + L.off_stage + ew * 4096;
        int acc = 0;
        uint32_t acc_phase = 0;
        for (int tile = blockIdx.x; tile < p.tiles; tile += gridDim.x) {
            const int n = tile / per_img, rem = tile - n * per_img;
            const int yt = rem / p.tx, xt = rem - yt * p.tx;
            const int y = yt * PH + q * (32 / PW), x = xt * PW;
            if (!__all_sync(0xffffffffu, bounded_wait(&tfull[acc], acc_phase, w, SITE_DW_TFULL))) break;
            tc_fence_after();
            const uint32_t tb = tmem_base + (static_cast<uint32_t>(q * 32) << 16) + static_cast<uint32_t>(acc * ncols);
            if (y < p.H) {
                for (int c = c_first; c < cout; c += 64) {
                    uint32_t r[32];
                    if (cout - c >= 32)
                        tmem_ld32(tb + c, r);
                    else
                        tmem_ld16(tb + c, *reinterpret_cast<uint32_t(*)[16]>(&r[0]));
                    if (lead) bulk_wait_read<0>();  // the previous store has read the buffer
                    __syncwarp();
                    tmem_ld_wait(r);
#pragma unroll
                    for (int ch = 0; ch < 8; ++ch)
                        *reinterpret_cast<uint4 *>(sb + lane * 128 + ((ch ^ (lane & 7)) << 4)) =
                            make_uint4(r[4 * ch], r[4 * ch + 1], r[4 * ch + 2], r[4 * ch + 3]);
                    fence_proxy_async_smem();
                    __syncwarp();
                    if (lead) {
                        tma_store_4d(&tmOut, sb, c0 + c, x, y, n);
                        bulk_commit();
                    }
                    __syncwarp();
                }
            }
            tc_fence_before();
            __syncwarp();
            if (lead) mbar_arrive(&tempty[acc]);
            __syncwarp();
            if (++acc == 2) {
                acc = 0;
                acc_phase ^= 1u;
            }
        }
        if (lead) bulk_wait_all<0>();
        __syncwarp();
    }

    tc_fence_before();
    __syncthreads();
    if (warp == kPMmaWarp) {
        tc_fence_after();
        tmem_dealloc(tmem_base, tmem_cols);
    }
}

using DwPatchKernel = void (*)(const CUtensorMap, const CUtensorMap, const CUtensorMap, const DwPatchParams);

DwPatchKernel dw_patch_kernel_for(int pw) {
    return pw == 8 ? dwsep_patch_kernel<8> : pw == 16 ? dwsep_patch_kernel<16> : dwsep_patch_kernel<32>;
}

// ---------------------------------------------------------------- host side
bool dw_channels_ok(int Cin, int Cout) {
    return Cin % 16 == 0 && Cin >= 16 && Cin <= 256 && Cout % 16 == 0 && Cout >= 16 && Cout <= 256;
}

// Channels of a block when `blocks` share them out (one block has them all).
int dw_step(int Cout, int blocks) { return blocks == 1 ? Cout : ((Cout + blocks - 1) / blocks + 31) / 32 * 32; }

// Fewest blocks of the output channels whose weights fit beside two patch chunks and
// two A chunks; 0 if none does.
int dw_fewest_blocks(int Cin, int Cout, int pw, int smem_optin) {
    int blocks = 1;
    while (dw_patch_layout(Cin, dw_step(Cout, blocks), pw, 2, 2).total > smem_optin) {
        if (dw_step(Cout, blocks) <= 32) return 0;
        ++blocks;
    }
    const int step = dw_step(Cout, blocks);
    return (Cout + step - 1) / step;
}

}  // namespace

int dwsep_plan(int N, int H, int W, int Cin, int Cout, int num_sms, int smem_optin, DwsepPlan *plan) {
    if (!dw_channels_ok(Cin, Cout))
        return set_error(ISAM_ERR_UNSUPPORTED,
                         "isam_dwsep_conv: needs Cin and Cout multiples of 16 in [16, 256] "
                         "(Cin=%d Cout=%d)",
                         Cin, Cout);
    const long long M = static_cast<long long>(N) * H * W;
    if (M > (1ll << 31) - 256)
        return set_error(ISAM_ERR_UNSUPPORTED, "isam_dwsep_conv: N*H*W too large");
    DwsepPlan p;
    p.patch_w = dw_patch_width(H, W);
    p.patch_h = kBM / p.patch_w;
    p.patches = N * ((H + p.patch_h - 1) / p.patch_h) * ((W + p.patch_w - 1) / p.patch_w);  // at most N * H * W
    // Blocks share the output channels out: as few as the resident weights allow,
    // since each recomputes the depthwise stage, but as many as idle SMs can take (a
    // CTA's start loads its share of the weights, and its tail drains its share of
    // the last tile: 32 x 14 x 14, 256 -> 256, 64 patches: 17.8 us as two launches, 9.2
    // as two grid rows).
    p.blocks = dw_fewest_blocks(Cin, Cout, p.patch_w, smem_optin);
    if (p.blocks < 1)
        return set_error(ISAM_ERR_UNSUPPORTED, "isam_dwsep_conv: Cin=%d does not fit shared memory", Cin);
    while (2LL * p.blocks * p.patches <= num_sms && dw_step(Cout, 2 * p.blocks) >= 64) p.blocks *= 2;
    p.block_cout = dw_step(Cout, p.blocks);
    p.blocks = (Cout + p.block_cout - 1) / p.block_cout;
    p.ctas = std::min(p.patches, std::max(1, num_sms / p.blocks));
    p.stages_p = kPatchStagesMax;
    p.stages_a = kAStagesMax;
    while (dw_patch_layout(Cin, p.block_cout, p.patch_w, p.stages_p, p.stages_a).total > smem_optin) {
        // The A ring gives way first: a patch takes longer to come.
        if (p.stages_a > 2)
            --p.stages_a;
        else
            --p.stages_p;
    }
    p.smem = dw_patch_layout(Cin, p.block_cout, p.patch_w, p.stages_p, p.stages_a).total;
    *plan = p;
    return ISAM_OK;
}

int dwsep_blocks(int W, int Cin, int Cout, int smem_optin, int *out) {
    if (!dw_channels_ok(Cin, Cout))
        return set_error(ISAM_ERR_UNSUPPORTED, "isam_dwsep_plan_info: needs Cin and Cout multiples of 16 in [16, 256]");
    const int blocks = dw_fewest_blocks(Cin, Cout, dw_patch_width(W, W), smem_optin);
    if (blocks < 1) return set_error(ISAM_ERR_UNSUPPORTED, "isam_dwsep_plan_info: Cin=%d does not fit shared memory", Cin);
    out[0] = 1;
    out[1] = 0;
    out[2] = blocks;
    out[3] = dw_step(Cout, blocks);
    return ISAM_OK;
}

int dwsep_launch(int N, int H, int W, int Cin, int Cout, const uint16_t *x, const uint16_t *dw,
                 const uint16_t *pw, float *out, DeviceState &ds, cudaStream_t stream) {
    DwsepPlan plan;
    int rc = dwsep_plan(N, H, W, Cin, Cout, ds.num_sms, ds.max_smem_optin, &plan);
    if (rc) return rc;
    if ((reinterpret_cast<uintptr_t>(x) | reinterpret_cast<uintptr_t>(dw) |
         reinterpret_cast<uintptr_t>(pw) | reinterpret_cast<uintptr_t>(out)) & 15u)
        return set_error(ISAM_ERR_UNSUPPORTED, "isam_dwsep_conv: pointers must be 16-byte aligned");
    CUtensorMap tmX, tmW, tmOut;
    auto nhwc = [&](int C, uint64_t elem, uint64_t (&dims)[4], uint64_t (&strides)[3]) {
        const uint64_t px = static_cast<uint64_t>(C) * elem;
        const uint64_t d[4] = {static_cast<uint64_t>(C), static_cast<uint64_t>(W), static_cast<uint64_t>(H),
                               static_cast<uint64_t>(N)};
        std::copy(d, d + 4, dims);
        strides[0] = px;
        strides[1] = px * W;
        strides[2] = px * W * H;
    };
    uint64_t dims[4], strides[3];
    const uint32_t box_x[4] = {64, static_cast<uint32_t>(plan.patch_w + 2), static_cast<uint32_t>(plan.patch_h + 2), 1};
    const uint32_t box_o[4] = {32, static_cast<uint32_t>(plan.patch_w), static_cast<uint32_t>(32 / plan.patch_w), 1};
    nhwc(Cin, 2, dims, strides);
    if ((rc = make_tmap_4d_bf16(&tmX, x, dims, strides, box_x, false))) return rc;
    nhwc(Cout, 4, dims, strides);
    if ((rc = make_tmap_4d_f32(&tmOut, out, dims, strides, box_o))) return rc;
    if ((rc = make_tmap_2d_bf16(&tmW, pw, static_cast<uint64_t>(Cout), static_cast<uint64_t>(Cin),
                                static_cast<uint64_t>(Cout) * 2, 64, 64)))
        return rc;
    DwPatchParams p{};
    p.H = H;
    p.W = W;
    p.Cin = Cin;
    p.Cout = Cout;
    p.step = plan.block_cout;
    p.ty = (H + plan.patch_h - 1) / plan.patch_h;
    p.tx = (W + plan.patch_w - 1) / plan.patch_w;
    p.tiles = plan.patches;
    p.atoms = (Cin + 63) / 64;
    p.nchunks = (plan.block_cout + 63) / 64;
    p.stages_p = plan.stages_p;
    p.stages_a = plan.stages_a;
    p.dw = dw;
    p.timeout_ns = wait_timeout_ns();
    p.err = ds.err_word;
    const DwPatchKernel kern = dw_patch_kernel_for(plan.patch_w);
    if ((rc = ensure_smem_optin(reinterpret_cast<const void *>(kern), ds.max_smem_optin, ds.device,
                                "cudaFuncSetAttribute(dwsep)")))
        return rc;
    cudaError_t e = launch_dependent(kern, dim3(static_cast<unsigned>(plan.ctas), static_cast<unsigned>(plan.blocks)),
                                     kPThreads, static_cast<size_t>(plan.smem), stream, 1, tmX, tmW, tmOut, p);
    if (e != cudaSuccess) return cuda_error(e, "launch dwsep_patch_kernel");
    return ISAM_OK;
}

}  // namespace isam
