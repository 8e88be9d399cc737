// gemm_common.cuh -- device helpers shared by the GEMM kernels.
#pragma once
#include "ptx.cuh"

namespace isam {

// Waits ignoring the abort flag (used only to let copies already issued land).
__device__ inline bool drain_wait(uint64_t *bar, uint32_t parity, unsigned long long timeout_ns) {
    const uint32_t a = smem_u32(bar);
    const unsigned long long t0 = globaltimer();
    while (!mbar_try_wait(a, parity)) {
        if (globaltimer() - t0 > timeout_ns) return false;
    }
    return true;
}

// bounded_wait by every lane of a warp, with a warp-uniform result.
template <bool cluster_scope = false>
__device__ __forceinline__ bool warp_wait(uint64_t *bar, uint32_t parity, const WaitCtx &w, uint32_t site) {
    const bool ok = bounded_wait<cluster_scope>(bar, parity, w, site);
    return __all_sync(0xffffffffu, ok) != 0;
}

// Rows of a tile (the MMA's M).
constexpr int kTileRows = 128;

// Columns of an epilogue chunk; the accumulators are whole chunks apart.
__host__ __device__ inline int chunk_cols(int bn) { return bn <= 16 ? 16 : 32; }
__host__ __device__ inline int acc_cols(int bn) { return (bn + 31) / 32 * 32; }

// A whole tile as partial rows: [chunk][128 rows][chunk columns] fp32.
__host__ __device__ inline int partial_bytes(int bn) {
    return (bn <= 16 ? 16 : acc_cols(bn)) * kTileRows * 4;
}

// ---- split tiles: S = 2^ls CTAs of a cluster hold partial sums of one tile;
// CTA `rank` of it owns rows rank * 128 / S on.
// 16-byte piece j of a staged row sits at j ^ split_swizzle(row): the rows that a
// quarter-warp stores or loads fall into different banks.
__device__ __forceinline__ int split_swizzle(int cw, int row) { return cw == 32 ? row & 7 : (row >> 1) & 3; }

// Sends lane quarter q of this CTA's partial tile to its owners: load(col, r)
// gives a lane 32 columns of its row, `stage` (partial_bytes, unused by now) takes
// the tile as [chunk][row], and lane i sends the rows of the quarter's i-th owner,
// one bulk copy per chunk, counted in bytes on the owner's barrier `full`.  The
// owner's `recv` is [rank][chunk][row of the slice].  The warp takes the chunks
// first, first + step, ...
template <typename Load>
__device__ __forceinline__ void split_push(uint8_t *stage, const void *recv, const uint64_t *full, int q, int lane,
                                           uint32_t rank, int ls, int cw, int nch, Load load, int first = 0,
                                           int step = 1) {
    const int lr = 7 - ls, rowb = cw * 4;          // log2 of the rows of a slice
    const int lper = min(5, lr);                   // and of one copy
    const int crow0 = q * 32 + (min(lane, (32 >> lper) - 1) << lper);
    const uint32_t owner = static_cast<uint32_t>(crow0 >> lr);
    const uint32_t dst = mapa_shared(
        smem_u32(recv) +
            static_cast<uint32_t>(((static_cast<int>(rank) * nch << lr) + (crow0 & ((1 << lr) - 1))) * rowb),
        owner);
    const uint32_t bar = mapa_shared(smem_u32(full), owner);
    const int row = q * 32 + lane;
#pragma unroll 1
    for (int c = first; c < nch; c += step) {
        uint32_t r[32];
        load(c * cw, r);
        uint8_t *chunk = stage + c * (kTileRows * rowb);
#pragma unroll
        for (int j = 0; j < 8; ++j)
            if (j < 4 || cw == 32)
                *reinterpret_cast<uint4 *>(chunk + row * rowb + ((j ^ split_swizzle(cw, row)) << 4)) =
                    make_uint4(r[4 * j], r[4 * j + 1], r[4 * j + 2], r[4 * j + 3]);
        fence_proxy_async_smem();
        __syncwarp();
        if (lane < (32 >> lper))
            bulk_copy_cluster(dst + static_cast<uint32_t>((c << lr) * rowb), smem_u32(chunk + crow0 * rowb),
                              static_cast<uint32_t>(rowb << lper), bar);
        __syncwarp();
    }
}

// The same without staging the tile: the warp turns a chunk of its 32 rows around
// in `buf` (4 KB) and stores it into the owners' `recv`, each instruction whole rows
// of the chunk, 16 bytes a thread.
template <typename Load>
__device__ __forceinline__ void split_store(uint8_t *buf, const void *recv, const uint64_t *full, int q, int lane,
                                            uint32_t rank, int ls, int cw, int nch, Load load, int first, int step) {
    const int lr = 7 - ls, rowb = cw * 4, lp = cw == 32 ? 3 : 2;
    const uint32_t slot = smem_u32(recv) + static_cast<uint32_t>((static_cast<int>(rank) * nch << lr) * rowb);
    const uint32_t bar = smem_u32(full);
#pragma unroll 1
    for (int c = first; c < nch; c += step) {
        uint32_t r[32];
        load(c * cw, r);
#pragma unroll
        for (int j = 0; j < 8; ++j)
            if (j < 4 || cw == 32)
                *reinterpret_cast<uint4 *>(buf + lane * rowb + ((j ^ split_swizzle(cw, lane)) << 4)) =
                    make_uint4(r[4 * j], r[4 * j + 1], r[4 * j + 2], r[4 * j + 3]);
        __syncwarp();
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            if (i >= 4 && cw != 32) break;
            const int at = i * 32 + lane, row = q * 32 + (at >> lp);  // the piece stays where the swizzle put it
            const float4 v = *reinterpret_cast<const float4 *>(buf + at * 16);
            const uint32_t owner = static_cast<uint32_t>(row >> lr);
            const uint32_t off = static_cast<uint32_t>(((c << lr) + (row & ((1 << lr) - 1))) * rowb + ((at & ((1 << lp) - 1)) << 4));
            st_async_f4(mapa_shared(slot + off, owner), v, mapa_shared(bar, owner));
        }
        __syncwarp();
    }
}

// Sums the slices this CTA received, in rank order, by `threads` threads (t), and
// stores alpha * sum + bias + beta * C: rows r0 on, `width` columns from col0 on.
__device__ __forceinline__ void split_sum(const void *recv, int t, int threads, int ls, int cw, int nch, int r0,
                                          int M, int N, int col0, int width, float alpha, float beta,
                                          const float *bias, float *C) {
    const int lr = 7 - ls, rowb = cw * 4, S = 1 << ls;
    const int lp = cw == 32 ? 3 : 2;
    const int groups = nch << (lr + lp);  // 16-byte pieces of the slice: [chunk][row][8 or 4]
    const bool vec4 = (N & 3) == 0;
    float cnext[4];
    auto load_piece = [&](int g) {
        const int rr = (g >> lp) & ((1 << lr) - 1);
        const int c4 = (((g >> (lr + lp)) << lp) + (g & ((1 << lp) - 1))) * 4;
        if (g >= groups || r0 + rr >= M) return;
        const float *src = C + static_cast<size_t>(r0 + rr) * N + col0 + c4;
#pragma unroll
        for (int j = 0; j < 4; ++j)
            if (c4 + j < width) cnext[j] = src[j];
    };
    if (beta != 0.0f) load_piece(t);
#pragma unroll 1
    for (int g = t; g < groups; g += threads) {
        const int j4 = g & ((1 << lp) - 1), rr = (g >> lp) & ((1 << lr) - 1), c = g >> (lr + lp);
        const int c4 = ((c << lp) + j4) * 4;
        float cin[4];
        if (beta != 0.0f) {
            // One piece ahead, so that the load's latency is hidden.
#pragma unroll
            for (int j = 0; j < 4; ++j) cin[j] = cnext[j];
            load_piece(g + threads);
        }
        const int left = width - c4;  // columns of the piece inside C
        if (left <= 0 || r0 + rr >= M) continue;
        const uint8_t *slice =
            static_cast<const uint8_t *>(recv) + ((c << lr) + rr) * rowb + ((j4 ^ split_swizzle(cw, rr)) << 4);
        float o[4] = {0.0f, 0.0f, 0.0f, 0.0f};
#pragma unroll 2
        for (int src = 0; src < S; ++src) {
            const float4 v = *reinterpret_cast<const float4 *>(slice + src * ((nch << lr) * rowb));
            o[0] += v.x;
            o[1] += v.y;
            o[2] += v.z;
            o[3] += v.w;
        }
        float *dst = C + static_cast<size_t>(r0 + rr) * N + col0 + c4;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            o[j] *= alpha;
            if (bias != nullptr && j < left) o[j] += bias[col0 + c4 + j];
            if (beta != 0.0f) o[j] += beta * cin[j];
        }
        if (vec4) {
            *reinterpret_cast<float4 *>(dst) = make_float4(o[0], o[1], o[2], o[3]);
        } else {
#pragma unroll
            for (int j = 0; j < 4; ++j)
                if (j < left) dst[j] = o[j];
        }
    }
}

// A warp's 32 rows of cw columns from its transpose buffer (tb, rows 33 floats
// apart) to rows row0 on of C, columns col0 on, by plain stores: a row per store
// (two of 16 columns), sixteen at a time.  Their loads, from C and from the
// buffer, are written ahead of the stores, which the compiler may not move them
// over: 7056 x 3453 x 224 46.9 -> 34.4 us, with beta 193 -> 103 (eight at a time and
// interleaved before; storing each thread's row straight from TMEM in shifted
// 16-byte pieces instead took 57 and 307).
__device__ __forceinline__ void store_rows(const float *tb, int lane, int cw, int row0, int M, int N, int col0, int width,
                                           float alpha, float beta, const float *bias, float *C) {
    const int col = lane & (cw - 1);
    const int sub = cw == 32 ? 0 : lane >> 4;  // row within a store
    const int rpi = cw == 32 ? 1 : 2;
    if (col >= width) return;
    const float bv = bias != nullptr ? bias[col0 + col] : 0.0f;
    const int rows = min(32, M - row0);
    const size_t step = static_cast<size_t>(rpi) * N;
    const float *src = tb + sub * 33 + col;
    float *dst = C + static_cast<size_t>(row0 + sub) * N + col0 + col;
    int rr = sub;
    if (beta != 0.0f) {
#pragma unroll 1
        for (; rr + 15 * rpi < rows; rr += 16 * rpi) {
            float v[16], u[16];
#pragma unroll
            for (int i = 0; i < 16; ++i) v[i] = dst[i * step];
#pragma unroll
            for (int i = 0; i < 16; ++i) u[i] = alpha * src[i * rpi * 33] + bv;
#pragma unroll
            for (int i = 0; i < 16; ++i) dst[i * step] = u[i] + beta * v[i];
            src += 16 * rpi * 33;
            dst += 16 * step;
        }
    } else {
#pragma unroll 1
        for (; rr + 15 * rpi < rows; rr += 16 * rpi) {
            float v[16];
#pragma unroll
            for (int i = 0; i < 16; ++i) v[i] = src[i * rpi * 33];
#pragma unroll
            for (int i = 0; i < 16; ++i) dst[i * step] = alpha * v[i] + bv;
            src += 16 * rpi * 33;
            dst += 16 * step;
        }
    }
#pragma unroll 1
    for (; rr < rows; rr += rpi) {
        float o = alpha * *src + bv;
        if (beta != 0.0f) o += beta * *dst;
        *dst = o;
        src += rpi * 33;
        dst += step;
    }
}

}  // namespace isam
