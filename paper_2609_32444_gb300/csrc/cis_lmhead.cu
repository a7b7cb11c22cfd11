// cis_lmhead.cu -- the CIS token pass fused with the LM head (sm_103a).
//
// Logits z = H W^T (H: [T, Hd] hidden states, W: [V, Hd] unembedding, bf16)
// are computed tile by tile on the tensor cores (tcgen05.mma, fp32 in TMEM)
// and never written to global memory.  One persistent GEMM kernel, its tile
// epilogue chosen at compile time, serves every pass:
//
//   FWD  z tiles [128 tokens x 256 vocab] -> per token, (max, sum e^{z - max})
//        over the tile's entries j != y, and z_y.
//   TOK  per token: combine the pairs, then log p, the weight (Algorithm 1 /
//        Table 8) and the token loss (Eq. 1) with the same device code as the
//        logits entry points; gives lse_t and c_t.
//   then for each vocabulary chunk [v0, v0 + w):
//   DZ   recompute the chunk's z tiles, form dz = c (softmax - onehot) in bf16
//        and write it as dz [Tp, w];
//   DH   dH (+)= dz W[v0 : v0 + w]   (K = w, fp32 accumulator);
//   DW   dW[v0 : v0 + w] = dz^T H    (K = T);
//   DH and DW of a chunk run as one launch with a balanced schedule; with few
//   tokens DH's contraction is cut into ranges (split_for).
// Masked tokens are left out of all four products (cis_lmhead_compact_kernel).
//
// dz exists one chunk at a time (the chunk width follows the workspace the
// caller gives); z never exists outside TMEM.  Every operand is read where
// it lies: FWD and DZ take H and W K-major; DH takes dz K-major and W
// MN-major (its columns are the output's); DW takes dz and H MN-major (the
// contraction runs over their rows, the tokens).  An MN-major operand tile
// arrives as boxes of 64 MN entries x 64 K rows (128-byte swizzle): the
// canonical MN-major layout of the shared-memory descriptor, with LBO the
// stride between 64-entry MN blocks and SBO the stride between 8-row K
// groups; the instruction descriptor marks it transposed (bits 15, 16).
//
// The GEMM kernel: 128 x 256 tiles, K blocks of 64 (one 128-byte swizzled row
// of bf16), a 4-stage ring of 48 KB (A 16 KB + B 32 KB), two 256-column fp32
// accumulators in TMEM so that the epilogue of one tile overlaps the main loop
// of the next; persistent CTAs take tiles i, i + grid, i + 2 grid, ...  Warp
// roles: warp 0 issues TMA loads, warp 1 issues tcgen05.mma (one thread) and
// owns TMEM, warps 2..9 are the epilogue: two warps per TMEM lane quadrant
// (one tile row per thread), each taking one 128-column half of the tile, so
// that a tile's epilogue fits in the next tile's main loop.  Epilogue stores
// are 32 bytes per thread (one whole sector of its row) where the output is
// 32-byte aligned.  All waits are bounded: a wait that runs out sets
// CIS_ERR_DEVICE_TIMEOUT, and the CTA drains its own loads and MMAs and runs
// to its end, so that TMEM is always released.
#include <cuda.h>
#include <cudaTypedefs.h>
#include <algorithm>
#include <mutex>

#include "cis_kernels.h"
#include "cis_tc.cuh"
#include "cis_nvtx.h"

namespace cis {
namespace lm {

constexpr int kBM = 128;                // tile rows (M)
constexpr int kBN = 256;                // tile columns (N)
constexpr int kBK = 64;                 // K block: one 128-byte swizzled row of bf16
constexpr int kStages = 4;
constexpr int kStageA = kBM * kBK * 2;  // 16 KB
constexpr int kStageB = kBN * kBK * 2;  // 32 KB
constexpr int kStageBytes = kStageA + kStageB;
constexpr int kEpiWarps = 8;            // two per TMEM lane quadrant, one per column half
constexpr int kEpiThreads = 32 * kEpiWarps;
constexpr int kThreads = 64 + kEpiThreads;
constexpr int kHalf = kBN / 2;          // columns per epilogue half
constexpr uint32_t kTmemCols = 2 * kBN;  // two accumulators
constexpr size_t kSmemBytes = (size_t)kStages * kStageBytes + 1024;
constexpr int kStageOut = 32 * 128;      // an epilogue warp's staging of dW: 32 rows of 128 bytes
constexpr size_t kDualSmem = kSmemBytes + (size_t)kEpiWarps * kStageOut;
constexpr int kMnBox = 64 * kBK * 2;     // one MN-major box: 64 MN entries x 64 K rows, 8 KB
// dz of one chunk takes 2 Tp bytes per vocabulary column; the default chunk
// keeps it within this many bytes.
constexpr int64_t kDefaultChunkBytes = 1ll << 30;

enum Epi { kStats = 0, kDz = 1, kStore = 2, kAccum = 3 };

// OR of `pred` over the epilogue threads (named barrier 1), so that the
// epilogue warps leave their loop together.
__device__ __forceinline__ int __syncthreads_or_epi(int pred)
{
    int r;
    asm volatile(
        "{\n\t.reg .pred p, q;\n\tsetp.ne.s32 p, %1, 0;\n\t"
        "bar.red.or.pred q, 1, %2, p;\n\tselp.s32 %0, 1, 0, q;\n\t}"
        : "=r"(r)
        : "r"(pred), "n"(kEpiThreads)
        : "memory");
    return r;
}

// 32-byte global accesses (sm_100 and later): one full sector per thread, so
// that a warp's store into 32 rows writes 32 whole sectors.  The address must
// be 32-byte aligned.
__device__ __forceinline__ void st_v8(void *p, const uint32_t *w)
{
    asm volatile("st.global.v8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(p), "r"(w[0]),
                 "r"(w[1]), "r"(w[2]), "r"(w[3]), "r"(w[4]), "r"(w[5]), "r"(w[6]), "r"(w[7])
                 : "memory");
}
// The same with the streaming (evict-first) hint.
__device__ __forceinline__ void st_v8_cs(void *p, const uint32_t *w)
{
    asm volatile("st.global.cs.v8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(p), "r"(w[0]),
                 "r"(w[1]), "r"(w[2]), "r"(w[3]), "r"(w[4]), "r"(w[5]), "r"(w[6]), "r"(w[7])
                 : "memory");
}
__device__ __forceinline__ void ld_v8(const void *p, float *r)
{
    asm volatile("ld.global.v8.f32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                 : "=f"(r[0]), "=f"(r[1]), "=f"(r[2]), "=f"(r[3]), "=f"(r[4]), "=f"(r[5]),
                   "=f"(r[6]), "=f"(r[7])
                 : "l"(p));
}

__device__ __forceinline__ uint32_t pack_bf16x2(float lo, float hi)
{
    __nv_bfloat162 h = __floats2bfloat162_rn(lo, hi);
    return *reinterpret_cast<uint32_t *>(&h);
}

// One launch of the GEMM kernel: C[M, N] = A[M, K] B[N, K]^T over tiles
// (m, n) of 128 x 256, with TMA coordinates offset by a_row0 / b_row0 along
// M / N and a_k0 / b_k0 along K.  Whether an operand's tensor map runs along
// M / N in its inner dimension (MN-major) rather than along K is a template
// parameter of the kernel (A_MN, B_MN).
struct GemmArgs {
    int nMt, nNt, nK;
    int raster_n;  // 1: tile i -> (m = i % nMt, n = i / nMt); 0: (m = i / nNt, n = i % nNt)
    // Batches with masked tokens: the valid ones' number, on the device (null:
    // every token counts).  It replaces the host's row count, along M (FWD, DZ,
    // DH: nMt, rows_valid) or along K (DW: nK).
    const int *count;
    int count_k;
    // kStats, kDz: token of a row, for ids; kStore, kAccum: output row of a row
    // (null: the row itself)
    const int *rowmap;
    // kStore, kAccum: the contraction in `splits` ranges of ksplit K blocks,
    // range i stored split_stride elements after range i - 1
    int splits, ksplit;
    int64_t split_stride;
    int a_row0, a_k0, b_row0, b_k0;
    // kStats, kDz: rows are tokens (rows_valid of them), columns vocabulary
    // entries col0 + n 256 + c; T: row stride of part and part_u
    int T, V, col0;
    const int32_t *ids;
    const float *lse, *cvec;
    float2 *part;     // kStats: [2 nNt, T] (max, sum) over j != y per 128-column half
    float *part_u;    // kStats: [2 nNt, T] sum e^{z - max} (z - max), or null (no entropy)
    float *zy;        // kStats: z at the sampled token
    uint16_t *dz;     // kDz: bf16 [Tp, ld_dz], column = chunk-local vocabulary index
    int64_t ld_dz;
    // kStore, kAccum: rows m 128 + r < rows_valid of out [., ld_out] (fp32; dW, which
    // may be bf16, goes through its tensor map); out_v8: out is 32-byte aligned
    // (32-byte accesses), else 16-byte ones
    void *out;
    int out_bf16, rows_valid, out_v8;
    int64_t ld_out;
    int32_t *status;
};

struct Barriers {
    uint64_t full[kStages], empty[kStages];
    uint64_t accfull[2], accempty[2];
    uint64_t done;
};

// A wait that runs out marks the CTA (shared flag) and the grid (status word)
// as aborted: the roles then stop waiting and run to the end, so a broken
// pipeline costs one bounded wait per role instead of one per tile.  on()
// reads the shared flag only; the status word (global memory, one L2 round
// trip) is consulted inside waits that are already taking long.
struct Abort {
    volatile int *local;
    int32_t *status;
    __device__ __forceinline__ bool on() const { return *local != 0; }
    // False once the CTA has aborted (now or earlier): the caller stops.  A
    // phase that has already completed returns at the first poll, without
    // reading the flag (the MMA thread waits once per stage, and every
    // instruction of its loop counts).
    __device__ __forceinline__ bool wait(uint64_t *bar, uint32_t parity) const
    {
        if (tc::bar_try(bar, parity))
            return true;
        if (*local)
            return false;
        if (!tc::bar_wait(bar, parity, status)) {
            *local = 1;
            set_status(status, kStatusTimeout);
            return false;
        }
        return true;
    }
};

// Tile order.  raster_n: groups of kGroupN vocabulary tiles, token tiles
// inside a group, so that the tiles in flight at one time (one per SM) share
// about 152 / kGroupN token tiles of A and kGroupN tiles of B in L2;
// otherwise m-major (the nNt column blocks of a row block together).  16 and
// 32 measured 0.5% faster than 8 on the full-size call, 4 slower.
constexpr int kGroupN = 16;
__device__ __forceinline__ void tile_mn(const GemmArgs &g, int i, int &m, int &n)
{
    if (g.raster_n) {
        const int per = kGroupN * g.nMt;
        const int grp = i / per, j = i - grp * per;
        const int n0 = grp * kGroupN;
        const int gw = g.nNt - n0 < kGroupN ? g.nNt - n0 : kGroupN;
        m = j / gw;
        n = n0 + (j - m * gw);
    } else {
        m = i / g.nNt;
        n = i - m * g.nNt;
    }
}
// The launch's arguments with the device's token count in place of the host's.
// At least one row tile (one K block) is kept, so that every output is written
// when no token is valid: its rows are dead, and their dz zero.
__device__ __forceinline__ GemmArgs live_args(const GemmArgs &in)
{
    GemmArgs g = in;
    if (in.count) {
        const int n = *in.count;
        if (in.count_k) {
            g.nK = n > 0 ? (n + kBK - 1) / kBK : 1;
            g.ksplit = g.nK;
        } else {
            g.nMt = n > 0 ? (n + kBM - 1) / kBM : 1;
            g.rows_valid = n;
        }
    }
    return g;
}
// Work unit u of a launch: a tile (in one K range), or with MC (2-CTA clusters) a pair of
// tiles in row tiles 2 mp and 2 mp + 1 of one column tile, CTA `rank` of the
// cluster taking row tile 2 mp + rank.  The pair shares its B tile: each CTA
// loads one half of it and multicasts it to both.  With an odd number of row
// tiles the last pair's second tile lies past the rows (m == nMt): its CTA
// still loads and multicasts its half of B, and its A reads as zeros (or, with
// masked tokens left out, whatever lies there), but its epilogue writes nothing.
template <bool MC> __device__ __forceinline__ int n_tiles(const GemmArgs &g)
{
    return MC ? ((g.nMt + 1) >> 1) * g.nNt : g.nMt * g.nNt;
}
// Unit u: its tile and its K range [k0, k0 + nk), in blocks.
struct Unit {
    int m, n, split, k0, nk;
};
template <bool MC>
__device__ __forceinline__ Unit unit_at(const GemmArgs &g, int u, int rank)
{
    Unit w;
    const int tiles = n_tiles<MC>(g);
    w.split = g.splits > 1 ? u / tiles : 0;
    u -= w.split * tiles;
    w.k0 = w.split * g.ksplit;
    w.nk = g.nK - w.k0 < g.ksplit ? g.nK - w.k0 : g.ksplit;
    if (!MC) {
        tile_mn(g, u, w.m, w.n);
        return w;
    }
    GemmArgs gp = g;
    gp.nMt = (g.nMt + 1) >> 1;  // the pairs' own grid of (row pair, column) units
    int mp;
    tile_mn(gp, u, mp, w.n);
    w.m = 2 * mp + rank;
    return w;
}

// Where the producer, or the MMA thread, is in the ring of stages.
struct Ring {
    int stage = 0;
    uint32_t phase = 0;
    __device__ __forceinline__ void next()
    {
        if (++stage == kStages) {
            stage = 0;
            phase ^= 1;
        }
    }
};

// The producer's loads for unit w: w.nk stages.  `used` and `last` record
// per stage whether it was ever loaded and the parity of its last load, for
// the drain before the CTA leaves.  Returns early once the CTA aborted.
template <bool A_MN, bool B_MN, bool MC>
__device__ __forceinline__ void load_tile(const CUtensorMap &tmA, const CUtensorMap &tmB,
                                          const GemmArgs &g, const Unit &w, int rank,
                                          uint8_t *ring, Barriers &bars, const Abort &ab,
                                          Ring &p, uint32_t &used, uint32_t &last)
{
    const int m = w.m, n = w.n;
    for (int kb = w.k0; kb < w.k0 + w.nk; ++kb) {
        if (!ab.wait(&bars.empty[p.stage], p.phase ^ 1))
            return;
        uint64_t *full = &bars.full[p.stage];
        tc::bar_expect_tx(full, kStageBytes);
        used |= 1u << p.stage;
        last = (last & ~(1u << p.stage)) | (p.phase << p.stage);
        uint8_t *st = ring + p.stage * kStageBytes;
        const int ka = g.a_k0 + kb * kBK, kbb = g.b_k0 + kb * kBK;
        if (A_MN) {  // MN-major: boxes of 64 rows of M along the inner dimension
#pragma unroll
            for (int i = 0; i < kBM / 64; ++i)
                tc::tma_load_2d(st + i * kMnBox, &tmA, g.a_row0 + m * kBM + 64 * i, ka, full);
        } else {
            tc::tma_load_2d(st, &tmA, ka, g.a_row0 + m * kBM, full);
        }
        if (MC) {  // this CTA's half of B, to both CTAs
            if (B_MN) {
#pragma unroll
                for (int i = 2 * rank; i < 2 * rank + 2; ++i)
                    tc::tma_load_2d_mc(st + kStageA + i * kMnBox, &tmB,
                                       g.b_row0 + n * kBN + 64 * i, kbb, full, 0x3);
            } else {
                tc::tma_load_2d_mc(st + kStageA + rank * (kStageB / 2), &tmB, kbb,
                                   g.b_row0 + n * kBN + rank * (kBN / 2), full, 0x3);
            }
        } else if (B_MN) {
#pragma unroll
            for (int i = 0; i < kBN / 64; ++i)
                tc::tma_load_2d(st + kStageA + i * kMnBox, &tmB, g.b_row0 + n * kBN + 64 * i,
                                kbb, full);
        } else {
            tc::tma_load_2d(st + kStageA, &tmB, kbb, g.b_row0 + n * kBN, full);
        }
        p.next();
    }
}

// The MMAs of one unit into the accumulator at TMEM column d: nk stages of
// four K=16 steps.  Returns early once the CTA aborted.
template <bool A_MN, bool B_MN, bool MC>
__device__ __forceinline__ void mma_tile(int nk, uint32_t d, uint8_t *ring,
                                         Barriers &bars, const Abort &ab, Ring &p)
{
    constexpr uint32_t kId =
        tc::idesc_bf16(kBM, kBN) | ((uint32_t)A_MN << 15) | ((uint32_t)B_MN << 16);
    // a K step of 16: 32 bytes along a K-major row, 16 rows (2 K groups) of an
    // MN-major tile
    constexpr uint32_t a_step = A_MN ? 16 * 128 : 32, b_step = B_MN ? 16 * 128 : 32;
    // Descriptors of stage 0's A and B tiles; a stage, and a K step inside
    // it, only move the start address, which sits in the low bits (address
    // >> 4, below 2^14 for any shared-memory address), so they are added
    // there.
    const uint32_t s0 = tc::smem_addr(ring);
    const uint64_t da0 = A_MN ? tc::desc_sw128_mn(s0, kMnBox) : tc::desc_sw128(s0);
    const uint64_t db0 =
        B_MN ? tc::desc_sw128_mn(s0 + kStageA, kMnBox) : tc::desc_sw128(s0 + kStageA);
    for (int kb = 0; kb < nk; ++kb) {
        if (!ab.wait(&bars.full[p.stage], p.phase))
            return;
        tc::fence_after_sync();
        const uint64_t so = (uint64_t)((p.stage * kStageBytes) >> 4);
#pragma unroll
        for (int kk = 0; kk < kBK / 16; ++kk)
            tc::mma_bf16(d, da0 + so + (kk * a_step >> 4), db0 + so + (kk * b_step >> 4), kId,
                         (kb | kk) != 0);
        if (MC)  // the stage is free in this CTA and in the peer
            tc::mma_commit_mc(&bars.empty[p.stage], 0x3);
        else
            tc::mma_commit(&bars.empty[p.stage]);
        p.next();
    }
}

// The epilogue of one tile for one thread: TMEM lane r (tile row r of row
// tile m), column half `half` of column tile n; taddr addresses the lane's
// first column of the tile's accumulator.
template <int EPI>
__device__ __forceinline__ void epilogue_tile(const GemmArgs &g, uint32_t taddr, int m, int n,
                                              int split, int r, int half)
{
    const int cbeg = half * kHalf;
    if (EPI == kStats) {
        const int row = m * kBM + r;  // token
        const int y_r = row < g.rows_valid ? g.ids[row] : -1;
        const bool ent = g.part_u != nullptr;
        float mx = -INFINITY, s = 0.0f, u = 0.0f, zyv = 0.0f;
        bool got_y = false;
        for (int c0 = cbeg; c0 < cbeg + kHalf; c0 += 32) {
            float v[32];
            tc::tmem_ld32(taddr + c0, v);
            const int base = g.col0 + n * kBN + c0;
            if (y_r >= base && y_r < base + 32) {
#pragma unroll
                for (int q = 0; q < 32; ++q)
                    if (base + q == y_r)
                        zyv = v[q];
                got_y = true;
            }
            float cm = -INFINITY;
#pragma unroll
            for (int q = 0; q < 32; ++q) {
                const int col = base + q;
                v[q] = (col == y_r || col >= g.V) ? -INFINITY : v[q];
                cm = fmaxf(cm, v[q]);
            }
            if (cm > mx) {
                if (mx == -INFINITY) {
                    s = 0.0f;
                    u = 0.0f;
                } else {
                    const float d = mx - cm, f = ex2_ftz(d * kLog2e);
                    u = fmaf(d, s, u) * f;
                    s *= f;
                }
                mx = cm;
            }
            if (mx != -INFINITY) {
                float a = 0.0f, au = 0.0f;
                if (ent) {  // the entropy term, e (z - max)
#pragma unroll
                    for (int q = 0; q < 32; ++q) {
                        const float d = v[q] - mx, e = ex2_ftz(d * kLog2e);
                        a += e;
                        au = fmaf(e, fmaxf(d, -1024.0f), au);
                    }
                } else {
#pragma unroll
                    for (int q = 0; q < 32; ++q)
                        a += ex2_ftz((v[q] - mx) * kLog2e);
                }
                s += a;
                u += au;
            }
        }
        if (row < g.rows_valid) {  // one (max, sum) per 128-column half
            const int64_t pi = (int64_t)(2 * n + half) * g.T + row;
            g.part[pi] = make_float2(mx, s);
            if (ent)
                g.part_u[pi] = u;
            if (got_y)
                g.zy[row] = zyv;
        }
    } else if (EPI == kDz) {
        const int row = m * kBM + r;  // token; rows up to Tp are allocated
        const bool live = row < g.rows_valid;
        // tokens with c = 0 (masked, clipped, past the last) give 0 without
        // touching the exponential (their lse is a placeholder)
        const float c_r = live ? g.cvec[row] : 0.0f;
        const float lse_r = live ? g.lse[row] : 0.0f;
        const int y_r = live ? g.ids[g.rowmap ? g.rowmap[row] : row] : -1;
        const int cl0 = n * kBN;  // chunk-local column of the tile
        for (int c0 = cbeg; c0 < cbeg + kHalf; c0 += 32) {
            float v[32];
            tc::tmem_ld32(taddr + c0, v);
            const int gc0 = g.col0 + cl0 + c0;  // vocabulary index of v[0]
            uint32_t w[16];
#pragma unroll
            for (int q = 0; q < 32; q += 2) {
                float d[2];
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const int gc = gc0 + q + h;
                    d[h] = (gc < g.V && c_r != 0.0f)
                               ? c_r * ex2_ftz((v[q + h] - lse_r) * kLog2e) -
                                     (gc == y_r ? c_r : 0.0f)
                               : 0.0f;
                }
                w[q >> 1] = pack_bf16x2(d[0], d[1]);
            }
            // 64 bytes of the row in two full-sector stores (read back by
            // the next two launches, DH and DW)
            uint16_t *drow = g.dz + (int64_t)row * g.ld_dz + cl0 + c0;
            st_v8_cs(drow, w);
            st_v8_cs(drow + 16, w + 8);
        }
    } else {
        const int lr = m * kBM + r;  // row of the output block
        const bool live = lr < g.rows_valid;
        const int orow = live && g.rowmap ? g.rowmap[lr] : lr;
        const int64_t o =
            (int64_t)split * g.split_stride + (int64_t)orow * g.ld_out + (int64_t)n * kBN;
        for (int c0 = cbeg; c0 < cbeg + kHalf; c0 += 32) {
            float v[32];
            tc::tmem_ld32(taddr + c0, v);
            if (!live)
                continue;
            if (g.out_v8) {
                float *dst = reinterpret_cast<float *>(g.out) + o + c0;
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    float x[8];
#pragma unroll
                    for (int e = 0; e < 8; ++e)
                        x[e] = v[8 * q + e];
                    if (EPI == kAccum) {
                        float old[8];
                        ld_v8(dst + 8 * q, old);
#pragma unroll
                        for (int e = 0; e < 8; ++e)
                            x[e] += old[e];
                    }
                    st_v8_cs(dst + 8 * q, reinterpret_cast<const uint32_t *>(x));
                }
            } else {
                float4 *dst = reinterpret_cast<float4 *>(
                    reinterpret_cast<float *>(g.out) + o + c0);
#pragma unroll
                for (int q = 0; q < 8; ++q) {
                    float4 x = make_float4(v[4 * q], v[4 * q + 1], v[4 * q + 2],
                                           v[4 * q + 3]);
                    if (EPI == kAccum) {
                        const float4 old = dst[q];
                        x.x += old.x;
                        x.y += old.y;
                        x.z += old.z;
                        x.w += old.w;
                    }
                    __stcs(dst + q, x);
                }
            }
        }
    }
}

// dW's epilogue for one warp: its 32 rows and 128 columns of the tile go through
// `stage` (128-byte rows, the tensor map's swizzle) to the copy engine, which
// writes whole lines.  A tile of few K blocks is bound by its 128 KB of output, which
// stores of 32 bytes to 32 rows a warp wrote at half the rate: T=512,
// H=2048, V=151936: dH and dW take 527 us against 552, T=1024 with a quarter masked 681
// against 729.
template <bool kBf16>
__device__ __forceinline__ void epilogue_staged(const GemmArgs &g, const CUtensorMap &tm,
                                                uint32_t taddr, int m, int n, int lg, int lane,
                                                int half, uint8_t *stage)
{
    constexpr int kCols = kBf16 ? 64 : 32;  // of a 128-byte row
    const int y = m * kBM + lg * 32;
    uint8_t *row = stage + lane * 128;
#pragma unroll
    for (int c0 = half * kHalf; c0 < (half + 1) * kHalf; c0 += kCols) {
        uint32_t w[32];
        float v[32];
        tc::tmem_ld32(taddr + c0, v);
        if (kBf16) {
#pragma unroll
            for (int q = 0; q < 16; ++q)
                w[q] = pack_bf16x2(v[2 * q], v[2 * q + 1]);
            tc::tmem_ld32(taddr + c0 + 32, v);
#pragma unroll
            for (int q = 0; q < 16; ++q)
                w[16 + q] = pack_bf16x2(v[2 * q], v[2 * q + 1]);
        } else {
#pragma unroll
            for (int q = 0; q < 32; ++q)
                w[q] = __float_as_uint(v[q]);
        }
        if (lane == 0)
            tc::tma_store_wait_read();  // the last box has left the staging rows
        __syncwarp();
#pragma unroll
        for (int q = 0; q < 8; ++q)
            *reinterpret_cast<uint4 *>(row + ((q ^ (lane & 7)) << 4)) =
                make_uint4(w[4 * q], w[4 * q + 1], w[4 * q + 2], w[4 * q + 3]);
        tc::fence_async_shared();
        __syncwarp();
        if (lane == 0 && y < g.rows_valid)
            tc::tma_store_2d(&tm, n * kBN + c0, y, stage);
    }
}

// Shared memory of a GEMM CTA besides the ring.
struct GemmShared {
    Barriers bars;
    uint32_t tmem_base;
    int aborted;
};

// Barriers, TMEM and (MC) the cluster, before the roles start.
template <bool MC> __device__ __forceinline__ void gemm_setup(GemmShared &sh, int warp)
{
    if (threadIdx.x == 0) {
        sh.aborted = 0;
        for (int s = 0; s < kStages; ++s) {
            tc::bar_init(&sh.bars.full[s], 1);
            // with MC both CTAs' MMAs release a stage: the peer's multicast
            // writes into this CTA's copy of it
            tc::bar_init(&sh.bars.empty[s], MC ? 2 : 1);
        }
        for (int b = 0; b < 2; ++b) {
            tc::bar_init(&sh.bars.accfull[b], 1);
            tc::bar_init(&sh.bars.accempty[b], kEpiThreads);
        }
        tc::bar_init(&sh.bars.done, 1);
        tc::bar_init_fence();
    }
    if (warp == 1)
        tc::tmem_alloc(&sh.tmem_base, kTmemCols);
    tc::fence_before_sync();
    __syncthreads();
    if (MC)
        tc::cluster_sync();  // the peer's barriers exist before anything signals them
    tc::fence_after_sync();
}

// The producer's last step: no load may still be landing when the CTA leaves.
__device__ __forceinline__ void drain_loads(Barriers &bars, uint32_t used, uint32_t last)
{
    for (int s = 0; s < kStages; ++s)
        if (used & (1u << s))
            tc::bar_wait(&bars.full[s], (last >> s) & 1);
}

// The MMA thread's last step: every MMA of this CTA is done before TMEM is
// released.
__device__ __forceinline__ void drain_mmas(Barriers &bars)
{
    tc::mma_commit(&bars.done);
    tc::bar_wait(&bars.done, 0);
}

// Every thread, after its role: TMEM freed once nothing uses it; with MC
// neither CTA leaves while the other may still signal its barriers.
template <bool MC> __device__ __forceinline__ void gemm_teardown(GemmShared &sh, int warp)
{
    __syncwarp();
    tc::fence_before_sync();
    __syncthreads();
    if (MC) {
        tc::cluster_sync();
        // after a wait ran out the peer may have issued one more multicast
        // into a stage this CTA no longer waits for: give it time to land
        if (sh.aborted && threadIdx.x == 0) {
            const long long t0 = clock64();
            while (clock64() - t0 < (1ll << 20)) {
            }
        }
        __syncthreads();
    }
    if (warp == 1) {
        tc::fence_after_sync();
        tc::tmem_dealloc(sh.tmem_base, kTmemCols);
    }
}

// The epilogue warps' part of one tile: wait for its accumulator, drain it,
// hand it back.  Warps 2..9: TMEM lane quadrant warp % 4 (one tile row per
// thread), column half (warp - 2) / 4 of the 256-column tile.
template <int EPI, bool MC>
__device__ __forceinline__ void epilogue_unit(const GemmArgs &g, const Unit &w, int i,
                                              uint32_t tmem, int warp, int lane, Barriers &bars,
                                              const Abort &ab)
{
    const int lg = warp & 3;
    const int half = (warp - 2) >> 2;
    const uint32_t lane_off = (uint32_t)(lg * 32) << 16;
    const int acc = i & 1;
    ab.wait(&bars.accfull[acc], (i >> 1) & 1);
    tc::fence_after_sync();
    // with MC, the padding tile of an odd row count has nothing to write
    if (!(MC && w.m >= g.nMt))
        epilogue_tile<EPI>(g, tmem + lane_off + acc * kBN, w.m, w.n, w.split, lg * 32 + lane,
                           half);
    tc::fence_before_sync();
    tc::bar_arrive(&bars.accempty[acc]);
}

// The same for a tile of dW, staged.
template <bool MC>
__device__ __forceinline__ void epilogue_dw(const GemmArgs &g, const CUtensorMap &tm,
                                            const Unit &w, int i, uint32_t tmem, int warp,
                                            int lane, Barriers &bars, const Abort &ab,
                                            uint8_t *stage)
{
    const int lg = warp & 3;
    const int half = (warp - 2) >> 2;
    const int acc = i & 1;
    ab.wait(&bars.accfull[acc], (i >> 1) & 1);
    tc::fence_after_sync();
    if (!(MC && w.m >= g.nMt)) {
        const uint32_t taddr = tmem + ((uint32_t)(lg * 32) << 16) + acc * kBN;
        if (g.out_bf16)
            epilogue_staged<true>(g, tm, taddr, w.m, w.n, lg, lane, half, stage);
        else
            epilogue_staged<false>(g, tm, taddr, w.m, w.n, lg, lane, half, stage);
    }
    tc::fence_before_sync();
    tc::bar_arrive(&bars.accempty[acc]);
}

// The MMA thread's part of one tile: a free accumulator, the tile's MMAs,
// then the accumulator handed to the epilogue.
template <bool A_MN, bool B_MN, bool MC>
__device__ __forceinline__ void mma_unit(int nk, int i, uint32_t tmem, uint8_t *ring,
                                         Barriers &bars, const Abort &ab, Ring &p)
{
    const int acc = i & 1;
    ab.wait(&bars.accempty[acc], ((i >> 1) & 1) ^ 1);
    tc::fence_after_sync();
    mma_tile<A_MN, B_MN, MC>(nk, tmem + acc * kBN, ring, bars, ab, p);
    tc::mma_commit(&bars.accfull[acc]);
}

// FWD and DZ: z tiles of H W^T, both operands K-major.
template <int EPI, bool MC>
__global__ void __launch_bounds__(kThreads, 1)
    cis_lmhead_gemm_kernel(const __grid_constant__ CUtensorMap tmA,
                           const __grid_constant__ CUtensorMap tmB, const GemmArgs args)
{
    extern __shared__ __align__(1024) uint8_t dsm[];
    uint8_t *ring = dsm + ((1024 - (tc::smem_addr(dsm) & 1023)) & 1023);
    __shared__ __align__(8) GemmShared sh;

    const GemmArgs g = live_args(args);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int nUnits = n_tiles<MC>(g);
    const int rank = MC ? (int)tc::cluster_ctarank() : 0;
    const int unit0 = MC ? (int)(blockIdx.x >> 1) : (int)blockIdx.x;
    const int ustep = MC ? (int)(gridDim.x >> 1) : (int)gridDim.x;

    gemm_setup<MC>(sh, warp);
    const uint32_t tmem = sh.tmem_base;
    const Abort ab{&sh.aborted, g.status};

    if (warp == 0) {
        if (lane == 0) {  // producer
            Ring p;
            uint32_t used = 0, last = 0;
            for (int u = unit0; u < nUnits && !ab.on(); u += ustep) {
                load_tile<false, false, MC>(tmA, tmB, g, unit_at<MC>(g, u, rank), rank, ring,
                                            sh.bars, ab, p, used, last);
            }
            drain_loads(sh.bars, used, last);
        }
    } else if (warp == 1) {
        if (lane == 0) {  // MMA issue
            Ring p;
            int i = 0;
            for (int u = unit0; u < nUnits && !ab.on(); u += ustep, ++i)
                mma_unit<false, false, MC>(g.nK, i, tmem, ring, sh.bars, ab, p);
            drain_mmas(sh.bars);
        }
    } else {  // epilogue
        int i = 0;
        for (int u = unit0; u < nUnits; u += ustep, ++i) {
            if (__syncthreads_or_epi(ab.on()))
                break;
            epilogue_unit<EPI, MC>(g, unit_at<MC>(g, u, rank), i, tmem, warp, lane, sh.bars, ab);
        }
    }
    gemm_teardown<MC>(sh, warp);
}

// The dH and dW GEMMs of one vocabulary chunk in one launch.  Launched one
// after the other, each ends in a partial wave: at T=16384 dH has 512 pair units
// of 512 K blocks for 76 clusters (6.7 waves), dW 1024 of 256 (13.5 waves), and
// few tokens leave most clusters without any dH unit.  Here group c of G (a
// cluster with MC, else a CTA) takes dH units c, c + G, ...; the L groups that
// got one fewer then take dW units alone, until they have caught up by K blocks
// (A units in all); the rest of dW goes round all groups, those L first.  The
// units of one GEMM go out in order, so the groups at work at any time hold
// neighbouring units, which share their operands in L2.  Every group works its
// list out for itself, so the token count may be the device's.
// A dW unit is taken to cost at least kDwBlocks K blocks: with few of them, what
// its 256 KB of output costs (T=512: 5.7 us a unit, 8 blocks' worth being 2.7).
constexpr int kDwBlocks = 16;
struct DualList {
    int c, G, n_dh, n_a, n_b, pos, L, A;
    __device__ __forceinline__ int size() const { return n_dh + n_a + n_b; }
    // Item i: a dH unit (true) or a dW unit, and its index.
    __device__ __forceinline__ bool item(int i, int &u) const
    {
        if (i < n_dh) {
            u = c + i * G;
            return true;
        }
        i -= n_dh;
        u = i < n_a ? pos + i * L : A + pos + (i - n_a) * G;
        return false;
    }
};
// n0 dH units of k0 K blocks and n1 dW units of k1.
__host__ __device__ __forceinline__ DualList list_of(int n0, int k0, int n1, int k1, int c, int G)
{
    const int q = n0 / G, r = n0 - q * G;
    DualList d;
    d.c = c;
    d.G = G;
    d.L = r ? G - r : 0;
    d.pos = c >= r ? c - r : c - r + G;
    d.n_dh = q + (c < r);
    const int cost1 = k1 > kDwBlocks ? k1 : kDwBlocks;
    const int x = d.L ? k0 / cost1 : 0;
    d.A = d.L * x < n1 ? d.L * x : n1;
    d.n_a = d.pos < d.L && d.A > d.pos ? (d.A - d.pos + d.L - 1) / d.L : 0;
    const int rest = n1 - d.A - d.pos;
    d.n_b = rest > 0 ? (rest + G - 1) / G : 0;
    return d;
}
template <bool MC>
__device__ __forceinline__ DualList dual_list(const GemmArgs &g0, const GemmArgs &g1, int c,
                                              int G)
{
    return list_of(n_tiles<MC>(g0) * g0.splits, g0.ksplit, n_tiles<MC>(g1) * g1.splits, g1.ksplit,
                   c, G);
}

// GEMM 0: dH (+)= dz W_c (A = dz K-major, B = W MN-major, EPI0 = kStore on
// the first chunk, kAccum after); GEMM 1: dW_c = dz^T H (A = dz MN-major,
// B = H MN-major, kStore).  A GEMM without units (nNt = 0) is left out.
template <int EPI0, bool MC>
__global__ void __launch_bounds__(kThreads, 1)
    cis_lmhead_dual_kernel(const __grid_constant__ CUtensorMap tmA0,
                           const __grid_constant__ CUtensorMap tmB0,
                           const __grid_constant__ CUtensorMap tmA1,
                           const __grid_constant__ CUtensorMap tmB1,
                           const __grid_constant__ CUtensorMap tmC1, const GemmArgs args0,
                           const GemmArgs args1)
{
    extern __shared__ __align__(1024) uint8_t dsm[];
    uint8_t *ring = dsm + ((1024 - (tc::smem_addr(dsm) & 1023)) & 1023);
    __shared__ __align__(8) GemmShared sh;

    const GemmArgs g0 = live_args(args0), g1 = live_args(args1);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int rank = MC ? (int)tc::cluster_ctarank() : 0;
    const DualList list = dual_list<MC>(g0, g1, MC ? (int)(blockIdx.x >> 1) : (int)blockIdx.x,
                                        MC ? (int)(gridDim.x >> 1) : (int)gridDim.x);
    const int items = list.size();

    gemm_setup<MC>(sh, warp);
    const uint32_t tmem = sh.tmem_base;
    const Abort ab{&sh.aborted, g0.status};

    if (warp == 0) {
        if (lane == 0) {  // producer
            Ring p;
            uint32_t used = 0, last = 0;
            for (int i = 0; i < items && !ab.on(); ++i) {
                int u;
                if (list.item(i, u))
                    load_tile<false, true, MC>(tmA0, tmB0, g0, unit_at<MC>(g0, u, rank), rank,
                                               ring, sh.bars, ab, p, used, last);
                else
                    load_tile<true, true, MC>(tmA1, tmB1, g1, unit_at<MC>(g1, u, rank), rank,
                                              ring, sh.bars, ab, p, used, last);
            }
            drain_loads(sh.bars, used, last);
        }
    } else if (warp == 1) {
        if (lane == 0) {  // MMA issue
            Ring p;
            for (int i = 0; i < items && !ab.on(); ++i) {
                int u;
                if (list.item(i, u))
                    mma_unit<false, true, MC>(unit_at<MC>(g0, u, rank).nk, i, tmem, ring,
                                              sh.bars, ab, p);
                else
                    mma_unit<true, true, MC>(g1.nK, i, tmem, ring, sh.bars, ab, p);
            }
            drain_mmas(sh.bars);
        }
    } else {  // epilogue
        for (int i = 0; i < items; ++i) {
            if (__syncthreads_or_epi(ab.on()))
                break;
            int u;
            if (list.item(i, u))
                epilogue_unit<EPI0, MC>(g0, unit_at<MC>(g0, u, rank), i, tmem, warp, lane,
                                        sh.bars, ab);
            else
                epilogue_dw<MC>(g1, tmC1, unit_at<MC>(g1, u, rank), i, tmem, warp, lane, sh.bars,
                                ab, ring + kStages * kStageBytes + (warp - 2) * kStageOut);
        }
        if (lane == 0)
            tc::tma_store_wait();
    }
    gemm_teardown<MC>(sh, warp);
}

// Masked tokens (the prompts and the padding of a batch) have no gradient, so
// the products are formed over the valid ones only: their hidden states are
// copied together, in token order, and every GEMM's tiles and K blocks are
// counted from their number, which stays on the device.  At T=16384, H=2048,
// V=151936 with 40% masked the call takes 15.8 ms against 25.0 for
// multiplying the masked rows as well; the copy and the scan take 33 us.
// Smaller calls are multiplied as they are (kPackWork).
//
// One CTA: pos[t] = the place of token t among the valid ones (-1: masked),
// their ids in that order, and their number.
constexpr int kCompactThreads = 1024;
__global__ void __launch_bounds__(kCompactThreads)
    cis_lmhead_compact_kernel(const uint8_t *mask, int T, const int32_t *ids, int *pos,
                              int32_t *ids_c, int *count)
{
    __shared__ int wsum[kCompactThreads / 32];
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    // warp w takes `per` groups of 32 tokens from group w per on
    const int groups = (T + 31) / 32;
    const int per = (groups + kCompactThreads / 32 - 1) / (kCompactThreads / 32);
    const int g0 = wid * per < groups ? wid * per : groups;
    const int g1 = groups - g0 < per ? groups : g0 + per;
    auto valid = [&](int grp) {
        const int t = grp * 32 + lane;
        return t < T && mask[t] != 0;
    };
    int n = 0;
#pragma unroll 8
    for (int grp = g0; grp < g1; ++grp)
        n += valid(grp);
    n = __reduce_add_sync(0xffffffffu, n);
    if (lane == 0)
        wsum[wid] = n;
    __syncthreads();
    int at = 0;
    for (int w = 0; w < wid; ++w)
        at += wsum[w];
#pragma unroll 8
    for (int grp = g0; grp < g1; ++grp) {
        const int t = grp * 32 + lane;
        const int32_t y = t < T ? ids[t] : 0;
        const bool on = valid(grp);
        const unsigned m = __ballot_sync(0xffffffffu, on);
        const int p = at + __popc(m & ((1u << lane) - 1));
        if (t < T)
            pos[t] = on ? p : -1;
        if (on)
            ids_c[p] = y;
        at += __popc(m);
    }
    if (tid == kCompactThreads - 1)
        *count = at;
}

// The valid tokens' rows of src to their places in dst, one warp per token;
// the rows after the last, up to the end of its row tile, are zeroed (dW's
// last K block reads them against dz's zeros).
__global__ void cis_lmhead_gather_kernel(const uint4 *src, const uint8_t *mask, const int *pos,
                                         const int *count, int T, int row16, uint4 *dst)
{
    const int r = (int)(blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5));
    const int lane = threadIdx.x & 31;
    if (r >= T)
        return;
    const int n = *count;
    if (mask[r]) {
        const uint4 *in = src + (int64_t)r * row16;
        uint4 *out = dst + (int64_t)pos[r] * row16;
        for (int c = lane; c < row16; c += 32)
            out[c] = __ldcs(in + c);
    }
    if (r >= n && r < (n > 0 ? (n + kBM - 1) / kBM : 1) * kBM)
        for (int c = lane; c < row16; c += 32)
            dst[(int64_t)r * row16 + c] = make_uint4(0, 0, 0, 0);
}

// dhidden from the products' fp32 rows (splits of them, `stride` elements
// apart, added in order), row r to row rowmap[r]; the masked tokens' rows are
// zeroed.  parts null: only those.  A CTA takes kFinishCols columns of 8 rows.
constexpr int kFinishCols = 256;
__global__ void __launch_bounds__(256)
    cis_lmhead_finish_kernel(const float *parts, int splits, int64_t stride, const int *rowmap,
                             const int *count, const uint8_t *mask, int T, int H, void *out,
                             int out_bf16)
{
    const int r = (int)(blockIdx.x * 8 + (threadIdx.x >> 5));
    if (r >= T)
        return;
    const int c0 = (int)blockIdx.y * kFinishCols + 4 * (threadIdx.x & 31);
    auto store = [&](int64_t row, int c, float4 v) {
        const int64_t o = row * H + c;
        if (out_bf16)
            __stcs(reinterpret_cast<uint2 *>(static_cast<uint16_t *>(out) + o),
                   make_uint2(pack_bf16x2(v.x, v.y), pack_bf16x2(v.z, v.w)));
        else
            __stcs(reinterpret_cast<float4 *>(static_cast<float *>(out) + o), v);
    };
    if (parts && r < (count ? *count : T)) {
        const int64_t row = count ? rowmap[r] : r;
#pragma unroll
        for (int c = c0; c < c0 + kFinishCols; c += 128) {
            const float *p = parts + (int64_t)r * H + c;
            float4 v = __ldcs(reinterpret_cast<const float4 *>(p));
#pragma unroll 4
            for (int k = 1; k < splits; ++k) {
                const float4 w = __ldcs(reinterpret_cast<const float4 *>(p + k * stride));
                v.x += w.x;
                v.y += w.y;
                v.z += w.z;
                v.w += w.w;
            }
            store(row, c, v);
        }
    }
    if (count && mask[r] == 0)
        for (int c = c0; c < c0 + kFinishCols; c += 128)
            store(r, c, make_float4(0.0f, 0.0f, 0.0f, 0.0f));
}

// Per token: combine the FWD pairs, then log p, weight, loss, c_t.  A CTA takes
// 8 tokens: lanes l, l + 8, ... of a warp hold the same token, so a warp's load
// of one half tile's pairs covers whole sectors (one warp per token, each lane
// a half tile of its own, read a sector per pair: 23 us at T=512, V=151936,
// now 10).
//
// With masked tokens (pos): the pairs and zy lie at the token's place among
// the valid ones, and so do lse and c; afterwards zy holds the token's index
// (the row map of the later GEMMs).  pos shares its memory with a.ws_logk: each
// token's place is read before its log k is written, by the same CTA.
constexpr int kTokCta = 8;
constexpr int kTokThreads = 256;
__global__ void __launch_bounds__(kTokThreads)
    cis_lmhead_token_kernel(const __grid_constant__ PassArgs a, const float2 *part, const float *part_u, float *zy,
                            int nHalf, float *lse_out, float *c_out, const int *pos)
{
    constexpr int kGroups = kTokThreads / kTokCta;
    __shared__ MaxSumU red[kTokThreads / 32][kTokCta];
    const int tid = threadIdx.x, ti = tid & (kTokCta - 1), lane = tid & 31, wid = tid >> 5;
    const int64_t t = blockIdx.x * (int64_t)kTokCta + ti;
    const bool in = t < a.T;
    const bool valid = in && (a.mask == nullptr || a.mask[t] != 0);
    const int64_t y = in ? a.ids[t] : -1;
    const bool live = valid && y >= 0 && y < a.V;
    // the token's place; -1: none (past the end, or masked and left out)
    const int64_t at = !in ? -1 : (pos == nullptr ? t : (valid ? pos[t] : -1));
    MaxSumU o{-INFINITY, 0.0f, 0.0f};
    if (live) {
        constexpr int kU = 8;  // loads in flight
        for (int j0 = tid / kTokCta; j0 < nHalf; j0 += kU * kGroups) {
            float2 q[kU];
            float u[kU];
#pragma unroll
            for (int k = 0; k < kU; ++k) {
                const int j = j0 + k * kGroups;
                q[k] = j < nHalf ? part[(int64_t)j * a.T + at] : make_float2(-INFINITY, 0.0f);
                u[k] = part_u && j < nHalf ? part_u[(int64_t)j * a.T + at] : 0.0f;
            }
#pragma unroll
            for (int k = 0; k < kU; ++k) {
                if (part_u) {
                    o = msu_combine(o, MaxSumU{q[k].x, q[k].y, u[k]});
                } else {
                    const MaxSum ms = ms_combine(MaxSum{o.m, o.s}, MaxSum{q[k].x, q[k].y});
                    o.m = ms.m;
                    o.s = ms.s;
                }
            }
        }
    }
#pragma unroll
    for (int d = kTokCta; d < 32; d <<= 1) {
        MaxSumU w;
        w.m = __shfl_xor_sync(0xffffffffu, o.m, d);
        w.s = __shfl_xor_sync(0xffffffffu, o.s, d);
        w.u = __shfl_xor_sync(0xffffffffu, o.u, d);
        o = msu_combine(o, w);
    }
    if (lane < kTokCta)
        red[wid][lane] = o;
    __syncthreads();
    if (tid >= kTokCta || !in)
        return;
    // a sequence operator's first sweep: log p only (the response's weight
    // needs every token of the response)
    const bool first = is_seq_mode(a.P.mode) && a.w_in == nullptr;
    auto place = [&](float lse, float c) {
        if (at < 0)
            return;
        lse_out[at] = lse;
        c_out[at] = c;
        if (pos)
            zy[at] = __int_as_float((int)t);
    };
    if (!live) {
        if (first)
            return;
        if (valid)
            set_status(a.status, kStatusBadId);
        const float lp = valid ? NAN : 0.0f;
        if (a.lp_out) a.lp_out[t] = lp;
        if (a.w_out) a.w_out[t] = 0.0f;
        if (a.trunc_out) a.trunc_out[t] = 0;
        a.ws_w[t] = 0.0f;
        a.ws_trunc[t] = 0;
        a.ws_logk[t] = 0.0f;
        a.ws_terms[t] = valid ? (double)NAN : 0.0;
        if (a.entropy_out) a.entropy_out[t] = lp;
        place(0.0f, 0.0f);
        return;
    }
#pragma unroll
    for (int w = 1; w < kTokThreads / 32; ++w)
        o = msu_combine(o, red[w][ti]);
    const float z = zy[at];
    const RowScalars rs = row_scalars(MaxSum{o.m, o.s}, z);
    if (part_u && a.entropy_out)
        a.entropy_out[t] = row_entropy(o, z, rs.lp);
    if (first) {
        if (a.lp64_out)
            a.lp64_out[t] = rs.lp64();
        return;
    }
    const bool has_old = a.lp_old != nullptr;
    const float lold = has_old ? a.lp_old[t] : 0.0f;
    TokenWeight tw = token_weight(has_old ? lold : rs.lp, has_old ? 0.0f : rs.lp_lo, a.lp_inf[t],
                                  a.P, has_old ? -1.0f : rs.omp);
    if (a.w_in) {
        tw.w = a.w_in[t];
        tw.trunc = a.trunc_in[t];
    }
    const TokenLoss tl =
        token_loss(rs.lp, rs.lp_lo, has_old, lold, a.adv[t], a.scale[t], tw.w, a.P);
    if (a.lp_out) a.lp_out[t] = rs.lp;
    if (a.w_out) a.w_out[t] = tw.w;
    if (a.trunc_out) a.trunc_out[t] = tw.trunc;
    a.ws_w[t] = tw.w;
    a.ws_trunc[t] = tw.trunc;
    a.ws_logk[t] = tw.logk;
    a.ws_terms[t] = tl.term;
    place(rs.lse, tl.c);
}

// ------------------------------------------------------------------ host side
PFN_cuTensorMapEncodeTiled_v12000 encoder()
{
    static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
    static std::once_flag once;
    std::call_once(once, [] {
        cudaDriverEntryPointQueryResult q;
        void *f = nullptr;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &f, 12000,
                                             cudaEnableDefault, &q) == cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(f);
    });
    return fn;
}

// 2-D bf16 tensor map: inner extent `inner`, `outer` rows, row stride `ld`
// elements, box {64, box_rows}, 128-byte swizzle, zero fill out of bounds.
bool make_map(CUtensorMap *m, const void *ptr, int64_t inner, int64_t outer, int64_t ld,
              int box_rows)
{
    auto enc = encoder();
    if (!enc)
        return false;
    cuuint64_t dims[2] = {(cuuint64_t)inner, (cuuint64_t)outer};
    cuuint64_t strides[1] = {(cuuint64_t)(ld * 2)};
    cuuint32_t box[2] = {(cuuint32_t)kBK, (cuuint32_t)box_rows};
    cuuint32_t es[2] = {1, 1};
    return enc(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void *>(ptr), dims, strides,
               box, es, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
               CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
               CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// dW [rows, inner] as a store's target: boxes of 128 bytes x 32 rows, 128-byte
// swizzle in shared memory.
bool make_out_map(CUtensorMap *m, void *ptr, int64_t inner, int64_t rows, bool bf16)
{
    auto enc = encoder();
    if (!enc)
        return false;
    const cuuint64_t es = bf16 ? 2 : 4;
    cuuint64_t dims[2] = {(cuuint64_t)inner, (cuuint64_t)rows};
    cuuint64_t strides[1] = {(cuuint64_t)inner * es};
    cuuint32_t box[2] = {(cuuint32_t)(128 / es), 32};
    cuuint32_t one[2] = {1, 1};
    return enc(m, bf16 ? CU_TENSOR_MAP_DATA_TYPE_BFLOAT16 : CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 2,
               ptr, dims, strides, box, one, CU_TENSOR_MAP_INTERLEAVE_NONE,
               CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_NONE,
               CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// The groups that run at once: co-resident 2-CTA clusters (MC), else SMs.
template <typename K>
cudaError_t resident_groups(K kern, bool mc, size_t smem, int *groups)
{
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)smem);
    if (e != cudaSuccess)
        return e;
    if (!mc) {
        int dev = 0;
        if ((e = cudaGetDevice(&dev)) != cudaSuccess)
            return e;
        return cudaDeviceGetAttribute(groups, cudaDevAttrMultiProcessorCount, dev);
    }
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = 2;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(2);
    cfg.blockDim = dim3(kThreads);
    cfg.dynamicSmemBytes = smem;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    if ((e = cudaOccupancyMaxActiveClusters(groups, kern, &cfg)) != cudaSuccess)
        return e;
    return *groups > 0 ? cudaSuccess : cudaErrorNotSupported;
}

// A persistent launch: one group (a cluster, or a CTA) per resident place, or
// per unit where there are fewer.
template <bool MC, typename K, typename... Args>
cudaError_t launch_groups(K kern, int64_t units, size_t smem, cudaStream_t s,
                          const Args &...args)
{
    int groups = 0;
    cudaError_t e = resident_groups(kern, MC, smem, &groups);
    if (e != cudaSuccess)
        return e;
    if (units <= 0)
        return cudaSuccess;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = 2;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)((units < groups ? units : groups) * (MC ? 2 : 1)));
    cfg.blockDim = dim3(kThreads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cfg.attrs = attr;
    cfg.numAttrs = MC ? 1 : 0;
    e = cudaLaunchKernelEx(&cfg, kern, args...);
    return e != cudaSuccess ? e : cudaGetLastError();
}

// Units of a GEMM by the host's counts (the device's token count may lower
// them).
template <bool MC> int64_t host_units(const GemmArgs &g)
{
    return (int64_t)(MC ? (g.nMt + 1) / 2 : g.nMt) * g.nNt * g.splits;
}

// FWD and DZ.  With MC `b` must be a map whose box is half of B's tile.
template <int EPI, bool MC>
cudaError_t launch_gemm(const CUtensorMap &a, const CUtensorMap &b, const GemmArgs &g,
                        cudaStream_t s)
{
    return launch_groups<MC>(cis_lmhead_gemm_kernel<EPI, MC>, host_units<MC>(g), kSmemBytes, s, a,
                             b, g);
}

// dH and dW of a chunk in one launch: the maps of dz and W, of dz and H, and of dW.
struct DualMaps {
    CUtensorMap dz, w, dz_mn, h, dw;
};
template <bool MC>
cudaError_t launch_dual(bool first, const DualMaps &m, const GemmArgs &g0, const GemmArgs &g1,
                        cudaStream_t s)
{
    const int64_t units = host_units<MC>(g0) + host_units<MC>(g1);
    return first ? launch_groups<MC>(cis_lmhead_dual_kernel<kStore, MC>, units, kDualSmem, s, m.dz,
                                     m.w, m.dz_mn, m.h, m.dw, g0, g1)
                 : launch_groups<MC>(cis_lmhead_dual_kernel<kAccum, MC>, units, kDualSmem, s, m.dz,
                                     m.w, m.dz_mn, m.h, m.dw, g0, g1);
}

// Whether a chunk's dH and dW run as one launch (CIS_LMHEAD_DUAL=0: one after
// the other, each with the other left out; the results are the same either way).
static bool dual_on()
{
    const char *e = getenv("CIS_LMHEAD_DUAL");
    return !(e && e[0] == '0');
}

// Which GEMMs run on 2-CTA multicast clusters: a bit mask over FWD (1), DZ
// (2), DH (4) and DW (8); all by default, CIS_LMHEAD_MC overrides it.  The
// results are bit for bit the same either way: each tile's MMAs and epilogue
// are unchanged, only where half of B comes from differs.  Multicast loads are for
// programs on one GPU (their tensor maps cover that GPU's memory alone): a process
// of a job of several ranks (WORLD_SIZE above 1) does without, whatever the mask.
static int mc_mask()
{
    const char *w = getenv("WORLD_SIZE");
    if (w && atol(w) > 1)
        return 0;
    const char *e = getenv("CIS_LMHEAD_MC");
    return e && e[0] ? (int)strtol(e, nullptr, 0) & 15 : 15;
}

}  // namespace lm

// Workspace of cis_lmhead_fused, after the token-pass layout of ws_layout(T),
// for vocabulary chunks of Vc columns (a multiple of 256).
struct LmLayout {
    WsLayout base;
    size_t lse, c, zy, part, part_u, dh, dz, total;
    int64_t Tp, Vc;
};

static int64_t round_up(int64_t x, int64_t m) { return (x + m - 1) / m * m; }

LmLayout lm_layout(int64_t T, int64_t V, int64_t Hd, int64_t Vc)
{
    auto up = [](size_t x) { return (x + 1023) / 1024 * 1024; };
    LmLayout L;
    L.base = ws_layout(T);
    const int64_t nVt = (V + lm::kBN - 1) / lm::kBN;
    L.Tp = round_up(T, lm::kBM);
    L.Vc = Vc;
    size_t o = up(L.base.total);
    L.lse = o;
    o = up(o + 4 * (size_t)T);
    L.c = o;
    o = up(o + 4 * (size_t)T);
    L.zy = o;
    o = up(o + 4 * (size_t)T);
    L.part = o;  // one (max, sum) per 128-column half tile
    o = up(o + 8 * (size_t)T * (size_t)(2 * nVt));
    L.part_u = o;
    o = up(o + 4 * (size_t)T * (size_t)(2 * nVt));
    L.dh = o;
    o = up(o + 4 * (size_t)T * (size_t)Hd);
    L.dz = o;
    o = up(o + 2 * (size_t)L.Tp * (size_t)Vc);
    L.total = o;
    return L;
}

// The widest chunk: every vocabulary column at once.
static int64_t max_chunk(int64_t V) { return round_up(V, lm::kBN); }

// The default chunk: dz within kDefaultChunkBytes.
static int64_t default_chunk(int64_t T, int64_t V)
{
    const int64_t Tp = round_up(T, lm::kBM);
    int64_t c = Tp > 0 ? lm::kDefaultChunkBytes / (2 * Tp) / lm::kBN * lm::kBN : max_chunk(V);
    if (c < lm::kBN)
        c = lm::kBN;
    return c < max_chunk(V) ? c : max_chunk(V);
}

// The widest chunk whose layout fits in `bytes`; 0 if not even 256 columns do.
static int64_t chunk_for_bytes(int64_t T, int64_t V, int64_t Hd, size_t bytes)
{
    const size_t fixed = lm_layout(T, V, Hd, 0).total;
    if (bytes < fixed)
        return 0;
    const size_t per = 2 * (size_t)round_up(T, lm::kBM);
    int64_t c = per > 0 ? (int64_t)((bytes - fixed) / per) / lm::kBN * lm::kBN : max_chunk(V);
    if (c > max_chunk(V))
        c = max_chunk(V);
    while (c >= lm::kBN && lm_layout(T, V, Hd, c).total > bytes)
        c -= lm::kBN;
    return c >= lm::kBN ? c : 0;
}

// dH has few, long units: (T / 256)(H / 256) pairs of tiles contracting the
// whole chunk, so that with few tokens most SMs would wait for it (T=512,
// H=2048, V=151936: 16 units of 2374 K blocks against dW's 4752 of 8, on 76
// clusters).  Its contraction is then cut into ranges of at most half a
// cluster's share of the launch, each with fp32 products of its own, added at
// the end in order.  The products take the room of a narrower chunk's dz, or
// what the caller's workspace has beyond the layout.  T=512, H=2048, V=151936:
// dH and dW take 527 us (two chunks) against 1123 one after the other, the call
// 1054 against 1600; ranges of a share took 5% longer, of a third 13%, of a sixth
// 5%.  T=300, H=1024, V=32003: 68 against 212.
// Leaving masked tokens out costs a call about 20 us (a scan, a copy, the zeroed
// rows), whether or not many are masked: T=1244, V=1040, H=3072 with 40% masked took
// 107 us against 93.  It is done from here on, where the products take 400 us.
// (CIS_LMHEAD_PACK=1: always; =0: never.)
constexpr double kPackWork = 8e10;  // tokens x vocabulary x hidden size
static bool pack_on(int64_t T, int64_t V, int64_t Hd)
{
    const char *e = getenv("CIS_LMHEAD_PACK");
    if (e && (e[0] == '0' || e[0] == '1'))
        return e[0] == '1';
    return (double)T * (double)V * (double)Hd >= kPackWork;
}
constexpr int64_t kSplitSms = 152;  // the split follows the shape alone
constexpr int kMaxSplits = 16;
struct Split {
    int64_t Vc;
    int splits;
    size_t parts;  // offset of the products
};
static int split_count(int64_t T, int64_t w, int64_t Hd)
{
    const int64_t nH = Hd / lm::kBN, nM = (T + lm::kBM - 1) / lm::kBM;
    const int64_t nV = (w + lm::kBM - 1) / lm::kBM;
    const bool pairs = nM > 1;
    const int64_t G = pairs ? kSplitSms / 2 : kSplitSms;
    const int64_t n0 = (pairs ? (nM + 1) / 2 : nM) * nH, c0 = (w + lm::kBK - 1) / lm::kBK;
    const int64_t n1 = (pairs ? (nV + 1) / 2 : nV) * nH, c1 = std::max<int64_t>((T + lm::kBK - 1) / lm::kBK, lm::kDwBlocks);
    const int64_t share = (n0 * c0 + n1 * c1) / G;
    if (share < 1)  // less than a K block a group: nothing to share out
        return 1;
    int64_t S = (2 * c0 + share - 1) / share;
    S = S < c0 / 16 ? S : c0 / 16;
    S = S < kMaxSplits ? S : kMaxSplits;
    return S > 1 ? (int)S : 1;
}
// The K blocks of the longest list (cis_lmhead_dual_kernel) that dH and dW of a chunk of w
// columns give a group: the first group's, or that of the first with a unit of dH less.
static int64_t dual_blocks(int64_t T, int64_t w, int64_t Hd, int splits)
{
    const int64_t nH = Hd / lm::kBN, nM = (T + lm::kBM - 1) / lm::kBM;
    const int64_t nV = (w + lm::kBM - 1) / lm::kBM;
    const bool pairs = nM > 1;
    const int64_t c0 = (w + lm::kBK - 1) / lm::kBK, c1 = (T + lm::kBK - 1) / lm::kBK;
    const int64_t k0 = (c0 + splits - 1) / splits;
    const int64_t n0 = (pairs ? (nM + 1) / 2 : nM) * nH * ((c0 + k0 - 1) / k0);
    const int64_t n1 = (pairs ? (nV + 1) / 2 : nV) * nH;
    const int64_t G = std::min<int64_t>(pairs ? kSplitSms / 2 : kSplitSms, n0 + n1);
    int64_t most = 0;
    for (const int64_t c : {(int64_t)0, n0 % G}) {
        const lm::DualList l = lm::list_of((int)n0, (int)k0, (int)n1, (int)c1, (int)c, (int)G);
        most = std::max(most, l.n_dh * k0 + (l.n_a + l.n_b) * std::max<int64_t>(c1, lm::kDwBlocks));
    }
    return most;
}
// What a plan costs beside the logits' products, in K blocks of 0.34 us: the chunks' lists;
// 28 us a chunk for its two launches' ends; 0.5 us a MB for dH's products where there are
// several.  (Fitted to 106 shapes; the lists alone differ from the measured times by these.)
static double plan_blocks(int64_t T, int64_t V, int64_t Hd, int64_t Vc, int splits)
{
    const int64_t whole = V / Vc, w = V - whole * Vc;
    double b = (double)whole * (85.0 + (double)dual_blocks(T, Vc, Hd, splits));
    if (w > 0)
        b += 85.0 + (double)dual_blocks(T, w, Hd, splits);
    return splits > 1 ? b + 1.5e-6 * 4.0 * (double)T * (double)Hd * (double)splits : b;
}
// The chunk and the split for a workspace that holds chunks of `widest` columns.  A split
// that plan_blocks puts more than 5% above none is not made: with 0.3 units of dH and more a
// cluster (T=2000, V=8000, H=1024: 166 us against 136; T=6000, V=20000, H=512: 468, 392;
// T=8192, V=32000, H=256: 689, 604; T=3739, V=45176, H=1024: 990, 925) or short chunks
// (T=768, V=8000, H=1536: 198, 125; T=532, V=7136, H=256: 91, 83).  Up to 5% above, what it leaves out (dz in L2) pays:
// T=512, V=151936, H=4096 1959 against 2082.
static Split split_for(int64_t T, int64_t V, int64_t Hd, int64_t widest, size_t bytes)
{
    if (T <= 0 || split_count(T, widest < V ? widest : V, Hd) == 1)
        return {widest, 1, 0};
    for (int64_t chunks = 1; chunks <= 4; ++chunks) {
        const int64_t Vc = round_up((V + chunks - 1) / chunks, lm::kBN);
        const size_t base = lm_layout(T, V, Hd, Vc).total;
        if (Vc > widest || base > bytes)
            continue;
        const int64_t want = split_count(T, Vc < V ? Vc : V, Hd);
        const int64_t fit = (int64_t)((bytes - base) / (4 * (size_t)T * (size_t)Hd));
        const int64_t S = want < fit ? want : fit;
        if (S > 1 && 2 * S >= want) {
            if (plan_blocks(T, V, Hd, Vc, (int)S) > 1.05 * plan_blocks(T, V, Hd, widest, 1))
                break;
            return {Vc, (int)S, base};
        }
    }
    return {widest, 1, 0};
}

}  // namespace cis

using namespace cis;

extern "C" {

CIS_API cis_status_t cis_lmhead_workspace_size(int64_t T, int64_t V, int64_t H, size_t *bytes)
{
    if (bytes == nullptr || T < 0 || V <= 0 || H <= 0)
        return CIS_ERR_INVALID_ARG;
    *bytes = lm_layout(T, V, H, default_chunk(T, V)).total;
    return CIS_OK;
}

CIS_API cis_status_t cis_lmhead_workspace_size_chunk(int64_t T, int64_t V, int64_t H,
                                                     int64_t chunk, size_t *bytes)
{
    if (bytes == nullptr || T < 0 || V <= 0 || H <= 0 || chunk <= 0 || chunk % lm::kBN != 0)
        return CIS_ERR_INVALID_ARG;
    *bytes = lm_layout(T, V, H, chunk < max_chunk(V) ? chunk : max_chunk(V)).total;
    return CIS_OK;
}

CIS_API cis_status_t cis_lmhead_fused(const void *hidden, const void *weight, int64_t T,
                                      int64_t H, int64_t V, const int32_t *ids,
                                      const float *lp_infer, const float *lp_old,
                                      const float *adv, const uint8_t *mask,
                                      const int32_t *cu_seqlens, int64_t B,
                                      const cis_params_t *params, void *dhidden, void *dweight,
                                      int32_t grad_dtype, float *lp_out, float *w_out,
                                      uint8_t *trunc_out, float *entropy_out,
                                      cis_stats_t *stats_out, double *loss_out, void *workspace,
                                      size_t workspace_bytes, void *stream)
{
    NvtxRange nvtx_range("cis_lmhead_fused");
    if (T < 0 || T > (1LL << 30) || V <= 0 || V > (1LL << 30) || H <= 0 || H > (1LL << 20))
        return CIS_ERR_INVALID_ARG;
    if (grad_dtype != CIS_F32 && grad_dtype != CIS_BF16)
        return CIS_ERR_INVALID_ARG;
    if (!params_ok(params))
        return CIS_ERR_INVALID_ARG;
    if ((params->agg == CIS_AGG_SEQ_MEAN_TOKEN_MEAN || is_seq_mode(params->mode)) &&
        (cu_seqlens == nullptr || B < 0))
        return CIS_ERR_INVALID_ARG;
    if (H % lm::kBN != 0)
        return CIS_ERR_UNSUPPORTED;  // Hd in blocks of 256 (and so of the 64-wide K blocks)
    if (workspace == nullptr || (reinterpret_cast<uintptr_t>(workspace) & 1023))
        return CIS_ERR_INVALID_ARG;
    const int64_t widest = chunk_for_bytes(T, V, H, workspace_bytes);
    if (widest == 0)
        return CIS_ERR_INVALID_ARG;  // smaller than the layout for 256-column chunks
    const Split sp = split_for(T, V, H, widest, workspace_bytes);
    const int64_t Vc = sp.Vc;
    const LmLayout L = lm_layout(T, V, H, Vc);
    if (T > 0 && (hidden == nullptr || weight == nullptr || ids == nullptr ||
                  lp_infer == nullptr || adv == nullptr || dhidden == nullptr ||
                  dweight == nullptr))
        return CIS_ERR_INVALID_ARG;
    if ((reinterpret_cast<uintptr_t>(hidden) & 15) || (reinterpret_cast<uintptr_t>(weight) & 15) ||
        (reinterpret_cast<uintptr_t>(dhidden) & 15) || (reinterpret_cast<uintptr_t>(dweight) & 15))
        return CIS_ERR_INVALID_ARG;
    const cis_params_t P = *params;
    cudaStream_t s = (cudaStream_t)stream;
    uint8_t *ws = static_cast<uint8_t *>(workspace);
    PassArgs a = {};
    a.T = T;
    a.V = V;
    a.ids = ids;
    a.lp_inf = lp_infer;
    a.lp_old = lp_old;
    a.adv = adv;
    a.mask = mask;
    a.scale = reinterpret_cast<float *>(ws + L.base.scale);
    a.lp_out = lp_out;
    a.w_out = w_out;
    a.trunc_out = trunc_out;
    a.entropy_out = entropy_out;
    a.ws_w = reinterpret_cast<float *>(ws + L.base.w);
    a.ws_trunc = ws + L.base.trunc;
    a.ws_logk = reinterpret_cast<float *>(ws + L.base.logk);
    a.ws_terms = reinterpret_cast<double *>(ws + L.base.terms);
    a.status = reinterpret_cast<int32_t *>(ws + L.base.status);
    a.P = make_dev_params(P);
    float *lse = reinterpret_cast<float *>(ws + L.lse);
    float *cv = reinterpret_cast<float *>(ws + L.c);
    float *zy = reinterpret_cast<float *>(ws + L.zy);
    float2 *part = reinterpret_cast<float2 *>(ws + L.part);
    float *part_u = entropy_out ? reinterpret_cast<float *>(ws + L.part_u) : nullptr;
    uint16_t *dz = reinterpret_cast<uint16_t *>(ws + L.dz);
    float *scale = reinterpret_cast<float *>(ws + L.base.scale);
    a.red_parts = ws + L.base.parts;
    a.red_ticket = reinterpret_cast<uint32_t *>(ws + L.base.ticket);
    cudaError_t e = launch_scales(mask, T, cu_seqlens, B, P.agg, scale, a.status, a.red_ticket, s,
                                  P.global_counts);
    if (e != cudaSuccess)
        return e == cudaErrorNotSupported ? CIS_ERR_UNSUPPORTED : CIS_ERR_CUDA;
    if (T > 0) {
        const int nTt = (int)((T + lm::kBM - 1) / lm::kBM);
        const int nVt = (int)((V + lm::kBN - 1) / lm::kBN);
        const int nHt = (int)(H / lm::kBN);
        const bool bf16 = grad_dtype == CIS_BF16;
        // one row tile has no partner to share B with
        const int mc = nTt == 1 ? 0 : lm::mc_mask();
        // Masked tokens are left out of the products of larger calls
        // (kPackWork).  What that needs lives in memory that is free
        // until the token step, each token's entry where the step itself writes
        // that token's value: the places in ws_logk, the ids in lse, afterwards
        // the row map in zy.  The valid tokens' hidden states take dH's fp32
        // rows' room, or dhidden's own where those rows are in use.
        // (A dhidden that shares memory with hidden is written last: not packed.)
        const uintptr_t h0 = reinterpret_cast<uintptr_t>(hidden), hb = (uintptr_t)(T * H) * 2;
        const uintptr_t d0 = reinterpret_cast<uintptr_t>(dhidden),
                        db = (uintptr_t)(T * H) * (bf16 ? 2 : 4);
        const bool packed = mask != nullptr && nTt > 1 && pack_on(T, V, H) &&
                            !(h0 < d0 + db && d0 < h0 + hb);
        int *count = packed ? reinterpret_cast<int *>(ws + L.base.status + 128) : nullptr;
        int *pos = packed ? reinterpret_cast<int *>(a.ws_logk) : nullptr;
        int32_t *ids_c = reinterpret_cast<int32_t *>(lse);
        const int *rowmap = packed ? reinterpret_cast<const int *>(zy) : nullptr;
        const bool direct = sp.splits == 1 && !bf16;  // dH's products are dhidden's rows
        float *dh_rows = direct ? static_cast<float *>(dhidden)
                                : reinterpret_cast<float *>(ws + (sp.splits > 1 ? sp.parts : L.dh));
        const void *h = hidden;
        if (packed) {
            void *hc = sp.splits == 1 && bf16 ? dhidden : static_cast<void *>(ws + L.dh);
            lm::cis_lmhead_compact_kernel<<<1, lm::kCompactThreads, 0, s>>>(mask, (int)T, ids, pos,
                                                                            ids_c, count);
            if (cudaGetLastError() != cudaSuccess)
                return CIS_ERR_CUDA;
            lm::cis_lmhead_gather_kernel<<<(unsigned)((T + 7) / 8), 256, 0, s>>>(
                static_cast<const uint4 *>(hidden), mask, pos, count, (int)T, (int)(H / 8),
                static_cast<uint4 *>(hc));
            if (cudaGetLastError() != cudaSuccess)
                return CIS_ERR_CUDA;
            h = hc;
        }
        // K-major maps of H and W (FWD, DZ) and MN-major ones (boxes of 64
        // rows: W as DH's B operand, H as DW's)
        // (mWh: W in boxes of half a B tile, for the multicast clusters)
        CUtensorMap mH, mW, mWh, mWmn, mHmn;
        if (!lm::make_map(&mH, h, H, T, H, lm::kBM) ||
            !lm::make_map(&mW, weight, H, V, H, lm::kBN) ||
            !lm::make_map(&mWh, weight, H, V, H, lm::kBN / 2) ||
            !lm::make_map(&mWmn, weight, H, V, H, 64) ||
            !lm::make_map(&mHmn, h, H, T, H, 64))
            return CIS_ERR_UNSUPPORTED;
        lm::GemmArgs g = {};
        g.T = (int)T;
        g.V = (int)V;
        g.ids = packed ? ids_c : ids;
        g.lse = lse;
        g.cvec = cv;
        g.part = part;
        g.part_u = part_u;
        g.zy = zy;
        g.dz = dz;
        g.ld_dz = Vc;
        g.rows_valid = (int)T;
        g.count = count;
        g.status = a.status;
        // FWD: z tiles of H W^T, row statistics
        g.nMt = nTt;
        g.nNt = nVt;
        g.nK = (int)(H / lm::kBK);
        g.splits = 1;
        g.ksplit = g.nK;
        g.raster_n = 1;
        if (((mc & 1) ? lm::launch_gemm<lm::kStats, true>(mH, mWh, g, s)
                      : lm::launch_gemm<lm::kStats, false>(mH, mW, g, s)) != cudaSuccess)
            return CIS_ERR_CUDA;
        // per-token scalars
        const unsigned tok_grid = (unsigned)((T + lm::kTokCta - 1) / lm::kTokCta);
        if (is_seq_mode(P.mode)) {
            // sequence operator: log p of every token (fp64, into the terms
            // array, which the second sweep then overwrites), the responses'
            // weights, then the token scalars with those weights
            if (lp_old == nullptr) {
                PassArgs f = a;
                f.lp64_out = a.ws_terms;
                lm::cis_lmhead_token_kernel<<<tok_grid, lm::kTokThreads, 0, s>>>(
                    f, part, part_u, zy, 2 * nVt, lse, cv, pos);
                if ((e = cudaGetLastError()) != cudaSuccess)
                    return CIS_ERR_CUDA;
            }
            if (cudaMemsetAsync(a.ws_w, 0, L.base.trunc - L.base.w + (size_t)T, s) != cudaSuccess)
                return CIS_ERR_CUDA;
            if (launch_seq_weights(lp_old ? nullptr : a.ws_terms, lp_old, lp_infer, ids, V, mask,
                                   cu_seqlens, B, T, a.P, a.ws_w, a.ws_trunc, s) != cudaSuccess)
                return CIS_ERR_CUDA;
            a.w_in = a.ws_w;
            a.trunc_in = a.ws_trunc;
        }
        lm::cis_lmhead_token_kernel<<<tok_grid, lm::kTokThreads, 0, s>>>(
            a, part, part_u, zy, 2 * nVt, lse, cv, pos);
        if ((e = cudaGetLastError()) != cudaSuccess)
            return CIS_ERR_CUDA;
        g.ids = ids;
        int splits = sp.splits;
        for (int64_t v0 = 0; v0 < V; v0 += Vc) {
            const int64_t w = V - v0 < Vc ? V - v0 : Vc;
            // DZ: recompute the chunk's z tiles, write dz
            g.nNt = (int)((w + lm::kBN - 1) / lm::kBN);
            g.rowmap = rowmap;
            g.b_row0 = (int)v0;
            g.col0 = (int)v0;
            if (((mc & 2) ? lm::launch_gemm<lm::kDz, true>(mH, mWh, g, s)
                          : lm::launch_gemm<lm::kDz, false>(mH, mW, g, s)) != cudaSuccess)
                return CIS_ERR_CUDA;
            // dz K-major (DH's A: rows are tokens) and MN-major (DW's A: its
            // M runs along dz's columns; rows past T read as zeros)
            CUtensorMap mDz, mDzmn;
            if (!lm::make_map(&mDz, dz, w, L.Tp, Vc, lm::kBM) ||
                !lm::make_map(&mDzmn, dz, w, T, Vc, 64))
                return CIS_ERR_UNSUPPORTED;
            // DH (+)= dz W[chunk]: A = dz [Tp, w] K-major, B = W rows v0 .. v0 + w
            // MN-major (N along Hd, K along the vocabulary), in `splits` ranges
            // (as many as the first chunk fills)
            lm::GemmArgs gdh = g;
            gdh.nNt = nHt;
            gdh.nK = (int)((w + lm::kBK - 1) / lm::kBK);
            gdh.ksplit = (gdh.nK + splits - 1) / splits;
            gdh.splits = (gdh.nK + gdh.ksplit - 1) / gdh.ksplit;
            if (v0 == 0)
                splits = gdh.splits;
            gdh.split_stride = T * H;
            gdh.raster_n = 0;
            gdh.b_row0 = 0;
            gdh.b_k0 = (int)v0;
            gdh.rowmap = direct ? rowmap : nullptr;
            gdh.out = dh_rows;
            gdh.out_v8 = (reinterpret_cast<uintptr_t>(dh_rows) & 31) == 0;
            gdh.ld_out = H;
            // DW[chunk] = dz^T H: A = dz MN-major (M along the chunk's columns,
            // K along the tokens), B = H MN-major (N along Hd, K along tokens)
            lm::GemmArgs gdw = g;
            gdw.count_k = 1;
            gdw.rowmap = nullptr;
            gdw.nMt = (int)((w + lm::kBM - 1) / lm::kBM);
            gdw.nNt = nHt;
            gdw.nK = (int)((T + lm::kBK - 1) / lm::kBK);
            gdw.ksplit = gdw.nK;
            gdw.raster_n = 0;
            gdw.b_row0 = 0;
            gdw.out = static_cast<uint8_t *>(dweight) + (size_t)v0 * (size_t)H * (bf16 ? 2 : 4);
            gdw.out_bf16 = bf16;
            gdw.rows_valid = (int)w;
            gdw.ld_out = H;
            // both in one launch if both take the same CTA grouping, else each
            // in one that leaves the other out
            lm::DualMaps maps{mDz, mWmn, mDzmn, mHmn, {}};
            if (!lm::make_out_map(&maps.dw, gdw.out, H, w, bf16))
                return CIS_ERR_UNSUPPORTED;
            const bool first = v0 == 0;
            if (lm::dual_on() && ((mc & 12) == 12 || (mc & 12) == 0)) {
                e = (mc & 12) ? lm::launch_dual<true>(first, maps, gdh, gdw, s)
                              : lm::launch_dual<false>(first, maps, gdh, gdw, s);
            } else {
                lm::GemmArgs no_dh = gdh, no_dw = gdw;
                no_dh.nNt = no_dw.nNt = 0;
                e = (mc & 4) ? lm::launch_dual<true>(first, maps, gdh, no_dw, s)
                             : lm::launch_dual<false>(first, maps, gdh, no_dw, s);
                if (e == cudaSuccess)
                    e = (mc & 8) ? lm::launch_dual<true>(true, maps, no_dh, gdw, s)
                                 : lm::launch_dual<false>(true, maps, no_dh, gdw, s);
            }
            if (e != cudaSuccess)
                return CIS_ERR_CUDA;
        }
        if (!direct || packed) {
            lm::cis_lmhead_finish_kernel<<<dim3((unsigned)((T + 7) / 8),
                                                (unsigned)(H / lm::kFinishCols)),
                                           256, 0, s>>>(
                direct ? nullptr : dh_rows, splits, T * H, rowmap, count, mask, (int)T, (int)H,
                dhidden, bf16);
            if ((e = cudaGetLastError()) != cudaSuccess)
                return CIS_ERR_CUDA;
        }
    }
    return launch_reduce(a, stats_out, loss_out, s) == cudaSuccess ? CIS_OK : CIS_ERR_CUDA;
}

}  // extern "C"
