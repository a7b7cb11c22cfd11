// cis_cluster.cuh -- the fused pass's cluster kernel and its launch; the launches
// are instantiated in cis_cluster.cu, cis_cluster_ragged.cu,
// cis_cluster_given.cu and cis_cluster_all.cu.
//
// A bf16 row of the 151,936-entry vocabulary is 303,872 bytes, more than one
// CTA's shared memory.  A cluster of CS CTAs (1 <= CS <= 8) therefore
// splits each row into CS contiguous slices.  Per row:
//   1. each CTA copies its slice from HBM into shared memory with bulk
//      asynchronous copies (cp.async.bulk, two chunks, each completing on its
//      own mbarrier so that pass 1 starts on the first chunk; no multicast);
//   2. pass 1 over shared memory: per thread the exact maximum of its entries
//      (j != y; bf16 pairs compared packed), then the sum of e^{z - max}; a
//      block reduction gives the CTA's pair (m_c, s_c);
//   3. every CTA stores its pair into slot [rank] of every CTA of the cluster
//      (st.async into distributed shared memory, counted on the receiver's
//      mbarrier, so a CTA waits for the data only, not for a cluster barrier);
//      each CTA combines the CS pairs in rank order, so all CTAs hold
//      bit-identical row scalars;
//   4. thread 0 forms log p (log-odds form, cis_common.cuh), the weight
//      (Algorithm 1 / Table 8) and the token loss (Eq. 1);
//   5. pass 2 over shared memory writes dz = c (softmax - onehot) with 16-byte
//      streaming stores.
// HBM traffic is one read of the logits and one write of dz.  Rows are
// independent; several clusters share an SM, so one cluster's copy overlaps
// another's arithmetic.
#pragma once

#include <cooperative_groups.h>

#include "cis_dsmem.cuh"
#include "cis_kernels.h"

namespace cg = cooperative_groups;

namespace cis {

// Cluster size and slice (entries, a multiple of 8) for a row of V entries.
struct ClusterPlan {
    int cs;
    int64_t slice;
    size_t smem;
    int nt;  // CTA width: 0 for the default (CIS_CLUSTER_THREADS, else plan_threads)
};


// What a variant of the kernel can do, least code first.  The code of operators
// that are not in use slows the others: the serial section's instructions
// compete for the cache (T=16384, V=1000, CIS: 109 us with all of them, 88 without;
// T=16384, V=151936: 1539 us a step with l_old's, 1463 without).
enum class Ops {
    kPlain,  // no l_old: CIS, TIS, exact, none
    kGiven,  // those with l_old, and the sequence operators (weights given)
    kAll     // every operator
};

// The launches, by form and operators, one translation unit each.
cudaError_t launch_cluster_aligned(const PassArgs &a, int dtype, int out_dtype,
                                   const ClusterPlan &p, cudaStream_t s);
cudaError_t launch_cluster_ragged(const PassArgs &a, int dtype, int out_dtype,
                                  const ClusterPlan &p, cudaStream_t s);
cudaError_t launch_cluster_given(const PassArgs &a, int dtype, int out_dtype, bool aligned,
                                 const ClusterPlan &p, cudaStream_t s);
cudaError_t launch_cluster_all(const PassArgs &a, int dtype, int out_dtype, bool aligned,
                               const ClusterPlan &p, cudaStream_t s);

namespace {


template <typename T> __device__ __forceinline__ T from_f32(float v);
template <> __device__ __forceinline__ float from_f32<float>(float v) { return v; }
template <> __device__ __forceinline__ __nv_bfloat16 from_f32<__nv_bfloat16>(float v)
{
    return __float2bfloat16_rn(v);
}

// 8 or 4 results to global memory with a streaming (evict-first) store.
__device__ __forceinline__ void store_group(__nv_bfloat16 *dst, const float (&v)[8])
{
    uint4 q;
    __nv_bfloat162 h;
    h = __floats2bfloat162_rn(v[0], v[1]); q.x = *reinterpret_cast<uint32_t *>(&h);
    h = __floats2bfloat162_rn(v[2], v[3]); q.y = *reinterpret_cast<uint32_t *>(&h);
    h = __floats2bfloat162_rn(v[4], v[5]); q.z = *reinterpret_cast<uint32_t *>(&h);
    h = __floats2bfloat162_rn(v[6], v[7]); q.w = *reinterpret_cast<uint32_t *>(&h);
    __stcs(reinterpret_cast<uint4 *>(dst), q);
}
__device__ __forceinline__ void store_group(float *dst, const float (&v)[4])
{
    __stcs(reinterpret_cast<float4 *>(dst), make_float4(v[0], v[1], v[2], v[3]));
}
__device__ __forceinline__ void store_group(__nv_bfloat16 *dst, const float (&v)[4])
{
    uint2 q;
    __nv_bfloat162 h;
    h = __floats2bfloat162_rn(v[0], v[1]); q.x = *reinterpret_cast<uint32_t *>(&h);
    h = __floats2bfloat162_rn(v[2], v[3]); q.y = *reinterpret_cast<uint32_t *>(&h);
    __stcs(reinterpret_cast<uint2 *>(dst), q);
}
// Group g of a slab, of 8 entries or 4.
template <typename InT>
__device__ __forceinline__ void load_group(const uint8_t *slab, int g, float (&z)[8])
{
    load8<InT>(slab, g, z);
}
template <typename InT>
__device__ __forceinline__ void load_group(const uint8_t *slab, int g, float (&z)[4])
{
    if constexpr (sizeof(InT) == 4) {
        const float4 q = reinterpret_cast<const float4 *>(slab)[g];
        z[0] = q.x; z[1] = q.y; z[2] = q.z; z[3] = q.w;
    } else {
        const uint2 q = reinterpret_cast<const uint2 *>(slab)[g];
        z[0] = bf16_lo(q.x); z[1] = bf16_hi(q.x);
        z[2] = bf16_lo(q.y); z[3] = bf16_hi(q.y);
    }
}

// Zero the n entries at dst (any alignment), 16 bytes a store between the ends.
template <typename OutT, int kThreads> __device__ __forceinline__ void zero_run(OutT *dst, int n)
{
    constexpr int EV = 16 / sizeof(OutT);
    int head = (int)((16 - (reinterpret_cast<uintptr_t>(dst) & 15)) & 15) / (int)sizeof(OutT);
    head = head < n ? head : n;
    const int nvec = (n - head) / EV, tail = head + nvec * EV;
    for (int v = threadIdx.x; v < nvec; v += kThreads)
        __stcs(reinterpret_cast<uint4 *>(dst + head) + v, make_uint4(0, 0, 0, 0));
    if ((int)threadIdx.x < head)
        dst[threadIdx.x] = from_f32<OutT>(0.0f);
    else if ((int)threadIdx.x - head < n - tail)
        dst[tail + threadIdx.x - head] = from_f32<OutT>(0.0f);
}

// Ragged form, rows with maxima beyond z log2e's range (kHugeLogit), or NaN:
// exponents from z - m.  Rare, and kept out of the kernel's own code (the same
// in the aligned form costs 0.5% at T=16384, V=151936, so there only threads
// that see nothing but masked entries are provided for).
// This thread's sums of e^{z - m} and e^{z - m} (z - m).
template <typename InT, int kThreads>
static __device__ __noinline__ float2 slow_sums(const uint8_t *slab, int ng, float m)
{
    float s = 0.0f, u = 0.0f;
#pragma unroll 1
    for (int g = threadIdx.x; g < ng; g += kThreads) {
        float z[8];
        load8<InT>(slab, g, z);
#pragma unroll 1
        for (int i = 0; i < 8; ++i) {
            const float d = z[i] - m, e = ex2_ftz(d * kLog2e);
            s += e;
            u = fmaf(e, fmaxf(d, -1024.0f), u);
        }
    }
    return make_float2(s, u);
}
// Pass 2, entry by entry; slow: the row's offset m and bias.
template <typename InT, typename OutT, int kThreads>
static __device__ __noinline__ void slow_gradient(const uint8_t *slab, int pad, int n, int yl,
                                                  OutT *orow, float c, float dzy, float2 slow)
{
    const InT *sl = reinterpret_cast<const InT *>(slab) + pad;
#pragma unroll 1
    for (int e = threadIdx.x; e < n; e += kThreads)
        orow[e] = from_f32<OutT>(
            e == yl ? dzy : c * ex2_full(fmaf(to_f32(sl[e]) - slow.x, kLog2e, -slow.y)));
}

// kEnt: the entropy variant exchanges (m, s, u) instead of (m, s).
template <bool kEnt> struct ClusterShared {
    alignas(8) uint64_t bar[kChunks];  // completion of each copy chunk
    alignas(8) uint64_t xbar;          // arrival of the cluster's (m, s) pairs
    alignas(16) float2 part[kMaxCluster];
    MaxSum red[512 / 32];
    float4 row;  // pass 2's multiplier, exponent offset and c (p - 1): one load
    float2 slow; // row.w != 0: pass 2's offset m and bias
};
template <> struct ClusterShared<true> {
    alignas(8) uint64_t bar[kChunks];
    alignas(8) uint64_t xbar;          // arrival of the cluster's (m, s, u) triples
    float4 part[kMaxCluster];
    MaxSumU red[512 / 32];
    float4 row;
    float2 slow;
};

// kRagged: rows of any alignment and any V.  The slab then starts at the 8-entry
// boundary of global memory at or before the slice: `pad` entries before the
// slice, and those after it up to a whole group, are -inf.  Bulk copies bring
// the 16-byte blocks that lie inside the slice, plain loads the few entries at
// its two ends, and nothing outside the slice is read.  Groups of 8 then are
// 16-byte aligned in the output too wherever its rows have the input's phase.
template <typename InT, typename OutT, int kThreads, bool kEnt, bool kRagged, Ops kOps>
__global__ void __launch_bounds__(kThreads) cis_fused_cluster_kernel(const __grid_constant__ PassArgs a, int64_t slice)
{
    extern __shared__ __align__(128) uint8_t dyn_smem[];
    __shared__ ClusterShared<kEnt> sh;
    // the bulk copy needs a 16-byte aligned destination; 128 bytes of slack
    // are allocated so the slab can start on a 128-byte boundary
    uint8_t *slab = dyn_smem + ((128 - (smem_u32(dyn_smem) & 127)) & 127);
    cg::cluster_group cluster = cg::this_cluster();
    const unsigned rank = cluster.block_rank();
    const unsigned cs = cluster.num_blocks();
    const int64_t t = blockIdx.x / cs;
    const int64_t v0 = (int64_t)rank * slice;
    const int64_t n = v0 < a.V ? (a.V - v0 < slice ? a.V - v0 : slice) : 0;  // multiple of 8
    const InT *irow = reinterpret_cast<const InT *>(a.logits) + t * a.ld + v0;
    const int pad = kRagged ? (int)(reinterpret_cast<uintptr_t>(irow) / sizeof(InT) & 7) : 0;
    const int ng = kRagged ? (n > 0 ? (int)((pad + n + 7) / 8) : 0) : (int)(n / 8);
    constexpr int kGroupBytes = 8 * sizeof(InT);
    constexpr bool kExact = kRagged && sizeof(OutT) == 4;  // pass 2's exponents, below
    OutT *orow = reinterpret_cast<OutT *>(a.dz) + t * a.ld_out + v0;

    const bool valid = a.mask == nullptr || a.mask[t] != 0;
    const int64_t y = a.ids[t];
    const bool id_ok = y >= 0 && y < a.V;
    if (threadIdx.x == 0)
        allow_next_grid();
    if (!valid || !id_ok) {  // same branch in every CTA of the cluster
        if constexpr (kRagged) {
            zero_run<OutT, kThreads>(orow, (int)n);
        } else {
            constexpr int ZV = 16 / sizeof(OutT);
            float zero[ZV];
#pragma unroll
            for (int i = 0; i < ZV; ++i)
                zero[i] = 0.0f;
            for (int g = threadIdx.x; g < ng * (8 / ZV); g += kThreads)
                store_group(orow + ZV * g, zero);
        }
        if (threadIdx.x == 0)
            grid_wait();  // in every CTA, so that this grid ends after the one before
        if (rank == 0 && threadIdx.x == 0) {
            const float lp = valid ? NAN : 0.0f;
            if (valid)
                set_status(a.status, kStatusBadId);
            if (a.lp_out) a.lp_out[t] = lp;
            if (kEnt) a.entropy_out[t] = lp;
            if (a.w_out) a.w_out[t] = 0.0f;
            if (a.trunc_out) a.trunc_out[t] = 0;
            a.ws_w[t] = 0.0f;
            a.ws_trunc[t] = 0;
            a.ws_logk[t] = 0.0f;
            a.ws_terms[t] = valid ? (double)NAN : 0.0;
        }
        return;
    }

    // Copy the slice in kChunks pieces, each completing on its own mbarrier.
    const int qg = (ng + kChunks - 1) / kChunks;  // groups per chunk
    const uint32_t xbar = smem_u32(&sh.xbar);
    // kRagged: the slice's bytes [b0, b1) and the 16-byte blocks inside them
    const uintptr_t b0 = reinterpret_cast<uintptr_t>(irow);
    const uintptr_t b1 = b0 + (uintptr_t)n * sizeof(InT), base = b0 - (uintptr_t)pad * sizeof(InT);
    const uintptr_t a1 = b1 & ~(uintptr_t)15;
    const uintptr_t a0 = ((b0 + 15) & ~(uintptr_t)15) < a1 ? (b0 + 15) & ~(uintptr_t)15 : a1;
    if (threadIdx.x == 0) {
        for (int c = 0; c < kChunks; ++c)
            mbar_init_only(smem_u32(&sh.bar[c]), 1);
        mbar_init_only(xbar, 1);
        mbar_init_fence();
        // the one local arrival on xbar; the peers' stores bring the bytes
        mbar_expect_tx(xbar, (uint32_t)(cs * (kEnt ? sizeof(float4) : sizeof(float2))));
        const uint8_t *src = reinterpret_cast<const uint8_t *>(irow);
        for (int c = 0; c < kChunks; ++c) {
            const int g0 = c * qg, g1 = min(ng, g0 + qg);
            if (g0 >= g1)
                break;
            const uint32_t b = smem_u32(&sh.bar[c]);
            if constexpr (kRagged) {
                uintptr_t lo = base + (uintptr_t)g0 * kGroupBytes;
                uintptr_t hi = base + (uintptr_t)g1 * kGroupBytes;
                lo = lo < a0 ? a0 : lo;
                hi = hi > a1 ? a1 : hi;
                const uint32_t bytes = hi > lo ? (uint32_t)(hi - lo) : 0u;
                mbar_expect_tx(b, bytes);
                if (bytes)
                    bulk_g2s(smem_u32(slab) + (uint32_t)(lo - base),
                             reinterpret_cast<const void *>(lo), bytes, b);
            } else {
                const uint32_t bytes = (uint32_t)((g1 - g0) * kGroupBytes);
                mbar_expect_tx(b, bytes);
                bulk_g2s(smem_u32(slab) + g0 * kGroupBytes, src + (int64_t)g0 * kGroupBytes,
                         bytes, b);
            }
        }
    }
    if constexpr (kRagged) {  // the ends: entries outside [a0, a1), at most 7 each, and the padding
        InT *sl = reinterpret_cast<InT *>(slab);
        if (threadIdx.x >= 32 && threadIdx.x < 64 && n > 0) {
            const int k = (int)threadIdx.x - 32;
            const int he = (int)((a0 > b0 ? a0 - b0 : 0) / sizeof(InT));
            const int te = (int)((a1 > b0 ? a1 - b0 : 0) / sizeof(InT));
            const int e = k < 16 ? k : te + (k - 16);  // lanes 0..15 the head, 16..31 the tail
            if (k < 16 ? e < he : e < (int)n)
                sl[pad + e] = irow[e];
            if (k < pad)
                poke_neg_inf<InT>(slab, k);
            if (k < 8 * ng - pad - (int)n)
                poke_neg_inf<InT>(slab, pad + (int)n + k);
        }
    }
    // Arrive now, wait before the first remote store: every CTA of the
    // cluster has started and initialised its barriers by then.
    cluster_arrive_relaxed();

    // Per-token inputs, fetched while the copy is in flight.
    // The weight is known here where it does not depend on the row (l_old, or a
    // sequence operator's weight).
    float zy = 0.0f, linf = 0.0f, lold = 0.0f, adv = 0.0f, sc = 0.0f, qinv = 0.0f, qinv_lo = 0.0f;
    TokenWeight tw{0.0f, 0.0f, 0};
    KpopSide kq{0.0f, 0.0f, 0.0f, 0.0f};
    constexpr bool kAll = kOps == Ops::kAll;
    const bool has_old = kOps != Ops::kPlain && a.lp_old != nullptr;
    const bool given = kOps != Ops::kPlain && a.w_in != nullptr;
    if (threadIdx.x == 0) {
        zy = to_f32(irow[y - v0]);
        linf = a.lp_inf[t];
        adv = a.adv[t];
        qinv = expf(-linf);  // 1 / q, off the row's serial path
        if (has_old) {
            lold = a.lp_old[t];
            tw = token_weight<kAll>(lold, 0.0f, linf, a.P);
        } else if (kAll || kRagged) {
            // 1 / q as a pair: q as one, its reciprocal's residual from FMAs
            float ql;
            const float qh = exp_pair(linf, 0.0f, ql);
            if (qh > 0.0f && linf >= -70.0f) {
                qinv = 1.0f / qh;
                qinv_lo = -qinv * fmaf(ql, qinv, fmaf(qh, qinv, -1.0f));
            }
            if (kAll && a.P.mode == CIS_MODE_KPOP)
                kq = kpop_side(linf);
        }
        // the workspace is the kernel before's until it has ended; with the
        // launch gaps that saves 6 us of 94 at T=4096, V=32000
        grid_wait();
        sc = a.scale[t];
        if (given) {  // a sequence operator: the response's weight
            tw.w = a.w_in[t];
            tw.trunc = a.trunc_in[t];
        }
    }
    __syncthreads();  // barriers initialised before anyone polls them

    // The sampled entry takes no part in the sums over j != y: the thread that
    // owns its 8-entry group (the only thread that reads that group in pass
    // 1) overwrites it with -inf in shared memory once its chunk has landed.
    const int64_t yl = y - v0;
    const int gy = (yl >= 0 && yl < n) ? (int)((yl + pad) >> 3) : -1;
    const int iy = (int)((yl + pad) & 7);

    // Pass 1a: exact maximum of this thread's entries, chunk by chunk as the
    // copy lands.
    MaxAcc<InT> macc;
    for (int c = 0; c < kChunks; ++c) {
        const int g0 = c * qg, g1 = min(ng, g0 + qg);
        if (g0 >= g1)
            break;
        wait_or_flag(smem_u32(&sh.bar[c]), false, a.status);
        if (gy >= g0 && gy < g1 && gy % kThreads == (int)threadIdx.x)
            poke_neg_inf<InT>(slab, 8 * gy + iy);
        const int first = g0 + (int)(((unsigned)threadIdx.x + kThreads - (unsigned)(g0 % kThreads)) %
                                     kThreads);
        macc.consume(slab, first, g1, kThreads);
    }
    const float m = macc.result();

    // Pass 1b: sum of e^{z - max} (8 exponentials added pairwise per group).
    // 2^{(z - m) log2e} is formed with one FMA as 2^{z log2e - cm}, cm = fl(m log2e);
    // the rounding residual of cm is exact (an FMA) and is taken out once at
    // the end, so the sum equals the one over (z - m) log2e.
    float s = 0.0f, u = 0.0f;
    if (kRagged ? fabsf(m) < kHugeLogit : m != -INFINITY) {
        // Aligned form: a thread's entries may all be masked ones, so low that
        // the residual of cm leaves the exponential's range; their exponents
        // are then taken from 0, which makes them count as 0, not NaN.
        const bool far = !kRagged && m < kFarLogit;
        const float cm = far ? 0.0f : m * kLog2e;
        const float cm_err = far ? 0.0f : fmaf(m, kLog2e, -cm);  // m log2e - cm, exactly
        const auto sum8_u = [](const float (&z)[8], float off, float &u) {
            return sizeof(InT) == 4 ? sum8_exp2_off_u2(z, off, u) : sum8_exp2_off_u(z, off, u);
        };
        auto add = [&](int g) {
            float z[8];
            load8_any<InT>(slab, g, z);
            return kEnt ? sum8_u(z, cm, u) : sum8_exp2_off(z, cm);
        };
        if constexpr (kThreads == 128) {
            // twice as many groups a thread as with 256: two at a time, added to
            // each other first, so that the growing sum is added to as often
            // (fp32 slices are long and the warps few: two such pairs in flight)
            int g = threadIdx.x;
#pragma unroll sizeof(InT) == 4 ? 2 : 1
            for (; g + kThreads < ng; g += 2 * kThreads) {
                const float a = add(g);
                s += a + add(g + kThreads);
            }
            if (g < ng)
                s += add(g);
        } else {
#pragma unroll 2
            for (int g = threadIdx.x; g < ng; g += kThreads)
                s += add(g);
        }
        const float f = ex2_ftz(-cm_err);
        if (kEnt)  // sum e (z - m) = f ln2 (sum e x - cm_err sum e)
            u = f * kLn2 * fmaf(-cm_err, s, u);
        s *= f;
    } else if (kRagged && m != -INFINITY) {
        const float2 su = slow_sums<InT, kThreads>(slab, ng, m);
        s = su.x;
        u = su.y;
    }
    // Exchange the CTA pairs (triples): lane r of warp 0 stores this CTA's
    // values into slot [rank] of CTA r, counted on CTA r's xbar.
    if constexpr (kEnt) {
        const MaxSumU mine = block_msu<kThreads, false>(MaxSumU{m, s, u}, sh.red);
        cluster_wait();
        if (threadIdx.x < cs)
            st_async_quad(map_rank(smem_u32(&sh.part[rank]), threadIdx.x), mine.m, mine.s,
                          mine.u, map_rank(xbar, threadIdx.x));
    } else {
        const MaxSum mine = block_ms<kThreads, false>(MaxSum{m, s}, sh.red);
        cluster_wait();
        if (threadIdx.x < cs)
            st_async_pair(map_rank(smem_u32(&sh.part[rank]), threadIdx.x), mine.m, mine.s,
                          map_rank(xbar, threadIdx.x));
    }
    wait_or_flag(xbar, true, a.status);
    // Everything addressed to this CTA has landed; tell the cluster, and wait
    // for the others' word only at exit (so no CTA leaves while stores into
    // its shared memory may be in flight).
    cluster_arrive_relaxed();

    // Thread 0 forms the row's scalars: the serial part of every row, which
    // the other threads wait for, and which shares the SM's issue slots with
    // the other CTAs' streaming loops, so its instruction count sets its
    // length.  Without l_old the weight comes from the row's statistics without
    // logarithms (row_direct) in the common case, and log p, log k and the fp64
    // loss term are formed after the barrier by rank 0 alone, which stores them.
    // Otherwise the log-domain path forms everything here.
    MaxSumU ou{0.0f, 0.0f, 0.0f};
    double term = 0.0;
    float lp = 0.0f, tdir = 0.0f;
    bool direct = false;
    if (threadIdx.x == 0) {
        MaxSum o;
        if constexpr (kEnt) {
            ou = combine_flat(sh.part, cs);
            o = MaxSum{ou.m, ou.s};
        } else {
            o = cs == 4 ? combine4(sh.part) : combine_flat(sh.part, cs);
        }
        float c, omp, bias_log2, scale = 1.0f;
        DirectRow dw;
        direct = !has_old && row_direct<(kAll || kRagged)>(o, zy, dw);
        if (direct && !given)
            direct = weight_direct<kAll, kAll || kRagged>(dw, linf, qinv, qinv_lo, kq, a.P, tw.w, tw.trunc);
        if (direct) {
            omp = dw.omp;
            tdir = dw.t;
            c = sc * tw.w * adv;  // s w A rho with rho = 1, g = 1 (Eq. 1 without l_old)
            // The softmax's 1 / (s' + e^{z_y - m'}) = e^{m' - z_y} p, in
            // [2^-102, 1] within the closed forms' range, replaces a logarithm:
            // its binary exponent -J goes into the exponent offset (as the
            // integer "bias" J) and its mantissa 2^J / (...) in [1, 2) into
            // the multiplier, so that every product stays a normal number.
            const float inv = dw.E * dw.p;
            const int J = 127 - (int)((__float_as_uint(inv) >> 23) & 0xff);
            bias_log2 = (float)J;
            scale = inv * __int_as_float((127 + J) << 23);
        } else {
            // a row that low throughout has lost its count: NaN
            if (!kRagged && o.s == 0.0f && zy < kFarLogit)
                o.s = NAN;
            const RowScalars rs = row_scalars(o, zy);
            if (!has_old) {
                const TokenWeight tn = token_weight<kAll>(rs.lp, rs.lp_lo, linf, a.P, rs.omp);
                tw.logk = tn.logk;
                if (!given) {
                    tw.w = tn.w;
                    tw.trunc = tn.trunc;
                }
            }
            const TokenLoss tl = token_loss(rs.lp, rs.lp_lo, has_old, lold, adv, sc, tw.w, a.P);
            term = tl.term;
            lp = rs.lp;
            c = tl.c;
            omp = rs.omp;
            bias_log2 = rs.bias_log2;
        }
        // Pass 2 forms c softmax_j as cs 2^{z_j log2e - B}: with the power-of-two
        // scale K = clamp(ilogb(c) + 25, 0, 127) (below), B = fl(m log2e + bias
        // - K), and the rounding residual of B folded into cs (with the direct
        // path's scale).  The residual is exact: the product's error from an
        // FMA, the two sums' errors from two-sums (fp32 throughout: fp64
        // operations take 64 cycles each here).
        const int kexp = (int)((__float_as_uint(c) >> 23) & 0xff) - 127 + 25;
        const int K = kexp < 0 ? 0 : (kexp > 127 ? 127 : kexp);
        // c 2^-K exactly: two power-of-two factors, each normal for K <= 127,
        // and every product normal (c 2^-K has exponent -25 unless K is 0)
        float cs = c * __int_as_float((127 - K / 2) << 23) *
                   __int_as_float((127 - (K - K / 2)) << 23);
        float B = INFINITY;
        const float m = o.m == -INFINITY ? 0.0f : o.m;  // row_scalars' offset
        if (bias_log2 != INFINITY) {
            const float p = m * kLog2e, pe = fmaf(m, kLog2e, -p);  // p + pe = m log2e
            float qe, se;
            const float q = two_sum(bias_log2, -(float)K, qe);      // q + qe = bias - K
            B = two_sum(p, q, se);                                   // B + se = p + q
            cs *= ex2_ftz(-(se + pe + qe));
        }
        sh.row = make_float4(cs * scale, B, c * (0.0f - omp), 0.0f);  // c (p - 1): +0 if p = 1
        if (kExact || (kRagged && !(fabsf(m) < kHugeLogit))) {
            sh.row.x = c * scale;
            sh.row.w = 1.0f;
            sh.slow = make_float2(m, bias_log2);
        }
    }
    __syncthreads();
    if (threadIdx.x == 0 && rank == 0) {
        if (direct) {  // log p, log k and the loss term, off the serial path
            lp = -log1pf(tdir);  // p = 1 / (1 + t)
            tw.logk = lp - linf;
            term = -(double)sc * (double)tw.w * (double)adv;
        }
        if (a.lp_out) a.lp_out[t] = lp;
        if (a.w_out) a.w_out[t] = tw.w;
        if (a.trunc_out) a.trunc_out[t] = tw.trunc;
        a.ws_w[t] = tw.w;
        a.ws_trunc[t] = tw.trunc;
        a.ws_logk[t] = tw.logk;
        a.ws_terms[t] = term;
        if (kEnt)
            a.entropy_out[t] = row_entropy(ou, zy, lp);
    }

    // Pass 2: dz = c (softmax - onehot) from the slice in shared memory.
    // c softmax_j is formed as (c 2^-K) 2^(x_j + K) with the flushing
    // exponential.  With K = clamp(ilogb(c) + 25, 0, 127): wherever
    // 2^(x_j + K) would be subnormal, |c softmax_j| < 2^-150 rounds to zero in
    // fp32 and bf16 anyway; c 2^-K stays normal and 2^(x_j + K) finite.  The
    // final multiply keeps subnormal products.
    // With an fp32 side a thread takes W = 4 entries at a time, so that a warp's
    // accesses are to neighbouring bytes (8 fp32 entries a thread left gaps between
    // its vectors: two-way bank conflicts, and every sector written in halves).
    // T=1024, V=151936 fp32 with the entropy and KPop: the pass takes 217 us against
    // 264 (pass 1's loads likewise, load8_any); T=4096, V=32000: fp32 to bf16 133
    // against 155, bf16 to fp32 120 against 128.
    // kExact: exponents from the exact z - m, without the power of two, whose
    // place in the exponent's argument costs it up to 4 bits (fp32 gradients of a row
    // are within 1.1e-7, else 1.6e-7; the aligned form has no issue slots to spare).
    const float4 row = sh.row;
    const float2 exact = kExact ? sh.slow : make_float2(0.0f, 0.0f);
    const auto grad = [&](float z, float c2, float b) {
        return kExact ? c2 * ex2_full(fmaf(z - exact.x, kLog2e, -exact.y))
                      : c2 * ex2_ftz(fmaf(z, kLog2e, -b));
    };
    const float cs2 = row.x, B = row.y, dzy = row.z;
    constexpr int W = sizeof(InT) == 4 || sizeof(OutT) == 4 ? 4 : 8;
    constexpr int kUnroll = 16 / W;
    const int gw = W == 8 ? gy : 2 * gy + (iy >> 2), iw = iy & (W - 1);  // (gy < 0: gw < 0)
    if (kRagged && !kExact && row.w != 0.0f) {
        slow_gradient<InT, OutT, kThreads>(slab, pad, (int)n, (int)yl, orow, cs2, dzy, sh.slow);
    } else if constexpr (!kRagged) {
#pragma unroll kUnroll
        for (int g = threadIdx.x; g < ng * (8 / W); g += kThreads) {
            float z[W], v[W];
            load_group<InT>(slab, g, z);
#pragma unroll
            for (int i = 0; i < W; ++i)
                v[i] = cs2 * ex2_ftz(fmaf(z[i], kLog2e, -B));
            if (g == gw) {  // the sampled entry: c (p - 1)
#pragma unroll
                for (int i = 0; i < W; ++i)
                    v[i] = i == iw ? dzy : v[i];
            }
            store_group(orow + W * g, v);
        }
    } else {
        // Groups whose entries all exist go out whole where the output has the
        // slab's phase (dlogits laid out as the logits are), the others entry
        // by entry.
        constexpr int EV = 16 / sizeof(OutT);
        const InT *sl = reinterpret_cast<const InT *>(slab);
        const int phase = (int)(reinterpret_cast<uintptr_t>(orow) / sizeof(OutT)) - pad;
        const bool whole = (phase & (EV - 1)) == 0;
        const int g0 = whole ? (pad + W - 1) / W : 0;
        const int g1 = whole ? (int)((pad + n) / W) : 0;
#pragma unroll kUnroll
        for (int g = g0 + threadIdx.x; g < g1; g += kThreads) {
            float z[W], v[W];
            load_group<InT>(slab, g, z);
#pragma unroll
            for (int i = 0; i < W; ++i)
                v[i] = grad(z[i], cs2, B);
            if (g == gw) {
#pragma unroll
                for (int i = 0; i < W; ++i)
                    v[i] = i == iw ? dzy : v[i];
            }
            store_group(orow + (W * g - pad), v);
        }
        // entries [0, e0) and [e1, n) of the slice
        const int e0 = whole ? min((int)n, W * g0 - (g0 ? pad : 0)) : 0;
        const int e1 = whole ? max(e0, W * g1 - pad) : 0;
        for (int k = threadIdx.x; k < e0 + ((int)n - e1); k += kThreads) {
            const int e = k < e0 ? k : e1 + (k - e0);
            orow[e] = from_f32<OutT>(e == (int)yl ? dzy
                                                 : grad(to_f32(sl[pad + e]), cs2, B));
        }
    }
    cluster_wait();
}

template <typename InT, typename OutT, int NT, bool kEnt, bool kRagged, Ops kOps>
cudaError_t launch_cluster_nt(const PassArgs &a, const ClusterPlan &p, cudaStream_t s)
{
    auto kern = cis_fused_cluster_kernel<InT, OutT, NT, kEnt, kRagged, kOps>;
    // a ragged slice has up to 15 entries of padding
    const size_t smem = p.smem + (kRagged ? 16 * sizeof(InT) : 0);
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)smem);
    if (e != cudaSuccess)
        return e;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(a.T * p.cs), 1, 1);
    cfg.blockDim = dim3(NT, 1, 1);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = (unsigned)p.cs;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = a.overlap ? 2 : 1;
    return cudaLaunchKernelEx(&cfg, kern, a, p.slice);
}

// The entropy variant: 128 threads, or for bf16 rows 256 too.
template <typename InT, typename OutT, bool kRagged, Ops kOps>
cudaError_t launch_cluster_ent(const PassArgs &a, const ClusterPlan &p, cudaStream_t s)
{
    if constexpr (sizeof(InT) == 2)
        if (p.nt != 128)
            return launch_cluster_nt<InT, OutT, 256, true, kRagged, kOps>(a, p, s);
    return launch_cluster_nt<InT, OutT, 128, true, kRagged, kOps>(a, p, s);
}

// f(InT, OutT) for the two element types.
template <template <typename, typename> class F>
cudaError_t by_type(int dtype, int out_dtype, const PassArgs &a, const ClusterPlan &p,
                    cudaStream_t s)
{
    if (dtype == CIS_BF16)
        return out_dtype == CIS_BF16 ? F<__nv_bfloat16, __nv_bfloat16>::run(a, p, s)
                                     : F<__nv_bfloat16, float>::run(a, p, s);
    return out_dtype == CIS_BF16 ? F<float, __nv_bfloat16>::run(a, p, s)
                                 : F<float, float>::run(a, p, s);
}

}  // namespace
}  // namespace cis
