// k_select.cu -- K1: Spatiotemporal Stability Criterion scoring and
// lowest-c selection (Sec. 4.1 V_i and Eq. ICE; Sec. 4.2 Eq. ssc and
// Eq. normalize; Algorithm 1 function SSC), fused with the row plan of the
// step (Sec. 4.2 index-based token compaction).
//
// One cluster of kSelCS = 8 CTAs (256 threads each) per sample; CTA r of
// the cluster owns tokens [r N / 8, (r + 1) N / 8).  Each CTA streams its
// tokens' two newest velocity slots (16 B + 16 B per token, coalesced uint4
// loads, four tokens of a thread in flight at once), keeps V and A in
// shared memory and reduces their min / max; the cluster combines the eight
// partial ranges through distributed shared memory.  Each CTA then forms
// the score in the same fp32 operation order as the definition and an
// order-preserving 32-bit key per token (in place of V), and a 4 x 8-bit
// radix select finds the c-th smallest key of the sample: every CTA counts
// its keys into a 256-bin histogram, the cluster sums the eight histograms
// bin by bin (each CTA redundantly, so all take the same digit), and the
// search ends at the first digit whose keys are all cached.  Finally each CTA
// caches its keys below the threshold plus the lowest-index ties
// and compacts its active tokens in ascending order, starting from the
// counts of the lower-ranked CTAs.  With a third history slot (SSC with
// three predictions) the acceleration term is the second difference of the
// velocity and each token reads 48 B.
//
// What bounds it: at large batches the load of all samples at once, then the
// passes over shared memory (batch 64 on the 32^3 grid, 73 MB: 40.7 us with
// scalar sums and divisions, four full radix passes and outputs written one at
// a time; 32.2 us = 2.3 TB/s now).  For one sample the chain of cluster barriers
// (16^3, one after another: 9.9 -> 7.9 us per call; the search ends at the first
// digit whose keys are all cached, usually the third).  Device time of the parts
// at batch 64: paired norms, shared reciprocals and wide outputs 39.0 -> 30.9 us,
// the early end 29.3, the keys' spacing and one histogram after the first pass
// 28.4.  Measured slower: 3 x 10-bit digits (45.7 us: every CTA reads eight
// histograms of 1024 bins per pass).
#include <atomic>

#include "common.cuh"
#include "kernels.h"

namespace f3dc {

namespace {

constexpr int kSelCS = 8;             // CTAs per sample (one cluster)
constexpr int kSelThreads = 256;      // one thread per histogram bin
constexpr int kSelWarps = kSelThreads / 32;
constexpr int kSelMaxTokens = 49152;  // per sample: 8 B of shared memory per token over 8 CTAs (48 KB each)
constexpr int kSelUnroll = 4;         // tokens of a thread whose loads are in flight together

// V = |v1|, A = |v1 - v2| (Sec. 4.1), or with v3 the second difference
// |(v1 - v2) - (v2 - v3)|, each channel term in that fp32 order.  The two sums
// of squares run side by side in paired instructions.
template <bool kThird>
F3DC_DEV void token_va(const uint4 &p, const uint4 &q, const uint4 &r, float neg_zero, float &V, float &A)
{
    const uint32_t pw[4] = {p.x, p.y, p.z, p.w};
    const uint32_t qw[4] = {q.x, q.y, q.z, q.w};
    const uint32_t rw[4] = {r.x, r.y, r.z, r.w};
    f32x2 s = {0.0f, 0.0f};
#pragma unroll
    for (int c = 0; c < 8; ++c) {
        auto at = [&](const uint32_t(&w)[4]) {
            return __uint_as_float(c & 1 ? w[c >> 1] & 0xFFFF0000u : w[c >> 1] << 16);
        };
        const float x = at(pw), y = at(qw);
        float d = __fsub_rn(x, y);
        if (kThird) d = __fsub_rn(d, __fsub_rn(y, at(rw)));
        s = fadd2(s, fmul2_alone({x, d}, {x, d}, neg_zero));
    }
    V = __fsqrt_rn(s.x);
    A = __fsqrt_rn(s.y);
}

// min-max normalisation; NaN stays NaN, a degenerate range gives 0.
F3DC_DEV float norm1(float x, float mn, float mx)
{
    if (isnan(x)) return x;
    if (!(mx > mn)) return 0.0f;
    return __fdiv_rn(__fsub_rn(x, mn), __fsub_rn(mx, mn));
}

// The same division for both norms of a token when both ranges d lie in
// [2^-98, 2^20] (`inv` = 1 / d, correctly rounded): n inv, then twice a
// residual and its correction (Markstein, "Computation of elementary functions
// on the IBM RISC System/6000 processor", 1990): with a correctly rounded
// reciprocal and a quotient within one unit, RN(q + RN(n - q d) inv) is the
// correctly rounded quotient.  Nothing underflows on the way: a norm is 0 or at
// least 2^-74.5 (the root of a bf16 square's fp32 sum), so n is 0 or at least
// 2^-98, the quotient at least 2^-118 and the residual a multiple of 2^-145.
F3DC_DEV f32x2 div_by_range(f32x2 n, f32x2 d, f32x2 inv)
{
    const f32x2 nd = {-d.x, -d.y};
    f32x2 q = fmul2(n, inv);
    q = ffma2(ffma2(q, nd, n), inv, q);
    return ffma2(ffma2(q, nd, n), inv, q);
}

// Order-preserving key of a score, 0 <= score < 1 + 2^-20: its bits, with the
// distances above 2^-6 stretched 64 times, so that a binade there covers 32
// values of the first radix digit (as the bits stand it would cover one half)
// and the largest key stays below 2^32; every NaN gives the largest key (never
// cached before a number).
F3DC_DEV uint32_t score_key(float s)
{
    constexpr uint32_t kKnee = 0x3C800000u;  // 2^-6
    const uint32_t u = __float_as_uint(s);
    return isnan(s) ? 0xFFFFFFFFu : (u < kKnee ? u : kKnee + ((u - kKnee) << 6));
}

F3DC_DEV int pad_tile(int a) { return (a + kTileRows - 1) / kTileRows * kTileRows; }

// pairs of tiles that n active tokens fill
F3DC_DEV int tile_pairs(int n) { return (n + 2 * kTileRows - 1) / (2 * kTileRows); }

F3DC_DEV int clamp_quota(int q, int N) { return q < 0 ? 0 : (q > N ? N : q); }

// Distributed shared memory: the address of a variable in CTA `rank` of the
// cluster, and loads through it.
F3DC_DEV uint32_t dsmem_u32(const void *p, uint32_t rank) { return mapa_shared(smem_u32(p), rank); }
F3DC_DEV uint32_t ld_dsmem_u32(uint32_t addr)
{
    uint32_t v;
    asm volatile("ld.shared::cluster.u32 %0, [%1];" : "=r"(v) : "r"(addr) : "memory");
    return v;
}
F3DC_DEV float ld_dsmem_f32(uint32_t addr) { return __uint_as_float(ld_dsmem_u32(addr)); }
F3DC_DEV void cluster_arrive() { asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory"); }
F3DC_DEV void cluster_wait() { asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory"); }

// Row offset of sample b, total padded rows, and the sample's tiles and pairs
// of tiles.  The first warp sums the padded row counts of all samples (B <= 64:
// two per lane) in one round of loads, and the pairs of those that come before
// (more active tokens, then the lower number; a guided step's copy follows its
// sample).  Every CTA of the cluster computes the
// offset; only the cluster's first CTA (`writer`) writes the plan.
static_assert(kMaxBatch <= 64, "write_plan covers two samples per lane");
F3DC_DEV void write_plan(const SelectArgs &a, int b, int na, bool writer, int &off)
{
    __shared__ int s_off, s_tot_rows, s_pair0;
    if (threadIdx.x < 32) {
        const int lane = threadIdx.x;
        const int n0 = lane < a.B ? a.N - clamp_quota(a.quota[lane], a.N) : 0;
        const int n1 = lane + 32 < a.B ? a.N - clamp_quota(a.quota[lane + 32], a.N) : 0;
        const int r0 = pad_tile(n0), r1 = pad_tile(n1), p0 = tile_pairs(n0), p1 = tile_pairs(n1);
        int before = (lane < b ? r0 : 0) + (lane + 32 < b ? r1 : 0), tot = r0 + r1;
        int pair0 = (n0 > na || (n0 == na && lane < b) ? p0 : 0) + (n1 > na || (n1 == na && lane + 32 < b) ? p1 : 0);
        int pairs = p0 + p1;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            before += __shfl_xor_sync(0xffffffffu, before, o);
            tot += __shfl_xor_sync(0xffffffffu, tot, o);
            pair0 += __shfl_xor_sync(0xffffffffu, pair0, o);
            pairs += __shfl_xor_sync(0xffffffffu, pairs, o);
        }
        if (lane == 0) {
            s_off = before;
            s_pair0 = pair0;
            s_tot_rows = tot;
            if (a.plan && writer) {
                a.plan->n_active[b] = na;
                a.plan->row_off[b] = before;
                if (a.cfg_dup) {  // the unguided copy of sample b
                    a.plan->n_active[a.B + b] = na;
                    a.plan->row_off[a.B + b] = tot + before;
                }
                if (b == 0) {
                    const int all = a.cfg_dup ? 2 * tot : tot;
                    a.plan->m_rows = all;
                    a.plan->n_tiles = all / kTileRows;
                    a.plan->n_pairs = a.cfg_dup ? 2 * pairs : pairs;
                }
            }
        }
    }
    __syncthreads();
    off = s_off;
    if (a.tile_sample && writer) {
        const int t0 = off / kTileRows, nt = pad_tile(na) / kTileRows;
        for (int t = threadIdx.x; t < nt; t += blockDim.x) a.tile_sample[t0 + t] = b;
        if (a.cfg_dup) {
            const int t1 = (s_tot_rows + off) / kTileRows;
            for (int t = threadIdx.x; t < nt; t += blockDim.x) a.tile_sample[t1 + t] = a.B + b;
        }
        const int np = (nt + 1) / 2, copies = a.cfg_dup ? 2 : 1;
        for (int i = threadIdx.x; i < copies * np; i += blockDim.x) {
            const int copy = i >= np, j = 2 * (i - copy * np);
            a.pair_tiles[copies * s_pair0 + i] =
                tile_pair(t0 + copy * (s_tot_rows / kTileRows) + j, b + copy * a.B, j + 1 < nt);
        }
    }
}

// Inclusive scan of one value per thread over the CTA (256 threads); returns
// the inclusive prefix and leaves the total in *total.
F3DC_DEV uint32_t block_scan(uint32_t v, uint32_t *wsum, uint32_t *total)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    uint32_t incl = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t n = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += n;
    }
    if (lane == 31) wsum[warp] = incl;
    __syncthreads();
    uint32_t before = 0, all = 0;
#pragma unroll
    for (int w = 0; w < kSelWarps; ++w) {
        const uint32_t x = wsum[w];
        before += w < warp ? x : 0u;
        all += x;
    }
    __syncthreads();  // wsum may be reused by the next scan
    *total = all;
    return before + incl;
}

template <bool kThird>
__global__ void __cluster_dims__(kSelCS, 1, 1) __launch_bounds__(kSelThreads, 4)
    k_ssc_select(const SelectArgs a, float neg_zero)
{
    griddep_launch();
    griddep_wait();
    extern __shared__ __align__(16) float sva[];  // V, A of this CTA's tokens; the key later replaces V
    __shared__ uint32_t whist[kSelWarps / 2][256];  // one histogram per warp pair
    // this CTA's histogram of the current radix pass (read by the cluster);
    // two buffers: pass p + 1 writes the buffer that pass p - 1's readers
    // finished with before they reached pass p's cluster barrier
    __shared__ uint32_t hist[2][256];
    __shared__ float part[4];                 // this CTA's min V, max V, min A, max A (read by the cluster)
    __shared__ uint32_t cnt[2];               // this CTA's keys below / at the threshold (read by the cluster)
    __shared__ float red[4][kSelWarps];
    __shared__ float gmm[4];
    __shared__ uint32_t wsum[kSelWarps];
    __shared__ uint32_t s_digit, s_rank, s_ties;

    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const uint32_t rk = cluster_rank();
    const int b = blockIdx.x / kSelCS;
    const int N = a.N, nl = N / kSelCS, lo = (int)rk * nl;
    const int c = clamp_quota(a.quota[b], N);
    const int na = N - c;
    const size_t base = (size_t)b * N;

    int off = 0;
    write_plan(a, b, na, rk == 0, off);
    if (a.n_active && rk == 0 && tid == 0) a.n_active[b] = na;

    // every CTA of the cluster takes the same branch here (c is per sample),
    // so none waits at a cluster barrier the others skip
    if (c == 0) {  // nothing cached: every token active, no scoring needed
        for (int i = lo + tid; i < lo + nl; i += kSelThreads) {
            a.active_idx[base + i] = i;
            if (a.mask) a.mask[base + i] = 0;
            if (a.row_of_token) a.row_of_token[base + i] = off + i;
        }
        return;
    }
    if (c == N) {  // everything cached
        for (int i = lo + tid; i < lo + nl; i += kSelThreads) {
            if (a.mask) a.mask[base + i] = 1;
            if (a.row_of_token) a.row_of_token[base + i] = -1;
        }
        return;
    }
    float *sV = sva, *sA = sva + nl;
    uint32_t *keys = reinterpret_cast<uint32_t *>(sva);  // key i overwrites V i

    // ---- V and A of this CTA's tokens, min / max (NaN never wins a comparison)
    const uint4 *g1 = reinterpret_cast<const uint4 *>(a.v1) + base + lo;
    const uint4 *g2 = reinterpret_cast<const uint4 *>(a.v2) + base + lo;
    const uint4 *g3 = kThird ? reinterpret_cast<const uint4 *>(a.v3) + base + lo : nullptr;
    float mnV = INFINITY, mxV = -INFINITY, mnA = INFINITY, mxA = -INFINITY;
    for (int i0 = tid; i0 < nl; i0 += kSelUnroll * kSelThreads) {
        uint4 p[kSelUnroll], q[kSelUnroll], r[kSelUnroll];
#pragma unroll
        for (int u = 0; u < kSelUnroll; ++u) {
            const int i = i0 + u * kSelThreads;
            if (i < nl) {
                p[u] = __ldg(g1 + i);
                q[u] = __ldg(g2 + i);
                r[u] = kThird ? __ldg(g3 + i) : make_uint4(0, 0, 0, 0);
            }
        }
#pragma unroll
        for (int u = 0; u < kSelUnroll; ++u) {
            const int i = i0 + u * kSelThreads;
            if (i < nl) {
                float V, A;
                token_va<kThird>(p[u], q[u], r[u], neg_zero, V, A);
                sV[i] = V;
                sA[i] = A;
                mnV = fminf(mnV, V);
                mxV = fmaxf(mxV, V);
                mnA = fminf(mnA, A);
                mxA = fmaxf(mxA, A);
            }
        }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        mnV = fminf(mnV, __shfl_xor_sync(0xffffffffu, mnV, o));
        mxV = fmaxf(mxV, __shfl_xor_sync(0xffffffffu, mxV, o));
        mnA = fminf(mnA, __shfl_xor_sync(0xffffffffu, mnA, o));
        mxA = fmaxf(mxA, __shfl_xor_sync(0xffffffffu, mxA, o));
    }
    if (lane == 0) {
        red[0][warp] = mnV;
        red[1][warp] = mxV;
        red[2][warp] = mnA;
        red[3][warp] = mxA;
    }
    __syncthreads();
    if (tid < 4) {
        float v = red[tid][0];
        for (int w = 1; w < kSelWarps; ++w) v = (tid & 1) ? fmaxf(v, red[tid][w]) : fminf(v, red[tid][w]);
        part[tid] = v;
    }
    cluster_sync();  // every CTA's partial range is in its shared memory
    if (warp == 0) {
        // lane = 4 rank + k reads entry k (min V, max V, min A, max A) of CTA rank
        float v = ld_dsmem_f32(dsmem_u32(&part[lane & 3], (uint32_t)(lane >> 2)));
#pragma unroll
        for (int o = 4; o < 32; o <<= 1) {
            const float w = __shfl_xor_sync(0xffffffffu, v, o);
            v = (lane & 1) ? fmaxf(v, w) : fminf(v, w);
        }
        if (lane < 4) gmm[lane] = v;
    }
    __syncthreads();
    mnV = gmm[0];
    mxV = gmm[1];
    mnA = gmm[2];
    mxA = gmm[3];

    // ---- C_i = w_a norm(A_i) + w_v norm(V_i) -> ordered keys, and the
    // histogram of their top digit (the first radix pass)
    for (int q = tid; q < kSelWarps / 2 * 256; q += kSelThreads) (&whist[0][0])[q] = 0;
    __syncthreads();
    const f32x2 d = {__fsub_rn(mxV, mnV), __fsub_rn(mxA, mnA)};
    auto plain = [](float x) { return x >= 0x1p-98f && x <= 0x1p20f; };
    if (plain(d.x) && plain(d.y)) {
        const f32x2 inv = {__frcp_rn(d.x), __frcp_rn(d.y)};
        for (int i = tid; i < nl; i += kSelThreads) {
            const f32x2 q = div_by_range({__fsub_rn(sV[i], mnV), __fsub_rn(sA[i], mnA)}, d, inv);
            const uint32_t k = score_key(__fadd_rn(__fmul_rn(a.wa, q.y), __fmul_rn(a.wv, q.x)));
            keys[i] = k;
            atomicAdd(&whist[warp >> 1][k >> 24], 1u);
        }
    } else {
        for (int i = tid; i < nl; i += kSelThreads) {
            const float sc =
                __fadd_rn(__fmul_rn(a.wa, norm1(sA[i], mnA, mxA)), __fmul_rn(a.wv, norm1(sV[i], mnV, mxV)));
            const uint32_t k = score_key(sc);
            keys[i] = k;
            atomicAdd(&whist[warp >> 1][k >> 24], 1u);
        }
    }
    __syncthreads();

    // ---- radix select of the c-th smallest key (1-based rank c) over the
    // cluster: each pass counts this CTA's keys matching the digits found so
    // far into its histogram; every CTA sums the eight CTAs' histograms bin by bin (thread
    // = bin), scans, and takes the digit of the bin that holds the rank
    uint32_t prefix = 0, hi_mask = 0;
    uint32_t rank = (uint32_t)c;
#pragma unroll 1
    for (int pass = 0; pass < 4; ++pass) {
        const int shift = 24 - 8 * pass;
        if (pass > 0) {
            whist[0][tid] = 0;  // few keys are left: one histogram
            __syncthreads();
            for (int i = tid; i < nl; i += kSelThreads) {
                const uint32_t k = keys[i];
                if ((k & hi_mask) == prefix) atomicAdd(&whist[0][(k >> shift) & 255u], 1u);
            }
            __syncthreads();
        }
        uint32_t v = whist[0][tid];
        if (pass == 0) {
#pragma unroll
            for (int w = 1; w < kSelWarps / 2; ++w) v += whist[w][tid];
        }
        hist[pass & 1][tid] = v;
        cluster_sync();  // every CTA's histogram of this pass is complete
        uint32_t tot = 0;
#pragma unroll
        for (int r2 = 0; r2 < kSelCS; ++r2) tot += ld_dsmem_u32(dsmem_u32(&hist[pass & 1][tid], (uint32_t)r2));
        uint32_t all;
        const uint32_t incl = block_scan(tot, wsum, &all);
        const uint32_t excl = incl - tot;
        if (excl < rank && rank <= incl) {
            s_digit = (uint32_t)tid;
            s_rank = rank - excl;
            s_ties = tot;
        }
        __syncthreads();
        prefix |= s_digit << shift;
        hi_mask |= 255u << shift;
        rank = s_rank;
        const uint32_t ties = s_ties;
        __syncthreads();  // rewritten by the next pass
        if (ties == rank) break;  // every key with these digits is cached: the rest cannot matter
    }
    // keys below thr in the digits found are cached, plus the first `rank` ties of the sample
    const uint32_t thr = prefix;

    // ---- this CTA's keys below / at the threshold; the lower-ranked CTAs'
    // counts give the sample-wide counts before this CTA's first token
    uint32_t nlt = 0, neq = 0;
    for (int i = tid; i < nl; i += kSelThreads) {
        const uint32_t k = keys[i];
        nlt += (k & hi_mask) < thr;
        neq += (k & hi_mask) == thr;
    }
    uint32_t all_lt, all_eq;
    block_scan(nlt, wsum, &all_lt);
    block_scan(neq, wsum, &all_eq);
    if (tid == 0) {
        cnt[0] = all_lt;
        cnt[1] = all_eq;
    }
    cluster_sync();
    uint32_t run_lt = 0, run_eq = 0, sum_lt = 0, sum_eq = 0;
    if (tid < kSelCS) {
        sum_lt = ld_dsmem_u32(dsmem_u32(&cnt[0], (uint32_t)tid));
        sum_eq = ld_dsmem_u32(dsmem_u32(&cnt[1], (uint32_t)tid));
    }
    // no CTA reads another's shared memory after this: arrive now, wait at exit
    cluster_arrive();
    {
        // prefix over ranks below rk (lanes 0..7 of warp 0), broadcast
        __shared__ uint32_t s_run[4];
        if (warp == 0) {
            uint32_t bl = (uint32_t)lane < rk ? sum_lt : 0u, be = (uint32_t)lane < rk ? sum_eq : 0u;
            uint32_t tl = sum_lt, te = sum_eq;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                bl += __shfl_xor_sync(0xffffffffu, bl, o);
                be += __shfl_xor_sync(0xffffffffu, be, o);
                tl += __shfl_xor_sync(0xffffffffu, tl, o);
                te += __shfl_xor_sync(0xffffffffu, te, o);
            }
            if (lane == 0) {
                s_run[0] = bl;
                s_run[1] = be;
                s_run[2] = tl;
                s_run[3] = te;
            }
        }
        __syncthreads();
        run_lt = s_run[0];
        run_eq = s_run[1];
        if (rk == 0 && tid == 0 && (uint32_t)N - s_run[2] - min(s_run[3], rank) != (uint32_t)na)
            raise_error(a.err, kDevBadPlan);
    }

    // ---- index-ordered compaction.  For token i with L(i) smaller keys and
    // E(i) ties before it in the sample, the tie is cached iff E(i) < rank, and
    // an active token lands at position i - L(i) - min(E(i), rank).  Each
    // thread takes four consecutive tokens per round of 1024.
    for (int j0 = 0; j0 < nl; j0 += 4 * kSelThreads) {
        const int j = j0 + 4 * tid;
        // nl is a multiple of 4: a thread's four tokens exist or none does
        uint32_t ltb = 0, eqb = 0;
        if (j < nl) {
            uint4 kk = *reinterpret_cast<const uint4 *>(keys + j);
            kk = make_uint4(kk.x & hi_mask, kk.y & hi_mask, kk.z & hi_mask, kk.w & hi_mask);
            ltb = (kk.x < thr ? 1u : 0u) | (kk.y < thr ? 2u : 0u) | (kk.z < thr ? 4u : 0u) | (kk.w < thr ? 8u : 0u);
            eqb = (kk.x == thr ? 1u : 0u) | (kk.y == thr ? 2u : 0u) | (kk.z == thr ? 4u : 0u) | (kk.w == thr ? 8u : 0u);
        }
        const uint32_t cnt4 = (uint32_t)__popc(ltb) | ((uint32_t)__popc(eqb) << 16);
        uint32_t tot;
        const uint32_t pre = block_scan(cnt4, wsum, &tot) - cnt4;
        if (j < nl) {
            uint32_t plt = run_lt + (pre & 0xFFFFu), peq = run_eq + (pre >> 16);
            const int i0 = lo + j;
            uint32_t mask4 = 0;
            int row[4];
#pragma unroll
            for (int r2 = 0; r2 < 4; ++r2) {
                const uint32_t lt = (ltb >> r2) & 1u, eq = (eqb >> r2) & 1u;
                const bool cached = lt || (eq && peq < rank);
                row[r2] = -1;
                if (cached) {
                    mask4 |= 1u << (8 * r2);
                } else {
                    const uint32_t pos = (uint32_t)(i0 + r2) - plt - min(peq, rank);
                    if (pos >= (uint32_t)na) {
                        raise_error(a.err, kDevBadPlan);
                    } else {
                        a.active_idx[base + pos] = i0 + r2;
                        row[r2] = off + (int)pos;
                    }
                }
                plt += lt;
                peq += eq;
            }
            if (a.mask) {
                uint8_t *m = a.mask + base + i0;
                if (((uintptr_t)a.mask & 3) == 0) {
                    *reinterpret_cast<uint32_t *>(m) = mask4;
                } else {  // the caller's mask may start anywhere
#pragma unroll
                    for (int r2 = 0; r2 < 4; ++r2) m[r2] = (uint8_t)((mask4 >> (8 * r2)) & 1u);
                }
            }
            if (a.row_of_token) *reinterpret_cast<int4 *>(a.row_of_token + base + i0) = make_int4(row[0], row[1], row[2], row[3]);
        }
        run_lt += tot & 0xFFFFu;
        run_eq += tot >> 16;
    }
    cluster_wait();  // the other CTAs have read this CTA's shared memory
}

__global__ void k_plan_from_counts(const int32_t *n_active, int B, int N, Plan *plan, int32_t *tile_sample,
                                   int32_t *pair_tiles, uint32_t *err)
{
    griddep_launch();
    griddep_wait();
    __shared__ int offs[kMaxBatch + 1], s_na[kMaxBatch], pair0[kMaxBatch];
    if (threadIdx.x == 0) {
        int o = 0, pairs = 0;
        for (int b = 0; b < B; ++b) {
            int na = n_active[b];
            if (na < 0 || na > N) {
                raise_error(err, kDevBadIndex);
                na = na < 0 ? 0 : N;
            }
            offs[b] = o;
            plan->n_active[b] = na;
            plan->row_off[b] = o;
            s_na[b] = na;
            o += pad_tile(na);
            pairs += tile_pairs(na);
        }
        offs[B] = o;
        plan->m_rows = o;
        plan->n_tiles = o / kTileRows;
        plan->n_pairs = pairs;
    }
    __syncthreads();
    if (threadIdx.x < B) {
        const int b = threadIdx.x;
        int p = 0;
        for (int o = 0; o < B; ++o)
            if (s_na[o] > s_na[b] || (s_na[o] == s_na[b] && o < b)) p += tile_pairs(s_na[o]);
        pair0[b] = p;
    }
    __syncthreads();
    for (int b = 0; b < B; ++b) {
        const int t0 = offs[b] / kTileRows, t1 = offs[b + 1] / kTileRows;
        for (int t = t0 + threadIdx.x; t < t1; t += blockDim.x) tile_sample[t] = b;
        for (int t = t0 + 2 * threadIdx.x; t < t1; t += 2 * blockDim.x)
            pair_tiles[pair0[b] + (t - t0) / 2] = tile_pair(t, b, t + 1 < t1);
    }
}

template <bool kThird>
cudaError_t launch_select(const SelectArgs &a, size_t smem, cudaStream_t s)
{
    // the shared-memory attribute is per device: set it on each device's first launch
    static std::atomic<uint64_t> attr_devices{0};
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    const uint64_t bit = 1ull << (dev & 63);
    if (!(attr_devices.load(std::memory_order_acquire) & bit)) {
        e = cudaFuncSetAttribute(k_ssc_select<kThird>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 kSelMaxTokens / kSelCS * 2 * (int)sizeof(float));
        if (e != cudaSuccess) return e;
        attr_devices.fetch_or(bit, std::memory_order_acq_rel);
    }
    launch_k(k_ssc_select<kThird>, dim3(a.B * kSelCS), dim3(kSelThreads), smem, s, a, -0.0f);
    return cudaGetLastError();
}

}  // namespace

int ssc_select_max_tokens() { return kSelMaxTokens; }

cudaError_t launch_ssc_select(const SelectArgs &a, cudaStream_t s)
{
    if (a.N > kSelMaxTokens || a.N % (4 * kSelCS) != 0 || a.B < 1 || a.B > kMaxBatch ||
        (a.cfg_dup && 2 * a.B > kMaxBatch))
        return cudaErrorInvalidValue;
    // V and A of a CTA's tokens (the key later replaces V)
    const size_t smem = (size_t)(a.N / kSelCS) * 2 * sizeof(float);
    return a.v3 ? launch_select<true>(a, smem, s) : launch_select<false>(a, smem, s);
}

cudaError_t launch_plan_from_counts(const int32_t *n_active, const int32_t *active_idx, int B, int N,
                                    Plan *plan, int32_t *tile_sample, int32_t *pair_tiles, int32_t *row_of_token,
                                    uint32_t *err, cudaStream_t s)
{
    (void)active_idx;
    (void)row_of_token;
    if (B < 1 || B > kMaxBatch) return cudaErrorInvalidValue;
    launch_k(k_plan_from_counts, dim3(1), dim3(256), 0, s, n_active, B, N, plan, tile_sample, pair_tiles,
             err);
    return cudaGetLastError();
}

}  // namespace f3dc
