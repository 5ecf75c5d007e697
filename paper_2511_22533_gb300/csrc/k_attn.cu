// k_attn.cu -- K5 / K6: multi-head attention softmax(Q K^T / sqrt(dh)) V on
// 5th-generation tensor cores, flash style (online softmax), for
//   mode 0  self-attention of every sample among its ACTIVE tokens only
//           (Sec. 4.2: attention runs on the compacted active subset)
//   mode 1  cross-attention of the active tokens to the sample's condition
//           tokens (Supp. Sec. F cross-attention)
//   mode 2  one sequence (diagnostic entry point)
//
// Persistent kernel, one CTA per SM (384 threads).  A work item is two
// 128-query tiles A and B of one head that share their keys: the K / V tiles
// are loaded once for both, and the two tiles' score / softmax / P V chains
// run side by side, so while one tile's softmax works the tensor core serves
// the other's MMAs.
//   warp 0     TMA producer: the item's two Q tiles (double-buffered across
//              items), K / V tiles of 128 keys into a 4-deep ring
//   warps 1, 2 tcgen05.mma issuers of tile A and of tile B (the whole warp
//              runs the loop and votes on every barrier outcome; elect.sync
//              issues), so neither tile's chain waits behind the other's.
//              Per key tile g: S_t(g + 1) = Q_t K^T (N=128, K=dh; once the
//              softmax has loaded S_t(g); also across items), then
//              O_t += P_t V(g) (N=dh, K=128; once P_t is written; P read
//              straight from TMEM).  Warp 1 allocates TMEM.
//   warp 3     idle (completes the warpgroup whose registers are given away)
//   warps 4-7  softmax of tile A, warps 8-11 of tile B: one thread per query
//              row (TMEM lane = row).  The row's 128 scores of a key tile
//              are loaded into registers at once and S_t is released for
//              the next key tile's MMA; P = exp2(S scale - m) goes to TMEM
//              P_t as bf16 pairs; l sums P in fp32.  O_t stays in TMEM for
//              the whole item; at its end O_t / l is stored as bf16.
// The reference m is the row's maximum over the item's first key tile (and
// the ragged last one, if it is 2^8 above).  A later score above m is no
// loss: P, l and O are floating point, with the same 8 exponent bits, so only
// an overflow would be, and a ragged tile's raise whose factor underflows.  Both
// are seen at the item's end (l above 2^64, O not finite; such a raise makes l
// infinite).  The CTA then does those items a second time with the maximum of
// every key tile, m raised (O_t and l rescaled in place) when a tile's maximum
// is 2^8 above it, and stores the rows that asked for it alone (they stored
// nothing before): the others keep the first pass's bits, whatever the rows of
// their item or the CTA's other items hold.  So the loop over the key tiles takes
// no maximum and has no branch on the data.
// What bounds it: the softmax warps.  Per key tile of 128 x 128 scores an SM's
// exponent unit needs 512 clocks (32 per clock) and the tensor core 512; the
// kernel takes ~950 (4096 x 4096 x 16 heads, dh 64, back to back: 63.4 us = 1083
// TFLOP/s; before -- one issuer warp, a maximum of every half tile, ~1250 clocks
// -- 79.1 us; 1229 x 1374: 17.6 -> 15.5 us).  A softmax warp alone needs ~730
// clocks per tile (load, exponents, store), and the two of an SM sub-partition
// mostly compete for the exponent unit at the same time.  Measured slower: 16
// softmax warps with half a row each (73 us: the waits' instructions double),
// turn-taking of the two warps through mbarriers, loading the next tile's
// scores under this one's exponents.
// TMEM: S_A S_B (fp32, 128 columns each) | O_A O_B (dh each) | P_A P_B (64).
// V is the MN-major B operand of the P V MMA straight from its row-major
// TMA tile.  Keys beyond a sample's count are masked to -inf before the
// exponent; padding rows are finite by construction, so 0 * pad = 0.
#include <atomic>

#include "common.cuh"
#include "kernels.h"

namespace f3dc {

namespace {

constexpr int kAttnThreads = 384;  // producer, two MMA issuers, an idle warp, 2 x 4 softmax warps
constexpr int kKVStages = 4;
// Registers per thread after the split.  The launch has 384 x 168 = 64512; a
// softmax thread holds a whole score row of a key tile (128 floats).
constexpr int kCtrlRegs = 72, kSoftmaxRegs = 216;
static_assert(128 * kCtrlRegs + 256 * kSoftmaxRegs <= 384 * 168, "register split above the launch's total");

template <int DH>
struct AttnCfg {
    static constexpr int kRowBytes = DH * 2;            // 128 (DH 64) or 64 (DH 32)
    static constexpr int kTileBytes = 128 * kRowBytes;  // Q, K or V tile
    static constexpr uint32_t kAtom = 8 * kRowBytes;    // 8-row swizzle atom
    static constexpr uint32_t kSwz = DH == 64 ? kSwizzle128 : kSwizzle64;
    static constexpr size_t kSmem = 1024 + kTileBytes * (4 + 2 * kKVStages) + 256 + 256 * 4;
    // TMEM columns: S_A S_B (fp32, 128 each) | O_A O_B (fp32, DH each) |
    // P_A P_B (bf16 pairs, 64 each)
    static constexpr uint32_t kColO = 256, kColP = 256 + 2 * DH;
    static constexpr uint32_t kTmemCols = 512;
    static_assert(kColP + 128 <= kTmemCols, "TMEM layout");
};

// A CTA's items run in windows of this many: a first pass over the window, then a
// second one over the items in which a row asked for it (a bit for each).  Against
// a second pass over all of a CTA's items that stores all their rows, so that one
// sample's data changes another's bits, this costs code and registers: 4096 x 4096
// 64.7 -> 65.3 us (L2 flushed), 1229 x 1374 15.7 -> 15.9, a sample of the 8^3 model
// 947 -> 957.  Measured slower still: the range from the first to the last such item
// instead of bits (66.8 us, 16.6, 962), item data kept in shared memory over the key
// loop (65.8, 16.0, 962).
constexpr int kWindow = 32;

struct Item {
    int q_row0, kv_row0, nk, h;  // q_row0: tile A's first row (B follows)
    bool both;                              // tile B is the pair's too (else computed, never stored)
};

// Work item w: pair w / heads of query tiles, head w % heads.  The tiles of a
// pair share their keys: the plan lists pairs within one sample, at most one of
// them half empty, and every listed sample has active tokens.  Pairs of
// neighbours in the packed rows, run twice where two samples meet, did up to 20 %
// more key tiles: a guided step of eight samples with 400 - 4096 active tokens
// took 2636 us, with these pairs 2557 (self-attention 295 -> 270 us,
// cross-attention 188 -> 170).  Items come longest first, one of every gridDim.x
// for a CTA; walking them forwards and backwards in turn measured the same there
// and 0.5 us slower at 4096 x 4096.
// kEarly: before griddep_wait (the plan is read from L2).
template <bool kEarly = false>
F3DC_DEV void decode_item(const AttnParams &p, int w, int n_tiles, Item &it)
{
    auto ld = [](const int32_t *q) { return kEarly ? ld_plan(q) : *q; };
    const int pt = w / p.heads;
    it.h = w - pt * p.heads;
    if (p.mode == 2) {  // one sequence
        it.q_row0 = 256 * pt;
        it.both = 2 * pt + 1 < n_tiles;
        it.kv_row0 = 0;
        it.nk = p.nk_fixed;
        return;
    }
    const int e = ld(p.pair_tiles + pt), b = (e & ~kPairBoth) >> kPairSampleShift;
    it.q_row0 = (e & kPairTileMask) * 128;
    it.both = (e & kPairBoth) != 0;
    if (p.mode == 0) {  // the sample's active tokens
        it.kv_row0 = ld(p.plan->row_off + b);
        it.nk = ld(p.plan->n_active + b);
    } else {  // the sample's condition tokens
        it.kv_row0 = (p.kv_null_from > 0 && b >= p.kv_null_from ? p.kv_null_sample : b) * p.nk_fixed;
        it.nk = p.nk_fixed;
    }
}

F3DC_DEV bool wait_bounded(uint64_t *bar, uint32_t parity, uint64_t ns)
{
    const uint64_t t0 = globaltimer();
    while (!mbar_try_wait(bar, parity))
        if (globaltimer() - t0 > ns) return false;
    return true;
}

template <int DH>
__global__ void __launch_bounds__(kAttnThreads, 1)
    k_attn(const __grid_constant__ CUtensorMap tmq, const __grid_constant__ CUtensorMap tmk,
           const __grid_constant__ CUtensorMap tmv, const AttnParams p)
{
    using Cfg = AttnCfg<DH>;
    extern __shared__ uint8_t smem_raw[];
    uint8_t *smem = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    // Q: two items' pairs of tiles (item i in buffer i % 2, tile A then B)
    uint8_t *sQ = smem;
    uint8_t *sK = sQ + 4 * Cfg::kTileBytes;
    uint8_t *sV = sK + kKVStages * Cfg::kTileBytes;
    uint64_t *bars = reinterpret_cast<uint64_t *>(sV + kKVStages * Cfg::kTileBytes);
    uint64_t *q_full = bars, *q_empty = bars + 2;
    uint64_t *kv_full = bars + 4, *kv_empty = kv_full + kKVStages;
    // per query tile t (0 = A, 1 = B), once per key tile: S_t written
    // (s_full), S_t read by the softmax (s_free), P_t written (p_full), P_t V
    // done (pv_done); once per item: O_t read (o_free)
    uint64_t *s_full = kv_empty + kKVStages, *s_free = s_full + 2, *p_full = s_free + 2, *pv_done = p_full + 2;
    uint64_t *o_free = pv_done + 2;
    uint64_t *drain = o_free + 2;
    uint32_t *tmem_holder = reinterpret_cast<uint32_t *>(drain + 1);
    volatile int *abort_flag = reinterpret_cast<volatile int *>(tmem_holder + 1);
    // items of a window that run again (of windows by turns), and of each softmax
    // thread's row the items of the window that it asked for
    uint32_t *redo_items = tmem_holder + 2, *redo_row = tmem_holder + 4;

    const int warp = __shfl_sync(0xffffffffu, threadIdx.x >> 5, 0), lane = threadIdx.x & 31;
    griddep_launch();

    if (threadIdx.x == 0) {
        for (int b = 0; b < 2; ++b) {
            mbar_init(&q_full[b], 1);
            mbar_init(&q_empty[b], 2);  // both MMA warps
        }
        for (int s = 0; s < kKVStages; ++s) {
            mbar_init(&kv_full[s], 1);
            mbar_init(&kv_empty[s], 2);
        }
        for (int t = 0; t < 2; ++t) {
            mbar_init(&s_full[t], 1);
            mbar_init(&s_free[t], 4);  // the four softmax warps of tile t
            mbar_init(&p_full[t], 4);
            mbar_init(&pv_done[t], 1);
            mbar_init(&o_free[t], 4);
        }
        mbar_init(drain, 2);
        *abort_flag = 0;
        redo_items[0] = redo_items[1] = 0;
        fence_mbar_init();
    }
    if (warp == 1) {
        tmem_alloc(tmem_holder, Cfg::kTmemCols);
        tmem_relinquish();
    }
    if (warp == 0 && lane == 0) {
        tma_prefetch(&tmq);
        tma_prefetch(&tmk);
        tma_prefetch(&tmv);
    }
    if (p.kv_prefetch_rows > 0 && warp == 0 && lane == 0) {
        // keys / values written long before this launch (the condition's):
        // pull this CTA's share into L2 while the previous kernel finishes
        const int rb = (p.kv_prefetch_rows + 127) / 128, boxes = rb * p.heads * 2;
        for (int i = blockIdx.x; i < boxes; i += gridDim.x) {
            const int r = i % rb, hk = i / rb, h = hk >> 1;
            tma_prefetch_l2_2d(hk & 1 ? &tmv : &tmk, (hk & 1 ? p.v_col0 : p.k_col0) + h * DH, r * 128);
        }
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = __shfl_sync(0xffffffffu, *tmem_holder, 0);
    const int n_tiles = __shfl_sync(0xffffffffu, p.n_tiles_dev ? ld_plan(p.n_tiles_dev) : p.n_tiles, 0);
    const int total =
        (p.n_tiles_dev ? __shfl_sync(0xffffffffu, ld_plan(&p.plan->n_pairs), 0) : (n_tiles + 1) >> 1) * p.heads;
    // the producer's first item is looked up early: its loads are the first
    // thing after the wait
    Item first_item;
    if (warp == 0 && (int)blockIdx.x < total) decode_item<true>(p, blockIdx.x, n_tiles, first_item);
    // the previous kernel's outputs (Q / K / V) are complete
    griddep_wait();

    // work item number n of this CTA, and whether a pass over the window at n0
    // comes to it
    auto item_of = [&](int n) { return (int)blockIdx.x + n * (int)gridDim.x; };
    auto in_window = [&](int n, int n0) { return n < n0 + kWindow && item_of(n) < total; };
    auto skipped = [&](int n, int pass) {
        return pass != 0 && (redo_items[n / kWindow & 1] >> (n % kWindow) & 1) == 0;
    };
    // Every warp ends a pass over a window here, also when the kernel is aborting
    // (each role's waits are bounded), and all take the same next step: stop, the
    // window's second pass, or the next window.
    auto end_pass = [&](int &n0, int &pass, bool &stop) {
        uint32_t any;
        asm volatile("{\n .reg .pred p, q;\n setp.ne.s32 p, %1, 0;\n bar.red.or.pred q, 1, %2, p;\n"
                     " selp.u32 %0, 1, 0, q;\n}\n"
                     : "=r"(any)
                     : "r"(*abort_flag), "n"(kAttnThreads)
                     : "memory");
        stop = any != 0;
        const bool again = pass == 0 && redo_items[n0 / kWindow & 1] != 0;
        pass = again ? 1 : 0;
        n0 += again ? 0 : kWindow;
    };
    bool stop = false;

    if (warp == 0) {
        // ------------------------------------------------ TMA producer
        reg_dec<kCtrlRegs>();
        uint32_t kv_it = 0, item_it = 0;
#pragma unroll 1
        for (int n0 = 0, pass = 0; !stop && item_of(n0) < total; end_pass(n0, pass, stop)) {
            if (lane == 0) {
                bool ok = true;
#pragma unroll 1
                for (int n = n0; ok && in_window(n, n0); ++n) {
                    if (skipped(n, pass)) continue;
                    Item it = first_item;
                    if (n) decode_item(p, item_of(n), n_tiles, it);
                    const uint32_t my_it = item_it++;
                    // Q buffer qb holds items qb, qb + 2, ...: its (my_it / 2)-th use
                    const uint32_t qb = my_it & 1, qph = (my_it >> 1) & 1;
                    if (!mbar_wait(&q_empty[qb], qph ^ 1, abort_flag, p.err)) break;
                    mbar_arrive_expect_tx(&q_full[qb], 2 * Cfg::kTileBytes);
                    for (int t = 0; t < 2; ++t)
                        tma_load_2d(sQ + (2 * qb + t) * Cfg::kTileBytes, &tmq, p.q_col0 + it.h * DH,
                                    it.q_row0 + 128 * t, &q_full[qb]);
                    const int nkt = (it.nk + 127) / 128;
#pragma unroll 1
                    for (int j = 0; j < nkt; ++j, ++kv_it) {
                        const int s = kv_it % kKVStages;
                        const uint32_t ph = (kv_it / kKVStages) & 1;
                        if (!mbar_wait(&kv_empty[s], ph ^ 1, abort_flag, p.err)) {
                            ok = false;
                            break;
                        }
                        // fault injection (tests of the failure path): the last
                        // key tile of CTA 0's first item is never loaded, so the
                        // waits on it (and on what follows it) run out while the
                        // earlier tiles went through, and the kernel aborts
                        if (p.fault_skip_kv && blockIdx.x == 0 && my_it == 0 && j == nkt - 1) continue;
                        mbar_arrive_expect_tx(&kv_full[s], 2 * Cfg::kTileBytes);
                        tma_load_2d(sK + s * Cfg::kTileBytes, &tmk, p.k_col0 + it.h * DH, it.kv_row0 + j * 128,
                                    &kv_full[s]);
                        tma_load_2d(sV + s * Cfg::kTileBytes, &tmv, p.v_col0 + it.h * DH, it.kv_row0 + j * 128,
                                    &kv_full[s]);
                    }
                }
            }
            __syncwarp();
        }
    } else if (warp <= 2) {
        // ------------------------------------------------ MMA issuer of one query tile
        reg_dec<kCtrlRegs>();
        // Every lane runs the loop (a converged warp keeps the descriptors
        // warp-uniform) and takes each barrier outcome as a warp vote;
        // elect.sync issues.  Key tile g (counted over the CTA's whole run)
        // sits in K/V stage g % kKVStages; every barrier here completes once
        // per key tile (or per item), so its phase parity follows from g.
        {
            constexpr uint32_t idesc_s = make_idesc_bf16(128, 128, 0, 0);
            constexpr uint32_t idesc_o = make_idesc_bf16(128, DH, 0, 1);
            // descriptors of the stage bases; a K step of 16 elements inside a
            // 128B / 64B swizzle atom advances the start address by 32 bytes,
            // i.e. the descriptor by 2
            const int t = warp - 1;
            const uint64_t q_desc0 = make_sdesc(smem_u32(sQ + t * Cfg::kTileBytes), 16, Cfg::kAtom, Cfg::kSwz);
            const uint64_t k_desc0 = make_sdesc(smem_u32(sK), 16, Cfg::kAtom, Cfg::kSwz);
            const uint64_t v_desc0 = make_sdesc(smem_u32(sV), Cfg::kAtom, Cfg::kAtom, Cfg::kSwz);
            constexpr uint64_t kStageStep = Cfg::kTileBytes >> 4, kVRowStep = (16 * Cfg::kRowBytes) >> 4;
            auto wait = [&](uint64_t *bar, uint32_t ph) { return warp_wait(bar, ph, abort_flag, p.err); };
            // One loop, S one key tile ahead of P V (also across items), so
            // that each is in the code once: the instruction cache is what
            // ten warps at different places of a long kernel share.
            uint32_t g = 0, item = 0;  // S: key tile g of the CTA's run, in its item number item
#pragma unroll 1
            for (int n0 = 0, pass = 0; !stop && item_of(n0) < total; end_pass(n0, pass, stop)) {
                int n = n0 - 1;
                uint32_t nkt = 0, j = 0;                // key tiles of the item, S's within it
                bool pending = false, p_first = false;  // P V of key tile g - 1, the first of its item
                uint32_t p_par = 0;                     // o_free's phase for that item
#pragma unroll 1
                while (true) {
                    if (j == nkt) {  // the next real work item
                        if (nkt) ++item;
                        nkt = j = 0;
                        do ++n;
                        while (in_window(n, n0) && skipped(n, pass));
                        if (in_window(n, n0)) {
                            Item it;
                            decode_item(p, item_of(n), n_tiles, it);
                            nkt = __shfl_sync(0xffffffffu, (uint32_t)((it.nk + 127) / 128), 0);
                        }
                    }
                    if (nkt) {
                        // S_t, once the softmax has loaded the previous S_t
                        const uint32_t st = g % kKVStages, qb = item & 1;
                        if (j == 0 && !wait(&q_full[qb], (item >> 1) & 1)) break;
                        if (!wait(&kv_full[st], (g / kKVStages) & 1)) break;
                        if (!wait(&s_free[t], (g & 1) ^ 1)) break;
                        tc_fence_after();
                        const uint64_t kd = k_desc0 + st * kStageStep, qd = q_desc0 + (uint64_t)(2 * qb) * kStageStep;
#pragma unroll
                        for (int kk = 0; kk < DH / 16; ++kk)
                            mma_bf16_elect(tmem + t * 128, qd + 2 * kk, kd + 2 * kk, idesc_s, kk > 0);
                        mma_commit_elect(&s_full[t]);
                        if (j + 1 == nkt) mma_commit_elect(&q_empty[qb]);  // every S_t of the item issued
                    }
                    if (pending) {
                        // P_t V, once P_t is written; the item's first overwrites
                        // O_t, which the softmax must have read for the previous item
                        const uint32_t gp = g - 1, st = gp % kKVStages;
                        if (p_first && !wait(&o_free[t], p_par)) break;
                        if (!wait(&p_full[t], gp & 1)) break;
                        tc_fence_after();
                        const uint64_t vd = v_desc0 + st * kStageStep;
#pragma unroll
                        for (int kk = 0; kk < 8; ++kk)
                            mma_bf16_ts_elect(tmem + Cfg::kColO + t * DH, tmem + Cfg::kColP + t * 64 + kk * 8,
                                              vd + kk * kVRowStep, idesc_o, kk > 0 || !p_first);
                        mma_commit_elect(&pv_done[t]);
                        mma_commit_elect(&kv_empty[st]);
                    }
                    if (!nkt) break;
                    pending = true;
                    p_first = j == 0;
                    p_par = (item & 1) ^ 1;
                    ++j;
                    ++g;
                }
            }
        }
    } else if (warp < 4) {
        // gives its registers to the softmax warps; clears the next window's bits
        reg_dec<kCtrlRegs>();
#pragma unroll 1
        for (int n0 = 0, pass = 0; !stop && item_of(n0) < total; end_pass(n0, pass, stop)) {
            if (lane == 0) redo_items[(n0 / kWindow + 1) & 1] = 0;
            __syncwarp();
        }
    } else {
        // ------------------------------------------------ softmax warps
        reg_inc<kSoftmaxRegs>();
        const int q = warp & 3;              // TMEM lane quarter of this warp
        const int t = (warp - 4) >> 2;       // query tile: warps 4-7 A, 8-11 B
        const int row = q * 32 + lane;
        const uint32_t tl = (uint32_t)(q * 32) << 16;
        const uint32_t s_addr = tmem + tl + t * 128;
        const uint32_t o_addr = tmem + tl + Cfg::kColO + t * DH;
        const uint32_t p_addr = tmem + tl + Cfg::kColP + t * 64;
        auto wait = [&](uint64_t *bar, uint32_t ph) { return warp_wait(bar, ph, abort_flag, p.err); };
        // S_t of key tile g completes s_full[t] (phase g), the four warps'
        // arrivals on s_free[t] / p_full[t] complete phase g once S_t is
        // loaded / P_t written, and P_t V of tile g completes pv_done[t]; a
        // wait that gives up (the kernel is aborting) ends this warp's loop
        const float scale = p.scale_log2;
        const f32x2 sc2 = {scale, scale};
        float m_ref = -INFINITY, l_run = 0.f;
        // S_t of key tile g into registers; S_t is released at once, so the
        // next key tile's S runs under this one's exponents
        auto load_s = [&](uint32_t g, float (&sv)[128]) {
            if (!wait(&s_full[t], g & 1)) return false;
            tc_fence_after();
            uint32_t r[4][32];
#pragma unroll
            for (int c = 0; c < 4; ++c) tmem_ld32(s_addr + 32 * c, r[c]);
            tmem_wait_ld();
#pragma unroll
            for (int c = 0; c < 128; ++c) sv[c] = __uint_as_float(r[c / 32][c % 32]);
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(&s_free[t]);
            return true;
        };
        // exponents of 64 scores against the reference -nm, their sum added to
        // s0, s1, as bf16 pairs
        auto exps = [&](const float (&sv)[128], int hb, float nm, f32x2 &s0, f32x2 &s1, uint32_t (&pw)[32]) {
            const f32x2 nm2 = {nm, nm};
#pragma unroll
            for (int c = 0; c < 32; c += 2) {
                const int k0 = 64 * hb + 2 * c;
                const f32x2 x0 = ffma2({sv[k0], sv[k0 + 1]}, sc2, nm2);
                const f32x2 x1 = ffma2({sv[k0 + 2], sv[k0 + 3]}, sc2, nm2);
                const f32x2 e0 = {exp2_fast(x0.x), exp2_fast(x0.y)};
                const f32x2 e1 = {exp2_fast(x1.x), exp2_fast(x1.y)};
                s0 = fadd2(s0, e0);
                s1 = fadd2(s1, e1);
                pw[c] = pack_bf16x2(e0.x, e0.y);
                pw[c + 1] = pack_bf16x2(e1.x, e1.y);
            }
        };
        auto p_written = [&]() {
            tmem_wait_st();
            tc_fence_before();  // P (and a rescaled O) written before P V may start
            __syncwarp();
            if (lane == 0) mbar_arrive(&p_full[t]);
        };
        // A key tile against the reference as it stands: no maximum, no check.
        auto plain_tile = [&](uint32_t g) {
            float sv[128];
            if (!load_s(g, sv)) return false;
            f32x2 s0 = {0.f, 0.f}, s1 = {0.f, 0.f};
            uint32_t pw0[32], pw1[32];
            exps(sv, 0, -m_ref, s0, s1, pw0);
            if (!wait(&pv_done[t], (g - 1) & 1)) return false;  // P_t read by P V of the previous key tile
            tc_fence_after();
            tmem_st32(p_addr, pw0);
            exps(sv, 1, -m_ref, s0, s1, pw1);
            tmem_st32(p_addr + 32, pw1);
            l_run += (s0.x + s0.y) + (s1.x + s1.y);
            p_written();
            return true;
        };
        // A key tile with its maximum (of its `valid` first keys): the item's
        // first and a ragged last one, and every one of a second pass.  The
        // reference is raised (O_t and l rescaled) when it grew by more than 2^8.
        // In a first pass the plain tiles before a ragged last one may lie far
        // above the reference, up to this tile's maximum: a raise above 2^126,
        // whose factor ex2.approx.ftz flushes to 0, would erase what they
        // summed, so l becomes infinite instead and the item's end asks for the
        // second pass.  (There an erased key is below 2^-118 of the row.)
        auto max_tile = [&](uint32_t g, bool first, int valid, bool second_pass) {
            float sv[128];
            if (!load_s(g, sv)) return false;
            if (valid < 128) {
#pragma unroll
                for (int c = 0; c < 128; ++c)
                    if (c >= valid) sv[c] = -INFINITY;
            }
            float mx4[4] = {-INFINITY, -INFINITY, -INFINITY, -INFINITY};
#pragma unroll
            for (int c = 0; c < 128; c += 8) {
#pragma unroll
                for (int e = 0; e < 4; ++e) mx4[e] = fmax3(mx4[e], sv[c + e], sv[c + 4 + e]);
            }
            const float mx = fmax3(mx4[0], mx4[1], fmaxf(mx4[2], mx4[3])) * scale;
            if (g > 0 && !wait(&pv_done[t], (g - 1) & 1)) return false;  // P_t, O_t free
            tc_fence_after();
            if (__any_sync(0xffffffffu, mx > m_ref + 8.0f)) {
                const float m_new = fmaxf(m_ref, mx);
                const float alpha = exp2_fast(m_ref - m_new);
                if (!first && !second_pass && m_new - m_ref > 126.0f) l_run = INFINITY;
                else l_run *= alpha;
                m_ref = m_new;
                if (!first) {  // O_t holds this item's earlier tiles
#pragma unroll 1
                    for (int d0 = 0; d0 < DH; d0 += 16) {
                        uint32_t r[16];
                        tmem_ld16(o_addr + d0, r);
                        tmem_wait_ld();
#pragma unroll
                        for (int e = 0; e < 16; ++e) r[e] = __float_as_uint(__uint_as_float(r[e]) * alpha);
                        tmem_st16(o_addr + d0, r);
                    }
                }
            }
            const float nm = m_ref == -INFINITY ? 0.f : -m_ref;
            f32x2 s0 = {0.f, 0.f}, s1 = {0.f, 0.f};
            uint32_t pw[2][32];
            exps(sv, 0, nm, s0, s1, pw[0]);
            exps(sv, 1, nm, s0, s1, pw[1]);
            tmem_st32(p_addr, pw[0]);
            tmem_st32(p_addr + 32, pw[1]);
            l_run += (s0.x + s0.y) + (s1.x + s1.y);
            p_written();
            return true;
        };
        uint32_t g = 0;  // key tiles of this CTA's earlier items
        uint32_t *const row_bits = redo_row + 128 * t + row;
#pragma unroll 1
        for (int n0 = 0, pass = 0; !stop && item_of(n0) < total; end_pass(n0, pass, stop)) {
            if (pass == 0) *row_bits = 0;
#pragma unroll 1
            for (int n = n0; in_window(n, n0); ++n) {
                if (skipped(n, pass)) continue;
                Item it;
                decode_item(p, item_of(n), n_tiles, it);
                const int nk = __shfl_sync(0xffffffffu, it.nk, 0);
                m_ref = -INFINITY;
                l_run = 0.f;
                bool ok = true;
                // The plain tiles run in a loop of their own, with as few values
                // kept over it as can be: one loop that picks each tile's form,
                // and one more value in it, cost register moves (4096 x 4096:
                // 66.5 us, here 63.9).
                int left = nk;
                bool first = true;
                do {
                    ok = max_tile(g++, first, left, pass != 0);
                    left -= 128;
                    first = false;
                    if (pass == 0) {
#pragma unroll 1
                        for (; ok && left >= 128; left -= 128) ok = plain_tile(g++);
                    }
                } while (ok && left > 0);
                if (!ok) break;
                // every P V of the item done: O_t / l, stored as bf16
                if (!wait(&pv_done[t], (g - 1) & 1)) break;
                tc_fence_after();
                float acc[DH];
#pragma unroll
                for (int d0 = 0; d0 < DH; d0 += 32) {
                    uint32_t r[32];
                    tmem_ld32(o_addr + d0, r);
                    tmem_wait_ld();
#pragma unroll
                    for (int d = 0; d < 32; ++d) acc[d0 + d] = __uint_as_float(r[d]);
                }
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(&o_free[t]);
                const int orow = it.q_row0 + 128 * t + row;
                if ((t == 0 || it.both) && orow < p.q_rows) {
                    // The first pass takes the reference from the item's first
                    // key tile.  P, l and O carry it exactly as long as no
                    // exponent overflows (all three have 8 exponent bits), and
                    // a later score 2^64 above it shows in l, a sum of
                    // positive terms; anything not finite in O is looked at
                    // again too.
                    float zero = 0.f;
#pragma unroll
                    for (int d = 0; d < DH; ++d) zero = fmaf(acc[d], 0.f, zero);  // NaN if any is inf or NaN
                    // A row that asks for the second pass stores nothing now (out
                    // may be q's buffer, whose row it needs again).
                    const bool redo = pass == 0 && !(l_run <= 0x1p64f && zero == 0.f);
                    if (redo) {
                        *row_bits |= 1u << (n % kWindow);
                        atomicOr(redo_items + (n / kWindow & 1), 1u << (n % kWindow));
                    }
                    if (pass == 0 ? !redo : (*row_bits >> (n % kWindow) & 1) != 0) {
                        const float inv = 1.0f / l_run;
                        uint4 *dst = reinterpret_cast<uint4 *>(p.out + (size_t)orow * p.ldo + it.h * DH);
#pragma unroll
                        for (int d = 0; d < DH; d += 8) {
                            uint4 u;
                            u.x = pack_bf16x2(acc[d] * inv, acc[d + 1] * inv);
                            u.y = pack_bf16x2(acc[d + 2] * inv, acc[d + 3] * inv);
                            u.z = pack_bf16x2(acc[d + 4] * inv, acc[d + 5] * inv);
                            u.w = pack_bf16x2(acc[d + 6] * inv, acc[d + 7] * inv);
                            dst[d / 8] = u;
                        }
                    }
                }
                __syncwarp();
            }
        }
    }
    __syncthreads();
    if (*abort_flag) {
        if (warp == 1 || warp == 2) {
            mma_commit_elect(drain);  // the MMAs' issuing lane
            if (lane == 0) wait_bounded(drain, 0, 100000000ull);
        }
        if (threadIdx.x == 0) spin_ns(200000);
        __syncthreads();
    }
    if (warp == 1) {
        tc_fence_after();
        tmem_dealloc(tmem, Cfg::kTmemCols);
    }
}

template <int DH>
cudaError_t launch_dh(const CUtensorMap *tq, const CUtensorMap *tk, const CUtensorMap *tv, const AttnParams &p,
                      int grid, cudaStream_t s)
{
    // the shared-memory attribute is per device: set it on each device's first launch
    static std::atomic<uint64_t> attr_devices{0};
    const size_t smem = AttnCfg<DH>::kSmem;
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    const uint64_t bit = 1ull << (dev & 63);
    if (!(attr_devices.load(std::memory_order_acquire) & bit)) {
        e = cudaFuncSetAttribute(k_attn<DH>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
        attr_devices.fetch_or(bit, std::memory_order_acq_rel);
    }
    launch_k(k_attn<DH>, dim3(grid), dim3(kAttnThreads), smem, s, *tq, *tk, *tv, p);
    return cudaGetLastError();
}

}  // namespace

size_t attn_smem_bytes(int dh) { return dh == 64 ? AttnCfg<64>::kSmem : AttnCfg<32>::kSmem; }

cudaError_t launch_attention(const CUtensorMap *tq, const CUtensorMap *tk, const CUtensorMap *tv,
                             const AttnParams &p, int grid, cudaStream_t s)
{
    if (grid < 1) return cudaErrorInvalidValue;
    if (p.dh == 64) return launch_dh<64>(tq, tk, tv, p, grid, s);
    if (p.dh == 32) return launch_dh<32>(tq, tk, tv, p, grid, s);
    return cudaErrorInvalidValue;
}

}  // namespace f3dc
